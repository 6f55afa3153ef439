// Interpolated PSF Hessian (App. D) on the GPU.
//
// The PSF image L^T L comb of a spike comb (nodes s/2 + k s along both axes)
// holds a localised column of the Hessian around every node. The column at a
// point c between the nodes is the bilinear interpolation (Eq. trilinear in
// its 2D form) of the windows of the four surrounding nodes, each taken
// relative to its own node:
//     H(c + a, c) = sum_corners w_corner(c) P_corner(a),  |a_z|, |a_x| <= half,
//     P_k(a) = Q(node_k + a) (0 outside the image),
// with the 1D weights (1 - w, w), w = (c - node_k0) / s, between the first and
// the last node and a single node (w = 0) beyond them. Two parameters give
// 2 x 2 blocks: block (i, j) takes plane i of the PSF of the comb in
// parameter j. The parameter mask restricts the operator to P H P.
//
// k_psfh_patches: the node windows, packed per (node, offset) as one float4
//   of the four blocks (00, 01, 10, 11), so one 16-byte load serves all four.
// k_psfh_apply<MASK, TR, R>: one thread per output column and R consecutive
//   rows (R = the largest of 8, 4, 2, 1 not above s), CTAs of 32 columns x
//   2 R rows (small CTAs spread the one wave evenly over the SMs). The input
//   planes over the tile plus a half-wide halo and the corner tables of the
//   halo's rows and columns sit in shared memory. Per
//   window offset a thread reads the six node windows covering its rows
//   (three node rows, two node columns; R <= s rows cross at most one node
//   row) through L1, interpolates along x once and along z per row: one
//   loaded value serves R pixels, which keeps the L1 return path (the limit
//   of a one-pixel-per-thread form) below the FMA pipe. A warp's rows are the
//   same for all its lanes, and most warps' (12 of 20 positions at s = 20, R = 8)
//   lie between two node rows: those load four node values an offset, not six,
//   and interpolate with one multiply-add. 300 x 2000, s = 20, 19 x 19 windows,
//   two parameters: 239 -> 199 us an application, by this and the interpolation
//   in packed FP32x2 (with two offsets loaded ahead 300: 160 registers). What
//   bounds it now: the L1 return path and its latency.
//   TR = false: y(r) = sum_a H(r, r - a) x(r - a), the columns gathered at r;
//   TR = true:  y(c) = sum_a H(c + a, c) x(c + a), the transpose.
// k_psfh3_patches, k_psfh3_rows: the same for 3D images, with the eight
//   corners of Eq. (trilinear) and (y, x) columns of R z rows.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "lsrtm_internal.cuh"
#include "psfhess3d.cuh"

namespace lsrtm {

namespace {

constexpr int kTX = 32;

struct Corner {
    int k0, k1;
    float w;
};

// Corner nodes and weight of coordinate c (clamped into [0, n)) on an axis
// with nk nodes at s/2 + k s.
__device__ __forceinline__ Corner corner_of(int c, int n, int s, int nk)
{
    c = min(max(c, 0), n - 1);
    const int c0 = s >> 1, last = c0 + (nk - 1) * s;
    Corner r;
    if (c <= c0) {
        r.k0 = r.k1 = 0;
        r.w = 0.f;
    } else if (c >= last) {
        r.k0 = r.k1 = nk - 1;
        r.w = 0.f;
    } else {
        const int k = (c - c0) / s;
        r.k0 = k;
        r.k1 = k + 1;
        r.w = (float)(c - c0 - k * s) / (float)s;
    }
    return r;
}

__global__ void k_psfh_patches(const float *psf_vp, const float *psf_ip, int nz, int nx, int s, int half,
                               int nkz, int nkx, int mask, float4 *pt)
{
    const int L = 2 * half + 1, LL = L * L;
    const long long plane = (long long)nz * nx;
    const long long n = (long long)nkz * nkx * LL;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const int node = (int)(i / LL), ai = (int)(i - (long long)node * LL);
        const int kz = node / nkx, kx = node - kz * nkx;
        const int z = (s >> 1) + kz * s + ai / L - half;
        const int x = (s >> 1) + kx * s + ai % L - half;
        const bool inside = z >= 0 && z < nz && x >= 0 && x < nx;
        float v[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int po = b >> 1, pi = b & 1;   // output plane, input (comb) plane
            const float *src = pi ? psf_ip : psf_vp;
            const bool use = inside && src && ((mask >> po) & 1) && ((mask >> pi) & 1);
            v[b] = use ? src[po * plane + (long long)z * nx + x] : 0.f;
        }
        pt[i] = make_float4(v[0], v[1], v[2], v[3]);
    }
}

// Parameter-block values: the four blocks (two parameters) as two pairs, or the
// one block of a single-parameter mask. Pairs are interpolated with packed FP32x2
// arithmetic: with scalars the kernel was bound by issue slots.
struct Pairs {
    float2 a, b;
};
template <int MASK>
struct Blk {
    using T = float;
};
template <>
struct Blk<3> {
    using T = Pairs;
};
__device__ __forceinline__ float2 dup(float a) { return make_float2(a, a); }
// The four blocks unpacked: for y = H x in 3D, but for four rows a thread.
// There the packed pairs cost more than they save (60 x 60 x 70: s = 10 762 us
// for 689, s = 8 377 for 345, s = 3 91 for 79; four rows, s = 5, 164 for 173).
// For y = H^T x they save or cost nothing (s = 8: 302 us for 391).
using Quad = float4;

template <int BM>
__device__ __forceinline__ float load_blk(const float4 *pt, int i, float)
{
    return __ldg(reinterpret_cast<const float *>(pt) + 4 * i + BM);
}
template <int BM>
__device__ __forceinline__ Pairs load_blk(const float4 *pt, int i, Pairs)
{
    const float4 v = __ldg(pt + i);
    return Pairs{make_float2(v.x, v.y), make_float2(v.z, v.w)};
}
template <int BM>
__device__ __forceinline__ Quad load_blk(const float4 *pt, int i, Quad)
{
    return __ldg(pt + i);
}
// p0 + w (p1 - p0)
__device__ __forceinline__ float sub_(float a, float b) { return a - b; }
__device__ __forceinline__ float2 sub_(float2 a, float2 b) { return __ffma2_rn(dup(-1.f), b, a); }
__device__ __forceinline__ Pairs sub_(Pairs a, Pairs b) { return Pairs{sub_(a.a, b.a), sub_(a.b, b.b)}; }
__device__ __forceinline__ float lerp_(float p0, float p1, float w) { return fmaf(w, p1 - p0, p0); }
__device__ __forceinline__ float2 lerp_(float2 p0, float2 p1, float w) { return __ffma2_rn(dup(w), sub_(p1, p0), p0); }
__device__ __forceinline__ Pairs lerp_(Pairs p0, Pairs p1, float w) { return Pairs{lerp_(p0.a, p1.a, w), lerp_(p0.b, p1.b, w)}; }
__device__ __forceinline__ Quad sub_(Quad a, Quad b) { return make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w); }
__device__ __forceinline__ Quad lerp_(Quad p0, Quad p1, float w)
{
    return make_float4(lerp_(p0.x, p1.x, w), lerp_(p0.y, p1.y, w), lerp_(p0.z, p1.z, w), lerp_(p0.w, p1.w, w));
}
// q0 + b d1 + c d2 (= (1 - b - c) q0 + b q1 + c q2 with d1 = q1 - q0, d2 = q2 - q0)
__device__ __forceinline__ float mix3(float q0, float d1, float d2, float b, float c)
{
    return fmaf(c, d2, fmaf(b, d1, q0));
}
__device__ __forceinline__ float2 mix3(float2 q0, float2 d1, float2 d2, float2 b, float2 c)
{
    return __ffma2_rn(c, d2, __ffma2_rn(b, d1, q0));
}
__device__ __forceinline__ Pairs mix3(Pairs q0, Pairs d1, Pairs d2, float2 b, float2 c)
{
    return Pairs{mix3(q0.a, d1.a, d2.a, b, c), mix3(q0.b, d1.b, d2.b, b, c)};
}
__device__ __forceinline__ Quad mix3(Quad q0, Quad d1, Quad d2, float b, float c)
{
    return make_float4(mix3(q0.x, d1.x, d2.x, b, c), mix3(q0.y, d1.y, d2.y, b, c), mix3(q0.z, d1.z, d2.z, b, c),
                       mix3(q0.w, d1.w, d2.w, b, c));
}
// q0 + b d1: rows that no node row separates
__device__ __forceinline__ float mix2(float q0, float d1, float b) { return fmaf(b, d1, q0); }
__device__ __forceinline__ Pairs mix2(Pairs q0, Pairs d1, float2 b)
{
    return Pairs{__ffma2_rn(b, d1.a, q0.a), __ffma2_rn(b, d1.b, q0.b)};
}
// Row weights: a scalar, or the pair both of a Pairs' products take.
template <int MASK>
struct Wgt {
    using T = float;
    static __device__ __forceinline__ T of(float w) { return w; }
};
template <>
struct Wgt<3> {
    using T = float2;
    static __device__ __forceinline__ T of(float w) { return dup(w); }
};
// One output pixel's products, plane 1's input first: unpacked, so that each
// plane is one chain of sums whose rounding does not depend on the packing (one
// sum per input plane, added at the end, took 180 us for 199 but moves the CG's
// misfits by up to 4e-9).
template <bool TR>
__device__ __forceinline__ void accum(float &a0, float &, float C, float x) { a0 = fmaf(C, x, a0); }
template <bool TR>
__device__ __forceinline__ void accum(float &a0, float &a1, Pairs C, float2 x)
{
    a0 = fmaf(C.a.x, x.x, fmaf(TR ? C.b.x : C.a.y, x.y, a0));
    a1 = fmaf(TR ? C.a.y : C.b.x, x.x, fmaf(C.b.y, x.y, a1));
}
template <bool TR>
__device__ __forceinline__ void accum(float &a0, float &a1, Quad C, float2 x)
{
    accum<TR>(a0, a1, Pairs{make_float2(C.x, C.y), make_float2(C.z, C.w)}, x);
}

// Weights of R consecutive rows (first corner row kf) on the node rows
// kf + 1 and kf + 2 (the rest, on kf, is implied): row r puts 1 - w on its k0
// and w on its k1. R <= s keeps every k0 in {kf, kf + 1} and every k1 in
// {kf, .., kf + 2}.
template <int MASK, int R>
__device__ __forceinline__ void row_weights(const Corner *zc, int kf, typename Wgt<MASK>::T (&wb)[R],
                                            typename Wgt<MASK>::T (&wc)[R])
{
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const Corner Z = zc[r];
        const int s0 = Z.k0 - kf, s1 = Z.k1 - kf;
        const float u = 1.f - Z.w, w = Z.w;
        wb[r] = Wgt<MASK>::of((s0 == 1 ? u : 0.f) + (s1 == 1 ? w : 0.f));
        wc[r] = Wgt<MASK>::of(s1 == 2 ? w : 0.f);
    }
}

// Whether a node row separates the R rows (a weight on kf + 2). The rows of a
// warp are the same for all its lanes.
__device__ __forceinline__ bool nonzero(float w) { return w != 0.f; }
__device__ __forceinline__ bool nonzero(float2 w) { return w.x != 0.f; }
template <int MASK, int R>
__device__ __forceinline__ bool any_weight(const typename Wgt<MASK>::T (&wc)[R])
{
    bool any = false;
#pragma unroll
    for (int r = 0; r < R; ++r) any |= nonzero(wc[r]);
    return any;
}

// One thread per column and R consecutive rows; CTAs of 32 columns x kRowThreads
// thread rows (32 x kRowThreads R pixels). Per window offset a thread loads the
// six node windows (three node rows x two node columns) that cover its R
// rows, interpolates along x once, then along z per row, so a loaded value
// serves R pixels.
constexpr int kRowThreads = 2, kApplyThreads = kTX * kRowThreads;

template <int MASK, bool TR, int R>
__global__ void __launch_bounds__(kApplyThreads) k_psfh_apply(const PsfHessDev a, const float *__restrict__ in,
                                                               float *__restrict__ out)
{
    using V = typename Blk<MASK>::T;
    constexpr int NP = MASK == 3 ? 2 : 1;
    constexpr int P0 = MASK == 2 ? 1 : 0;    // first plane in the mask
    constexpr int BM = MASK == 2 ? 3 : 0;    // the block of a single-parameter mask
    constexpr int TZ = kRowThreads * R;      // rows of the CTA tile
    extern __shared__ __align__(16) float sm[];
    const int h = a.half, L = 2 * h + 1, LL = L * L;
    const int TRW = TZ + 2 * h, TCW = kTX + 2 * h;
    float *tile = sm;   // [TRW][TCW] of the input, plane pairs interleaved for two parameters
    Corner *zc = reinterpret_cast<Corner *>(tile + NP * TRW * TCW);    // [TRW]
    Corner *xc = zc + TRW;                                             // [TCW]
    const int t = threadIdx.x, tx = t % kTX, ty = t / kTX;
    const int Z0 = (int)blockIdx.y * TZ, X0 = (int)blockIdx.x * kTX;
    const long long plane = (long long)a.nz * a.nx;

    for (int i = t; i < TRW * TCW; i += kApplyThreads) {
        const int r = i / TCW, c = i - r * TCW;
        const int gz = Z0 - h + r, gx = X0 - h + c;
        const bool ok = gz >= 0 && gz < a.nz && gx >= 0 && gx < a.nx;
        const long long g = ok ? (long long)gz * a.nx + gx : 0;
        if (MASK == 3)
            reinterpret_cast<float2 *>(tile)[i] = ok ? make_float2(in[g], in[plane + g]) : make_float2(0.f, 0.f);
        else
            tile[i] = ok ? in[P0 * plane + g] : 0.f;
    }
    for (int i = t; i < TRW + TCW; i += kApplyThreads) {
        if (i < TRW) zc[i] = corner_of(Z0 - h + i, a.nz, a.s, a.nkz);
        else xc[i - TRW] = corner_of(X0 - h + (i - TRW), a.nx, a.s, a.nkx);
    }
    __syncthreads();
    const int rz0 = Z0 + ty * R, rx = X0 + tx;   // this thread: rows rz0 .. rz0 + R - 1, column rx
    if (rz0 >= a.nz || rx >= a.nx) return;

    const float4 *pt = a.pt;
    const int nkx = a.nkx, nkz1 = a.nkz - 1;
    const V zero = V{};
    using X = typename std::conditional<MASK == 3, float2, float>::type;
    const X *in_t = reinterpret_cast<const X *>(tile);
    float acc0[R], acc1[R];
#pragma unroll
    for (int r = 0; r < R; ++r) acc0[r] = acc1[r] = 0.f;
    typename Wgt<MASK>::T wb[R], wc[R];

    if (!TR) {
        // y(r) = sum_a [sum_corners(c) w P(a)] x(c), c = r - a: for offset
        // row dz the thread's input rows c are rz0 - dz .. + R - 1
        for (int dz = -h; dz <= h; ++dz) {
            const int row0 = ty * R + h - dz;   // tile row of c = rz0 - dz
            const int kf = zc[row0].k0;
            row_weights<MASK, R>(zc + row0, kf, wb, wc);
            const int n0 = kf * nkx, n1 = min(kf + 1, nkz1) * nkx, n2 = min(kf + 2, nkz1) * nkx;
            const int arow = (dz + h) * L + h;
            // node values of offset dx = -h, then of dx + 1 while dx is used
            const float4 *q0 = pt + n0 * LL + arow, *q1 = pt + n1 * LL + arow, *q2 = pt + n2 * LL + arow;
            auto sweep = [&](auto cross) {
                constexpr bool CROSS = decltype(cross)::value;
                V p00, p01, p10, p11, p20 = V{}, p21 = V{};
                float wx;
                auto load = [&](int dx) {
                    const Corner Xc = xc[tx + h - dx];
                    const int k0 = Xc.k0 * LL + dx, k1 = Xc.k1 * LL + dx;
                    wx = Xc.w;
                    p00 = load_blk<BM>(q0, k0, zero), p01 = load_blk<BM>(q0, k1, zero);
                    p10 = load_blk<BM>(q1, k0, zero), p11 = load_blk<BM>(q1, k1, zero);
                    if (CROSS) p20 = load_blk<BM>(q2, k0, zero), p21 = load_blk<BM>(q2, k1, zero);
                };
                load(-h);
                const X *xin = in_t + row0 * TCW + tx + 2 * h;   // input of offset dx = -h
                for (int dx = -h; dx <= h; ++dx) {
                    const V m0 = lerp_(p00, p01, wx), d1 = sub_(lerp_(p10, p11, wx), m0);
                    V d2 = V{};
                    if (CROSS) d2 = sub_(lerp_(p20, p21, wx), m0);
                    load(min(dx + 1, h));
#pragma unroll
                    for (int r = 0; r < R; ++r)
                        accum<TR>(acc0[r], acc1[r], CROSS ? mix3(m0, d1, d2, wb[r], wc[r]) : mix2(m0, d1, wb[r]), xin[r * TCW]);
                    --xin;
                }
            };
            if (any_weight<MASK, R>(wc)) sweep(std::true_type{});
            else sweep(std::false_type{});
        }
    } else {
        // y(c) = sum_a [sum_corners(c) w P(a)] x(c + a): the thread's rows c
        // and column are fixed, so are their corners
        const int row0 = ty * R + h;   // tile row of c = rz0
        const int kf = zc[row0].k0;
        row_weights<MASK, R>(zc + row0, kf, wb, wc);
        const int xk0 = xc[tx + h].k0, xk1 = xc[tx + h].k1;
        const float wx = xc[tx + h].w;
        const int n0 = kf * nkx, n1 = min(kf + 1, nkz1) * nkx, n2 = min(kf + 2, nkz1) * nkx;
        const int b00 = (n0 + xk0) * LL, b01 = (n0 + xk1) * LL, b10 = (n1 + xk0) * LL;
        const int b11 = (n1 + xk1) * LL, b20 = (n2 + xk0) * LL, b21 = (n2 + xk1) * LL;
        // the window offsets in storage order, the next offset's node values
        // loaded while the current one's are used
        const float4 *q00 = pt + b00, *q01 = pt + b01, *q10 = pt + b10, *q11 = pt + b11, *q20 = pt + b20, *q21 = pt + b21;
        auto sweep = [&](auto cross) {
            constexpr bool CROSS = decltype(cross)::value;
            V p00 = load_blk<BM>(q00, 0, zero), p01 = load_blk<BM>(q01, 0, zero);
            V p10 = load_blk<BM>(q10, 0, zero), p11 = load_blk<BM>(q11, 0, zero);
            V p20 = V{}, p21 = V{};
            if (CROSS) p20 = load_blk<BM>(q20, 0, zero), p21 = load_blk<BM>(q21, 0, zero);
            const X *xin = in_t + (row0 - h) * TCW + tx;   // input of offset (-h, -h)
            int dx = -h;
            for (int ai = 0; ai < LL; ++ai) {
                const V m0 = lerp_(p00, p01, wx), d1 = sub_(lerp_(p10, p11, wx), m0);
                V d2 = V{};
                if (CROSS) d2 = sub_(lerp_(p20, p21, wx), m0);
                const int an = min(ai + 1, LL - 1);
                p00 = load_blk<BM>(q00, an, zero), p01 = load_blk<BM>(q01, an, zero);
                p10 = load_blk<BM>(q10, an, zero), p11 = load_blk<BM>(q11, an, zero);
                if (CROSS) p20 = load_blk<BM>(q20, an, zero), p21 = load_blk<BM>(q21, an, zero);
#pragma unroll
                for (int r = 0; r < R; ++r)
                    accum<TR>(acc0[r], acc1[r], CROSS ? mix3(m0, d1, d2, wb[r], wc[r]) : mix2(m0, d1, wb[r]), xin[r * TCW]);
                ++xin;
                if (++dx > h) dx = -h, xin += TCW - L;
            }
        };
        if (any_weight<MASK, R>(wc)) sweep(std::true_type{});
        else sweep(std::false_type{});
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int z = rz0 + r;
        if (z >= a.nz) break;
        const long long o = (long long)z * a.nx + rx;
        if (MASK == 3) {
            out[o] = acc0[r];
            out[plane + o] = acc1[r];
        } else {
            out[P0 * plane + o] = acc0[r];
            out[(1 - P0) * plane + o] = 0.f;
        }
    }
}

size_t apply_smem(int mask, int half, int R)
{
    const int np = mask == 3 ? 2 : 1;
    const size_t rows = kRowThreads * R + 2 * half, cols = kTX + 2 * half;
    return np * rows * cols * sizeof(float) + (rows + cols) * sizeof(Corner);
}

template <int MASK, bool TR, int R>
cudaError_t launch_t(const PsfHessDev &a, const float *in, float *out, cudaStream_t s)
{
    const size_t sm = apply_smem(MASK, a.half, R);
    dim3 grid((a.nx + kTX - 1) / kTX, (a.nz + kRowThreads * R - 1) / (kRowThreads * R));
    k_psfh_apply<MASK, TR, R><<<grid, kApplyThreads, sm, s>>>(a, in, out);
    return cudaGetLastError();
}

template <int MASK, bool TR>
cudaError_t launch_r(const PsfHessDev &a, const float *in, float *out, cudaStream_t s)
{
    // rows per thread: the largest of 8, 4, 2, 1 not above the node spacing
    if (a.s >= 8) return launch_t<MASK, TR, 8>(a, in, out, s);
    if (a.s >= 4) return launch_t<MASK, TR, 4>(a, in, out, s);
    if (a.s >= 2) return launch_t<MASK, TR, 2>(a, in, out, s);
    return launch_t<MASK, TR, 1>(a, in, out, s);
}

// ---------------------------------------------------------------------------
// 3D (Eq. trilinear as printed: eight corners, products of the three 1D
// weights). CTAs of 32 x 4 (y, x) columns of R z rows; the corner tables of
// the z, y and x coordinates the CTA's windows reach sit in shared memory,
// inputs and node windows are read through L1.
// ---------------------------------------------------------------------------
constexpr int k3X = 32, k3Y = 4, k3Threads = k3X * k3Y;

__global__ void k_psfh3_patches(const float *psf_vp, const float *psf_ip, const PsfHess3Dev a, float4 *pt)
{
    const int L = 2 * a.half + 1, LL = L * L, LLL = LL * L;
    const long long vol = (long long)a.nz * a.ny * a.nx;
    const long long n = (long long)a.nkz * a.nky * a.nkx * LLL;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const int node = (int)(i / LLL), ai = (int)(i - (long long)node * LLL);
        const int kz = node / (a.nky * a.nkx), ky = (node / a.nkx) % a.nky, kx = node % a.nkx;
        const int z = (a.s >> 1) + kz * a.s + ai / LL - a.half;
        const int y = (a.s >> 1) + ky * a.s + (ai / L) % L - a.half;
        const int x = (a.s >> 1) + kx * a.s + ai % L - a.half;
        const bool inside = z >= 0 && z < a.nz && y >= 0 && y < a.ny && x >= 0 && x < a.nx;
        const long long v = inside ? ((long long)z * a.ny + y) * a.nx + x : 0;
        float e[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int po = b >> 1, pi = b & 1;
            const float *src = pi ? psf_ip : psf_vp;
            const bool use = inside && src && ((a.mask >> po) & 1) && ((a.mask >> pi) & 1);
            e[b] = use ? src[po * vol + v] : 0.f;
        }
        pt[i] = make_float4(e[0], e[1], e[2], e[3]);
    }
}

// The 3D kernel with the row blocking of the 2D one: each thread owns one
// (y, x) column and R consecutive z rows (R <= s, so its rows span at most
// three node rows); per window offset it loads the twelve node values
// covering them (3 node rows x 2 x 2), interpolates along x and y once and
// along z per row. Inputs are read through L1.
template <int MASK, bool TR, int R>
__global__ void __launch_bounds__(k3Threads) k_psfh3_rows(const PsfHess3Dev a, const float *__restrict__ in,
                                                           float *__restrict__ out)
{
    constexpr bool QUAD = MASK == 3 && !TR && R != 4;
    constexpr int PK = QUAD ? 1 : MASK;   // weights as the blocks take them
    using V = typename std::conditional<QUAD, Quad, typename Blk<MASK>::T>::type;
    constexpr int P0 = MASK == 2 ? 1 : 0;
    constexpr int BM = MASK == 2 ? 3 : 0;
    __shared__ Corner zc[8 + 2 * kPsfHessMaxHalf], yc[k3Y + 2 * kPsfHessMaxHalf], xc[k3X + 2 * kPsfHessMaxHalf];
    const int h = a.half, L = 2 * h + 1, LL = L * L, LLL = LL * L;
    const int t = threadIdx.x, tx = t % k3X, ty = t / k3X;
    const int X0 = (int)blockIdx.x * k3X, Y0 = (int)blockIdx.y * k3Y, Z0 = (int)blockIdx.z * R;
    const int NZ = R + 2 * h, NY = k3Y + 2 * h, NX = k3X + 2 * h;
    for (int i = t; i < NZ + NY + NX; i += k3Threads) {
        if (i < NZ) zc[i] = corner_of(Z0 - h + i, a.nz, a.s, a.nkz);
        else if (i < NZ + NY) yc[i - NZ] = corner_of(Y0 - h + (i - NZ), a.ny, a.s, a.nky);
        else xc[i - NZ - NY] = corner_of(X0 - h + (i - NZ - NY), a.nx, a.s, a.nkx);
    }
    __syncthreads();
    const int y = Y0 + ty, x = X0 + tx;
    if (y >= a.ny || x >= a.nx) return;
    const long long vol = (long long)a.nz * a.ny * a.nx, rowz = (long long)a.ny * a.nx;
    const float *in0 = in + P0 * vol, *in1 = in + vol;
    const float4 *pt = a.pt;
    const int nky = a.nky, nkx = a.nkx, nkz1 = a.nkz - 1;
    const V zero = V{};
    float acc0[R], acc1[R];
    typename Wgt<PK>::T wb[R], wc[R];
#pragma unroll
    for (int r = 0; r < R; ++r) acc0[r] = acc1[r] = 0.f;
    if (!TR) {
        for (int dz = -h; dz <= h; ++dz) {
            const int row0 = h - dz;   // zc index of c_z = Z0 - dz
            const int kf = zc[row0].k0;
            row_weights<PK, R>(zc + row0, kf, wb, wc);
            const int nq[3] = {kf, min(kf + 1, nkz1), min(kf + 2, nkz1)};
            for (int dy = -h; dy <= h; ++dy) {
                const int cy = y - dy;
                if (cy < 0 || cy >= a.ny) continue;
                const Corner Y = yc[ty + h - dy];
                for (int dx = -h; dx <= h; ++dx) {
                    const int cx = x - dx;
                    if (cx < 0 || cx >= a.nx) continue;
                    const Corner X = xc[tx + h - dx];
                    const int ai = ((dz + h) * L + (dy + h)) * L + (dx + h);
                    V Q[3];
#pragma unroll
                    for (int q = 0; q < 3; ++q) {
                        const int b0 = (nq[q] * nky + Y.k0) * nkx, b1 = (nq[q] * nky + Y.k1) * nkx;
                        const V v0 = lerp_(load_blk<BM>(pt, (b0 + X.k0) * LLL + ai, zero),
                                           load_blk<BM>(pt, (b0 + X.k1) * LLL + ai, zero), X.w);
                        const V v1 = lerp_(load_blk<BM>(pt, (b1 + X.k0) * LLL + ai, zero),
                                           load_blk<BM>(pt, (b1 + X.k1) * LLL + ai, zero), X.w);
                        Q[q] = lerp_(v0, v1, Y.w);
                    }
                    const V d1 = sub_(Q[1], Q[0]), d2 = sub_(Q[2], Q[0]);
                    const long long cb = (long long)cy * a.nx + cx;
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const int cz = Z0 + r - dz;
                        if (cz < 0 || cz >= a.nz) continue;
                        const V C = mix3(Q[0], d1, d2, wb[r], wc[r]);
                        const long long c = cz * rowz + cb;
                        if constexpr (MASK == 3) accum<TR>(acc0[r], acc1[r], C, make_float2(__ldg(in0 + c), __ldg(in1 + c)));
                        else accum<TR>(acc0[r], acc1[r], C, __ldg(in0 + c));
                    }
                }
            }
        }
    } else {
        const int kf = zc[h].k0;
        row_weights<PK, R>(zc + h, kf, wb, wc);
        const Corner Y = yc[ty + h], X = xc[tx + h];
        int base[3][2][2];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const int kz = min(kf + q, nkz1);
            base[q][0][0] = ((kz * nky + Y.k0) * nkx + X.k0) * LLL;
            base[q][0][1] = ((kz * nky + Y.k0) * nkx + X.k1) * LLL;
            base[q][1][0] = ((kz * nky + Y.k1) * nkx + X.k0) * LLL;
            base[q][1][1] = ((kz * nky + Y.k1) * nkx + X.k1) * LLL;
        }
        for (int dz = -h; dz <= h; ++dz) {
            for (int dy = -h; dy <= h; ++dy) {
                const int cy = y + dy;
                if (cy < 0 || cy >= a.ny) continue;
                for (int dx = -h; dx <= h; ++dx) {
                    const int cx = x + dx;
                    if (cx < 0 || cx >= a.nx) continue;
                    const int ai = ((dz + h) * L + (dy + h)) * L + (dx + h);
                    V Q[3];
#pragma unroll
                    for (int q = 0; q < 3; ++q) {
                        const V v0 = lerp_(load_blk<BM>(pt, base[q][0][0] + ai, zero),
                                           load_blk<BM>(pt, base[q][0][1] + ai, zero), X.w);
                        const V v1 = lerp_(load_blk<BM>(pt, base[q][1][0] + ai, zero),
                                           load_blk<BM>(pt, base[q][1][1] + ai, zero), X.w);
                        Q[q] = lerp_(v0, v1, Y.w);
                    }
                    const V d1 = sub_(Q[1], Q[0]), d2 = sub_(Q[2], Q[0]);
                    const long long cb = (long long)cy * a.nx + cx;
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const int cz = Z0 + r + dz;
                        if (cz < 0 || cz >= a.nz) continue;
                        const V C = mix3(Q[0], d1, d2, wb[r], wc[r]);
                        const long long c = cz * rowz + cb;
                        if constexpr (MASK == 3) accum<TR>(acc0[r], acc1[r], C, make_float2(__ldg(in0 + c), __ldg(in1 + c)));
                        else accum<TR>(acc0[r], acc1[r], C, __ldg(in0 + c));
                    }
                }
            }
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int z = Z0 + r;
        if (z >= a.nz) break;
        const long long o = z * rowz + (long long)y * a.nx + x;
        if (MASK == 3) {
            out[o] = acc0[r];
            out[vol + o] = acc1[r];
        } else {
            out[P0 * vol + o] = acc0[r];
            out[(1 - P0) * vol + o] = 0.f;
        }
    }
}

template <int MASK, bool TR, int R>
cudaError_t launch3_r(const PsfHess3Dev &a, const float *in, float *out, cudaStream_t s)
{
    dim3 grid((a.nx + k3X - 1) / k3X, (a.ny + k3Y - 1) / k3Y, (a.nz + R - 1) / R);
    k_psfh3_rows<MASK, TR, R><<<grid, k3Threads, 0, s>>>(a, in, out);
    return cudaGetLastError();
}

template <int MASK, bool TR>
cudaError_t launch3_t(const PsfHess3Dev &a, const float *in, float *out, cudaStream_t s)
{
    if (a.s >= 8) return launch3_r<MASK, TR, 8>(a, in, out, s);
    if (a.s >= 4) return launch3_r<MASK, TR, 4>(a, in, out, s);
    if (a.s >= 2) return launch3_r<MASK, TR, 2>(a, in, out, s);
    return launch3_r<MASK, TR, 1>(a, in, out, s);
}

}  // namespace

int psfh_max_half() { return kPsfHessMaxHalf; }

cudaError_t launch_psfh3_patches(const float *psf_vp, const float *psf_ip, const PsfHess3Dev &a,
                                 float4 *pt, cudaStream_t st)
{
    const long long L = 2 * a.half + 1;
    const long long n = (long long)a.nkz * a.nky * a.nkx * L * L * L;
    const int blocks = (int)std::min<long long>((n + 255) / 256, 152 * 16);
    k_psfh3_patches<<<blocks, 256, 0, st>>>(psf_vp, psf_ip, a, pt);
    return cudaGetLastError();
}

cudaError_t launch_psfh3_apply(const PsfHess3Dev &a, bool transpose, const float *in, float *out, cudaStream_t s)
{
    switch (a.mask * 2 + (transpose ? 1 : 0)) {
    case 2: return launch3_t<1, false>(a, in, out, s);
    case 3: return launch3_t<1, true>(a, in, out, s);
    case 4: return launch3_t<2, false>(a, in, out, s);
    case 5: return launch3_t<2, true>(a, in, out, s);
    case 6: return launch3_t<3, false>(a, in, out, s);
    case 7: return launch3_t<3, true>(a, in, out, s);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_psfh_patches(const float *psf_vp, const float *psf_ip, int nz, int nx, int s, int half,
                                int nkz, int nkx, int mask, float4 *pt, cudaStream_t st)
{
    const long long n = (long long)nkz * nkx * (2 * half + 1) * (2 * half + 1);
    const int blocks = (int)std::min<long long>((n + 255) / 256, 4096);
    k_psfh_patches<<<blocks, 256, 0, st>>>(psf_vp, psf_ip, nz, nx, s, half, nkz, nkx, mask, pt);
    return cudaGetLastError();
}

cudaError_t launch_psfh_apply(const PsfHessDev &a, bool transpose, const float *in, float *out, cudaStream_t s)
{
    switch (a.mask * 2 + (transpose ? 1 : 0)) {
    case 2: return launch_r<1, false>(a, in, out, s);
    case 3: return launch_r<1, true>(a, in, out, s);
    case 4: return launch_r<2, false>(a, in, out, s);
    case 5: return launch_r<2, true>(a, in, out, s);
    case 6: return launch_r<3, false>(a, in, out, s);
    case 7: return launch_r<3, true>(a, in, out, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace lsrtm
