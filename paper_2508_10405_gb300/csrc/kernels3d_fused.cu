// Fused 3D time-step kernels: one launch advances every shot of a batch by
// one time step of the Born operator (Eq. scattereqln driven by Eq. 1) or of
// its exact transpose (App. A), reading each state field once from HBM and
// writing it once (ping-pong buffers).
//
// A CTA of 384 threads owns a 32 x 12 tile of (x, y) columns, one column per
// thread, and marches down a z-chunk (two CTAs per SM):
//   * z stencils: per-thread register rings of length 2M, shifted after every
//     row;
//   * x and y stencils: shared-memory tiles of the current row. Every tile a
//     row needs (the centre column block, the x-extended and y-extended
//     halo blocks, the model) arrives by TMA (cp.async.bulk.tensor, one or
//     two copies an elected lane of every warp) into a 2-deep stage ring
//     guarded by mbarriers, one row ahead of the compute; the tensor maps zero-fill outside the padded
//     array, which is the operators' boundary convention;
//   * the velocity (half-node) stage is recomputed on the x and y halos, so
//     the pressure stage of the same row needs nothing from other CTAs and a
//     step needs no grid-wide barrier.
// A background field and its partner (scattered or adjoint) are float2
// pairs, so one 8-byte access and one packed FFMA2 serve both.
//
// Every mbarrier wait is bounded: after kWaitLimit polls the CTA sets the
// error word, waits (bounded) for its copies in flight and returns; the host
// reports the error.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>
#include <mutex>
#include <type_traits>

#include "lsrtm_internal.cuh"
#include "tma.cuh"

namespace lsrtm {
namespace {

constexpr int TX = kTile3X, TY = kTile3Y, NTH = TX * TY;
constexpr int PD = 2;                       // stage ring depth
constexpr int kMinBlocks = 2;               // resident CTAs per SM the register budget targets

// ---- packed arithmetic
__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 fma2(float a, float2 b, float2 c) { return __ffma2_rn(f2(a), b, c); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float a, float2 b) { return __fmul2_rn(f2(a), b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(f2(-1.f), b, a); }

// sum_l c_l (fa(l) - fb(l)), l = 1..M: M independent differences, then one
// multiply-add chain of depth M.
template <int M, class FA, class FB>
__device__ __forceinline__ float2 st2(const float *c, FA fa, FB fb)
{
    float2 d[M];
#pragma unroll
    for (int l = 0; l < M; ++l) d[l] = sub2(fa(l + 1), fb(l + 1));
    float2 acc = mul2(c[0], d[0]);
#pragma unroll
    for (int l = 1; l < M; ++l) acc = fma2(c[l], d[l], acc);
    return acc;
}
template <int M, class FA, class FB>
__device__ __forceinline__ float st1(const float *c, FA fa, FB fb)
{
    float d[M];
#pragma unroll
    for (int l = 0; l < M; ++l) d[l] = fa(l + 1) - fb(l + 1);
    float acc = c[0] * d[0];
#pragma unroll
    for (int l = 1; l < M; ++l) acc = fmaf(c[l], d[l], acc);
    return acc;
}

// Free surface (method of images about row z0): ghost node rows r < z0 read
// their mirror row with the sign flipped (p odd), ghost half rows k < z0 their
// mirror half row (v_z even).
__device__ __forceinline__ int node_src_row(const GridDev &g, int r) { return (g.fs && r < g.z0) ? fs_node_row(g, r) : r; }
__device__ __forceinline__ int half_src_row(const GridDev &g, int k) { return (g.fs && k < g.z0) ? fs_half_row(g, k) : k; }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
// Half-node and node z CPML rows.
__device__ __forceinline__ bool zpml_half(const GridDev &g, int k)
{
    return k >= 0 && k < g.Nz && (k <= g.z0 - 2 || k >= g.z0 + g.nz);
}
__device__ __forceinline__ bool zpml_node(const GridDev &g, int r)
{
    return r >= 0 && r < g.Nz && (r <= g.z0 - 1 || r >= g.z0 + g.nz);
}

// ---- shared memory, mbarriers and TMA (tma.cuh)
using tma::al128;
using tma::kWaitLimit;
using tma::mbar_expect;
using tma::mbar_init;
using tma::mbar_wait;
using tma::su32;
__device__ __forceinline__ void tma4(void *dst, const CUtensorMap &m, int x, int y, int z, int q, uint64_t *b)
{
    tma::load4(dst, m, x, y, z, q, b);
}

// Tile geometry for half-width M. Box shapes (x extent in elements, rows):
//   core  TX x TY                      the thread block's own columns
//   xbox  XW1 x TY   from x0 - 4       half nodes [x0-M, x0+TX+M-2] and their rho pairs
//   ybox  TX x YH1   from y0 - M       half nodes [y0-M, y0+TY+M-2]
//   ybr   XW1 x YHB  from (x0-4, y0-M) rho pairs of both half-node directions
//   wide  XW2 x YH2  from (x0-XO2, y0-YO2) nodes feeding the halo stencils
// Every x start is a multiple of 4 elements, so each TMA copy starts on a
// 16-byte boundary for float and float2 elements alike.
template <int M>
struct Geo {
    static constexpr int W = 2 * M;
    static constexpr int XO1 = 4, XW1 = TX + 8;
    static constexpr int XO2 = (2 * M + 3) / 4 * 4, XW2 = TX + 2 * XO2;
    static constexpr int XH1 = TX + 2 * M - 1;   // half nodes [x0-M, x0+TX+M-2]
    static constexpr int YO1 = M, YH1 = TY + 2 * M - 1, YHB = TY + 2 * M;
    static constexpr int YO2 = 2 * M - 1, YH2 = TY + 4 * M - 2;
    static_assert(XO1 >= M && XO2 >= 2 * M - 1, "halo offsets");
};

// ---------------------------------------------------------------------------
// Born modelling step n -> n+1.
//
// What bounds it: 80 B a cell in one pass (105 measured: the tiles' halos come
// from DRAM again where neighbours run apart in z) and the issue slots of the
// halo work. So every warp issues one of a row's tile copies (one thread that
// issued all eleven was waited for by the CTA), the half nodes of a row are
// dealt to the threads once per launch (its own x and y half node and at most
// one of the halo's), tiles and rows away from the strips run a form without
// boundary tests, and strip tiles apply the CPML terms to all columns with
// profiles that are zero outside the strips. 2 shots of 168 x 296 x 296 cells,
// order 8: 107.2 -> 84.6 ms in 96 steps, 26.4 -> 33.4 G cell-updates/s in the
// same chunk of 168 rows; 73.7 ms = 38.4 G = 0.46 of the measured copy rate
// with march3d_rows' chunks.
// ---------------------------------------------------------------------------
template <int M>
struct BornSmem {
    using G = Geo<M>;
    // stage layout (bytes)
    static constexpr unsigned PA = 0;                                     // p, row z+W-1, core
    static constexpr unsigned VZ = PA + al128(TX * TY * 8);               // vz, half row z+M-1, core
    static constexpr unsigned BK = VZ + al128(TX * TY * 8);               // br pairs, row z+M, core
    static constexpr unsigned KD = BK + al128(TX * TY * 8);               // kd pairs, row z, core
    static constexpr unsigned PZ = KD + al128(TX * TY * 8);               // psi_pz, half row z+M-1, core
    static constexpr unsigned PW = PZ + al128(TX * TY * 8);               // p, row z, wide
    static constexpr unsigned VX = PW + al128(G::XW2 * G::YH2 * 8);       // vx, row z, xbox
    static constexpr unsigned VY = VX + al128(G::XW1 * TY * 8);           // vy, row z, ybox
    static constexpr unsigned BR = VY + al128(TX * G::YH1 * 8);           // br pairs, row z, ybr
    static constexpr unsigned PX = BR + al128(G::XW1 * G::YHB * 8);       // psi_px, row z, xbox
    static constexpr unsigned PY = PX + al128(G::XW1 * TY * 8);           // psi_py, row z, ybox
    static constexpr unsigned STAGE = PY + al128(TX * G::YH1 * 8);
    // after the stages: the new vx / vy of the row (half-node halos)
    static constexpr unsigned OVX = PD * STAGE;
    static constexpr unsigned OVY = OVX + al128(G::XW1 * TY * 8);
    // CPML profiles over the tile, zero outside the strips: a, b at the half
    // nodes along x and y (halo included), a, b at the nodes
    static constexpr unsigned TAB = OVY + al128(TX * G::YH1 * 8);
    static constexpr int HX = 0, HY = HX + 2 * G::XH1, NX = HY + 2 * G::YH1, NY = NX + 2 * TX, NTAB = NY + 2 * TY;
    static constexpr unsigned BAR = TAB + al128(NTAB * 4);
    static constexpr unsigned TOTAL = BAR + 64 + 128;   // + alignment slack
};

}  // namespace

size_t fused3d_born_smem(int M) { return M == 2 ? BornSmem<2>::TOTAL : BornSmem<4>::TOTAL; }

namespace {

// One of the row's copies per warp (called by whole warps).
template <int M>
__device__ __forceinline__ void born_issue(const Step3F &a, int warp, unsigned char *st, uint64_t *bar, int slot, int x0,
                                           int y0, int z, int zc0, bool px, bool py)
{
    using G = Geo<M>;
    using S = BornSmem<M>;
    const GridDev &g = a.g;
    const int k = z + M - 1, r = z + G::W - 1;
    const bool main = z >= zc0;
    const bool pzs = zpml_half(g, k);
    const int q = slot * a.in_pairs;   // pair-plane index of the slot's first field
    // x coordinates in floats (pairs x 2); each a multiple of 4 (16 bytes)
    const int xc = 2 * x0, x1 = 2 * (x0 - G::XO1), x2 = 2 * (x0 - G::XO2);
    if (warp == 0) {
        if (tma::elect_one()) tma4(st + S::PA, a.in_core, xc, y0, node_src_row(g, r), q + F3_P, bar);
    } else if (warp == 1) {
        if (tma::elect_one()) tma4(st + S::VZ, a.in_core, xc, y0, half_src_row(g, k), q + F3_VZ, bar);
    } else if (warp == 2) {
        if (tma::elect_one()) tma4(st + S::BK, a.m_core, xc, y0, k + 1, 1, bar);
    } else if (warp == 3) {
        if (pzs && tma::elect_one()) tma4(st + S::PZ, a.in_core, xc, y0, k, q + F3_PPZ, bar);
    } else if (warp == 4) {
        if (main && tma::elect_one()) tma4(st + S::KD, a.m_core, xc, y0, z, 0, bar);
    } else if (warp == 5) {
        if (main && tma::elect_one()) tma4(st + S::PW, a.in_wide, x2, y0 - G::YO2, z, q + F3_P, bar);
    } else if (warp == 6) {
        if (main && tma::elect_one()) tma4(st + S::VX, a.in_xbox, x1, y0, z, q + F3_VX, bar);
    } else if (warp == 7) {
        if (main && tma::elect_one()) tma4(st + S::VY, a.in_ybox, xc, y0 - G::YO1, z, q + F3_VY, bar);
    } else if (warp == 8) {
        if (main && tma::elect_one()) tma4(st + S::BR, a.m_ybr, x1, y0 - G::YO1, z, 1, bar);
    } else if (warp == 9) {
        if (main && px && tma::elect_one()) tma4(st + S::PX, a.in_xbox, x1, y0, z, q + F3_PPX, bar);
    } else if (warp == 10) {
        if (main && py && tma::elect_one()) tma4(st + S::PY, a.in_ybox, xc, y0 - G::YO1, z, q + F3_PPY, bar);
    } else if (tma::elect_one()) {
        unsigned bytes = 3 * TX * TY * 8 + (pzs ? TX * TY * 8 : 0);
        if (main) {
            bytes += TX * TY * 8 + G::XW2 * G::YH2 * 8 + G::XW1 * TY * 8 + TX * G::YH1 * 8 + G::XW1 * G::YHB * 8;
            if (px) bytes += G::XW1 * TY * 8;
            if (py) bytes += TX * G::YH1 * 8;
        }
        mbar_expect(bar, bytes);
    }
    __syncwarp();
}

template <int M>
__global__ void __launch_bounds__(NTH, kMinBlocks) k3f_born(const __grid_constant__ Step3F a)
{
    if (guard_tripped(a.g)) return;
    using G = Geo<M>;
    using S = BornSmem<M>;
    constexpr int W = G::W;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *sm = smem_raw + ((128u - (su32(smem_raw) & 127u)) & 127u);
    uint64_t *bar = reinterpret_cast<uint64_t *>(sm + S::BAR);
    float2 *oVX = reinterpret_cast<float2 *>(sm + S::OVX);
    float2 *oVY = reinterpret_cast<float2 *>(sm + S::OVY);

    const GridDev &g = a.g;
    const int t = threadIdx.x, tx = t % TX, ty = t / TX;
    const int warp = __shfl_sync(0xffffffffu, t >> 5, 0);   // (known to be uniform)
    const int nzc = (g.Nz + a.tzc - 1) / a.tzc;
    const int slot = blockIdx.z / nzc, zcn = blockIdx.z - slot * nzc;
    const int shot = a.shot0 + slot;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
    const int x = x0 + tx, y = y0 + ty;
    const bool colok = x < g.Nx && y < g.Ny;
    const int zc0 = zcn * a.tzc, zc1 = min(zc0 + a.tzc, g.Nz);
    const int zstart = zc0 - W;
    const float dt = g.dt;
    const long long plane = g.plane;
    const long long cxy = (long long)y * g.pitch + x;
    // CTA-uniform: does the tile's x (y) halo reach a CPML strip?
    const bool px = (x0 - M <= g.x0 - 2) || (x0 + TX + M - 2 >= g.x0 + g.nx);
    const bool py = (y0 - M <= g.y0 - 2) || (y0 + TY + M - 2 >= g.y0 + g.ny);
    const bool xyf = !px && !py;   // (then every node and half node of the tile and its halo is interior)
    float2 *out = reinterpret_cast<float2 *>(a.out) + slot * a.out_pairs * plane;
    float2 *psv = reinterpret_cast<float2 *>(a.psiv) + slot * a.psiv_pairs * plane;   // in place: x y z
    const int src = a.src_cell[shot];
    const float wsrc = a.wav[(a.wav_per_shot ? (long long)shot * g.nt : 0) + a.n];

    float *tab = reinterpret_cast<float *>(sm + S::TAB);
    if (t == 0) {
        for (int i = 0; i < PD; ++i) mbar_init(bar + i);
        tma::mbar_init_fence();
    }
    for (int i = t; i < S::NTAB; i += NTH) {
        int d, e;   // axis, and entry in its (a, b) table
        const float *pa, *pb;
        if (i < S::NX) {
            d = i < S::HY ? 2 : 1;
            e = i < S::HY ? i : i - S::HY;
            pa = a.pml.ah[d], pb = a.pml.bh[d];
        } else {
            d = i < S::NY ? 2 : 1;
            e = i < S::NY ? i - S::NX : i - S::NY;
            pa = a.pml.ai[d], pb = a.pml.bi[d];
        }
        const int len = i < S::NX ? (d == 2 ? G::XH1 : G::YH1) : (d == 2 ? TX : TY);
        const int q = e % len, c0 = (d == 2 ? x0 : y0) - (i < S::NX ? M : 0) + q, N = d == 2 ? g.Nx : g.Ny;
        tab[i] = c0 >= 0 && c0 < N ? (e < len ? pa : pb)[c0] : 0.f;
    }
    __syncthreads();
    for (int j = 0; j < PD - 1; ++j)
        if (zstart + j < zc1) born_issue<M>(a, warp, sm + j * S::STAGE, bar + j, slot, x0, y0, zstart + j, zc0, px, py);

    // This thread's half nodes: its column's x and y ones (all offsets around
    // the centre of the wide and ybr tiles), and one of the halo's: vy rows
    // outside the tile for the first 2M - 1 warps, vx columns outside it for
    // the next threads. Half nodes before the array's start are zero (past its
    // end 1/rho reads zero), the last one replicates the last node's 1/rho.
    constexpr int NH = 2 * M - 1;
    static_assert(NH + (TY * NH + 31) / 32 <= TY, "one halo item per thread");
    const int wc = (ty + G::YO2) * G::XW2 + tx + G::XO2, bc = (ty + M) * G::XW1 + tx + G::XO1;
    const int vxi = ty * G::XW1 + tx + G::XO1, vyi = (ty + M) * TX + tx;
    const bool halo_y = warp < NH;
    const int he = (warp - NH) * 32 + tx;
    const bool halo_x = !halo_y && he < TY * NH;
    int hw = 0, hb = 0, hv = 0, ho = 0, hi = 0, hq = 0;   // entries in the wide, ybr, v and output tiles; index along the axis, in its table
    if (halo_y) {
        const int jy = warp < M ? warp : warp + TY;
        hw = (jy + M - 1) * G::XW2 + tx + G::XO2;
        hb = jy * G::XW1 + tx + G::XO1;
        hv = ho = jy * TX + tx;
        hi = y0 - M + jy;
        hq = S::HY + jy;
    } else if (halo_x) {
        const int iy = he / NH, q = he - iy * NH, jx = q < M ? q : q + TX;
        hw = (iy + G::YO2) * G::XW2 + (jx - M + G::XO2);
        hb = (iy + M) * G::XW1 + (jx - M + G::XO1);
        hv = iy * G::XW1 + (jx - M + G::XO1);
        ho = iy * G::XW1 + jx;
        hi = x0 - M + jx;
        hq = S::HX + jx;
    }
    const float hscale = hi >= 0 ? 0.5f : 0.f;

    // z rings, shifted by U entries after every U rows: entry u + m holds p^n
    // at row z + m (P) or vz^{n+1/2} at half row z + m - M (VZ) of the pass's
    // row u
    constexpr int U = 1, RL = W + U - 1;
    float2 P[RL], VZ[RL];
    {
        const float2 *pin = reinterpret_cast<const float2 *>(a.in) + slot * a.in_pairs * plane + F3_P * plane;
#pragma unroll
        for (int m = 0; m < RL; ++m) {
            P[m] = make_float2(0.f, 0.f);
            if (m < W - 1) {
                const int zr = zstart + m, zs = node_src_row(g, zr);
                const float2 v = (colok && zs >= 0 && zs < g.Nz) ? pin[zs * g.rowz + cxy] : make_float2(0.f, 0.f);
                P[m] = zs != zr ? neg2(v) : v;
            }
            VZ[m] = make_float2(0.f, 0.f);
        }
    }
    float2 br_old = make_float2(0.f, 0.f);
    {
        const int kk = zstart + M - 1;
        if (colok && kk >= 0 && kk < g.Nz) br_old = a.br2[kk * g.rowz + cxy];
    }

    // this column's strips of the node CPML memories
    const bool xp = colok && (x <= g.x0 - 1 || x >= g.x0 + g.nx), yp = colok && (y <= g.y0 - 1 || y >= g.y0 + g.ny);
    bool failed = false;
    int fail_row = 0;
    const int pl = (int)plane;   // in-slot offsets fit in 32 bits (checked by the host)
    const int rowz = (int)g.rowz, pitch = g.pitch;
    const int cxy32 = y * pitch + x;
    for (int zb = zstart; zb < zc1 && !failed; zb += U) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int z = zb + u;
            if (z >= zc1) break;
            const int j = z - zstart;
            const bool to = !mbar_wait(bar + j % PD, (unsigned)(j / PD) & 1u);
            // (this barrier also certifies that every thread is done with row
            // z-1, its stage and the vx / vy tiles)
            if (__syncthreads_or(to)) {
                failed = true;
                fail_row = z;
                break;
            }
            if (z + PD - 1 < zc1)   // refill the stage of row z-1 with row z+PD-1
                born_issue<M>(a, warp, sm + ((j + PD - 1) % PD) * S::STAGE, bar + (j + PD - 1) % PD, slot, x0, y0,
                              z + PD - 1, zc0, px, py);
            const unsigned char *st = sm + (j % PD) * S::STAGE;
            auto tile = [&](unsigned off) { return reinterpret_cast<const float2 *>(st + off); };
            const int k = z + M - 1, c = z * rowz + cxy32;
            const bool main = z >= zc0;
            const bool zf = main && z > g.z0 && z + W < g.z0 + g.nz;
            // node CPML memories, for the last stage
            float2 mx = make_float2(0.f, 0.f), my = mx, mz = mx;
            if (!xyf && main) {
                if (xp) mx = psv[c];
                if (yp) my = psv[pl + c];
            }
            const bool zs = main && !zf && zpml_node(g, z);
            if (zs && colok) mz = psv[2 * pl + c];
            // ---- vz at half row k (column-local), then the half nodes of row
            // z. ZF: rows without tests (the rows and all they reach are
            // interior); XY: tiles without strips. In strip tiles the CPML
            // terms run on every column, with zero profiles outside the strips.
            auto v_stage = [&](auto zc, auto xyc) {
                constexpr bool ZF = decltype(zc)::value, XY = decltype(xyc)::value;
                const float2 pa = tile(S::PA)[t];
                P[u + W - 1] = (!ZF && g.fs && z + W - 1 < g.z0) ? neg2(pa) : pa;   // ghost rows: -p(mirror)
                // (the last half row replicates the last node row's buoyancy)
                float2 brk1 = tile(S::BK)[t];
                if (!ZF && k + 1 >= g.Nz) brk1 = make_float2(br_old.x, 0.f);
                float2 vzn = make_float2(0.f, 0.f);
                if (ZF || (k >= 0 && k < g.Nz)) {
                    float2 Gz = st2<M>(g.cz, [&](int l) { return P[u + M - 1 + l]; }, [&](int l) { return P[u + M - l]; });
                    const bool own = (XY || colok) && (ZF || k >= zc0) && k < zc1;
                    if (!ZF && (k <= g.z0 - 2 || k >= g.z0 + g.nz)) {
                        const float2 ps = fma2(a.pml.bh[0][k], tile(S::PZ)[t], mul2(a.pml.ah[0][k], Gz));
                        if (own) out[F3_PPZ * pl + k * rowz + cxy32] = ps;
                        Gz = add2(Gz, ps);
                    }
                    const float bu = 0.5f * (br_old.x + brk1.x);
                    vzn = fma2(-dt * bu, Gz, tile(S::VZ)[t]);
                    vzn.y = fmaf(0.5f * dt * (br_old.y + brk1.y), Gz.x, vzn.y);
                    if (own) out[F3_VZ * pl + k * rowz + cxy32] = vzn;
                }
                br_old = brk1;
                VZ[u + W - 1] = vzn;
                if (!ZF && !main) return;
                // one half node: entries in the wide and ybr tiles, tap strides
                // there, the stored velocity; strip: its table entries a (at q)
                // and b (len further), its memory
                auto half = [&](const float *cf, int w, int ws, int b, int bst, float2 v0, float hs, bool last, bool strip,
                                int q, int len, const float2 *psi, float2 *ps_out) -> float2 {
                    const float2 *p = tile(S::PW) + w;
                    float2 Gd = st2<M>(cf, [&](int l) { return p[l * ws]; }, [&](int l) { return p[(1 - l) * ws]; });
                    if (!XY && strip) {
                        const float pb = tab[q + len];
                        const float2 ps = fma2(pb, *psi, mul2(tab[q], Gd));
                        if (ps_out && pb != 0.f) *ps_out = ps;
                        Gd = add2(Gd, ps);
                    }
                    const float2 b0 = tile(S::BR)[b];
                    float2 b1 = tile(S::BR)[b + bst];
                    if (!XY && last) b1 = make_float2(b0.x, 0.f);
                    float2 v = fma2(-dt * (hs * (b0.x + b1.x)), Gd, v0);
                    v.y = fmaf(hs * dt * (b0.y + b1.y), Gd.x, v.y);
                    return v;
                };
                {
                    const float2 v = half(g.cx, wc, 1, bc, 1, tile(S::VX)[vxi], 0.5f, x + 1 >= g.Nx, px, S::HX + tx + M, G::XH1,
                                          tile(S::PX) + vxi, colok ? out + F3_PPX * pl + c : nullptr);
                    oVX[ty * G::XW1 + tx + M] = v;
                    if (XY || colok) out[F3_VX * pl + c] = v;
                }
                {
                    const float2 v = half(g.cy, wc, G::XW2, bc, G::XW1, tile(S::VY)[vyi], 0.5f, y + 1 >= g.Ny, py,
                                          S::HY + ty + M, G::YH1, tile(S::PY) + vyi, colok ? out + F3_PPY * pl + c : nullptr);
                    oVY[vyi] = v;
                    if (XY || colok) out[F3_VY * pl + c] = v;
                }
                if (halo_y)
                    oVY[ho] = half(g.cy, hw, G::XW2, hb, G::XW1, tile(S::VY)[hv], XY ? 0.5f : hscale, hi + 1 >= g.Ny, py, hq,
                                   G::YH1, tile(S::PY) + hv, nullptr);
                else if (halo_x)
                    oVX[ho] = half(g.cx, hw, 1, hb, 1, tile(S::VX)[hv], XY ? 0.5f : hscale, hi + 1 >= g.Nx, px, hq, G::XH1,
                                   tile(S::PX) + hv, nullptr);
            };
            // ---- pressure at row z on the thread's own column
            auto p_stage = [&](auto zc, auto xyc) {
                constexpr bool ZF = decltype(zc)::value, XY = decltype(xyc)::value;
                const float2 *vxr = oVX + ty * G::XW1 + tx + M;
                const float2 *vyc = oVY + vyi;
                float2 Qx = st2<M>(g.cx, [&](int l) { return vxr[l - 1]; }, [&](int l) { return vxr[-l]; });
                float2 Qy = st2<M>(g.cy, [&](int l) { return vyc[(l - 1) * TX]; }, [&](int l) { return vyc[-l * TX]; });
                float2 Qz = st2<M>(g.cz, [&](int l) { return VZ[u + M + l - 1]; }, [&](int l) { return VZ[u + M - l]; });
                if (!XY && px) {
                    const float2 ps = fma2(tab[S::NX + TX + tx], mx, mul2(tab[S::NX + tx], Qx));
                    if (xp) psv[c] = ps;
                    Qx = add2(Qx, ps);
                }
                if (!XY && py) {
                    const float2 ps = fma2(tab[S::NY + TY + ty], my, mul2(tab[S::NY + ty], Qy));
                    if (yp) psv[pl + c] = ps;
                    Qy = add2(Qy, ps);
                }
                if (!ZF && zs) {
                    const float2 ps = fma2(a.pml.bi[0][z], mz, mul2(a.pml.ai[0][z], Qz));
                    if (colok) psv[2 * pl + c] = ps;
                    Qz = add2(Qz, ps);
                }
                const float2 Q = add2(add2(Qx, Qy), Qz);
                const float2 kd = tile(S::KD)[t];
                float2 pn = fma2(-kd.x, Q, P[u]);
                pn.y = fmaf(-kd.y, Q.x, pn.y);
                pn.x = fmaf(a.src_scale, c == src ? wsrc : 0.f, pn.x);
                if (!ZF && g.fs && z <= g.z0) pn = make_float2(0.f, 0.f);   // p = 0 on the free surface
                if (XY || colok) out[F3_P * pl + c] = pn;
            };
            const std::true_type Y{};
            const std::false_type N{};
            if (xyf) {
                if (zf) v_stage(Y, Y);
                else v_stage(N, Y);
            } else {
                if (zf) v_stage(Y, N);
                else v_stage(N, N);
            }
            if (!main) continue;
            __syncthreads();
            if (xyf) {
                if (zf) p_stage(Y, Y);
                else p_stage(N, Y);
            } else {
                if (zf) p_stage(Y, N);
                else p_stage(N, N);
            }
        }
#pragma unroll
        for (int m = 0; m < W - 1; ++m) {
            P[m] = P[m + U];
            VZ[m] = VZ[m + U];
        }
    }

    if (failed) {
        if (t == 0) {
            atomicOr(a.err, 1);
            // rows issued and not yet consumed: jf .. jf + PD - 2 (bounded waits)
            const int jf = fail_row - zstart;
            for (int jj = jf; jj < jf + PD - 1 && zstart + jj < zc1; ++jj)
                (void)mbar_wait(bar + jj % PD, (unsigned)(jj / PD) & 1u);
        }
        return;
    }
    // records dp^{n+1} at the receivers of this tile
    __syncthreads();
    const int ntile = (int)(gridDim.x * gridDim.y) * nzc;
    const int rt = shot * ntile + (zcn * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    const int b = a.trec.ptr[rt], e = a.trec.ptr[rt + 1];
    for (int i = b + t; i < e; i += NTH) {
        const int2 rc = a.trec.rec[i];
        a.dstage[(long long)rc.y * g.nt + a.n] = out[F3_P * plane + rc.x].y;   // (all rows written: barrier above)
    }
}

// ---------------------------------------------------------------------------
// Adjoint (migration) step n: the exact reverse-order transpose of the Born
// sub-steps, the zero-lag imaging condition and the reconstruction of the
// background p^{n-1}, v^{n-1/2} from p^n, v^{n+1/2} and the boundary bands
// (App. A), arranged as in the 2D kernel. State pairs (background, adjoint):
// (p, mu = dt kappa lambda_p) at nodes, (v_d, lambda_v_d) at half nodes; the
// lambda CPML memories as float planes. For the half-node stencils each node
// carries (p, u_d) with u_d = mu - a_d (lambda_psi_v_d - mu) (a_d nonzero only
// in the d strips, where u_d is formed once per node).
//
// What bounds it: 88 B a cell in one pass, but the kernel is held back by
// latencies and instructions (56% of the issue slots used): four outputs a half
// node instead of one. Against the form it replaces: mu in place of lambda_p
// needs no pass over the wide tile and no dt kappa there; the four values of a
// half node lie in one float4, read by one load a tap; the image comes by TMA
// (read where it was used, every row waited for it); band values of the strips
// are loaded a stage ahead at offsets formed once; registers that did not fit
// went to L2 (16 KB of L1 are left beside the tiles), so offsets are formed
// anew instead. 2 shots of 168 x 296 x 296, order 8, BF16 bands: 229.0 ->
// 154.2 ms in 96 steps in one chunk of 168 rows, 120.5 ms = 23.5 G
// cell-updates/s = 0.31 of the measured copy rate with march3d_rows' chunks.
// ---------------------------------------------------------------------------

// Face bands (as written by the 3D background kernels):
// [x faces 2M nz ny][y faces 2M nz nx][z faces 2M ny nx]; -1 if the interior
// offsets (iz, iy, ix) are not in the d face band.
__device__ __forceinline__ long long fband(const GridDev &g, int d, int iz, int iy, int ix)
{
    const int M = g.M;
    const int i = d == 0 ? iz : (d == 1 ? iy : ix);
    const int n = d == 0 ? g.nz : (d == 1 ? g.ny : g.nx);
    int sb;
    if (i >= -M && i < 0) sb = i + M;
    else if (i >= n && i < n + M) sb = M + (i - n);
    else return -1;
    if (d != 0 && (iz < 0 || iz >= g.nz)) return -1;
    if (d != 1 && (iy < 0 || iy >= g.ny)) return -1;
    if (d != 2 && (ix < 0 || ix >= g.nx)) return -1;
    if (d == 2) return ((long long)iz * g.ny + iy) * (2 * M) + sb;
    long long base = 2LL * M * g.nz * g.ny;
    if (d == 1) return base + ((long long)iz * (2 * M) + sb) * g.nx + ix;
    base += 2LL * M * g.nz * g.nx;
    return base + ((long long)sb * g.ny + iy) * g.nx + ix;
}

template <int M>
struct AdjSmem {
    using G = Geo<M>;
    static constexpr unsigned PA = 0;                                  // (p, mu) row z+W-1, core
    static constexpr unsigned LA = PA + al128(TX * TY * 8);            // lpsi_vz, row z+W-1 (strip)
    static constexpr unsigned VZ = LA + al128(TX * TY * 4);            // (vz, lvz) half row z+M-1
    static constexpr unsigned BK = VZ + al128(TX * TY * 8);            // 1/rho, row z+M
    static constexpr unsigned PZ = BK + al128(TX * TY * 4);            // lpsi_pz half row z+M-1 (strip)
    static constexpr unsigned KD = PZ + al128(TX * TY * 4);            // dt kappa, row z
    static constexpr unsigned PW = KD + al128(TX * TY * 4);            // (p, mu) row z, wide
    static constexpr unsigned LX = PW + al128(G::XW2 * G::YH2 * 8);    // lpsi_vx, x-wide (strip tiles), then u_x
    static constexpr unsigned LY = LX + al128(G::XW2 * TY * 4);        // lpsi_vy, y-wide (strip tiles), then u_y
    static constexpr unsigned VX = LY + al128(TX * G::YH2 * 4);        // (vx, lvx) xbox
    static constexpr unsigned VY = VX + al128(G::XW1 * TY * 8);        // (vy, lvy) ybox
    static constexpr unsigned BB = VY + al128(TX * G::YH1 * 8);        // 1/rho ybr
    static constexpr unsigned QX = BB + al128(G::XW1 * G::YHB * 4);    // lpsi_px xbox (strip tiles)
    static constexpr unsigned QY = QX + al128(G::XW1 * TY * 4);        // lpsi_py ybox (strip tiles)
    static constexpr unsigned IM = QY + al128(TX * G::YH1 * 4);        // image, row z, core (interior rows)
    static constexpr unsigned STAGE = IM + al128(TX * TY * 8);
    // the half nodes of the row: (v^{n+1/2}, w, v^{n-1/2}, G lambda_v)
    static constexpr unsigned OX = PD * STAGE;
    static constexpr unsigned OY = OX + al128(G::XW1 * TY * 16);
    // CPML profiles over the tile, zero outside the strips: a, b at the half
    // nodes along x and y, a at the nodes of the wide tile, b at the own nodes;
    // then the step's (p, v) band scales
    static constexpr unsigned TAB = OY + al128(TX * G::YH1 * 16);
    static constexpr int HX = 0, HY = HX + 2 * G::XH1, WX = HY + 2 * G::YH1, WY = WX + G::XW2, NX = WY + G::YH2,
                         NY = NX + TX, SC = NY + TY, NTAB = SC + 2;
    static constexpr unsigned BAR = TAB + al128(NTAB * 4);
    static constexpr unsigned TOTAL = BAR + 64 + 128;
};

// two CTAs of each fused kernel per SM: 228 KB per SM, 1 KB reserved per CTA
static_assert(2 * (AdjSmem<4>::TOTAL + 1024) <= 233472 && 2 * (BornSmem<4>::TOTAL + 1024) <= 233472,
              "fused 3D kernels must fit two CTAs per SM");

}  // namespace

size_t fused3d_adj_smem(int M) { return M == 2 ? AdjSmem<2>::TOTAL : AdjSmem<4>::TOTAL; }

namespace {

// A row's copies, dealt to the warps (called by whole warps).
template <int M>
__device__ __forceinline__ void adj_issue(const Adj3F &a, int warp, unsigned char *st, uint64_t *bar, int slot, int x0,
                                          int y0, int z, int zc0, bool px, bool py, bool px2, bool py2)
{
    using G = Geo<M>;
    using S = AdjSmem<M>;
    const GridDev &g = a.g;
    const int k = z + M - 1, r = z + G::W - 1;
    const bool main = z >= zc0, im = main && z >= g.z0 && z < g.z0 + g.nz;
    const bool rs = zpml_node(g, r), ks = zpml_half(g, k);
    const int qp = slot * (a.in_planes / 2), qf = slot * a.in_planes;
    constexpr unsigned C8 = TX * TY * 8, C4 = TX * TY * 4;
    const int xc = x0, x1 = x0 - G::XO1, x2 = x0 - G::XO2;   // floats, each a multiple of 4 (16 bytes); pairs use 2x
    if (warp == 0) {
        if (tma::elect_one()) tma4(st + S::PA, a.p_core, 2 * xc, y0, node_src_row(g, r), qp + A3F_PL / 2, bar);
    } else if (warp == 1) {
        if (tma::elect_one()) tma4(st + S::VZ, a.p_core, 2 * xc, y0, half_src_row(g, k), qp + A3F_VZ / 2, bar);
    } else if (warp == 2) {
        if (tma::elect_one()) {
            tma4(st + S::BK, a.m_core, xc, y0, k + 1, 1, bar);
            if (main) tma4(st + S::KD, a.m_core, xc, y0, z, 0, bar);
        }
    } else if (warp == 3) {
        if ((rs || ks || im) && tma::elect_one()) {
            if (im) tma4(st + S::IM, a.im, 2 * xc, y0, z, slot, bar);
            if (rs) tma4(st + S::LA, a.f_core, xc, y0, r, qf + A3F_LPVZ, bar);
            if (ks) tma4(st + S::PZ, a.f_core, xc, y0, k, qf + A3F_LPPZ, bar);
        }
    } else if (warp == 4) {
        if (main && tma::elect_one()) tma4(st + S::PW, a.p_wide, 2 * x2, y0 - G::YO2, z, qp + A3F_PL / 2, bar);
    } else if (warp == 5) {
        if (main && tma::elect_one()) tma4(st + S::VX, a.p_xbox, 2 * x1, y0, z, qp + A3F_VX / 2, bar);
    } else if (warp == 6) {
        if (main && tma::elect_one()) tma4(st + S::VY, a.p_ybox, 2 * xc, y0 - G::YO1, z, qp + A3F_VY / 2, bar);
    } else if (warp == 7) {
        if (main && tma::elect_one()) tma4(st + S::BB, a.m_ybr, x1, y0 - G::YO1, z, 1, bar);
    } else if (warp == 8) {
        if (main && px2 && tma::elect_one()) tma4(st + S::LX, a.f_xwide, x2, y0, z, qf + A3F_LPVX, bar);
    } else if (warp == 9) {
        if (main && py2 && tma::elect_one()) tma4(st + S::LY, a.f_ywide, xc, y0 - G::YO2, z, qf + A3F_LPVY, bar);
    } else if (warp == 10) {
        if (main && (px || py) && tma::elect_one()) {
            if (px) tma4(st + S::QX, a.f_xbox, x1, y0, z, qf + A3F_LPPX, bar);
            if (py) tma4(st + S::QY, a.f_ybox, xc, y0 - G::YO1, z, qf + A3F_LPPY, bar);
        }
    } else if (tma::elect_one()) {
        unsigned bytes = C8 + C8 + C4 + (rs ? C4 : 0) + (ks ? C4 : 0) + (im ? C8 : 0);
        if (main) {
            bytes += C4 + G::XW2 * G::YH2 * 8 + G::XW1 * TY * 8 + TX * G::YH1 * 8 + G::XW1 * G::YHB * 4;
            if (px2) bytes += G::XW2 * TY * 4;
            if (py2) bytes += TX * G::YH2 * 4;
            if (px) bytes += G::XW1 * TY * 4;
            if (py) bytes += TX * G::YH1 * 4;
        }
        mbar_expect(bar, bytes);
    }
    __syncwarp();
}

template <int M>
__global__ void __launch_bounds__(NTH, kMinBlocks) k3f_adj(const __grid_constant__ Adj3F a)
{
    if (guard_tripped(a.g)) return;
    using G = Geo<M>;
    using S = AdjSmem<M>;
    constexpr int W = G::W;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *sm = smem_raw + ((128u - (su32(smem_raw) & 127u)) & 127u);
    uint64_t *bar = reinterpret_cast<uint64_t *>(sm + S::BAR);
    float4 *oX = reinterpret_cast<float4 *>(sm + S::OX);
    float4 *oY = reinterpret_cast<float4 *>(sm + S::OY);

    const GridDev &g = a.g;
    const int t = threadIdx.x, tx = t % TX, ty = t / TX;
    const int warp = __shfl_sync(0xffffffffu, t >> 5, 0);   // (known to be uniform)
    const int nzc = (g.Nz + a.tzc - 1) / a.tzc;
    const int slot = blockIdx.z / nzc, zcn = blockIdx.z - slot * nzc;
    const int shot = a.shot0 + slot;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
    const int x = x0 + tx, y = y0 + ty;
    const bool colok = x < g.Nx && y < g.Ny;
    const int zc0 = zcn * a.tzc, zc1 = min(zc0 + a.tzc, g.Nz);
    const int zstart = zc0 - W;
    const float dt = g.dt;
    const int n = a.n;
    const bool recon = n > 0;
    const int pl = (int)g.plane, rowz = (int)g.rowz, pitch = g.pitch;
    const int cxy = y * pitch + x;
    const int ixg = x - g.x0, iyg = y - g.y0;
    const bool xin = ixg >= 0 && ixg < g.nx, yin = iyg >= 0 && iyg < g.ny;
    // CTA-uniform strip flags: half-node halos (px, py), node halos (px2, py2)
    const bool px = (x0 - M <= g.x0 - 2) || (x0 + TX + M - 2 >= g.x0 + g.nx);
    const bool py = (y0 - M <= g.y0 - 2) || (y0 + TY + M - 2 >= g.y0 + g.ny);
    const bool px2 = (x0 - 2 * M + 1 <= g.x0 - 1) || (x0 + TX + 2 * M - 2 >= g.x0 + g.nx);
    const bool py2 = (y0 - 2 * M + 1 <= g.y0 - 1) || (y0 + TY + 2 * M - 2 >= g.y0 + g.ny);
    const bool xyf = !px2 && !py2;   // every node and half node the tile reads is interior
    const float *in = a.in + (long long)slot * a.in_planes * g.plane;
    float *outf = a.out + (long long)slot * a.out_planes * g.plane;
    float2 *out2 = reinterpret_cast<float2 *>(outf);
    float2 *img = a.img + (long long)slot * g.plane;
    const long long rowprev = band_row(a.bands, shot, n - 1);
    const int src = a.src_cell[shot];
    const float wsrc = recon ? a.src_scale * a.wav[(a.wav_per_shot ? (long long)shot * g.nt : 0) + n - 1] : 0.f;

    float *tab = reinterpret_cast<float *>(sm + S::TAB);
    if (t == 0) {
        for (int i = 0; i < PD; ++i) mbar_init(bar + i);
        tma::mbar_init_fence();
        for (int f = 0; f < 2; ++f) tab[S::SC + f] = recon && a.bands.fmt != BAND_F32 ? a.bands.scale[rowprev * 2 + f] : 1.f;
    }
    for (int i = t; i < S::SC; i += NTH) {
        const float *pr;
        int c0, N;
        if (i < S::HY) pr = i < G::XH1 ? a.pml.ah[2] : a.pml.bh[2], c0 = x0 - M + i % G::XH1, N = g.Nx;
        else if (i < S::WX) pr = i - S::HY < G::YH1 ? a.pml.ah[1] : a.pml.bh[1], c0 = y0 - M + (i - S::HY) % G::YH1, N = g.Ny;
        else if (i < S::WY) pr = a.pml.ai[2], c0 = x0 - G::XO2 + i - S::WX, N = g.Nx;
        else if (i < S::NX) pr = a.pml.ai[1], c0 = y0 - G::YO2 + i - S::WY, N = g.Ny;
        else if (i < S::NY) pr = a.pml.bi[2], c0 = x0 + i - S::NX, N = g.Nx;
        else pr = a.pml.bi[1], c0 = y0 + i - S::NY, N = g.Ny;
        tab[i] = c0 >= 0 && c0 < N ? pr[c0] : 0.f;
    }
    __syncthreads();
    for (int j = 0; j < PD - 1; ++j)
        if (zstart + j < zc1)
            adj_issue<M>(a, warp, sm + j * S::STAGE, bar + j, slot, x0, y0, zstart + j, zc0, px, py, px2, py2);

    // this thread's half nodes (k3f_born): its own column's and at most one of
    // the halo's, whose offsets are formed anew in every row (the z rings leave
    // no registers to keep them; a spilled one comes from L2)
    constexpr int NH = 2 * M - 1;
    const int wc = (ty + G::YO2) * G::XW2 + tx + G::XO2, bc = (ty + M) * G::XW1 + tx + G::XO1;
    const bool halo_y = warp < NH;
    const int jy = warp < M ? warp : warp + TY;   // halo_y: its row of half nodes
    const int he = (warp - NH) * 32 + tx;
    const bool halo_x = !halo_y && he < TY * NH;
    const int hy0 = he / NH, hx0 = he - hy0 * NH < M ? he - hy0 * NH : he - hy0 * NH + TX;
    const int hpack = hy0 | hx0 << 8;   // halo_x: its row and half node, in one register
    // Strip band values of an interior row iz: those of this column (its v is
    // the strip's normal one, along x or y) at b_off + iz times the strip's
    // values a row, those of the halo item at h_off (-1: none)
    const int xstr = 2 * M * g.ny, ystr = 2 * M * g.nx;
    auto strip_off = [&](int jx, int jy) -> int {   // interior offsets of a half node or node
        const bool ix_in = jx >= 0 && jx < g.nx, iy_in = jy >= 0 && jy < g.ny;
        const int sx = jx < 0 ? jx + M : M + jx - g.nx, sy = jy < 0 ? jy + M : M + jy - g.ny;
        if (iy_in && !ix_in && sx >= 0 && sx < 2 * M) return jy * 2 * M + sx;
        if (ix_in && !iy_in && sy >= 0 && sy < 2 * M) return 2 * M * g.nz * g.ny + sy * g.nx + jx;
        return -1;
    };
    const int b_off = recon && colok && !xyf ? strip_off(ixg, iyg) : -1;
    const int h_off = !recon ? -1 : (halo_y ? strip_off(ixg, y0 - M + jy - g.y0)
                                            : (halo_x ? strip_off(x0 - M + hx0 - g.x0, y0 + hy0 - g.y0) : -1));
    auto band_raw = [&](int field, int o) -> float {
        const long long e = rowprev * a.bands.nb + o;
        const void *b = field ? a.bands.v : a.bands.p;
        if (a.bands.fmt == BAND_F32) return reinterpret_cast<const float *>(b)[e];
        if (a.bands.fmt == BAND_BF16S) return tab[S::SC + field] * __bfloat162float(reinterpret_cast<const __nv_bfloat16 *>(b)[e]);
        return tab[S::SC + field] * __half2float(reinterpret_cast<const __half *>(b)[e]);
    };

    // (p^n, u_z) at node row rr of this column
    // (pq holds the mirror row's values for a ghost row rr < z0; the surface
    // row carries p = 0 and mu = 0)
    auto pu_node = [&](int rr, float2 pq, float lpvz) -> float2 {
        if (g.fs && rr <= g.z0) return rr == g.z0 ? make_float2(0.f, 0.f) : neg2(pq);
        if (zpml_node(g, rr)) pq.y -= a.pml.ai[0][rr] * (lpvz - pq.y);
        return pq;
    };
    // z rings: PU[m] node row z + m; VW, VN half row z + m - M; PIZ half row z + m - 1
    float2 PU[W], VW[W];
    float VN[W], PIZ[M + 1];
#pragma unroll
    for (int m = 0; m < W; ++m) {
        VW[m] = make_float2(0.f, 0.f);
        VN[m] = 0.f;
    }
#pragma unroll
    for (int m = 0; m <= M; ++m) PIZ[m] = 0.f;
    {
        const float2 *pin = reinterpret_cast<const float2 *>(in) + (A3F_PL / 2) * (long long)pl;
#pragma unroll
        for (int m = 0; m < W - 1; ++m) {
            const int rr = zstart + m, rs = node_src_row(g, rr);
            const float2 pq = (colok && rs >= 0 && rs < g.Nz) ? pin[rs * rowz + cxy] : make_float2(0.f, 0.f);
            const float lv = colok && zpml_node(g, rr) ? in[A3F_LPVZ * (long long)pl + rr * rowz + cxy] : 0.f;
            PU[m] = pu_node(rr, pq, lv);
        }
    }
    float bz_old = 0.f;
    {
        const int kk = zstart + M - 1;
        if (colok && kk >= 0 && kk < g.Nz) bz_old = a.binv[kk * rowz + cxy];
    }

    bool failed = false;
    int fail_row = 0;
    for (int z = zstart; z < zc1; ++z) {
        const int j = z - zstart;
        const bool to = !mbar_wait(bar + j % PD, (unsigned)(j / PD) & 1u);
        if (__syncthreads_or(to)) {
            failed = true;
            fail_row = z;
            break;
        }
        if (z + PD - 1 < zc1)
            adj_issue<M>(a, warp, sm + ((j + PD - 1) % PD) * S::STAGE, bar + (j + PD - 1) % PD, slot, x0, y0, z + PD - 1,
                         zc0, px, py, px2, py2);
        unsigned char *st = sm + (j % PD) * S::STAGE;
        auto tile2 = [&](unsigned off) { return reinterpret_cast<const float2 *>(st + off); };
        auto tile1 = [&](unsigned off) { return reinterpret_cast<const float *>(st + off); };
        const int k = z + M - 1, c = z * rowz + cxy, izg = z - g.z0;
        const bool main = z >= zc0;
        const bool zin = izg >= 0 && izg < g.nz;
        const bool inner = xin && yin && zin;
        const bool zf = recon && main && z > g.z0 && z + W < g.z0 + g.nz;
        const bool surf = g.fs && z == g.z0;   // free-surface row: p = 0, mu = 0
        // band values of this thread's half nodes in the strips, loaded ahead
        float bv = 0.f, bvh = 0.f;
        if (main && !xyf && zin) {
            if (b_off >= 0) bv = band_raw(1, izg * (yin ? xstr : ystr) + b_off);
            if (h_off >= 0) {
                const int hy = (halo_y ? y0 - M + jy : y0 + (hpack & 255)) - g.y0;
                bvh = band_raw(1, izg * (hy >= 0 && hy < g.ny ? xstr : ystr) + h_off);
            }
        }
        // ---- strip tiles: u_x and u_y of every node the half nodes' stencils
        // reach, in place of the lambda CPML memories (after the own node's
        // are advanced)
        if (main && (px2 || py2)) {
            const float2 *wP = tile2(S::PW);
            const float mu = surf ? 0.f : wP[wc].y;
            if (px2) {
                float *LX = reinterpret_cast<float *>(st + S::LX);
                auto put = [&](int l, int w, int cc) {
                    const float u = wP[w].y;
                    LX[l] = u - tab[S::WX + cc] * (LX[l] - u);
                };
                const int lxc = ty * G::XW2 + tx + G::XO2;
                if (colok && !(ixg >= 0 && ixg < g.nx)) outf[A3F_LPVX * pl + c] = tab[S::NX + tx] * (LX[lxc] - mu);
                put(lxc, wc, tx + G::XO2);
                constexpr int NX2 = 2 * G::XO2;
                if (t < TY * NX2) {
                    const int iy = t / NX2, q = t - iy * NX2, cc = q < G::XO2 ? q : q + TX;
                    put(iy * G::XW2 + cc, (iy + G::YO2) * G::XW2 + cc, cc);
                }
            }
            if (py2) {
                float *LY = reinterpret_cast<float *>(st + S::LY);
                auto put = [&](int l, int w, int rr) {
                    const float u = wP[w].y;
                    LY[l] = u - tab[S::WY + rr] * (LY[l] - u);
                };
                const int lyc = (ty + G::YO2) * TX + tx;
                if (colok && !(iyg >= 0 && iyg < g.ny)) outf[A3F_LPVY * pl + c] = tab[S::NY + ty] * (LY[lyc] - mu);
                put(lyc, wc, ty + G::YO2);
                for (int q = warp; q < 2 * G::YO2; q += TY) {
                    const int rr = q < G::YO2 ? q : q + TY;
                    put(rr * TX + tx, rr * G::XW2 + tx + G::XO2, rr);
                }
            }
            // the generic-proxy writes to the stage must be ordered before the
            // TMA copy that refills it (issued after the next row's barrier)
            tma::fence_proxy_async();
            __syncthreads();
        }
        // ---- half row k along z: lambda_vz, lambda_psi_pz, background vz^{n-1/2}; half nodes of row z
        // (ZF: rows without tests, XY: tiles without strips, as in k3f_born)
        auto v_stage = [&](auto zc, auto xyc) {
            constexpr bool ZF = decltype(zc)::value, XY = decltype(xyc)::value;
            const float2 pq = tile2(S::PA)[t];
            if (ZF) PU[W - 1] = pq;
            else PU[W - 1] = pu_node(z + W - 1, pq, tile1(S::LA)[t]);
            const float2 v2z = tile2(S::VZ)[t];
            float bk1 = tile1(S::BK)[t];
            if (!ZF && k + 1 >= g.Nz) bk1 = bz_old;   // the last half row replicates the last node row
            float wz = 0.f, vn = 0.f, piz = 0.f;
            if (ZF || (k >= 0 && k < g.Nz)) {
                const bool own = (XY || colok) && (ZF || k >= zc0) && k < zc1;
                const int ck = k * rowz + cxy;
                const float2 D = st2<M>(g.cz, [&](int l) { return PU[M - 1 + l]; }, [&](int l) { return PU[M - l]; });
                const float lv = v2z.y + D.y;
                const float dtbu = dt * 0.5f * (bz_old + bk1);
                wz = dtbu * lv;
                if (!ZF && (k <= g.z0 - 2 || k >= g.z0 + g.nz)) {
                    const float l1 = tile1(S::PZ)[t] - dtbu * lv;
                    wz -= a.pml.ah[0][k] * l1;
                    if (own) outf[A3F_LPPZ * pl + ck] = a.pml.bh[0][k] * l1;
                }
                piz = D.x * lv;
                if (ZF) {
                    vn = XY || (xin && yin) ? v2z.x + dtbu * D.x : 0.f;
                } else if (recon && xin && yin) {
                    const int iz = k - g.z0;
                    if ((iz >= 0 || g.fs) && iz < g.nz) vn = v2z.x + dtbu * D.x;   // ghost half rows: mirrors
                    else {
                        const long long b = fband(g, 0, iz, iyg, ixg);
                        if (b >= 0) vn = band_get(a.bands, 1, rowprev, b);
                    }
                }
                if (own) out2[(A3F_VZ / 2) * pl + ck] = make_float2(vn, lv);
            }
            bz_old = bk1;
            VW[W - 1] = make_float2(v2z.x, wz);
            VN[W - 1] = vn;
            PIZ[M] = piz;
            if (!ZF && !main) return;
            // one half node: (v^{n+1/2}, w, v^{n-1/2}, G lambda_v). strip: its u
            // tile lt (entry l0) in node strip tiles, its table entries a (at q)
            // and b (len further) and memory psi in half-node strip tiles
            auto half = [&](const float *cf, int w, int ws, int b, int bst, float2 v2, float hs, bool last, bool p2,
                            const float *lt, int l0, bool strip, int q, int len, const float *psi, float *psi_out, bool vin,
                            float band, float2 *v_out) -> float4 {
                const float2 *p = tile2(S::PW) + w;
                float2 D;
                if (XY || !p2) {
                    D = st2<M>(cf, [&](int l) { return p[l * ws]; }, [&](int l) { return p[(1 - l) * ws]; });
                } else {
                    const int ls = ws == 1 ? 1 : TX;
                    D.x = st1<M>(cf, [&](int l) { return p[l * ws].x; }, [&](int l) { return p[(1 - l) * ws].x; });
                    D.y = st1<M>(cf, [&](int l) { return lt[l0 + l * ls]; }, [&](int l) { return lt[l0 + (1 - l) * ls]; });
                }
                if (!ZF && surf) D.y = 0.f;
                const float lv = v2.y + D.y;
                const float b0 = tile1(S::BB)[b];
                const float b1 = !XY && last ? b0 : tile1(S::BB)[b + bst];
                const float dtbu = dt * (hs * (b0 + b1));
                float wv = dtbu * lv;
                if (!XY && strip) {
                    const float ah = tab[q], bh = tab[q + len];
                    const float l1 = *psi - dtbu * lv;
                    wv -= ah * l1;
                    if (psi_out && bh != 0.f) *psi_out = bh * l1;
                }
                const float vn1 = (ZF && XY) || vin ? v2.x + dtbu * D.x : band;
                if (v_out) *v_out = make_float2(vn1, lv);
                return make_float4(v2.x, wv, vn1, D.x * lv);
            };
            const bool rz = ZF || (recon && zin);
            {
                const int vi = ty * G::XW1 + tx + G::XO1;
                oX[ty * G::XW1 + tx + M] =
                    half(g.cx, wc, 1, bc, 1, tile2(S::VX)[vi], 0.5f, x + 1 >= g.Nx, px2, tile1(S::LX),
                         ty * G::XW2 + tx + G::XO2, px, S::HX + tx + M, G::XH1, tile1(S::QX) + vi,
                         colok ? outf + A3F_LPPX * pl + c : nullptr, rz && xin && yin, yin ? bv : 0.f,
                         XY || colok ? out2 + (A3F_VX / 2) * pl + c : nullptr);
            }
            {
                const int vi = (ty + M) * TX + tx;
                oY[vi] = half(g.cy, wc, G::XW2, bc, G::XW1, tile2(S::VY)[vi], 0.5f, y + 1 >= g.Ny, py2, tile1(S::LY),
                              (ty + G::YO2) * TX + tx, py, S::HY + ty + M, G::YH1, tile1(S::QY) + vi,
                              colok ? outf + A3F_LPPY * pl + c : nullptr, rz && xin && yin, xin ? bv : 0.f,
                              XY || colok ? out2 + (A3F_VY / 2) * pl + c : nullptr);
            }
            if (halo_y) {
                const int hi = y0 - M + jy, vi = jy * TX + tx;
                const bool vin = rz && xin && hi >= g.y0 && hi < g.y0 + g.ny;
                oY[vi] = half(g.cy, (jy + M - 1) * G::XW2 + tx + G::XO2, G::XW2, jy * G::XW1 + tx + G::XO1, G::XW1,
                              tile2(S::VY)[vi], XY || hi >= 0 ? 0.5f : 0.f, hi + 1 >= g.Ny, py2, tile1(S::LY),
                              (jy + M - 1) * TX + tx, py, S::HY + jy, G::YH1, tile1(S::QY) + vi, nullptr, vin, bvh, nullptr);
            } else if (halo_x) {
                int h = hpack;
                const int hiy = h & 255, hjx = h >> 8, hi = x0 - M + hjx, hj = y0 + hiy, vi = hiy * G::XW1 + hjx - M + G::XO1;
                const bool vin = rz && hj >= g.y0 && hj < g.y0 + g.ny && hi >= g.x0 && hi < g.x0 + g.nx;
                oX[hiy * G::XW1 + hjx] =
                    half(g.cx, (hiy + G::YO2) * G::XW2 + hjx - M + G::XO2, 1, (hiy + M) * G::XW1 + hjx - M + G::XO1, 1,
                         tile2(S::VX)[vi], XY || hi >= 0 ? 0.5f : 0.f, hi + 1 >= g.Nx, px2, tile1(S::LX),
                         hiy * G::XW2 + hjx - M + G::XO2, px, S::HX + hjx, G::XH1, tile1(S::QX) + vi, nullptr, vin, bvh, nullptr);
            }
        };
        const std::true_type Y{};
        const std::false_type N{};
        if (xyf) {
            if (zf) v_stage(Y, Y);
            else v_stage(N, Y);
        } else {
            if (zf) v_stage(Y, N);
            else v_stage(N, N);
        }
        // the node's band value, or z strip memory
        float bp = 0.f;
        if (main && !(xyf && zf)) {
            if (zin) {
                if (b_off >= 0) bp = band_raw(0, izg * (yin ? xstr : ystr) + b_off);
            } else if (recon && colok) {
                const long long b = fband(g, 0, izg, iyg, ixg);
                if (b >= 0) bp = band_raw(0, (int)b);
            }
            if (!zf && colok && zpml_node(g, z))
                outf[A3F_LPVZ * pl + c] = a.pml.bi[0][z] * (in[A3F_LPVZ * pl + c] - (surf ? 0.f : tile2(S::PW)[wc].y));
        }
        if (main) {
            __syncthreads();
            // ---- node of the thread's own column at row z
            auto node_stage = [&](auto zc, auto xyc) {
                constexpr bool ZF = decltype(zc)::value, XY = decltype(xyc)::value;
                // (Q_n, D- w) and D- v^{n-1/2} along an axis, and the two adjacent G lambda_v products
                auto axis = [&](const float *cf, const float4 *o, int st_, float2 &E, float &q, float &pi) {
                    float2 d2[M];
                    float dn[M];
#pragma unroll
                    for (int l = 0; l < M; ++l) {
                        const float4 u = o[l * st_], v = o[-(l + 1) * st_];
                        d2[l] = sub2(make_float2(u.x, u.y), make_float2(v.x, v.y));
                        dn[l] = u.z - v.z;
                        if (l == 0) pi = u.w + v.w;
                    }
                    E = mul2(cf[0], d2[0]);
                    q = cf[0] * dn[0];
#pragma unroll
                    for (int l = 1; l < M; ++l) {
                        E = fma2(cf[l], d2[l], E);
                        q = fmaf(cf[l], dn[l], q);
                    }
                };
                float2 Ex, Ey;
                float qx, qy, pix, piy;
                axis(g.cx, oX + ty * G::XW1 + tx + M, 1, Ex, qx, pix);
                axis(g.cy, oY + (ty + M) * TX + tx, TX, Ey, qy, piy);
                const float2 Ez = st2<M>(g.cz, [&](int l) { return VW[M + l - 1]; }, [&](int l) { return VW[M - l]; });
                const float2 E = add2(add2(Ex, Ey), Ez);   // (Q_n = D- . v^{n+1/2}, D- . w)
                // D- . v^{n-1/2}, summed z, y, x as the background pass sums
                // it, so the rebuilt p^{n-1} undoes that pass's rounding
                const float qn = (st1<M>(g.cz, [&](int l) { return VN[M + l - 1]; }, [&](int l) { return VN[M - l]; }) + qy) + qx;
                float2 pm = tile2(S::PW)[wc];
                if (!ZF && surf) pm.y = 0.f;
                const float kd = tile1(S::KD)[t];
                const bool in_ = (ZF && XY) || inner;
                if (in_) {
                    float2 acc = tile2(S::IM)[t];
                    acc.x += E.x * pm.y;
                    // (on the free surface the half row above is a ghost: no product of its own)
                    acc.y += pix + piy + (PIZ[1] + (!ZF && surf ? 0.f : PIZ[0]));
                    img[c] = acc;
                }
                float pn = in_ && (ZF || recon) ? pm.x + kd * qn : bp;
                pn -= c == src ? wsrc : 0.f;   // (a source node is an interior one; wsrc = 0 at the last reverse step)
                float2 pmn = make_float2(pn, fmaf(kd, E.y, pm.y));
                if (!ZF && g.fs && z <= g.z0) pmn = make_float2(0.f, 0.f);
                if (XY || colok) out2[(A3F_PL / 2) * pl + c] = pmn;
            };
            if (xyf) {
                if (zf) node_stage(Y, Y);
                else node_stage(N, Y);
            } else {
                if (zf) node_stage(Y, N);
                else node_stage(N, N);
            }
        }
#pragma unroll
        for (int m = 0; m < W - 1; ++m) {
            PU[m] = PU[m + 1];
            VW[m] = VW[m + 1];
            VN[m] = VN[m + 1];
        }
#pragma unroll
        for (int m = 0; m < M; ++m) PIZ[m] = PIZ[m + 1];
    }

    if (failed) {
        if (t == 0) {
            atomicOr(a.err, 1);
            const int jf = fail_row - zstart;
            for (int jj = jf; jj < jf + PD - 1 && zstart + jj < zc1; ++jj)
                (void)mbar_wait(bar + jj % PD, (unsigned)(jj / PD) & 1u);
        }
        return;
    }
    if (recon) {
        // pre-add the residual of step n-1 at the receivers of this tile
        __syncthreads();
        const int ntile = (int)(gridDim.x * gridDim.y) * nzc;
        const int rt = shot * ntile + (zcn * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
        const int b = a.trec.ptr[rt], e = a.trec.ptr[rt + 1];
        for (int i = b + t; i < e; i += NTH) {
            const int2 rc = a.trec.rec[i];
            if (i > b && a.trec.rec[i - 1].x == rc.x) continue;   // run handled by its first entry
            float add = 0.f;
            for (int q = i; q < e && a.trec.rec[q].x == rc.x; ++q)
                add += a.dstage[(long long)a.trec.rec[q].y * g.nt + (n - 1)];
            out2[(A3F_PL / 2) * pl + rc.x].y += a.kdt[rc.x] * add;
        }
    }
}

// ---------------------------------------------------------------------------
// Tensor maps
// ---------------------------------------------------------------------------
PFN_cuTensorMapEncodeTiled_v12000 encode_fn()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
        else
            cudaGetLastError();
    });
    return fn;
}

}  // namespace

cudaError_t encode_tmap(CUtensorMap *m, CUtensorMapDataType type, int rank, const void *base, const cuuint64_t *dims,
                        const cuuint64_t *strides, const cuuint32_t *box)
{
    PFN_cuTensorMapEncodeTiled_v12000 fn = encode_fn();
    if (!fn) return cudaErrorNotSupported;
    cuuint32_t es[5] = {1, 1, 1, 1, 1};
    CUresult r = fn(m, type, (cuuint32_t)rank, const_cast<void *>(base), dims, strides, box, es,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// Tensor map over `nq` planes of `esz`-byte elements (4: float, 8: float2
// pair) starting at base: dims (x in floats, y, z, plane), box (bx elements,
// by rows, 1, 1); outside the padded grid the copy reads zeros.
cudaError_t make_tmap3(CUtensorMap *m, const void *base, const GridDev &g, int esz, long long nq, int bx, int by)
{
    PFN_cuTensorMapEncodeTiled_v12000 fn = encode_fn();
    if (!fn) return cudaErrorNotSupported;
    const int f = esz / 4;   // floats per element
    cuuint64_t dims[4] = {(cuuint64_t)g.Nx * f, (cuuint64_t)g.Ny, (cuuint64_t)g.Nz, (cuuint64_t)nq};
    cuuint64_t strides[3] = {(cuuint64_t)g.pitch * esz, (cuuint64_t)g.rowz * esz, (cuuint64_t)g.plane * esz};
    cuuint32_t box[4] = {(cuuint32_t)(bx * f), (cuuint32_t)by, 1, 1};
    cuuint32_t es[4] = {1, 1, 1, 1};
    if (((uintptr_t)base & 15) || box[0] > 256 || by > 256 || (box[0] * 4) % 16) return cudaErrorInvalidValue;
    CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, const_cast<void *>(base), dims, strides, box, es,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// Fills the tensor maps of a fused Born step reading `in` (pairs per slot
// in_pairs) with model pairs kd2 / br2.
cudaError_t fused3d_born_maps(Step3F &a, const float2 *kd2, const float2 *br2, int batch)
{
    const GridDev &g = a.g;
    cudaError_t e;
    const long long nq = (long long)batch * a.in_pairs;
    if (a.g.M == 2) {
        using G = Geo<2>;
        if ((e = make_tmap3(&a.in_wide, a.in, g, 8, nq, G::XW2, G::YH2)) != cudaSuccess) return e;
        if ((e = make_tmap3(&a.in_xbox, a.in, g, 8, nq, G::XW1, TY)) != cudaSuccess) return e;
        if ((e = make_tmap3(&a.in_ybox, a.in, g, 8, nq, TX, G::YH1)) != cudaSuccess) return e;
    } else {
        using G = Geo<4>;
        if ((e = make_tmap3(&a.in_wide, a.in, g, 8, nq, G::XW2, G::YH2)) != cudaSuccess) return e;
        if ((e = make_tmap3(&a.in_xbox, a.in, g, 8, nq, G::XW1, TY)) != cudaSuccess) return e;
        if ((e = make_tmap3(&a.in_ybox, a.in, g, 8, nq, TX, G::YH1)) != cudaSuccess) return e;
    }
    if ((e = make_tmap3(&a.in_core, a.in, g, 8, nq, TX, TY)) != cudaSuccess) return e;
    // model: plane 0 = kd2, plane 1 = br2 (one map over the two planes needs
    // them to be one plane apart)
    if (reinterpret_cast<const char *>(br2) - reinterpret_cast<const char *>(kd2) != (ptrdiff_t)(g.plane * 8))
        return cudaErrorInvalidValue;
    if ((e = make_tmap3(&a.m_core, kd2, g, 8, 2, TX, TY)) != cudaSuccess) return e;
    const int ybr = a.g.M == 2 ? Geo<2>::YHB : Geo<4>::YHB;
    return make_tmap3(&a.m_ybr, kd2, g, 8, 2, Geo<4>::XW1, ybr);
}

namespace {

// Start state of a fused reverse pass: pairs (p, 0), (vx, 0), (vy, 0), (vz, 0)
// from the saved background final state, whose planes are ordered
// [p][vz][vy][vx] (direction 0 = z in the background kernels).
__global__ void k3f_pack(const GridDev g, const float *final_state, int fs0, int batch, float *st,
                         long long sstride)
{
    const long long plane = g.plane;
    const long long n = batch * plane;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const long long s = i / plane, c = i - s * plane;
        const float *fs = final_state + (fs0 + s) * 4 * plane;
        float2 *o = reinterpret_cast<float2 *>(st + s * sstride);
        o[(A3F_PL / 2) * plane + c] = make_float2(fs[c], 0.f);
        o[(A3F_VZ / 2) * plane + c] = make_float2(fs[1 * plane + c], 0.f);
        o[(A3F_VY / 2) * plane + c] = make_float2(fs[2 * plane + c], 0.f);
        o[(A3F_VX / 2) * plane + c] = make_float2(fs[3 * plane + c], 0.f);
    }
}

}  // namespace

cudaError_t launch_pack3f(const GridDev &g, const float *final_state, int fs0, int batch, float *st,
                          long long sstride, cudaStream_t s)
{
    const long long n = batch * g.plane;
    const int blocks = (int)std::min<long long>((n + 255) / 256, 152 * 16);
    k3f_pack<<<blocks, 256, 0, s>>>(g, final_state, fs0, batch, st, sstride);
    return cudaGetLastError();
}

cudaError_t fused3d_adj_maps(Adj3F &a, const float *kdt, const float *binv, int batch)
{
    const GridDev &g = a.g;
    cudaError_t e;
    const long long nqp = (long long)batch * (a.in_planes / 2), nqf = (long long)batch * a.in_planes;
    const bool m2 = g.M == 2;
    const int XW2 = m2 ? Geo<2>::XW2 : Geo<4>::XW2, YH2 = m2 ? Geo<2>::YH2 : Geo<4>::YH2;
    const int XW1 = Geo<4>::XW1, YH1 = m2 ? Geo<2>::YH1 : Geo<4>::YH1, YHB = m2 ? Geo<2>::YHB : Geo<4>::YHB;
    if ((e = make_tmap3(&a.p_core, a.in, g, 8, nqp, TX, TY)) != cudaSuccess) return e;
    if ((e = make_tmap3(&a.p_wide, a.in, g, 8, nqp, XW2, YH2)) != cudaSuccess) return e;
    if ((e = make_tmap3(&a.p_xbox, a.in, g, 8, nqp, XW1, TY)) != cudaSuccess) return e;
    if ((e = make_tmap3(&a.p_ybox, a.in, g, 8, nqp, TX, YH1)) != cudaSuccess) return e;
    if ((e = make_tmap3(&a.f_core, a.in, g, 4, nqf, TX, TY)) != cudaSuccess) return e;
    if ((e = make_tmap3(&a.f_xwide, a.in, g, 4, nqf, XW2, TY)) != cudaSuccess) return e;
    if ((e = make_tmap3(&a.f_ywide, a.in, g, 4, nqf, TX, YH2)) != cudaSuccess) return e;
    if ((e = make_tmap3(&a.f_xbox, a.in, g, 4, nqf, XW1, TY)) != cudaSuccess) return e;
    if ((e = make_tmap3(&a.f_ybox, a.in, g, 4, nqf, TX, YH1)) != cudaSuccess) return e;
    // model: plane 0 dt kappa, plane 1 1/rho (adjacent)
    if (binv - kdt != (ptrdiff_t)g.plane) return cudaErrorInvalidValue;
    if ((e = make_tmap3(&a.m_core, kdt, g, 4, 2, TX, TY)) != cudaSuccess) return e;
    if ((e = make_tmap3(&a.im, a.img, g, 8, batch, TX, TY)) != cudaSuccess) return e;
    return make_tmap3(&a.m_ybr, kdt, g, 4, 2, XW1, YHB);
}

// A chunk of t rows marches t + 2M. A CTA that shares its SM with another one
// takes 1.25x its time alone; past two a SM the warm-up rows hide behind other
// CTAs and what counts is the work repeated and the last wave (0.6 of one on
// average): the model's relative costs a row, 1, 1.25 and 1.06 a wave, follow
// from a Born and migration step of 168 x 296 x 296 cells: 1 shot 1300 us in
// one chunk, 1253 in 84 rows, 1053 in 24, 1066 in 16; 2 shots 2449, 2090,
// 2002, 2076, and 1969 in 34; 16 shots 14415, 14250 (84), 15271, 16235; 100 x
// 120 x 130 cells, 1 shot: 658 in one chunk, 252 in 25 rows, 182 in 17.
int march3d_rows(int M, int Nz, long long ctas)
{
    constexpr double sms = 152.0;
    double best = 1e300;
    int rows = Nz;
    for (int nc = 1; nc <= Nz; ++nc) {
        const int t = (Nz + nc - 1) / nc;
        const double n = (double)ctas * ((Nz + t - 1) / t), q = std::ceil(n / sms);
        const double c = q <= 2.0 ? (t + 2 * M) * (q <= 1.0 ? 1.0 : 1.25) : (t + 0.5 * M) * 1.06 * (n / (2.0 * sms) + 0.6);
        if (c < best) {
            best = c;
            rows = t;
        }
    }
    return rows;
}

cudaError_t configure_3d_kernels()
{
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(k3f_born<2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)BornSmem<2>::TOTAL)) != cudaSuccess)
        return e;
    if ((e = cudaFuncSetAttribute(k3f_born<4>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)BornSmem<4>::TOTAL)) != cudaSuccess)
        return e;
    if ((e = cudaFuncSetAttribute(k3f_adj<2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)AdjSmem<2>::TOTAL)) != cudaSuccess)
        return e;
    return cudaFuncSetAttribute(k3f_adj<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)AdjSmem<4>::TOTAL);
}

cudaError_t launch_adj3f(const Adj3F &a, int batch, cudaStream_t s)
{
    const GridDev &g = a.g;
    const int nzc = (g.Nz + a.tzc - 1) / a.tzc;
    dim3 grid((g.Nx + TX - 1) / TX, (g.Ny + TY - 1) / TY, nzc * batch);
    if (g.M == 2) k3f_adj<2><<<grid, NTH, AdjSmem<2>::TOTAL, s>>>(a);
    else k3f_adj<4><<<grid, NTH, AdjSmem<4>::TOTAL, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_born3f(const Step3F &a, int batch, cudaStream_t s)
{
    const GridDev &g = a.g;
    const int nzc = (g.Nz + a.tzc - 1) / a.tzc;
    dim3 grid((g.Nx + TX - 1) / TX, (g.Ny + TY - 1) / TY, nzc * batch);
    if (g.M == 2) k3f_born<2><<<grid, NTH, BornSmem<2>::TOTAL, s>>>(a);
    else k3f_born<4><<<grid, NTH, BornSmem<4>::TOTAL, s>>>(a);
    return cudaGetLastError();
}

}  // namespace lsrtm
