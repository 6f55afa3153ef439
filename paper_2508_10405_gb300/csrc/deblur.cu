// Nonstationary deblurring filters (App. E) on the GPU.
//
// App. E relates the reference image m' and the remigrated image m'' = H m'
// by a convolution with the inverse of a locally translation-invariant
// Hessian, f * m'' ~= m'. Per comb node k (spacing s, nodes at s/2 + i s) a
// flen x flen FIR filter solves, over the window of pixels within s of the
// node (clipped to the image),
//     min_f  sum_p ((f * m'')(p) - m'(p))^2 + eps_k ||f||^2,
//     (f * g)(p) = sum_{|a|,|b|<=h} f[a,b] g(p - (a,b)), g = 0 outside,
//     eps_k = eps * trace(A^T A) / flen^2,
// through its FP64 normal equations (A^T A + eps_k I) f = A^T m'. The image
// delta m = sum_k w_k (f_k * m_rtm) / sum_k w_k blends the filtered blocks with
// bilinear valence weights w_k(p) = max(0, 1 - |z - z_k|/s) max(0, 1 - |x - x_k|/s).
//
// k_deblur_solve: one CTA per (node, parameter plane). The window's patch of
// m'' (window + h on each side, zero outside the image) sits in shared memory
// as double: a conversion costs the FP64 pipe as much as the multiply-add it
// feeds. Entry (u, v) of A^T A is the sum of P(q) P(q + d) over the window
// shifted to tap u's origin, d = origin(v) - origin(u): the products depend on
// the lag d only, so per lag and patch row a thread forms the running sums of
// the row's lagged products over the window width at every origin column (one
// pass along the row), and per lag and origin column a thread slides those
// along z over the window height at every origin row: 15x fewer FP64
// operations than summing each entry over the window (products of two floats
// are exact in FP64; sums in FP64). The (dz, row) pairs of one dx are dealt
// over all threads together: one lag's 41 to 51 rows fill two warps to 72%,
// and an FP64 instruction takes its 64 cycles of a scheduler whatever lanes it
// has. The matrix is kept as its packed lower triangle with the right-hand side
// as one more row (60 KB for flen = 11, two CTAs per SM: the serial parts of
// one run under the other's sums), factorised in panels of eight columns: the
// diagonal block in the registers of one warp, a panel row per thread, and one
// pass over the rest for all eight columns.
// Bound by the FP64 pipe (2 multiply-adds a clock and SM: about 1.1M of them a
// window; 5.3 ms for the two planes' 3000 windows of 300 x 2000, s = 20, flen =
// 11): 6.8 ms there, 26.7 with P in float, a lag a warp, the whole matrix and a
// column at a time; the rest are the Cholesky's and the sums' serial chains.
// Small windows are bound by those chains: they take CTAs of 64 threads, twelve
// an SM (launch_deblur).
// k_deblur_apply: one thread per pixel and plane; FP32 taps, at most four
// covering nodes.
// The paper's own Fourier form of the filter (per-block Wiener ratio) follows
// below the space-domain kernels.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "lsrtm_internal.cuh"
#include "wiener.cuh"

namespace lsrtm {

namespace {

constexpr int kSolveThreads = 256, kSolveFew = 64, kSolveFewCtas = 12, kSolvePanel = 8;

__device__ __forceinline__ int tri(int i) { return i * (i + 1) / 2; }

// Row of entry e of a packed lower triangle.
__device__ __forceinline__ int tri_row(int e)
{
    int i = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);
    if (tri(i) > e) --i;
    if (tri(i + 1) <= e) ++i;
    return i;
}

// ulen: doubles of the region U, at least one lag's row sums, PZ * flen. NT:
// threads, at least one a tap; few for small windows, whose sums are too short
// for more and whose serial parts then run under eleven other CTAs' (three or
// two of kSolveThreads).
template <int NT>
__global__ void __launch_bounds__(NT, NT == kSolveThreads ? 3 : kSolveFewCtas)
    k_deblur_solve(const float *mref, const float *mrem, int nz, int nx, int s, int flen, double eps, float *filt,
                   int *flag, int ulen)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int n = flen * flen, h = flen / 2, w2 = 2 * h;
    const int nkz = gridDim.y, nkx = gridDim.x;
    const int param = blockIdx.z;
    const int zk = s / 2 + (int)blockIdx.y * s, xk = s / 2 + (int)blockIdx.x * s;
    const int z0 = max(0, zk - s), z1 = min(nz, zk + s + 1);
    const int x0 = max(0, xk - s), x1 = min(nx, xk + s + 1);
    const int WZ = z1 - z0, WX = x1 - x0;
    const int PZ = WZ + w2, PX = WX + w2, PS = PX | 1;   // odd row stride: lanes on consecutive rows hit all banks
    double *G = reinterpret_cast<double *>(smem);   // rows 0..n packed; row n: the right-hand side
    double *red = G + tri(n + 1);                   // [2]: trace, pivot status
    double *U = red + 2;                            // row sums; then rows of m'; then the panel [8][n + 1]
    double *P = U + ulen;                           // [PZ][PS]
    const long long plane = (long long)nz * nx;
    const float *m2 = mrem + param * plane;
    const float *m1 = mref + param * plane;
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;

    for (int i = t; i < PZ * PX; i += NT) {
        const int pz = i / PX, px = i - pz * PX;
        const int z = z0 - h + pz, x = x0 - h + px;
        P[pz * PS + px] = (z >= 0 && z < nz && x >= 0 && x < nx) ? (double)m2[(long long)z * nx + x] : 0.0;
    }
    if (t == 0) red[1] = 0.0;
    __syncthreads();

    // A[p, u] = m''(p - (a, b)) = P[pz + oz_u][px + ox_u], u = (a + h) flen + (b + h),
    // origin (oz_u, ox_u) = (2h - u / flen, 2h - u % flen) in [0, 2h]^2. Lags dz > 0, or dz = 0 and dx >= 0.
    for (int dx = -w2; dx <= w2; ++dx) {
        const int ox0 = max(0, -dx), ox1 = min(w2, w2 - dx), nox = ox1 - ox0 + 1, nos = nox | 1;
        const int chunk = ulen / (PZ * nos);
        for (int d0 = dx < 0 ? 1 : 0; d0 <= w2; d0 += chunk) {
            const int cnt = min(chunk, w2 + 1 - d0);
            // rs[(dz, r)][ox] = sum_{c = ox}^{ox + WX - 1} P[r][c] P[r + dz][c + dx], the PZ - dz rows of each dz in turn
            const int items = cnt * (PZ - d0) - cnt * (cnt - 1) / 2;
            for (int e = t; e < items; e += NT) {
                int r = e, dz = d0;
                while (r >= PZ - dz) {
                    r -= PZ - dz;
                    ++dz;
                }
                const double *a = P + r * PS, *b = P + (r + dz) * PS + dx;
                double *rs = U + e * nos - ox0;
                double acc = 0.0;
#pragma unroll 4
                for (int c = ox0; c < ox0 + WX; ++c) acc = fma(a[c], b[c], acc);
                rs[ox0] = acc;
                for (int ox = ox0 + 1; ox <= ox1; ++ox) {
                    acc = fma(a[ox + WX - 1], b[ox + WX - 1], acc);
                    acc = fma(-a[ox - 1], b[ox - 1], acc);
                    rs[ox] = acc;
                }
            }
            __syncthreads();
            // S(oz, ox) = sum_{r = oz}^{oz + WZ - 1} rs[r][ox] -> G[u][v]; d >= 0 in the order of taps: v <= u
            for (int e = t; e < cnt * nox; e += NT) {
                const int j = e / nox, ox = ox0 + e - j * nox, dz = d0 + j;
                const double *rs = U + (j * (PZ - d0) - j * (j - 1) / 2) * nos + (ox - ox0);
                double acc = 0.0;
#pragma unroll 4
                for (int r = 0; r < WZ; ++r) acc += rs[r * nos];
                for (int oz = 0; oz <= w2 - dz; ++oz) {
                    if (oz > 0) acc += rs[(oz + WZ - 1) * nos] - rs[(oz - 1) * nos];
                    const int u = (w2 - oz) * flen + (w2 - ox);
                    G[tri(u) + u - dz * flen - dx] = acc;
                }
            }
            __syncthreads();
        }
    }
    // right-hand side: a thread per tap, m' in pieces
    {
        const int u = min(t, n - 1), ou = (w2 - u / flen) * PS + w2 - u % flen;
        double acc = 0.0;
        for (int q0 = 0; q0 < WZ * WX; q0 += ulen) {
            const int q1 = min(WZ * WX, q0 + ulen);
            for (int q = q0 + t; q < q1; q += NT) {
                const int pz = q / WX;
                U[q - q0] = (double)m1[(long long)(z0 + pz) * nx + x0 + q - pz * WX];
            }
            __syncthreads();
            if (warp * 32 < n) {
                int pz = q0 / WX, px = q0 - pz * WX;
                for (int q = q0; q < q1;) {
                    const int len = min(WX - px, q1 - q);
                    const double *ru = P + pz * PS + ou + px, *r1 = U + (q - q0);
#pragma unroll 4
                    for (int i = 0; i < len; ++i) acc = fma(ru[i], r1[i], acc);
                    q += len;
                    px = 0;
                    ++pz;
                }
            }
            __syncthreads();
        }
        if (t < n) G[tri(n) + t] = acc;
    }
    if (warp == 0) {
        double tr = 0.0;
        for (int u = lane; u < n; u += 32) tr += G[tri(u) + u];
        for (int o = 16; o; o >>= 1) tr += __shfl_xor_sync(~0u, tr, o);
        if (lane == 0) red[0] = tr;
    }
    __syncthreads();
    const double tr = red[0];
    float *out = filt + (((long long)param * nkz + blockIdx.y) * nkx + blockIdx.x) * n;
    if (tr == 0.0) {   // all-zero remigrated window: zero filter
        for (int u = t; u < n; u += NT) out[u] = 0.f;
        return;
    }
    for (int u = t; u < n; u += NT) G[tri(u) + u] += eps * tr / n;   // (the division by warps with taps only)
    __syncthreads();

    // Cholesky G = L L^T with 1 / L_kk on the diagonal; row n becomes y of L y = rhs
    double *panel = U;   // [8][m + 1]: the panel's rows below its diagonal block
    for (int k0 = 0; k0 < n; k0 += kSolvePanel) {
        const int nb = min(kSolvePanel, n - k0), k1 = k0 + nb, m = n - k1;
        if (warp == 0) {
            double g[kSolvePanel];
            double *row = G + tri(k0 + lane) + k0;
#pragma unroll
            for (int c = 0; c < kSolvePanel; ++c) g[c] = (lane < nb && c <= lane) ? row[c] : 0.0;
            bool bad = false;
#pragma unroll
            for (int c = 0; c < kSolvePanel; ++c) {
                if (c >= nb) break;
                double d = __shfl_sync(~0u, g[c], c);
                if (!(d > 0.0)) {
                    bad = true;
                    d = 1.0;
                }
                const double r = rsqrt(d);
                g[c] = lane == c ? r : g[c] * r;
#pragma unroll
                for (int j = c + 1; j < kSolvePanel; ++j)
                    g[j] = fma(-g[c], __shfl_sync(~0u, g[c], j), g[j]);
            }
#pragma unroll
            for (int c = 0; c < kSolvePanel; ++c)
                if (lane < nb && c <= lane) row[c] = g[c];
            if (bad && lane == 0) red[1] = 1.0;
        }
        __syncthreads();
        for (int i = t; i <= m; i += NT) {
            double *row = G + tri(k1 + i) + k0;
            double x[kSolvePanel];
#pragma unroll
            for (int c = 0; c < kSolvePanel; ++c) x[c] = c < nb ? row[c] : 0.0;
#pragma unroll
            for (int c = 0; c < kSolvePanel; ++c) {
                if (c >= nb) break;
                x[c] *= G[tri(k0 + c) + k0 + c];
                row[c] = x[c];
                panel[c * (m + 1) + i] = x[c];
#pragma unroll
                for (int j = c + 1; j < kSolvePanel; ++j)
                    if (j < nb) x[j] = fma(-x[c], G[tri(k0 + j) + k0 + c], x[j]);
            }
        }
        __syncthreads();
        // the rest, rows k1..n of columns k1..n-1; m > 0 only below a full panel
        const int rest = tri(m + 1) - 1;
        for (int e = t; e < rest; e += 2 * NT) {
            const bool two = e + NT < rest;   // two entries a thread, for two chains
            const int e1 = two ? e + NT : e;
            const int ia = tri_row(e), ja = e - tri(ia), ib = tri_row(e1), jb = e1 - tri(ib);
            double *ga = G + tri(k1 + ia) + k1 + ja, *gb = G + tri(k1 + ib) + k1 + jb;
            double va = *ga, vb = *gb;
#pragma unroll
            for (int c = 0; c < kSolvePanel; ++c) {
                const double *l = panel + c * (m + 1);
                va = fma(-l[ia], l[ja], va);
                vb = fma(-l[ib], l[jb], vb);
            }
            *ga = va;
            if (two) *gb = vb;
        }
        __syncthreads();
    }
    if (warp > 0) return;
    // L^T f = y: a warp, f[lane + 32 q] in its registers
    double f[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) f[q] = 32 * q + lane < n ? G[tri(n) + 32 * q + lane] : 0.0;
#pragma unroll
    for (int q = 3; q >= 0; --q) {
        for (int k = min(n, 32 * q + 32) - 1; k >= 32 * q; --k) {
            const double *row = G + tri(k);
            const double fk = __shfl_sync(~0u, f[q], k & 31) * row[k];
            if (lane == (k & 31)) f[q] = fk;
#pragma unroll
            for (int p = 0; p <= q; ++p)
                if (32 * p + lane < k) f[p] = fma(-row[32 * p + lane], fk, f[p]);
        }
    }
    const bool bad = red[1] != 0.0;
    if (bad && lane == 0) atomicOr(flag, 1);
#pragma unroll
    for (int q = 0; q < 4; ++q)
        if (32 * q + lane < n) out[32 * q + lane] = bad ? 0.f : (float)f[q];
}

__global__ void k_deblur_apply(const float *mref, const float *filt, int nz, int nx, int s, int flen, int nkz,
                               int nkx, float *out)
{
    const long long plane = (long long)nz * nx;
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= plane) return;
    const int param = blockIdx.y;
    const int z = (int)(i / nx), x = (int)(i - (long long)(i / nx) * nx);
    const int n = flen * flen, h = flen / 2;
    const float *m1 = mref + param * plane;
    // covering nodes: the nearest node at or above, and the next one, per axis
    int kz[2], kx[2];
    float wz[2], wx[2];
    const int iz = z >= s / 2 ? (z - s / 2) / s : -1, ix = x >= s / 2 ? (x - s / 2) / s : -1;
    for (int q = 0; q < 2; ++q) {
        kz[q] = iz + q;
        kx[q] = ix + q;
        wz[q] = (kz[q] >= 0 && kz[q] < nkz) ? fmaxf(0.f, 1.f - fabsf((float)(z - (s / 2 + kz[q] * s))) / s) : 0.f;
        wx[q] = (kx[q] >= 0 && kx[q] < nkx) ? fmaxf(0.f, 1.f - fabsf((float)(x - (s / 2 + kx[q] * s))) / s) : 0.f;
    }
    const float *fk[4];
    float w[4];
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    float den = 0.f;
    for (int q = 0; q < 4; ++q) {
        const int a = q >> 1, b = q & 1;
        w[q] = wz[a] * wx[b];
        fk[q] = w[q] > 0.f ? filt + (((long long)param * nkz + kz[a]) * nkx + kx[b]) * n : nullptr;
        den += w[q];
    }
    for (int a = -h; a <= h; ++a) {
        const int zz = z - a;
        if (zz < 0 || zz >= nz) continue;
        for (int b = -h; b <= h; ++b) {
            const int xx = x - b;
            if (xx < 0 || xx >= nx) continue;
            const float v = m1[(long long)zz * nx + xx];
            const int u = (a + h) * flen + (b + h);
            for (int q = 0; q < 4; ++q)
                if (fk[q]) acc[q] = fmaf(fk[q][u], v, acc[q]);
        }
    }
    float num = 0.f;
    for (int q = 0; q < 4; ++q) num = fmaf(w[q], acc[q], num);
    out[param * plane + i] = den > 0.f ? num / den : 0.f;
}

// ---------------------------------------------------------------------------
// Nonstationary Wiener filter (App. E, Fourier form). Per comb node a block of
// N x N = 2s x 2s pixels (z_k - s .. z_k + s - 1, the same in x; zero outside
// the image). With A = F m'' and B = F m_rtm (F the N x N DFT) the block's
// result is Re F^-1 [conj(A) B / (|A|^2 + eps_k) B], eps_k = eps mean|A|^2
// (zero when m'' is zero), and the blocks are blended with the bilinear
// valence of the space-domain filters.
//
// k_wiener_node (N = N1 N2 with both factors at most 8, every even N up to 64
// but those with a larger prime factor, 50, 54 and 60): one CTA per node, both
// planes. The blocks of m'' and m_rtm are real, so one complex transform of
// a + i b gives both spectra, A = (Z(k) + conj Z(-k)) / 2 and B = (Z(k) - conj
// Z(-k)) / 2i, and the two planes' results, real again, come from one inverse
// transform: three transforms a node where six were made. What is packed
// together is first scaled to about the same norm by powers of two, so neither
// part loses precision to the other; mean|A|^2 is sum a^2 (Parseval). A 2D transform is one Cooley-Tukey split per
// axis; a thread forms a whole length-N1 or N2 transform in registers, so a
// value is read once instead of N1 or N2 times. The inverse is the forward
// transform with real and imaginary parts exchanged before and after.
// Bound by issue slots and the shared memory around the twelve passes with a
// barrier after each (65% of issue, 65% of L1's data pipe): 300 x 2000, s = 20 (1500 nodes,
// N = 40) 100 us with the blend, at 64 registers a thread, three CTAs an SM
// (9% more at 81 registers, two); k_wiener_block took 533 us there.
// k_wiener_block: the other N; one CTA per (node, plane); the block, its
// spectra and a transform buffer sit in shared memory as complex FP32; each 2D
// DFT runs along the rows, then the columns, each as one Cooley-Tukey split
// (dft2) with a twiddle table and one output a thread.
// Both write blk[node][N*N][plane].
// k_wiener_blend: one thread per pixel, both planes, the (up to) four covering
// blocks.
// ---------------------------------------------------------------------------
constexpr int kWienerThreads = 256, kWienerMaxS = 32;
// m'' is packed 2^3 above m_rtm: the filter amplifies an error of A by up to
// 1 / sqrt(eps), one of B not at all (error 5.4e-6 with both alike, 4.0e-6 so,
// 6.8e-6 at 2^6, of the result at 300 x 2000).
constexpr int kWienerBias = 3;

// One Cooley-Tukey split of a length-N DFT, N = N1 N2 (N1 the divisor of N
// nearest sqrt N; 5 x 8 for N = 40): with n = N2 n1 + n2 and k = k1 + N1 k2,
//   X[k] = sum_n2 w^(N1 n2 k2) [ w^(n2 k1) sum_n1 x[N2 n1 + n2] w^(N2 n1 k1) ],
// w = exp(-+2 pi i / N): N1 + N2 terms per output instead of N. Pass A (the
// inner sums and the twiddle) writes tmp[row][n2 N1 + k1]; pass B the outputs.
// Applied to every row (stride 1 along a row, rows `rs` apart) or every
// column (stride N, columns 1 apart) of an N x N block.
__device__ int dft_split(int N)
{
    int best = 1;
    for (int d = 2; d <= N; ++d)
        if (N % d == 0 && fabsf((float)d * d - (float)N) < fabsf((float)best * best - (float)N)) best = d;
    return best;
}

__device__ void dft_pass_a(const float2 *src, float2 *tmp, const float2 *tw, int N, int N1, bool inverse, bool cols)
{
    const int N2 = N / N1, NN = N * N;
    for (int idx = threadIdx.x; idx < NN; idx += blockDim.x) {
        const int line = idx / N, e = idx - line * N;   // e = n2 N1 + k1
        const int n2 = e / N1, k1 = e - n2 * N1;
        const int st = cols ? N : 1, base = cols ? line : line * N;
        float re = 0.f, im = 0.f;
        int j = 0;
        for (int n1 = 0; n1 < N1; ++n1) {
            const float2 w = tw[j];
            const float wi = inverse ? w.y : -w.y;
            const float2 v = src[base + (N2 * n1 + n2) * st];
            re = fmaf(v.x, w.x, fmaf(-v.y, wi, re));
            im = fmaf(v.x, wi, fmaf(v.y, w.x, im));
            j += N2 * k1;
            while (j >= N) j -= N;
        }
        int jt = n2 * k1;
        while (jt >= N) jt -= N;
        const float2 w = tw[jt];
        const float wi = inverse ? w.y : -w.y;
        tmp[idx] = make_float2(re * w.x - im * wi, re * wi + im * w.x);
    }
    __syncthreads();
}

__device__ void dft_pass_b(const float2 *tmp, float2 *dst, const float2 *tw, int N, int N1, bool inverse, bool cols)
{
    const int N2 = N / N1, NN = N * N;
    for (int idx = threadIdx.x; idx < NN; idx += blockDim.x) {
        const int line = idx / N, k = idx - line * N;   // k = k1 + N1 k2
        const int k2 = k / N1, k1 = k - k2 * N1;
        float re = 0.f, im = 0.f;
        int j = 0;
        for (int n2 = 0; n2 < N2; ++n2) {
            const float2 w = tw[j];
            const float wi = inverse ? w.y : -w.y;
            const float2 v = tmp[line * N + n2 * N1 + k1];
            re = fmaf(v.x, w.x, fmaf(-v.y, wi, re));
            im = fmaf(v.x, wi, fmaf(v.y, w.x, im));
            j += N1 * k2;
            while (j >= N) j -= N;
        }
        dst[cols ? k * N + line : line * N + k] = make_float2(re, im);
    }
    __syncthreads();
}

// dst = DFT2(src) (sign -1) or the unscaled inverse (sign +1), rows then
// columns, via tmp (src is kept; dst and tmp are overwritten).
__device__ void dft2(const float2 *src, float2 *tmp, float2 *dst, const float2 *tw, int N, bool inverse)
{
    const int N1 = dft_split(N);
    dft_pass_a(src, tmp, tw, N, N1, inverse, false);
    dft_pass_b(tmp, dst, tw, N, N1, inverse, false);
    dft_pass_a(dst, tmp, tw, N, N1, inverse, true);
    dft_pass_b(tmp, dst, tw, N, N1, inverse, true);
}

__device__ void load_block(const float *g, int nz, int nx, int zc, int xc, int N, float2 *dst)
{
    const int s = N / 2;
    for (int idx = threadIdx.x; idx < N * N; idx += blockDim.x) {
        const int a = idx / N, b = idx - a * N;
        const int z = zc - s + a, x = xc - s + b;
        const float v = (z >= 0 && z < nz && x >= 0 && x < nx) ? g[(long long)z * nx + x] : 0.f;
        dst[idx] = make_float2(v, 0.f);
    }
}

__global__ void __launch_bounds__(kWienerThreads) k_wiener_block(const float *mref, const float *mrem, int nz, int nx,
                                                                 int s, int nkx, float eps, float *blk)
{
    extern __shared__ __align__(16) float2 wsm[];
    const int N = 2 * s, NN = N * N;
    float2 *tw = wsm;            // [N] (cos, sin)(2 pi k / N)
    float2 *P = tw + N;          // [NN] input / product
    float2 *Q = P + NN;          // [NN] transform buffer
    float2 *A = Q + NN;          // [NN] F m''
    float2 *B = A + NN;          // [NN] F m_rtm
    __shared__ float red[kWienerThreads / 32];
    const int node = blockIdx.x, plane = blockIdx.y;
    const int kz = node / nkx, kx = node - kz * nkx;
    const int zc = s / 2 + kz * s, xc = s / 2 + kx * s;
    const long long pl = (long long)nz * nx;
    for (int k = threadIdx.x; k < N; k += blockDim.x) {
        float sn, cs;
        sincospif(2.f * (float)k / (float)N, &sn, &cs);
        tw[k] = make_float2(cs, sn);
    }
    load_block(mrem + plane * pl, nz, nx, zc, xc, N, P);
    __syncthreads();
    dft2(P, Q, A, tw, N, false);
    load_block(mref + plane * pl, nz, nx, zc, xc, N, P);
    __syncthreads();
    dft2(P, Q, B, tw, N, false);
    // eps_k = eps * mean |A|^2
    float pw = 0.f;
    for (int idx = threadIdx.x; idx < NN; idx += blockDim.x) pw = fmaf(A[idx].x, A[idx].x, fmaf(A[idx].y, A[idx].y, pw));
    for (int o = 16; o > 0; o >>= 1) pw += __shfl_xor_sync(0xffffffffu, pw, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = pw;
    __syncthreads();
    float tot = 0.f;
    for (int w = 0; w < kWienerThreads / 32; ++w) tot += red[w];
    const float eps_k = eps * tot / (float)NN;
    // P = Lam^-1 B = conj(A) B B / (|A|^2 + eps_k)
    for (int idx = threadIdx.x; idx < NN; idx += blockDim.x) {
        float2 r = make_float2(0.f, 0.f);
        if (tot > 0.f) {
            const float2 a = A[idx], b = B[idx];
            const float den = fmaf(a.x, a.x, fmaf(a.y, a.y, eps_k));
            const float2 l = make_float2((a.x * b.x + a.y * b.y) / den, (a.x * b.y - a.y * b.x) / den);   // conj(a) b / den
            r = make_float2(l.x * b.x - l.y * b.y, l.x * b.y + l.y * b.x);
        }
        P[idx] = r;
    }
    __syncthreads();
    dft2(P, Q, A, tw, N, true);
    float *out = blk + (long long)node * NN * 2 + plane;
    const float scale = 1.f / (float)NN;
    for (int idx = threadIdx.x; idx < NN; idx += blockDim.x) out[2 * idx] = A[idx].x * scale;
}

// ---- forward DFTs of length R in registers, v[k] = sum_n v[n] exp(-2 pi i n k / R)
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b)
{
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
// a w, the twiddle w as a rounded value (x, y) and what rounding took off (z, w)
__device__ __forceinline__ float2 ctwiddle(float2 a, float4 w)
{
    return make_float2(fmaf(a.x, w.x, fmaf(-a.y, w.y, fmaf(a.x, w.z, -a.y * w.w))),
                       fmaf(a.x, w.y, fmaf(a.y, w.x, fmaf(a.x, w.w, a.y * w.z))));
}
// cos and sin of 2 pi j / R, j = 0 .. R - 1, for R = 3, 5, 7
template <int R>
__device__ constexpr float cos_of(int j)
{
    if (2 * j > R) j = R - j;
    if (j == 0) return 1.f;
    if (R == 3) return -0.5f;
    if (R == 5) return j == 1 ? 0.309016994374947424f : -0.809016994374947424f;
    return j == 1 ? 0.623489801858733531f : (j == 2 ? -0.222520933956314404f : -0.900968867902419126f);
}
template <int R>
__device__ constexpr float sin_of(int j)
{
    if (2 * j > R) return -sin_of<R>(R - j);
    if (j == 0) return 0.f;
    if (R == 3) return 0.866025403784438647f;
    if (R == 5) return j == 1 ? 0.951056516295153572f : 0.587785252292473129f;
    return j == 1 ? 0.781831482468029809f : (j == 2 ? 0.974927912181823607f : 0.433883739117558120f);
}
template <int R>
__device__ __forceinline__ void dft_reg(float2 (&v)[R])
{
    if constexpr (R == 2) {
        const float2 a = v[0];
        v[0] = cadd(a, v[1]);
        v[1] = csub(a, v[1]);
    } else if constexpr (R % 2 == 1) {
        // with p = v_j + v_{R-j}, m = v_j - v_{R-j}: V_k, V_{R-k} = (v_0 + sum c_jk p_j) -+ i sum s_jk m_j
        constexpr int H = (R - 1) / 2;
        float2 p[H], m[H], sum = v[0];
#pragma unroll
        for (int j = 0; j < H; ++j) {
            p[j] = cadd(v[j + 1], v[R - 1 - j]);
            m[j] = csub(v[j + 1], v[R - 1 - j]);
            sum = cadd(sum, p[j]);
        }
        const float2 v0 = v[0];
        v[0] = sum;
#pragma unroll
        for (int k = 1; k <= H; ++k) {
            float2 a = v0, b = make_float2(0.f, 0.f);
#pragma unroll
            for (int j = 1; j <= H; ++j) {
                const float c = cos_of<R>(j * k % R), s = sin_of<R>(j * k % R);
                a = make_float2(fmaf(c, p[j - 1].x, a.x), fmaf(c, p[j - 1].y, a.y));
                b = make_float2(fmaf(s, m[j - 1].x, b.x), fmaf(s, m[j - 1].y, b.y));
            }
            v[k] = make_float2(a.x + b.y, a.y - b.x);
            v[R - k] = make_float2(a.x - b.y, a.y + b.x);
        }
    } else {
        // even and odd halves, V_k = E_k + w^k O_k, V_{k+R/2} = E_k - w^k O_k
        constexpr int H = R / 2;
        float2 e[H], o[H];
#pragma unroll
        for (int j = 0; j < H; ++j) {
            e[j] = v[2 * j];
            o[j] = v[2 * j + 1];
        }
        dft_reg<H>(e);
        dft_reg<H>(o);
        constexpr float r2 = 0.707106781186547524f, r3 = 0.866025403784438647f;
#pragma unroll
        for (int k = 0; k < H; ++k) {
            float2 t = o[k];
            if (R == 4 && k == 1) t = make_float2(t.y, -t.x);
            if (R == 8 && k == 1) t = make_float2(r2 * (t.x + t.y), r2 * (t.y - t.x));
            if (R == 8 && k == 2) t = make_float2(t.y, -t.x);
            if (R == 8 && k == 3) t = make_float2(r2 * (t.y - t.x), -r2 * (t.x + t.y));
            if (R == 6 && k == 1) t = cmul(t, make_float2(0.5f, -r3));
            if (R == 6 && k == 2) t = cmul(t, make_float2(-0.5f, -r3));
            v[k] = cadd(e[k], t);
            v[k + H] = csub(e[k], t);
        }
    }
}

// One pass over every line of an N x N block (line stride ls, element stride
// es): with e = N2 n1 + n2, A forms the length-N1 transforms over n1 and the
// twiddle w^(n2 k1) into n2 N1 + k1; B the length-N2 transforms over n2 into
// k1 + N1 k2. Lanes run along the contiguous direction.
template <int N1, int N2, int P, bool COLS, bool PASS_B>
__device__ __forceinline__ void dft_lines(const float2 *src, float2 *dst, const float4 *tw)
{
    constexpr int N = N1 * N2, R = PASS_B ? N2 : N1, C = N / R;   // C transforms of length R a line
    constexpr int ls = COLS ? 1 : P, es = COLS ? P : 1;
    for (int i = threadIdx.x; i < N * C; i += blockDim.x) {
        const int line = COLS ? i % N : i / C, m = COLS ? i / N : i % C;   // m: n2 (A) or k1 (B)
        const float2 *a = src + line * ls;
        float2 *b = dst + line * ls;
        float2 v[R];
#pragma unroll
        for (int q = 0; q < R; ++q) v[q] = a[(PASS_B ? q * N1 + m : N2 * q + m) * es];
        dft_reg<R>(v);
#pragma unroll
        for (int q = 0; q < R; ++q) {
            if (PASS_B) b[(m + N1 * q) * es] = v[q];
            else b[(m * N1 + q) * es] = q == 0 ? v[q] : ctwiddle(v[q], tw[m * q]);
        }
    }
    __syncthreads();
}

// Block sum (or maximum) of two values; every thread gets both.
template <bool MAX>
__device__ __forceinline__ float2 block_reduce2(float a, float b, float2 *red)
{
    auto op = [](float u, float v) { return MAX ? fmaxf(u, v) : u + v; };
    for (int o = 16; o > 0; o >>= 1) {
        a = op(a, __shfl_xor_sync(0xffffffffu, a, o));
        b = op(b, __shfl_xor_sync(0xffffffffu, b, o));
    }
    __syncthreads();   // (red may still be read from an earlier reduction)
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = make_float2(a, b);
    __syncthreads();
    float2 t = red[0];
    for (unsigned w = 1; w < (blockDim.x + 31) / 32; ++w) t = make_float2(op(t.x, red[w].x), op(t.y, red[w].y));
    return t;
}
// The exponent e for which 2^e m is about one (0 for zero and non-finite m).
__device__ __forceinline__ int unit_exp(float m)
{
    return m > 0.f && isfinite(m) ? -ilogbf(m) : 0;
}
// v 2^e for |e| up to 252, as two factors in the normal range.
struct Scale {
    float a, b;
    __device__ __forceinline__ explicit Scale(int e) : a(ldexpf(1.f, e / 2)), b(ldexpf(1.f, e - e / 2)) {}
    __device__ __forceinline__ float operator*(float v) const { return v * a * b; }
};

// exp(-2 pi i k / N), each part as a float and the rest of it: the rounding of the
// twiddles was the largest part of the error (4.0e-6 -> 3.1e-6 of the result with
// the rests; with this form's packing, before it, 3.7e-6 for one DFT a plane).
template <int N>
struct WienerTwiddles {
    float4 w[N];
};

template <int N1, int N2>
struct WienerCfg {
    static constexpr int N = N1 * N2, P = N + 1;   // row pitch
    static constexpr int items = N * (N1 > N2 ? N1 : N2);
    static constexpr int threads = items >= 512 ? 512 : (items + 31) / 32 * 32;
    static constexpr size_t smem = N * sizeof(float4) + 3 * (size_t)N * P * sizeof(float2);
    static constexpr int blocks = 1024 / threads;   // 64 registers a thread
};

template <int N1, int N2>
__global__ void __launch_bounds__(WienerCfg<N1, N2>::threads, WienerCfg<N1, N2>::blocks) k_wiener_node(const float *mref, const float *mrem, int nz,
                                                                            int nx, int nkx, float eps, float *blk,
        const WienerTwiddles<N1 * N2> table)
{
    using C = WienerCfg<N1, N2>;
    constexpr int N = C::N, P = C::P, NN = N * N, s = N / 2, NT = C::threads, PER = (NN + NT - 1) / NT;
    extern __shared__ __align__(16) float4 wsm4[];
    float4 *tw = wsm4;                                  // [N] exp(-2 pi i k / N)
    float2 *X = reinterpret_cast<float2 *>(tw + N);     // [N][P]
    float2 *Y = X + N * P;         // [N][P]
    float2 *W = Y + N * P;         // [N][P] the first plane's product
    __shared__ float2 red[16];
    const int node = blockIdx.x, t = threadIdx.x;
    const int kz = node / nkx, kx = node - kz * nkx;
    const int zb = s / 2 + kz * s - s, xb = s / 2 + kx * s - s;   // first pixel of the block
    const long long pl = (long long)nz * nx;
    for (int k = t; k < N; k += NT) tw[k] = table.w[k];
    int out_exp[2];                               // the result's scale of each plane
    float pmax0 = 0.f;                            // the first product's largest part
    bool bad[2] = {false, false};                 // a plane's product is not finite
    float norm[2] = {1.f / (float)NN, 1.f / (float)NN};   // 1 / N^2, or what a plane without a result gets
    for (int q = 0; q < 3; ++q) {
        if (q < 2) {
            // the plane's two blocks, scaled, as a + i b
            float2 v[PER];
            float ma = 0.f, mb = 0.f;
#pragma unroll
            for (int i = 0; i < PER; ++i) {
                const int idx = t + i * NT, a = idx / N, b = idx - a * N, z = zb + a, x = xb + b;
                const bool ok = idx < NN && z >= 0 && z < nz && x >= 0 && x < nx;
                const long long g = q * pl + (long long)z * nx + x;
                v[i] = ok ? make_float2(mrem[g], mref[g]) : make_float2(0.f, 0.f);
                ma = fmaxf(ma, fabsf(v[i].x));
                mb = fmaxf(mb, fabsf(v[i].y));
            }
            // scaled to norms of about one (by the largest value first: sums
            // of squares could overflow)
            const float2 mx = block_reduce2<true>(ma, mb, red);
            const int ea = unit_exp(mx.x), eb = unit_exp(mx.y);
            const Scale fa(ea), fb(eb);
            float sa = 0.f, sb = 0.f;
#pragma unroll
            for (int i = 0; i < PER; ++i) {
                v[i] = make_float2(fa * v[i].x, fb * v[i].y);
                sa = fmaf(v[i].x, v[i].x, sa);
                sb = fmaf(v[i].y, v[i].y, sb);
            }
            const float2 sq = block_reduce2<false>(sa, sb, red);
            const int na = unit_exp(sqrtf(sq.x)) + kWienerBias, nb = unit_exp(sqrtf(sq.y));
            const float ga = ldexpf(1.f, na), gb = ldexpf(1.f, nb);
#pragma unroll
            for (int i = 0; i < PER; ++i) {
                const int idx = t + i * NT, a = idx / N, b = idx - a * N;
                if (idx < NN) X[a * P + b] = make_float2(v[i].x * ga, v[i].y * gb);
            }
            __syncthreads();
            const float eps_k = eps * (sq.x * ga * ga);   // sum a^2 = mean |A|^2 of the scaled block
            // (a zero or non-finite m'' gives zero, and so does a zero m_rtm)
            const bool live = sq.x > 0.f && isfinite(sq.x) && !(sq.y == 0.f);
            dft_lines<N1, N2, P, false, false>(X, Y, tw);
            dft_lines<N1, N2, P, false, true>(Y, X, tw);
            dft_lines<N1, N2, P, true, false>(X, Y, tw);
            dft_lines<N1, N2, P, true, true>(Y, X, tw);
            // conj(A) B B / (|A|^2 + eps_k)
            float2 *dst = q == 0 ? W : Y;
            float pm = 0.f;
            bool nf = false;
            for (int idx = t; idx < NN; idx += NT) {
                const int a = idx / N, b = idx - a * N;
                const float2 z1 = X[a * P + b], z2 = X[(a ? N - a : 0) * P + (b ? N - b : 0)];
                const float2 A = make_float2(0.5f * (z1.x + z2.x), 0.5f * (z1.y - z2.y));
                const float2 B = make_float2(0.5f * (z1.y + z2.y), 0.5f * (z2.x - z1.x));
                float2 r = make_float2(0.f, 0.f);
                if (live) {
                    const float den = fmaf(A.x, A.x, fmaf(A.y, A.y, eps_k));
                    const float2 l = make_float2((A.x * B.x + A.y * B.y) / den, (A.x * B.y - A.y * B.x) / den);
                    r = make_float2(l.x * B.x - l.y * B.y, l.x * B.y + l.y * B.x);
                }
                dst[a * P + b] = r;
                pm = fmaxf(pm, fmaxf(fabsf(r.x), fabsf(r.y)));
                nf |= !(isfinite(r.x) && isfinite(r.y));
            }
            bad[q] = __syncthreads_or(nf);
            // conj(A) B B / (|A|^2 + eps_k) goes as b^2 / a
            out_exp[q] = ea + na - 2 * (eb + nb);
            if (!live) norm[q] = 0.f;
            if (bad[q]) norm[q] = __int_as_float(0x7fffffff);
            if (q == 0) {
                pmax0 = pm;
            } else {
                // both planes' products as P0 + i P1, scaled to norms of about
                // one, parts exchanged; one that is not finite stays out of the
                // other's result (its own is then not a number)
                const float2 mp = block_reduce2<true>(pmax0, pm, red);
                const int e0 = unit_exp(mp.x), e1 = unit_exp(mp.y);
                const Scale f0(e0), f1(e1);
                float s0 = 0.f, s1 = 0.f;
                for (int idx = t; idx < NN; idx += NT) {
                    const int e = idx / N * P + idx % N;
                    const float2 p0 = W[e], p1 = Y[e];
                    const float2 u0 = make_float2(f0 * p0.x, f0 * p0.y), u1 = make_float2(f1 * p1.x, f1 * p1.y);
                    W[e] = u0, Y[e] = u1;
                    s0 = fmaf(u0.x, u0.x, fmaf(u0.y, u0.y, s0));
                    s1 = fmaf(u1.x, u1.x, fmaf(u1.y, u1.y, s1));
                }
                const float2 sp = block_reduce2<false>(s0, s1, red);
                const int n0 = unit_exp(sqrtf(sp.x)), n1 = unit_exp(sqrtf(sp.y));
                const float g0 = ldexpf(1.f, n0), g1 = ldexpf(1.f, n1);
                out_exp[0] -= e0 + n0;
                out_exp[1] -= e1 + n1;
                for (int idx = t; idx < NN; idx += NT) {
                    const int a = idx / N, b = idx - a * N;
                    const float2 zero = make_float2(0.f, 0.f);
                    const float2 p0 = bad[0] ? zero : W[a * P + b], p1 = bad[1] ? zero : Y[a * P + b];
                    X[a * P + b] = make_float2(g0 * p0.y + g1 * p1.x, g0 * p0.x - g1 * p1.y);
                }
                __syncthreads();
            }
        } else {
            dft_lines<N1, N2, P, false, false>(X, Y, tw);
            dft_lines<N1, N2, P, false, true>(Y, X, tw);
            dft_lines<N1, N2, P, true, false>(X, Y, tw);
            dft_lines<N1, N2, P, true, true>(Y, X, tw);
        }
    }
    float2 *out = reinterpret_cast<float2 *>(blk) + (long long)node * NN;
    for (int idx = t; idx < NN; idx += NT) {
        const int a = idx / N, b = idx - a * N;
        const float2 r = X[a * P + b];   // (imaginary, real) of the inverse: (plane 1, plane 0)
        out[idx] = make_float2(ldexpf(r.y * norm[0], out_exp[0]), ldexpf(r.x * norm[1], out_exp[1]));
    }
}

__global__ void k_wiener_blend(const float2 *blk, int nz, int nx, int s, int nkz, int nkx, float *out)
{
    const long long plane = (long long)nz * nx;
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= plane) return;
    const int z = (int)(i / nx), x = (int)(i - (long long)(i / nx) * nx);
    const int N = 2 * s, NN = N * N;
    const int iz = z >= s / 2 ? (z - s / 2) / s : -1, ix = x >= s / 2 ? (x - s / 2) / s : -1;
    float num0 = 0.f, num1 = 0.f, den = 0.f;
    for (int a = 0; a < 2; ++a) {
        const int kz = iz + a;
        if (kz < 0 || kz >= nkz) continue;
        const int dz = z - (s / 2 + kz * s);
        const float wz = fmaxf(0.f, 1.f - fabsf((float)dz) / s);
        for (int b = 0; b < 2; ++b) {
            const int kx = ix + b;
            if (kx < 0 || kx >= nkx) continue;
            const int dx = x - (s / 2 + kx * s);
            const float w = wz * fmaxf(0.f, 1.f - fabsf((float)dx) / s);
            if (w <= 0.f) continue;
            const float2 v = blk[((long long)kz * nkx + kx) * NN + (dz + s) * N + (dx + s)];
            num0 = fmaf(w, v.x, num0);
            num1 = fmaf(w, v.y, num1);
            den += w;
        }
    }
    out[i] = den > 0.f ? num0 / den : 0.f;
    out[plane + i] = den > 0.f ? num1 / den : 0.f;
}

template <int N1, int N2>
cudaError_t wiener_node(const float *mref, const float *mrem, int nz, int nx, int nkz, int nkx, double eps, float *blk,
                        cudaStream_t st)
{
    using C = WienerCfg<N1, N2>;
    const cudaError_t e = cudaFuncSetAttribute(k_wiener_node<N1, N2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::smem);
    if (e != cudaSuccess) return e;
    WienerTwiddles<C::N> tw;
    for (int k = 0; k < C::N; ++k) {
        const double a = 2.0 * M_PI * k / C::N, c = std::cos(a), s = -std::sin(a);
        tw.w[k] = make_float4((float)c, (float)s, (float)(c - (float)c), (float)(s - (float)s));
    }
    k_wiener_node<N1, N2><<<nkz * nkx, C::threads, C::smem, st>>>(mref, mrem, nz, nx, nkx, (float)eps, blk, tw);
    return cudaGetLastError();
}

}  // namespace

int wiener_max_spacing() { return kWienerMaxS; }

size_t wiener_smem(int s)
{
    const size_t N = 2 * (size_t)s;
    return (N + 4 * N * N) * sizeof(float2);
}

cudaError_t launch_wiener(const float *mref, const float *mrem, int nz, int nx, int s, double eps, float *blk,
                          float *out, cudaStream_t st)
{
    const int nkz = deblur_nodes(nz, s), nkx = deblur_nodes(nx, s);
    cudaError_t e = cudaSuccess;
    auto node = [&](auto f) { e = f(mref, mrem, nz, nx, nkz, nkx, eps, blk, st); };
    switch (2 * s) {   // the factors nearest the square root
    case 4: node(wiener_node<2, 2>); break;
    case 6: node(wiener_node<2, 3>); break;
    case 8: node(wiener_node<2, 4>); break;
    case 10: node(wiener_node<2, 5>); break;
    case 12: node(wiener_node<3, 4>); break;
    case 14: node(wiener_node<2, 7>); break;
    case 16: node(wiener_node<4, 4>); break;
    case 18: node(wiener_node<3, 6>); break;
    case 20: node(wiener_node<4, 5>); break;
    case 24: node(wiener_node<4, 6>); break;
    case 28: node(wiener_node<4, 7>); break;
    case 30: node(wiener_node<5, 6>); break;
    case 32: node(wiener_node<4, 8>); break;
    case 36: node(wiener_node<6, 6>); break;
    case 40: node(wiener_node<5, 8>); break;
    case 42: node(wiener_node<6, 7>); break;
    case 48: node(wiener_node<6, 8>); break;
    case 56: node(wiener_node<7, 8>); break;
    case 64: node(wiener_node<8, 8>); break;
    default: {
        const size_t sm = wiener_smem(s);
        e = cudaFuncSetAttribute(k_wiener_block, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        if (e != cudaSuccess) return e;
        k_wiener_block<<<dim3(nkz * nkx, 2), kWienerThreads, sm, st>>>(mref, mrem, nz, nx, s, nkx, (float)eps, blk);
        e = cudaGetLastError();
    }
    }
    if (e != cudaSuccess) return e;
    const long long plane = (long long)nz * nx;
    k_wiener_blend<<<(unsigned)((plane + 255) / 256), 256, 0, st>>>(reinterpret_cast<const float2 *>(blk), nz, nx, s, nkz, nkx,
                                                                    out);
    return cudaGetLastError();
}

// Doubles of k_deblur_solve's region U, and its shared memory in bytes. The
// patch and the matrix leave two CTAs an SM (three for flen <= 9) at the usual
// spacings; U, at least one lag's row sums and the panel, takes the rest of
// the share, up to what all lags of a dx need. most_ctas: CTAs an SM that the
// kernel's registers leave room for.
int deblur_solve_region(int nz, int nx, int s, int flen, int most_ctas, size_t *bytes)
{
    const int n = flen * flen, pz = std::min(nz, 2 * s + 1) + flen - 1, px = std::min(nx, 2 * s + 1) + flen - 1;
    const size_t fixed = ((size_t)(n + 1) * (n + 2) / 2 + 2 + (size_t)pz * (px | 1)) * sizeof(double);
    const int least = std::max(pz * flen, kSolvePanel * (n + 1)), most = std::max(least, pz * flen * flen);
    const int wish = std::max(least, 4 * pz * flen);
    int ulen = least;
    for (int ctas = most_ctas; ctas >= 1; --ctas) {
        const size_t share = std::min<size_t>(228 * 1024 / ctas - 1024, kDeblurSmemLimit);
        if (fixed + (size_t)(ctas > 1 ? wish : least) * sizeof(double) > share) continue;
        ulen = (int)std::min<size_t>(most, (share - fixed) / sizeof(double));
        break;
    }
    *bytes = fixed + (size_t)ulen * sizeof(double);
    return ulen;
}

int deblur_nodes(int n, int s) { return n > s / 2 ? (n - 1 - s / 2) / s + 1 : 0; }

cudaError_t launch_deblur(const float *mref, const float *mrem, int nz, int nx, int s, int flen, double eps,
                          float *filt, float *out, int *flag, cudaStream_t st)
{
    const int nkz = deblur_nodes(nz, s), nkx = deblur_nodes(nx, s);
    size_t sm = 0;
    // windows of at most 13 x 13 pixels and a thread a tap (300 x 2000: s = 2, one tap 1.45 ms for 5.29 of 256
    // threads, 49 taps 35.7 for 56.7; s = 6 0.55 for 1.45, 6.0 for 8.2; 90 x 130, s = 8, 49 taps 0.21 for 0.19)
    const bool few = s <= 6 && flen * flen <= kSolveFew;
    const int ulen = deblur_solve_region(nz, nx, s, flen, few ? kSolveFewCtas : 3, &sm);
    if (sm > kDeblurSmemLimit) return cudaErrorInvalidValue;
    auto k = few ? k_deblur_solve<kSolveFew> : k_deblur_solve<kSolveThreads>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    k<<<dim3(nkx, nkz, 2), few ? kSolveFew : kSolveThreads, sm, st>>>(mref, mrem, nz, nx, s, flen, eps, filt, flag, ulen);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const long long plane = (long long)nz * nx;
    k_deblur_apply<<<dim3((unsigned)((plane + 255) / 256), 2), 256, 0, st>>>(mref, filt, nz, nx, s, flen, nkz, nkx,
                                                                              out);
    return cudaGetLastError();
}

}  // namespace lsrtm
