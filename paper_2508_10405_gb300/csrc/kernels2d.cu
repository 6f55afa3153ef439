// Fused 2D time-step kernels for the staggered-grid Born operator and its
// exact transpose (Eq. 1, Eq. scattereqln, App. A).
//
// One launch advances every shot of a batch by one time step. A CTA of 256
// threads owns one x-column per thread (240 output columns plus 2M halo
// columns on each side for M = 4) and marches down a z-chunk of the padded
// grid, two rows (one group) at a time:
//   * along z the stencil operands live in per-thread register rings (the
//     march is unrolled by a few rows and the rings shift after every pass);
//   * along x each group passes through two shared-memory rows per field;
//   * the rows a group needs arrive by TMA: one thread issues each field's
//     two rows as one 256 x 2 tile copy on the mbarrier of the group's stage
//     while the previous group is computed. The tensor maps read zeros
//     outside the padded grid, which is the operators' boundary convention;
//   * a background field and its partner (the scattered field in Born
//     modelling, the adjoint field in migration) are interleaved as float2 in
//     HBM, so one 8-byte access and one packed FP32x2 FMA (FFMA2) serve both.
// For every group the velocity stage (half nodes) is computed on the output
// columns and the x halo, then the pressure stage (integer nodes), so a time
// step needs no grid-wide barrier. Inputs and outputs are separate (ping-pong)
// buffers; each state field is read once and written once per step from HBM.
//
// A stage is refilled only after a CTA barrier that follows every read of it:
// the first barrier of the next group (a warm-up group, which fills the z
// rings only, has one barrier of its own for this).
//
// Shots with aperture windows (WIN) have their own width, model planes (in
// their slot) and x CPML profiles; CTAs past a shot's width exit at once.
// Every state and model plane of a slot is zero past the shot's width.
#include <algorithm>
#include <cmath>
#include <mutex>
#include <type_traits>

#include "lsrtm_internal.cuh"
#include "tma.cuh"

namespace lsrtm {
namespace {

constexpr int NTH = kThreads2D;
constexpr int NS = 2;                    // stages: the group in use and the one in flight
constexpr int kBornMinBlocks = 3;        // resident CTAs per SM the register budgets target
constexpr int kPlainMinBlocks = 4;       // background step without bands or pseudo-Hessian (modelling)
constexpr int kBandsMinBlocks = 3;
constexpr int kAdjMinBlocks = 3;

// State layouts, as offsets in float planes within a shot slot.
// Born: float2 pairs (background, scattered).
enum { B_P = 0, B_VX = 2, B_VZ = 4, B_PPX = 6, B_PPZ = 8 };
// Background only (band saving, pseudo-Hessian): float.
enum { G_P = 0, G_VX = 1, G_VZ = 2, G_PPX = 3, G_PPZ = 4 };
// Adjoint: float2 pairs (p, dt kappa lambda_p), (v, lambda_v), float lambda
// CPML memories and lambda_p (a plane that holds forward passes' node CPML
// memories).
enum { A_PL = 0, A_VX = 2, A_VZ = 4, A_LPPX = 6, A_LPPZ = 7, A_LPVX = 8, A_LPVZ = 9, A_L = 10 };
// Slots of aperture-windowed shots carry the window's own model after the
// state: dt kappa and 1/rho (float planes), and the Born pairs (float2).
enum { W_KDT = 12, W_BINV = 13, W_KD2 = 14, W_BR2 = 16 };
static_assert(W_BR2 + 2 == kWinStatePlanes2D && A_L == kExtra2D, "slot layout");

// ---- packed arithmetic for T = float or float2
__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float fma_(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ float2 fma_(float a, float2 b, float2 c) { return __ffma2_rn(f2(a), b, c); }
__device__ __forceinline__ float add_(float a, float b) { return a + b; }
__device__ __forceinline__ float2 add_(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float mul_(float a, float b) { return a * b; }
__device__ __forceinline__ float2 mul_(float a, float2 b) { return __fmul2_rn(f2(a), b); }
template <class T> __device__ __forceinline__ T zero_();
template <> __device__ __forceinline__ float zero_<float>() { return 0.f; }
template <> __device__ __forceinline__ float2 zero_<float2>() { return make_float2(0.f, 0.f); }
__device__ __forceinline__ float sub_(float a, float b) { return a - b; }
__device__ __forceinline__ float2 sub_(float2 a, float2 b) { return __ffma2_rn(f2(-1.f), b, a); }
__device__ __forceinline__ float neg_(float a) { return -a; }
__device__ __forceinline__ float2 neg_(float2 a) { return make_float2(-a.x, -a.y); }

// Free surface (method of images about row z0): a ghost node row r < z0
// reads its mirror row with the sign flipped (p odd), a ghost half row k < z0
// its mirror half row (v_z even); other rows read themselves.
template <bool FS>
__device__ __forceinline__ int node_src_row(const GridDev &g, int r) { return (FS && r < g.z0) ? fs_node_row(g, r) : r; }
template <bool FS>
__device__ __forceinline__ int half_src_row(const GridDev &g, int k) { return (FS && k < g.z0) ? fs_half_row(g, k) : k; }

// Staggered first difference sum_l c_l (a_l - b_l): the M differences are
// independent, then one multiply-add chain of depth M (short critical path).
template <int M, class T, class FA, class FB>
__device__ __forceinline__ T stencil(const float *c, FA fa, FB fb)
{
    T d[M];
#pragma unroll
    for (int l = 0; l < M; ++l) d[l] = sub_(fa(l + 1), fb(l + 1));
    T acc = mul_(c[0], d[0]);
#pragma unroll
    for (int l = 1; l < M; ++l) acc = fma_(c[l], d[l], acc);
    return acc;
}
__device__ __forceinline__ float xof(float v) { return v; }
__device__ __forceinline__ float xof(float2 v) { return v.x; }
__device__ __forceinline__ float yof(float) { return 0.f; }
__device__ __forceinline__ float yof(float2 v) { return v.y; }

// ---- boundary bands
__device__ __forceinline__ long long band_xstrip(int iz, int ix, int M, int nz, int nx)
{
    return ix < 0 ? (long long)iz * M + (ix + M) : (long long)M * nz + (long long)iz * M + (ix - nx);
}

__device__ __forceinline__ long long band_zstrip(int iz, int ix, int M, int nz, int nx)
{
    long long base = 2LL * M * nz;
    return iz < 0 ? base + (long long)(iz + M) * nx + ix
                  : base + (long long)M * nx + (long long)(iz - nz) * nx + ix;
}

__device__ __forceinline__ bool in_xstrip(int ix, int M, int nx)
{
    return (ix >= -M && ix < 0) || (ix >= nx && ix < nx + M);
}

// Band slot of a node for the p band, -1 if the node is not in it.
__device__ __forceinline__ long long pband_index(int iz, int ix, int M, int nz, int nx)
{
    if (iz >= 0 && iz < nz) return in_xstrip(ix, M, nx) ? band_xstrip(iz, ix, M, nz, nx) : -1;
    if (ix >= 0 && ix < nx && in_xstrip(iz, M, nz)) return band_zstrip(iz, ix, M, nz, nx);
    return -1;
}


template <int M>
struct Cols {
    static constexpr int W = 2 * M;            // ring length along z
    static constexpr int HXP = 2 * M;          // halo columns per side
    static constexpr int TXO = NTH - 2 * HXP;  // output columns per CTA
    // every tile copy starts on a 16-byte boundary, for 4- and 8-byte elements
    static_assert(TXO % 4 == 0 && HXP % 4 == 0, "CTA column starts must be multiples of 4 elements");
};

// A launch's arguments: the step and the row maps of its input state.
struct Arg2D {
    Step2D a;
    Maps2D m;
};

// Copies field rows r0 and r1 (FR bytes each) of map plane q to dst and dst +
// FR: one 2-row tile when they are adjacent, else (mirror rows of a free
// surface, rows of different fields) one row each.
template <bool PAIR>
__device__ __forceinline__ void copy_rows(char *dst, unsigned FR, const CUtensorMap (&m)[2], int xs, int r0, int r1, int q,
                                          uint64_t *b)
{
    if (PAIR || r1 == r0 + 1) {
        tma::load3(dst, m[1], xs, r0, q, b);
    } else {
        tma::load3(dst, m[0], xs, r0, q, b);
        tma::load3(dst + FR, m[0], xs, r1, q, b);
    }
}

// Brings the line of *p into L1 ahead of its use by the same thread.
__device__ __forceinline__ void prefetch_l1(const void *p) { asm volatile("prefetch.global.L1 [%0];\n" ::"l"(p)); }

// Asynchronous copies of 4 bytes.
__device__ __forceinline__ void cp_async4(void *dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(tma::su32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// Half-node z CPML rows, node z CPML rows.
__device__ __forceinline__ bool zpml_half(const GridDev &g, int k)
{
    return k >= 0 && k < g.Nz && (k <= g.z0 - 2 || k >= g.z0 + g.nz);
}
__device__ __forceinline__ bool zpml_node(const GridDev &g, int r)
{
    return r >= 0 && r < g.Nz && (r <= g.z0 - 1 || r >= g.z0 + g.nz);
}

// ---------------------------------------------------------------------------
// Forward step from n to n+1. BORN: the background and the scattered field as
// float2 pairs (Eq. scattereqln driven by the background). Otherwise the
// background alone as float, with BANDS saving the boundary bands of p^n and
// v^{n+1/2} and HESS accumulating the pseudo-Hessian diagonal of App. B.
//
// What bounds it: the Born step moves 64 B a cell, 63.1 from DRAM (the shots
// of a batch share the model), and is held back by latencies between its
// barriers (55% of the issue slots used). A group of two rows halves the
// barriers; every warp issues one field's copy (one thread that issued all of
// a row's was waited for 600 to 1000 cycles); interior rows and warps run
// straight-line code, and what the strips need in the last stage comes with
// the copies (their warps took twice the others' time and set the CTA's pace).
// 96 shots of 424 x 1192 padded cells, order 8: 82.0 G cell-updates/s = 0.78
// of the measured copy rate (a row at a time, one issuing thread: 67.6); the
// background step with recording, 48 shots: 115.4 G (with per-thread copies:
// 70.8), with bands 75.9. Windowed shots: with k_adj2d 1.27x over per-thread
// copies.
// ---------------------------------------------------------------------------
template <int M, bool BORN, bool HESS>
struct FwdLay {
    using T = typename std::conditional<BORN, float2, float>::type;   // state (pair), (1/rho, rr), (dt kappa, dt kappa dlnk)
    static constexpr unsigned FR = NTH * sizeof(T);   // one field row
    static constexpr unsigned F = 2 * FR;             // a field's rows of a group
    // stage: p (rows z + 2M - 1), vz and psi_pz (half rows z + M - 1), vx, dt kappa and psi_px (rows z)
    static constexpr unsigned P = 0, VZ = F, VX = 2 * F, KD = 3 * F, PZ = 4 * F, PX = 5 * F, STAGE = 6 * F;
    // 1/rho: rows z + M of group j in slot j % NB; the x stage of group j reads group j - M/2's
    static constexpr int NB = M / 2 + NS;
    static constexpr unsigned BR = NS * STAGE;
    static constexpr unsigned SP = BR + NB * F;       // [2][NTH] p of the group's rows
    static constexpr unsigned SV = SP + F;            // [2][NTH] vx
    static constexpr unsigned SH = SV + F;            // [2][NTH] (b G_x)^2 (HESS)
    static constexpr unsigned BAR = SH + (HESS ? 2 * NTH * 4 : 0) + 128;
    static constexpr unsigned SMEM = BAR + 64 + 128;  // + alignment slack
    static_assert(STAGE % 128 == 0 && F % 128 == 0, "copy destinations stay 128-byte aligned");
};

// Issues the copies of the group of rows z, z + 1 on barrier b; called by
// whole warps, each of which issues its own field (a copy costs its issuing
// lane 30 to 100 cycles, and the other warps would wait for one that issued
// them all). tpn / tph: the CTA has node / half-node x CPML columns.
template <int M, bool BORN, bool FS, bool WIN>
__device__ __forceinline__ void fwd_issue(const Arg2D &p, int warp, char *st, char *brs, uint64_t *b, int slot, int xs,
                                          int z, int zc0, bool tpn, bool tph)
{
    using L = FwdLay<M, BORN, false>;
    const GridDev &g = p.a.g;
    const Maps2D &m = p.m;
    constexpr int W = 2 * M;
    const int q = slot * (BORN ? m.pps : m.fps);
    const CUtensorMap(&ms)[2] = BORN ? m.pr : m.fl;
    const CUtensorMap(&mm)[2] = WIN ? ms : (BORN ? m.mb : m.md);
    const int zr = z + W - 1, k = z + M - 1;
    const bool main = z >= zc0;
    const bool pz = zpml_half(g, k) || zpml_half(g, k + 1);
    if (warp == 0) {
        if (tma::elect_one()) {
            const int f = q + (BORN ? B_P / 2 : G_P);
            if (FS && zr < g.z0)
                copy_rows<false>(st + L::P, L::FR, ms, xs, node_src_row<FS>(g, zr), node_src_row<FS>(g, zr + 1), f, b);
            else
                copy_rows<true>(st + L::P, L::FR, ms, xs, zr, zr + 1, f, b);
        }
    } else if (warp == 1) {
        if (tma::elect_one()) {
            const int f = q + (BORN ? B_VZ / 2 : G_VZ);
            if (FS && k < g.z0)
                copy_rows<false>(st + L::VZ, L::FR, ms, xs, k < 0 ? -1 : half_src_row<FS>(g, k),
                                 k + 1 < 0 ? -1 : half_src_row<FS>(g, k + 1), f, b);
            else
                copy_rows<true>(st + L::VZ, L::FR, ms, xs, k, k + 1, f, b);
        }
    } else if (warp == 2) {
        if (tma::elect_one()) tma::load3(brs, mm[1], xs, k + 1, WIN ? q + (BORN ? W_BR2 / 2 : W_BINV) : 1, b);
    } else if (warp == 3) {
        if (main && tma::elect_one()) tma::load3(st + L::VX, ms[1], xs, z, q + (BORN ? B_VX / 2 : G_VX), b);
    } else if (warp == 4) {
        if (main && tma::elect_one()) tma::load3(st + L::KD, mm[1], xs, z, WIN ? q + (BORN ? W_KD2 / 2 : W_KDT) : 0, b);
    } else if (warp == 5) {
        if (main && tph && tma::elect_one()) tma::load3(st + L::PX, ms[1], xs, z, q + (BORN ? B_PPX / 2 : G_PPX), b);
    } else if (warp == 6) {
        if (pz) {
            if (tma::elect_one()) tma::load3(st + L::PZ, ms[1], xs, k, q + (BORN ? B_PPZ / 2 : G_PPZ), b);
        } else if (main && tpn) {   // node CPML memories along x, in the unused place of psi_pz
            if (tma::elect_one()) tma::load3(st + L::PZ, m.pv[BORN], xs, z, slot, b);
        }
    } else {
        if (tma::elect_one())
            tma::mbar_expect(b, (3 + (pz ? 1 : 0) + (main ? 2 + (tph ? 1 : 0) + (!pz && tpn ? 1 : 0) : 0)) * L::F);
    }
    __syncwarp();
}

template <int M, bool BORN, bool BANDS, bool HESS, bool WIN, bool FS>
__device__ __forceinline__ void fwd_body(const Arg2D &p)
{
    const Step2D &a = p.a;
    if (guard_tripped(a.g)) return;
    using C = Cols<M>;
    using L = FwdLay<M, BORN, HESS>;
    using T = typename L::T;
    constexpr int W = C::W, HXP = C::HXP, TXO = C::TXO, NB = L::NB;
    extern __shared__ unsigned char smraw[];
    char *sm = reinterpret_cast<char *>(smraw + ((128u - (tma::su32(smraw) & 127u)) & 127u));
    T *const sP = reinterpret_cast<T *>(sm + L::SP);
    T *const sV = reinterpret_cast<T *>(sm + L::SV);
    float *const sH = reinterpret_cast<float *>(sm + L::SH);
    uint64_t *bar = reinterpret_cast<uint64_t *>(sm + L::BAR);

    const GridDev &g = a.g;
    const int t = threadIdx.x;
    const int slot = blockIdx.z, shot = a.shot0 + slot;
    // padded and interior widths of this shot's grid (its aperture window)
    const int Nx = WIN ? a.win_nx[shot] + 2 * g.x0 : g.Nx;
    const int nx = WIN ? Nx - 2 * g.x0 : g.nx;
    if (WIN && (int)blockIdx.x * TXO >= Nx) return;   // no output column in this shot's window
    const int xs = (int)blockIdx.x * TXO - HXP;
    const int x = xs + t;
    const bool colok = x >= 0 && x < Nx;
    const bool outcol = colok && t >= HXP && t < HXP + TXO;
    const int zc0 = (int)blockIdx.y * a.tzc;
    const int zc1 = min(zc0 + a.tzc, g.Nz);
    const int zstart = zc0 - W;
    const long long plane = g.plane;
    const int pT = (int)plane;   // in-slot offsets fit 32 bits (checked by the host)
    const int pitch = g.pitch;
    const int xc = colok ? x : 0;
    const float *in = a.in + slot * a.sstride;
    T *out = reinterpret_cast<T *>(a.out + slot * a.sstride) + xc;
    T *psiv = reinterpret_cast<T *>(a.psiv + slot * a.vstride) + xc;   // along x; along z oPVZ planes further
    const float dt = g.dt;
    const int x0 = g.x0, x1 = g.x0 + nx, z0 = g.z0, z1 = g.z0 + g.nz;
    const int ix = x - x0;
    const bool pmlxh = colok && ((x <= x0 - 2) || (x >= x1));
    const bool pmlxn = outcol && ((x <= x0 - 1) || (x >= x1));
    const bool tph = (xs <= x0 - 2) || (xs + NTH - 1 >= x1);   // the CTA has half-node / node x CPML columns
    const bool tpn = (xs <= x0 - 1) || (xs + NTH - 1 >= x1);
    const int px = WIN ? shot * a.pml_xstride + x : x;         // x CPML profiles of this shot's window
    const float ahx = pmlxh ? a.pml.ah[2][px] : 0.f, bhx = pmlxh ? a.pml.bh[2][px] : 0.f;
    const float aix = pmlxn ? a.pml.ai[2][px] : 0.f, bix = pmlxn ? a.pml.bi[2][px] : 0.f;
    // half nodes left of the array are zero; past its end 1/rho reads zero,
    // and the last half node replicates the last node's
    const float hbx = x >= 0 ? 0.5f : 0.f;
    const bool lastx = x + 1 >= Nx;
    const long long bandoff = band_base(a.bands, shot, a.n);
    const int src = a.src_cell[shot];
    const float wsrc = a.wav[(a.wav_per_shot ? (long long)shot * g.nt : 0) + a.n];
    constexpr int oP = BORN ? B_P / 2 : G_P, oVX = BORN ? B_VX / 2 : G_VX, oVZ = BORN ? B_VZ / 2 : G_VZ;
    constexpr int oPPX = BORN ? B_PPX / 2 : G_PPX, oPPZ = BORN ? B_PPZ / 2 : G_PPZ;
    constexpr int oPVZ = BORN ? (WIN ? kWinStatePlanes2D : kStatePlanes2D) / 2 : 1;
    const int warp = __shfl_sync(0xffffffffu, t >> 5, 0);   // (known to be uniform)

    if (t == 0) {
        for (int i = 0; i < NS; ++i) tma::mbar_init(bar + i);
        tma::mbar_init_fence();
    }
    __syncthreads();
    for (int j = 0; j < NS && zstart + 2 * j < zc1; ++j)
        fwd_issue<M, BORN, FS, WIN>(p, warp, sm + j * L::STAGE, sm + L::BR + j * L::F, bar + j, slot, xs, zstart + 2 * j,
                                    zc0, tpn, tph);

    // z rings, shifted by U entries after every U rows (entry u + m holds row
    // z + m of P, or the half-row value written m - W + 1 rows earlier)
    constexpr int U = 2, RL = W + U - 1;
    static_assert(U % 2 == 0, "whole groups");
    T P[RL], VZ[RL];
    float HZ[HESS ? RL : 1];
#pragma unroll
    for (int j = 0; j < RL; ++j) {
        P[j] = zero_<T>();
        VZ[j] = zero_<T>();
        if (HESS) HZ[j] = 0.f;
    }
    {
        const T *pin = reinterpret_cast<const T *>(in) + oP * pT + xc;
#pragma unroll
        for (int j = 0; j < W - 1; ++j) {
            const int zr = zstart + j, zrs = node_src_row<FS>(g, zr);
            const T v = (colok && zrs >= 0 && zrs < g.Nz) ? pin[zrs * pitch] : zero_<T>();
            P[j] = zrs != zr ? neg_(v) : v;
        }
    }
    T br_old = zero_<T>();
    {
        const T *br = WIN ? reinterpret_cast<const T *>(in + (BORN ? W_BR2 : W_BINV) * plane)
                          : (BORN ? reinterpret_cast<const T *>(a.br2) : reinterpret_cast<const T *>(a.binv));
        const int k = zstart + M - 1;
        if (colok && k >= 0 && k < g.Nz) br_old = br[k * pitch + xc];
    }

    // Groups whose rows (with everything their stencils reach) are interior
    // take a form without tests of the rows (ZF), and there warps whose columns
    // are all interior one without any boundary test (XF): straight-line code
    // for the two rows, so their shared memory and FMA latencies overlap.
    const bool xf = !HESS && !BANDS && __all_sync(0xffffffffu, ix >= 0 && ix < nx);

    bool bad = false;      // this thread's wait gave up
    int fail_j = -1;       // group whose stage was not consumed
    int j = 0, bs = 0;     // group, its 1/rho slot
    for (int zb = zstart; zb < zc1; zb += U) {
#pragma unroll
        for (int u = 0; u < U; u += 2) {
            const int z = zb + u;
            if (z >= zc1) break;
            char *const st = sm + (j % NS) * L::STAGE;
            bad |= !tma::mbar_wait(bar + j % NS, (unsigned)(j / NS) & 1u);
            const char *const stt = st + t * sizeof(T);
            const char *const brk = sm + L::BR + bs * L::F + t * sizeof(T);
            bs = bs + 1 == NB ? 0 : bs + 1;   // (the next group's)
            const char *const brx = sm + L::BR + (bs + NS - 1 >= NB ? bs + NS - 1 - NB : bs + NS - 1) * L::F;
            const bool main = z >= zc0;
            const bool zf = !HESS && !BANDS && main && z > z0 && z + W < z1 && z + 1 < zc1;
            if (!zf && main && outcol) {
                // the node CPML memories of this group, read in its last stage
                const int zn = min(z + 1, zc1 - 1);
                if (pmlxn) {
                    prefetch_l1(psiv + z * pitch);
                    prefetch_l1(psiv + zn * pitch);
                }
                if (z <= z0 - 1 || zn >= z1) {
                    prefetch_l1(psiv + oPVZ * pT + z * pitch);
                    prefetch_l1(psiv + oPVZ * pT + zn * pitch);
                }
            }
            // ---- vz at half rows k = z + M - 1, z + M (column-local)
            auto vz_stage = [&](auto zc) {
                constexpr bool ZF = decltype(zc)::value;
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const int k = z + r + M - 1, sl = u + r + W - 1;
                    const T pc = *reinterpret_cast<const T *>(stt + L::P + r * L::FR);
                    P[sl] = (!ZF && FS && z + r + W - 1 < z0) ? neg_(pc) : pc;   // ghost rows hold -p(mirror)
                    T br1 = *reinterpret_cast<const T *>(brk + r * L::FR);
                    if (!ZF && k + 1 >= g.Nz) br1 = br_old;   // the last half row replicates the last node row
                    const float buz = 0.5f * (xof(br_old) + xof(br1));
                    const float rsum = yof(br_old) + yof(br1);
                    br_old = br1;
                    T vzn = zero_<T>();
                    float hzq = 0.f;
                    if (ZF || (k >= 0 && k < g.Nz)) {
                        const int ck = k * pitch;
                        const bool own = outcol && (ZF || k >= zc0) && k < zc1;
                        T G = stencil<M, T>(g.cz, [&](int l) { return P[u + r + M - 1 + l]; },
                                            [&](int l) { return P[u + r + M - l]; });
                        if (!ZF && ((k <= z0 - 2) || (k >= z1))) {
                            const T psz = *reinterpret_cast<const T *>(stt + L::PZ + r * L::FR);
                            const T ps = fma_(a.pml.bh[0][k], psz, mul_(a.pml.ah[0][k], G));
                            if (own) out[oPPZ * pT + ck] = ps;
                            G = add_(G, ps);
                        }
                        const float dtbu = dt * buz;
                        vzn = fma_(-dtbu, G, *reinterpret_cast<const T *>(stt + L::VZ + r * L::FR));
                        if constexpr (BORN) vzn.y = fmaf(0.5f * dt * rsum, G.x, vzn.y);
                        if (own) out[oVZ * pT + ck] = vzn;
                        if (BANDS && own) {
                            const int iz = k - z0;
                            if (ix >= 0 && ix < nx && in_xstrip(iz, M, g.nz))
                                band_put(a.bands, 1, slot, bandoff, band_zstrip(iz, ix, M, g.nz, nx), xof(vzn));
                        }
                        if (HESS) {
                            const float q = buz * xof(G);
                            hzq = q * q;
                        }
                    }
                    VZ[sl] = vzn;
                    if (HESS) HZ[sl] = hzq;
                }
            };
            if (main) {
#pragma unroll
                for (int r = 0; r < 2; ++r) sP[r * NTH + t] = P[u + r];
            }
            if (zf) vz_stage(std::true_type{});
            else vz_stage(std::false_type{});
            // every thread is past the previous group's reads: refill its stage
            if (__syncthreads_or(bad)) {
                fail_j = j;
                break;
            }
            if (j >= 1 && z + 2 * (NS - 1) < zc1) {
                const int jn = j + NS - 1;
                fwd_issue<M, BORN, FS, WIN>(p, warp, sm + (jn % NS) * L::STAGE, sm + L::BR + (jn % NB) * L::F, bar + jn % NS,
                                            slot, xs, z + 2 * (NS - 1), zc0, tpn, tph);
            }
            ++j;
            if (!main) continue;   // warm-up groups fill the z rings

            // ---- rows z, z + 1: vx on the output columns and the halo
            auto vx_stage = [&](auto zc, auto xc_) {
                constexpr bool ZF = decltype(zc)::value, XF = decltype(xc_)::value;
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const T *const pr = sP + r * NTH + t;
                    T G = stencil<M, T>(g.cx, [&](int l) { return pr[l]; }, [&](int l) { return pr[1 - l]; });
                    const T *const b = reinterpret_cast<const T *>(brx + r * L::FR) + t;
                    const T b0 = b[0], b1 = !XF && lastx ? b0 : b[1];
                    const float hb = XF ? 0.5f : hbx;
                    const float bux = hb * (xof(b0) + xof(b1));
                    const bool own = outcol && (ZF || z + r < zc1);
                    if (!XF && pmlxh) {
                        const T psx = *reinterpret_cast<const T *>(stt + L::PX + r * L::FR);
                        const T ps = fma_(bhx, psx, mul_(ahx, G));
                        if (own) out[oPPX * pT + (z + r) * pitch] = ps;
                        G = add_(G, ps);
                    }
                    const float dtbu = dt * bux;
                    T vxn = fma_(-dtbu, G, *reinterpret_cast<const T *>(stt + L::VX + r * L::FR));
                    if constexpr (BORN) {
                        const float rs = yof(b0) + (!XF && lastx ? 0.f : yof(b1));
                        vxn.y = fmaf(hb * dt * rs, G.x, vxn.y);
                    }
                    sV[r * NTH + t] = vxn;
                    if (own) out[oVX * pT + (z + r) * pitch] = vxn;
                    if (BANDS && own) {
                        const int iz = z + r - z0;
                        if (iz >= 0 && iz < g.nz && in_xstrip(ix, M, nx))
                            band_put(a.bands, 1, slot, bandoff, band_xstrip(iz, ix, M, g.nz, nx), xof(vxn));
                    }
                    if (HESS) {
                        const float q = bux * xof(G);
                        sH[r * NTH + t] = q * q;
                    }
                }
            };
            if (!zf) vx_stage(std::false_type{}, std::false_type{});
            else if (xf) vx_stage(std::true_type{}, std::true_type{});
            else vx_stage(std::true_type{}, std::false_type{});
            __syncthreads();

            // ---- rows z, z + 1: pressure on the output columns
            auto p_stage = [&](auto zc, auto xc_) {
                constexpr bool ZF = decltype(zc)::value, XF = decltype(xc_)::value;
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const int zr = z + r, cz = zr * pitch;
                    const T *const vr = sV + r * NTH + t;
                    T qx = stencil<M, T>(g.cx, [&](int l) { return vr[l - 1]; }, [&](int l) { return vr[-l]; });
                    T qz = stencil<M, T>(g.cz, [&](int l) { return VZ[u + r + M + l - 1]; },
                                         [&](int l) { return VZ[u + r + M - l]; });
                    const bool own = outcol && (ZF || zr < zc1);
                    if (!XF && own && pmlxn) {
                        const T pv = ZF ? *reinterpret_cast<const T *>(stt + L::PZ + r * L::FR) : psiv[cz];
                        const T ps = fma_(bix, pv, mul_(aix, qx));
                        psiv[cz] = ps;
                        qx = add_(qx, ps);
                    }
                    if (!ZF && own && ((zr <= z0 - 1) || (zr >= z1))) {
                        const T ps = fma_(a.pml.bi[0][zr], psiv[oPVZ * pT + cz], mul_(a.pml.ai[0][zr], qz));
                        psiv[oPVZ * pT + cz] = ps;
                        qz = add_(qz, ps);
                    }
                    const T Q = add_(qx, qz);
                    const T kd2 = *reinterpret_cast<const T *>(stt + L::KD + r * L::FR);
                    const float kd = xof(kd2);
                    const T p0 = P[u + r];
                    T pn = fma_(-kd, Q, p0);
                    const float sw = cz + x == src ? wsrc : 0.f;
                    if constexpr (BORN) {
                        pn.y = fmaf(-kd2.y, Q.x, pn.y);
                        pn.x = fmaf(a.src_scale, sw, pn.x);
                    } else {
                        pn = fmaf(a.src_scale, sw, pn);
                    }
                    if (!ZF && FS && zr <= z0) pn = zero_<T>();   // p = 0 on the free surface (ghost rows unused)
                    if (own) out[oP * pT + cz] = pn;
                    if (BANDS && own) {
                        const long long b = pband_index(zr - z0, ix, M, g.nz, nx);
                        if (b >= 0) band_put(a.bands, 0, slot, bandoff, b, xof(p0));
                    }
                    if (HESS && own) {
                        const int iz = zr - z0;
                        if (iz >= 0 && iz < g.nz && ix >= 0 && ix < nx) {
                            const float bx0 = xof(reinterpret_cast<const T *>(brx + r * L::FR)[t]);
                            const float *const h = sH + r * NTH + t;
                            const float hr = 0.5f * ((h[0] + h[-1]) + (HZ[u + r + M] + HZ[u + r + M - 1])) / (bx0 * bx0);
                            const float kq = kd * xof(Q) / dt;
                            (a.hess + slot * plane)[cz + xc] += dt * (hr + kq * kq);
                        }
                    }
                }
            };
            if (!zf) p_stage(std::false_type{}, std::false_type{});
            else if (xf) p_stage(std::true_type{}, std::true_type{});
            else p_stage(std::true_type{}, std::false_type{});
        }
        if (fail_j >= 0) break;
#pragma unroll
        for (int i = 0; i < W - 1; ++i) {
            P[i] = P[i + U];
            VZ[i] = VZ[i + U];
            if (HESS) HZ[i] = HZ[i + U];
        }
    }

    if (fail_j >= 0) {
        // a wait gave up: record it, let the copies in flight land, return
        if (t == NTH - 1) {
            atomicOr(a.err, 1);
            for (int jj = fail_j; jj <= max(NS - 1, fail_j + NS - 2) && zstart + 2 * jj < zc1; ++jj)
                (void)tma::mbar_wait(bar + jj % NS, (unsigned)(jj / NS) & 1u);
        }
        return;
    }

    if (BORN || a.rec_bg) {
        // record dp^{n+1} (Born) or the background p^{n+1} (nonlinear
        // modelling) at the receivers of this CTA
        __syncthreads();
        const int tile = shot * a.trec.ntiles + blockIdx.y * gridDim.x + blockIdx.x;
        const int b = a.trec.ptr[tile], e = a.trec.ptr[tile + 1];
        const T *po = reinterpret_cast<const T *>(a.out + slot * a.sstride) + oP * plane;
        for (int i = b + t; i < e; i += NTH) {
            const int2 rc = a.trec.rec[i];
            const T v = po[rc.x];
            a.dstage[(long long)rc.y * g.nt + a.n] = BORN && !a.rec_bg ? yof(v) : xof(v);
        }
    }
}

// The Born step of shots spanning the model, of shots with aperture windows,
// and the background steps.
template <int M, bool FS>
__global__ void __launch_bounds__(NTH, kBornMinBlocks) k_fwd2t(const __grid_constant__ Arg2D p)
{
    fwd_body<M, true, false, false, false, FS>(p);
}
template <int M, bool FS>
__global__ void __launch_bounds__(NTH, kBornMinBlocks) k_fwd2w(const __grid_constant__ Arg2D p)
{
    fwd_body<M, true, false, false, true, FS>(p);
}
template <int M, bool BANDS, bool HESS, bool WIN, bool FS>
__global__ void __launch_bounds__(NTH, (BANDS || HESS) ? kBandsMinBlocks : kPlainMinBlocks) k_fwd2d(const __grid_constant__ Arg2D p)
{
    fwd_body<M, false, BANDS, HESS, WIN, FS>(p);
}

// ---------------------------------------------------------------------------
// Reverse step n (n = nt-1 .. 0) of L^T. Input state: (background p^n,
// mu = dt kappa lambda_p) with the residual of step n already added,
// (v^{n+1/2}, lambda_v) and the lambda CPML memories. The step applies the
// transposed Born sub-steps (S4^T, S3^T on the half nodes from mu; S2^T, S1^T
// on the nodes from lambda_v), accumulates the two zero-lag images (discrete
// transposed forms of Eqs. gradkappa, gradrho; the kappa image as sum Q lambda_p),
// rebuilds p^{n-1}, v^{n-1/2} in the interior from the saved boundary bands,
// and pre-adds the residual of step n-1. The D+ stencils of (p^n, u) and the
// D- stencils of (v^{n+1/2}, w) run as packed pairs.
//
// The adjoint pressure is carried twice: as mu in the pairs, the quantity the
// D+ stencils take, and as lambda_p in a plane of its own (the first of the
// forward passes' node CPML planes), what the images and the update take. Away
// from the z strips the ring's entry of a row then is the row's own (p, mu): a
// row needs neither dt kappa of its look-ahead row nor a second copy of the
// pairs. (With mu alone, 72 B a cell: 55.2 G, and
// lambda_p is rounded as mu, which moves the 64-bit misfits of a CG by 1e-8.)
// Which products of the CPML terms are fused into the subtractions, and in the
// forward step the source's, is written out for the same reason: left to the
// compiler, it changes with the code around them.
//
// What bounds it: 80 B a cell (81.6 from DRAM), held back like the Born step; 3
// tile copies a row where a row at a time took 9; at order 8 three CTAs an SM
// leave 80 registers and 76 B of spills. The x strips' band values come one
// group ahead by asynchronous copies (read where they are used, they
// doubled the strip warps' time). 96 shots of 424 x 1192, order 8, FP16 bands:
// 56.0 G cell-updates/s = 0.67 of the measured copy rate (a row at a time with
// one issuing thread: 42.4; in groups without the straight-line form: 31.5).
// ---------------------------------------------------------------------------
struct AdjLay {
    static constexpr unsigned F2R = NTH * 8, F1R = NTH * 4, F2 = 2 * F2R, F1 = 2 * F1R;   // a row, a group's two rows
    // stage: (p, mu) rows z + 2M - 1; v_z half rows z + M - 1; v_x rows z; image (interior rows) or lambda psi_vz rows z
    static constexpr unsigned PL = 0, VZ = F2, VX = 2 * F2, IM = 3 * F2;
    // dt kappa and lambda_p rows z; lambda CPML memories psi_vx and psi_px rows z (CTAs with x strips), psi_vz rows
    // z + 2M - 1, psi_pz half rows z + M - 1 (groups with z strip rows)
    static constexpr unsigned KD = 4 * F2, LAM = KD + F1, LVX = LAM + F1, LPX = LVX + F1, LVZR = LPX + F1,
                              LPZ = LVZR + F1, STAGE = LPZ + F1;
    static constexpr unsigned B = NS * STAGE;   // 1/rho ring (FwdLay::BR)
};
template <int M>
struct AdjLayM : AdjLay {
    static constexpr int NB = M / 2 + NS;
    static constexpr unsigned SPU = B + NB * F1;   // [2][NTH] (p^n, mu - ai_x (lpsi_vx - mu))
    static constexpr unsigned SVW = SPU + F2;      // [2][NTH] (vx^{n+1/2}, dt*bu_x*lvx - ah_x*lpsi_px)
    static constexpr unsigned SVN = SVW + F2;      // [2][NTH] vx^{n-1/2}
    static constexpr unsigned SPI = SVN + F1;      // [2][8] Gx lvx of the last lane of each warp
    static constexpr unsigned SB = SPI + 64;       // [2 groups][p, v][2 rows][2 sides][M] band values of the x strips (16-bit: in the first half)
    static constexpr unsigned BAR = SB + 2 * 2 * 2 * 2 * M * 4 + 8;
    static constexpr unsigned SMEM = BAR + 64 + 128;
    static_assert(STAGE % 128 == 0, "copy destinations stay 128-byte aligned");
    // three CTAs per SM: 228 KB, 1 KB reserved per CTA
    static_assert(3 * (SMEM + 1024) <= 233472, "migration kernel must fit three CTAs per SM");
};

// Issues the copies of the group of rows z, z + 1 on barrier b (as fwd_issue).
template <int M, bool FS, bool WIN>
__device__ __forceinline__ void adj_issue(const Arg2D &p, int warp, char *st, char *bs, uint64_t *b, int slot, int xs, int z,
                                          int zc0, bool tpn, bool tph)
{
    using L = AdjLay;
    const GridDev &g = p.a.g;
    const Maps2D &m = p.m;
    constexpr int W = 2 * M;
    const int zr = z + W - 1, k = z + M - 1;
    const int qp = slot * m.pps, qf = slot * m.fps;
    const CUtensorMap(&mm)[2] = WIN ? m.fl : m.md;
    const bool main = z >= zc0;
    const bool lvr = zpml_node(g, zr) || zpml_node(g, zr + 1), lpz = zpml_half(g, k) || zpml_half(g, k + 1);
    const bool in0 = z >= g.z0 && z < g.z0 + g.nz, in1 = z + 1 >= g.z0 && z + 1 < g.z0 + g.nz;
    if (warp == 0) {
        if (tma::elect_one()) {
            if (FS && zr < g.z0)
                copy_rows<false>(st + L::PL, L::F2R, m.pr, xs, node_src_row<FS>(g, zr), node_src_row<FS>(g, zr + 1),
                                 qp + A_PL / 2, b);
            else
                copy_rows<true>(st + L::PL, L::F2R, m.pr, xs, zr, zr + 1, qp + A_PL / 2, b);
        }
    } else if (warp == 1) {
        if (tma::elect_one()) {
            if (FS && k < g.z0)
                copy_rows<false>(st + L::VZ, L::F2R, m.pr, xs, k < 0 ? -1 : half_src_row<FS>(g, k),
                                 k + 1 < 0 ? -1 : half_src_row<FS>(g, k + 1), qp + A_VZ / 2, b);
            else
                copy_rows<true>(st + L::VZ, L::F2R, m.pr, xs, k, k + 1, qp + A_VZ / 2, b);
        }
    } else if (warp == 2) {
        if (main && tma::elect_one()) tma::load3(st + L::VX, m.pr[1], xs, z, qp + A_VX / 2, b);
    } else if (warp == 3) {
        // the image of interior rows, lambda psi_vz of others
        if (main && tma::elect_one()) {
            if (in0 && in1) {
                tma::load3(st + L::IM, m.im[1], xs, z, slot, b);
            } else {
                tma::load3(st + L::IM, in0 ? m.im[0] : m.fl[0], xs, z, in0 ? slot : qf + A_LPVZ, b);
                tma::load3(st + L::IM + L::F2R, in1 ? m.im[0] : m.fl[0], xs, z + 1, in1 ? slot : qf + A_LPVZ, b);
            }
        }
    } else if (warp == 4) {
        if (tma::elect_one()) {
            tma::load3(bs, mm[1], xs, k + 1, WIN ? qf + W_BINV : 1, b);
            if (main) tma::load3(st + L::KD, mm[1], xs, z, WIN ? qf + W_KDT : 0, b);
        }
    } else if (warp == 5) {
        if ((lvr || lpz) && tma::elect_one()) {
            if (lvr) tma::load3(st + L::LVZR, m.fl[1], xs, zr, qf + A_LPVZ, b);
            if (lpz) tma::load3(st + L::LPZ, m.fl[1], xs, k, qf + A_LPPZ, b);
        }
    } else if (warp == 6) {
        if (main && tma::elect_one()) {
            tma::load3(st + L::LAM, m.fl[1], xs, z, qf + A_L, b);
            if (tpn) tma::load3(st + L::LVX, m.fl[1], xs, z, qf + A_LPVX, b);
            if (tph) tma::load3(st + L::LPX, m.fl[1], xs, z, qf + A_LPPX, b);
        }
    } else {
        if (tma::elect_one()) {
            unsigned bytes = 2 * L::F2 + (1 + (lvr ? 1 : 0) + (lpz ? 1 : 0)) * L::F1;
            if (main) bytes += L::F2 + (in0 ? L::F2R : L::F1R) + (in1 ? L::F2R : L::F1R) + (2 + (tpn ? 1 : 0) + (tph ? 1 : 0)) * L::F1;
            tma::mbar_expect(b, bytes);
        }
    }
    __syncwarp();
}

template <int M, bool WIN, bool FS>
__device__ __forceinline__ void adj_body(const Arg2D &p)
{
    const Step2D &a = p.a;
    if (guard_tripped(a.g)) return;
    using C = Cols<M>;
    using L = AdjLayM<M>;
    constexpr int W = C::W, HXP = C::HXP, TXO = C::TXO, NB = L::NB;
    extern __shared__ unsigned char smraw[];
    char *sm = reinterpret_cast<char *>(smraw + ((128u - (tma::su32(smraw) & 127u)) & 127u));
    float2 *const sPU = reinterpret_cast<float2 *>(sm + L::SPU);
    float2 *const sVW = reinterpret_cast<float2 *>(sm + L::SVW);
    float *const sVN = reinterpret_cast<float *>(sm + L::SVN);
    float *const sPi = reinterpret_cast<float *>(sm + L::SPI);
    char *const sB = sm + L::SB;
    float *const sScale = reinterpret_cast<float *>(sm + L::BAR - 8);   // this step's (p, v) band scales
    uint64_t *bar = reinterpret_cast<uint64_t *>(sm + L::BAR);

    const GridDev &g = a.g;
    const int t = threadIdx.x;
    const int slot = blockIdx.z, shot = a.shot0 + slot;
    // padded and interior widths of this shot's grid (its aperture window)
    const int Nx = WIN ? a.win_nx[shot] + 2 * g.x0 : g.Nx;
    const int nx = WIN ? Nx - 2 * g.x0 : g.nx;
    if (WIN && (int)blockIdx.x * TXO >= Nx) return;   // no output column in this shot's window
    const int xs = (int)blockIdx.x * TXO - HXP;
    const int x = xs + t;
    const bool colok = x >= 0 && x < Nx;
    const bool outcol = colok && t >= HXP && t < HXP + TXO;
    const int zc0 = (int)blockIdx.y * a.tzc;
    const int zc1 = min(zc0 + a.tzc, g.Nz);
    const int zstart = zc0 - W;
    const int pT = (int)g.plane;   // in-slot offsets fit 32 bits (checked by the host); the stride of a pair field in float2
    const int pitch = g.pitch;
    const int xc = colok ? x : 0;
    const float *in = a.in + slot * a.sstride;
    float *outf = a.out + slot * a.sstride + xc;
    float *outl = a.out + slot * a.sstride + A_L * g.plane + xc;
    float2 *out2 = reinterpret_cast<float2 *>(a.out + slot * a.sstride) + xc;
    const float dt = g.dt;
    const int n = a.n;
    const bool recon = n > 0;
    const int x0 = g.x0, x1 = g.x0 + nx, z0 = g.z0, z1 = g.z0 + g.nz;
    const int ix = x - x0;
    const bool xint = ix >= 0 && ix < nx;
    const bool xband = recon && in_xstrip(ix, M, nx);
    const bool cband = recon && (xs < x0 || xs + NTH > x1);    // the CTA may have x strip columns of the bands
    const int bc = ix < 0 ? ix + M : M + ix - nx;              // this column in a row's [2 sides][M] strip values
    const bool pmlxh = colok && ((x <= x0 - 2) || (x >= x1));
    const bool pmlxn = colok && ((x <= x0 - 1) || (x >= x1));
    const bool tph = (xs <= x0 - 2) || (xs + NTH - 1 >= x1);   // the CTA has half-node / node CPML columns
    const bool tpn = (xs <= x0 - 1) || (xs + NTH - 1 >= x1);
    const int px = WIN ? shot * a.pml_xstride + x : x;         // x CPML profiles of this shot's window
    const float ahx = pmlxh ? a.pml.ah[2][px] : 0.f, bhx = pmlxh ? a.pml.bh[2][px] : 0.f;
    const float aix = pmlxn ? a.pml.ai[2][px] : 0.f, bix = pmlxn ? a.pml.bi[2][px] : 0.f;
    const float hbx = x >= 0 ? 0.5f : 0.f;   // half nodes left of the array are zero (past its end 1/rho reads zero)
    const bool lastx = x + 1 >= Nx;
    const long long rowprev = band_row(a.bands, shot, n - 1);
    const int src = a.src_cell[shot];
    const float wsrc = recon ? a.src_scale * a.wav[(a.wav_per_shot ? (long long)shot * g.nt : 0) + n - 1] : 0.f;
    float2 *img = a.img + slot * g.plane + xc;
    const float *kdt = WIN ? in + W_KDT * g.plane : a.kdt;
    const int warp = __shfl_sync(0xffffffffu, t >> 5, 0);   // (known to be uniform)

    if (t == 0) {
        for (int i = 0; i < NS; ++i) tma::mbar_init(bar + i);
        tma::mbar_init_fence();
        if (cband && a.bands.fmt != BAND_F32)
            for (int f = 0; f < 2; ++f) sScale[f] = a.bands.scale[rowprev * 2 + f];
    }
    __syncthreads();
    for (int j = 0; j < NS && zstart + 2 * j < zc1; ++j)
        adj_issue<M, FS, WIN>(p, warp, sm + j * L::STAGE, sm + L::B + j * L::F1, bar + j, slot, xs, zstart + 2 * j, zc0, tpn,
                              tph);

    // z rings, shifted by U entries after every U rows: at row u of a pass,
    // entry u + m holds node row z + m (PU) or the half-row value written m -
    // W + 1 rows earlier (VW, VN), m = 0 .. W - 1; PIZ entry u + m half row z
    // - 1 + m, m = 0 .. M
    constexpr int U = 2, RL = W + U - 1, RP = M + U;
    float2 PU[RL], VW[RL];
    float VN[RL], PIZ[RP];
#pragma unroll
    for (int i = 0; i < RL; ++i) {
        PU[i] = make_float2(0.f, 0.f);
        VW[i] = make_float2(0.f, 0.f);
        VN[i] = 0.f;
    }
#pragma unroll
    for (int i = 0; i < RP; ++i) PIZ[i] = 0.f;
    // (p^n, mu - ai_z (lpsi_vz - mu)) at node row r of this column (pl holds
    // the mirror row's values for a ghost row r < z0; the surface row carries
    // p = 0 and mu = 0)
    auto pu_node = [&](int r, float2 pl, float lpvz) -> float2 {
        if (FS && r <= z0) {
            if (r == z0) return make_float2(0.f, 0.f);
            return make_float2(-pl.x, -pl.y);
        }
        if (zpml_node(g, r)) pl.y -= a.pml.ai[0][r] * (lpvz - pl.y);
        return pl;
    };
    {
        const float2 *in2 = reinterpret_cast<const float2 *>(in) + (A_PL / 2) * pT + xc;
#pragma unroll
        for (int i = 0; i < W - 1; ++i) {
            const int r = zstart + i, rs = node_src_row<FS>(g, r);
            const float2 plv = (colok && rs >= 0 && rs < g.Nz) ? in2[rs * pitch] : make_float2(0.f, 0.f);
            const float lpvz = colok && zpml_node(g, r) ? in[A_LPVZ * pT + r * pitch + xc] : 0.f;
            PU[i] = pu_node(r, plv, lpvz);
        }
    }
    float bz_old = 0.f;
    {
        const int k = zstart + M - 1;
        if (colok && k >= 0 && k < g.Nz) bz_old = (WIN ? in + W_BINV * g.plane : a.binv)[k * pitch + xc];
    }

    // forms without row (ZF) and column (XF) tests, as in fwd_body
    const bool xf = __all_sync(0xffffffffu, xint);

    // The x strips' band values of the group of rows zg, zg + 1 (buffer bf),
    // fetched one group ahead by asynchronous copies of 4 bytes: one value, or
    // two 16-bit ones by the even columns (rows of a strip hold M values, M
    // even, so their pairs are 4-byte aligned).
    auto band_fetch = [&](int zg, int bf) {
        const bool f32 = a.bands.fmt == BAND_F32;
        if (xband && (f32 || (bc & 1) == 0)) {
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const int iz = zg + r - z0;
                if (iz < 0 || iz >= g.nz) continue;
                const long long o = rowprev * a.bands.nb + band_xstrip(iz, ix, M, g.nz, nx);
                const int e = (bf * 4 + r) * 2 * M + bc;   // field 0; field 1 at + 2 * 2M
                const int sz = f32 ? 4 : 2;
                cp_async4(sB + e * sz, static_cast<const char *>(a.bands.p) + o * sz);
                cp_async4(sB + (e + 4 * M) * sz, static_cast<const char *>(a.bands.v) + o * sz);
            }
        }
    };
    auto band_val = [&](int field, int bf, int r) -> float {
        const int e = (bf * 4 + field * 2 + r) * 2 * M + bc;
        if (a.bands.fmt == BAND_F32) return reinterpret_cast<const float *>(sB)[e];
        if (a.bands.fmt == BAND_BF16S) return sScale[field] * __bfloat162float(reinterpret_cast<const __nv_bfloat16 *>(sB)[e]);
        return sScale[field] * __half2float(reinterpret_cast<const __half *>(sB)[e]);
    };

    bool bad = false;      // this thread's wait gave up
    int fail_j = -1;       // group whose stage was not consumed
    int j = 0, bs = 0;     // group, its 1/rho slot
    for (int z = zstart; z < zc1; z += U) {
        char *const st = sm + (j % NS) * L::STAGE;
        bad |= !tma::mbar_wait(bar + j % NS, (unsigned)(j / NS) & 1u);
        const char *const st2 = st + t * 8;
        const char *const st1 = st + t * 4;
        const char *const bk = sm + L::B + bs * L::F1 + t * 4;
        bs = bs + 1 == NB ? 0 : bs + 1;   // (the next group's)
        const char *const brx = sm + L::B + (bs + NS - 1 >= NB ? bs + NS - 1 - NB : bs + NS - 1) * L::F1;
        const bool main = z >= zc0;
        const bool zf = recon && main && z > z0 && z + W < z1 && z + 1 < zc1;
        // ---- rows z, z + 1: (p, mu) of the row itself (the ring's entries of rows in the z strips hold u != mu)
        float pr[2];
        auto own_lam = [&](int r, bool ZF) {   // zero on the free surface
            return (!ZF && FS && z + r == z0) ? 0.f : *reinterpret_cast<const float *>(st1 + L::LAM + r * L::F1R);
        };
        auto own_row = [&](auto zc, auto xc_) {
            constexpr bool ZF = decltype(zc)::value, XF = decltype(xc_)::value;
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                pr[r] = (!ZF && FS && z + r < z0) ? 0.f : PU[r].x;
                float u = PU[r].y;
                if (!ZF) u = __fmul_rn(*reinterpret_cast<const float *>(st1 + L::KD + r * L::F1R), own_lam(r, ZF));
                if (!XF && pmlxn) u = fmaf(-aix, *reinterpret_cast<const float *>(st1 + L::LVX + r * L::F1R) - u, u);
                sPU[r * NTH + t] = make_float2(pr[r], u);
            }
        };
        // ---- half rows k along z: lambda_vz, lambda_psi_pz, background vz^{n-1/2}
        auto vz_stage = [&](auto zc) {
            constexpr bool ZF = decltype(zc)::value;
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const int zr = z + r + W - 1, k = z + r + M - 1, sl = r + W - 1;
                const float2 pl = *reinterpret_cast<const float2 *>(st2 + L::PL + r * L::F2R);
                if (ZF) PU[sl] = pl;
                else PU[sl] = pu_node(zr, pl, *reinterpret_cast<const float *>(st1 + L::LVZR + r * L::F1R));
                float b1 = *reinterpret_cast<const float *>(bk + r * L::F1R);
                if (!ZF && k + 1 >= g.Nz) b1 = bz_old;   // the last half row replicates the last node row
                const float buz = 0.5f * (bz_old + b1);
                bz_old = b1;
                const float2 v2z = *reinterpret_cast<const float2 *>(st2 + L::VZ + r * L::F2R);
                float wz = 0.f, vn = 0.f, piz = 0.f;
                if (ZF || (k >= 0 && k < g.Nz)) {
                    const int ck = k * pitch;
                    const bool own = outcol && (ZF || k >= zc0) && k < zc1;
                    // (Gz, du/dz)
                    const float2 D = stencil<M, float2>(g.cz, [&](int l) { return PU[r + M - 1 + l]; },
                                                        [&](int l) { return PU[r + M - l]; });
                    const float lv = v2z.y + D.y;
                    const float dtbu = dt * buz;
                    wz = __fmul_rn(dtbu, lv);
                    if (!ZF && ((k <= z0 - 2) || (k >= z1))) {
                        const float l1 = *reinterpret_cast<const float *>(st1 + L::LPZ + r * L::F1R) - wz;
                        wz = fmaf(-a.pml.ah[0][k], l1, wz);
                        if (own) outf[A_LPPZ * pT + ck] = a.pml.bh[0][k] * l1;
                    }
                    piz = D.x * lv;
                    if (ZF) {
                        vn = xint ? v2z.x + dtbu * D.x : 0.f;
                    } else if (recon && xint) {
                        const int iz = k - z0;
                        if ((iz >= 0 || FS) && iz < g.nz) vn = v2z.x + dtbu * D.x;
                        else if (in_xstrip(iz, M, g.nz))
                            vn = band_get(a.bands, 1, rowprev, band_zstrip(iz, ix, M, g.nz, nx));
                    }
                    if (own) out2[(A_VZ / 2) * pT + ck] = make_float2(vn, lv);
                }
                VW[sl] = make_float2(v2z.x, wz);
                VN[sl] = vn;
                PIZ[r + M] = piz;
            }
        };
        if (!zf) {
            if (main) own_row(std::false_type{}, std::false_type{});
            vz_stage(std::false_type{});
        } else {
            if (xf) own_row(std::true_type{}, std::true_type{});
            else own_row(std::true_type{}, std::false_type{});
            vz_stage(std::true_type{});
        }
        if (cband) cp_async_wait();   // (the barrier makes this group's band values visible to the other lanes)
        // every thread is past the previous group's reads: refill its stage
        if (__syncthreads_or(bad)) {
            fail_j = j;
            break;
        }
        if (j >= 1 && z + 2 * (NS - 1) < zc1) {
            const int jn = j + NS - 1;
            adj_issue<M, FS, WIN>(p, warp, sm + (jn % NS) * L::STAGE, sm + L::B + (jn % NB) * L::F1, bar + jn % NS, slot, xs,
                                  z + 2 * (NS - 1), zc0, tpn, tph);
        }
        ++j;
        if (cband && z + 2 >= zc0) band_fetch(z + 2, j & 1);   // the next group's
        if (main) {
            // ---- rows z, z + 1: half nodes along x
            float pix[2];
            const int bf = (j - 1) & 1;   // band values of this group (j counts the next one by now)
            auto vx_stage = [&](auto zc, auto xc_) {
                constexpr bool ZF = decltype(zc)::value, XF = decltype(xc_)::value;
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const int zr = z + r, cz = zr * pitch, iz = zr - z0;
                    const float2 *const pu = sPU + r * NTH + t;
                    // (Gx, du/dx)
                    const float2 D = stencil<M, float2>(g.cx, [&](int l) { return pu[l]; }, [&](int l) { return pu[1 - l]; });
                    const float2 v2x = *reinterpret_cast<const float2 *>(st2 + L::VX + r * L::F2R);
                    const float *const b = reinterpret_cast<const float *>(brx + r * L::F1R) + t;
                    const float bux = (XF ? 0.5f : hbx) * (b[0] + (!XF && lastx ? b[0] : b[1]));
                    const float dtbu = dt * bux;
                    const float lv = v2x.y + D.y;
                    const bool own = outcol && (ZF || zr < zc1);
                    float wx = __fmul_rn(dtbu, lv);
                    if (!XF && pmlxh) {
                        const float l1 = *reinterpret_cast<const float *>(st1 + L::LPX + r * L::F1R) - wx;
                        // Two roundings of one product, each the one that its instances' results on record have (the
                        // order-8 instance without a free surface was contracted differently): one form for all would
                        // move that instance's images by 2e-7 and the 64-bit misfits of its CGs by 1e-7
                        wx = M == 4 && !FS ? fmaf(dtbu, lv, -__fmul_rn(ahx, l1)) : fmaf(-ahx, l1, wx);
                        if (own) outf[A_LPPX * pT + cz] = bhx * l1;
                    }
                    pix[r] = D.x * lv;
                    float vxn = 0.f;
                    if (XF) {
                        vxn = v2x.x + dtbu * D.x;
                    } else if (ZF || (recon && iz >= 0 && iz < g.nz)) {
                        if (xint) vxn = v2x.x + dtbu * D.x;
                        else if (xband) vxn = band_val(1, bf, r);
                    }
                    if (own) out2[(A_VX / 2) * pT + cz] = make_float2(vxn, lv);
                    sVW[r * NTH + t] = make_float2(v2x.x, wx);
                    sVN[r * NTH + t] = vxn;
                    if ((t & 31) == 31) sPi[r * (NTH / 32) + (t >> 5)] = pix[r];
                }
            };
            if (!zf) vx_stage(std::false_type{}, std::false_type{});
            else if (xf) vx_stage(std::true_type{}, std::true_type{});
            else vx_stage(std::true_type{}, std::false_type{});
            __syncthreads();
            // Gx lvx of the half node to the left: the lane below's, or the
            // last lane's of the warp below (the first warp's first lane
            // owns no output column)
            float pil[2];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                pil[r] = __shfl_up_sync(0xffffffffu, pix[r], 1);
                const float left = sPi[r * (NTH / 32) + max((t >> 5) - 1, 0)];
                if ((t & 31) == 0) pil[r] = left;
            }
            // ---- rows z, z + 1: nodes on the output columns
            auto node_stage = [&](auto zc, auto xc_) {
                constexpr bool ZF = decltype(zc)::value, XF = decltype(xc_)::value;
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const int zr = z + r, cz = zr * pitch, iz = zr - z0;
                    const bool own = outcol && (ZF || zr < zc1);
                    const bool surf = !ZF && FS && zr == z0;   // free-surface row: p = 0, mu = 0
                    const float2 *const vw = sVW + r * NTH + t;
                    const float *const vn = sVN + r * NTH + t;
                    // (Q_n, D- w) along x and z
                    const float2 Ex = stencil<M, float2>(g.cx, [&](int l) { return vw[l - 1]; }, [&](int l) { return vw[-l]; });
                    const float2 Ez = stencil<M, float2>(g.cz, [&](int l) { return VW[r + M + l - 1]; },
                                                         [&](int l) { return VW[r + M - l]; });
                    const float2 E = add_(Ex, Ez);
                    float qn = 0.f;
                    if (ZF || recon)
                        qn = stencil<M, float>(g.cx, [&](int l) { return vn[l - 1]; }, [&](int l) { return vn[-l]; }) +
                             stencil<M, float>(g.cz, [&](int l) { return VN[r + M + l - 1]; },
                                               [&](int l) { return VN[r + M - l]; });
                    const float kd = *reinterpret_cast<const float *>(st1 + L::KD + r * L::F1R);
                    const float lam = own_lam(r, ZF);
                    const bool inner = XF || (xint && (ZF || (iz >= 0 && iz < g.nz)));
                    if (inner) {
                        float2 acc = *reinterpret_cast<const float2 *>(st2 + L::IM + r * L::F2R);
                        acc.x += E.x * lam;
                        // (on the free surface the half row above is a ghost: no product of its own)
                        acc.y += (pix[r] + pil[r]) + (PIZ[r + 1] + (surf ? 0.f : PIZ[r]));
                        if (own) img[cz] = acc;
                    }
                    float pn = 0.f;
                    if (ZF || recon) {
                        if (inner) {
                            pn = pr[r] + kd * qn;
                            pn -= cz + x == src ? wsrc : 0.f;
                        } else if (ZF || (iz >= 0 && iz < g.nz)) {
                            if (xband) pn = band_val(0, bf, r);
                        } else if (xint && in_xstrip(iz, M, g.nz)) {
                            pn = band_get(a.bands, 0, rowprev, band_zstrip(iz, ix, M, g.nz, nx));
                        }
                    }
                    float ln = lam + E.y;
                    if (!ZF && FS && zr <= z0) pn = ln = 0.f;
                    if (own) {
                        out2[(A_PL / 2) * pT + cz] = make_float2(pn, kd * ln);
                        outl[cz] = ln;
                    }
                    const float kl = __fmul_rn(kd, lam);
                    if (!XF && own && pmlxn)
                        outf[A_LPVX * pT + cz] = bix * (*reinterpret_cast<const float *>(st1 + L::LVX + r * L::F1R) - kl);
                    if (!ZF && own && ((zr <= z0 - 1) || (zr >= z1)))
                        outf[A_LPVZ * pT + cz] =
                            a.pml.bi[0][zr] * (*reinterpret_cast<const float *>(st1 + L::IM + r * L::F2R) - kl);
                }
            };
            if (!zf) node_stage(std::false_type{}, std::false_type{});
            else if (xf) node_stage(std::true_type{}, std::true_type{});
            else node_stage(std::true_type{}, std::false_type{});
        }
#pragma unroll
        for (int i = 0; i < W - 1; ++i) {
            PU[i] = PU[i + U];
            VW[i] = VW[i + U];
            VN[i] = VN[i + U];
        }
#pragma unroll
        for (int i = 0; i < M; ++i) PIZ[i] = PIZ[i + U];
    }

    if (cband) cp_async_wait();
    if (fail_j >= 0) {
        // a wait gave up: record it, let the copies in flight land, return
        if (t == NTH - 1) {
            atomicOr(a.err, 1);
            for (int jj = fail_j; jj <= max(NS - 1, fail_j + NS - 2) && zstart + 2 * jj < zc1; ++jj)
                (void)tma::mbar_wait(bar + jj % NS, (unsigned)(jj / NS) & 1u);
        }
        return;
    }

    if (recon) {
        // pre-add the residual of step n-1 at the receivers of this CTA
        __syncthreads();
        const int tile = shot * a.trec.ntiles + blockIdx.y * gridDim.x + blockIdx.x;
        const int b = a.trec.ptr[tile], e = a.trec.ptr[tile + 1];
        float2 *plo = reinterpret_cast<float2 *>(a.out + slot * a.sstride) + (A_PL / 2) * pT;
        float *lo = a.out + slot * a.sstride + A_L * g.plane;
        for (int i = b + t; i < e; i += NTH) {
            const int2 rc = a.trec.rec[i];
            if (i > b && a.trec.rec[i - 1].x == rc.x) continue;  // run handled by its first entry
            float add = 0.f;
            for (int q = i; q < e && a.trec.rec[q].x == rc.x; ++q)
                add += a.dstage[(long long)a.trec.rec[q].y * g.nt + (n - 1)];
            const float l = lo[rc.x] + add;
            lo[rc.x] = l;
            plo[rc.x].y = kdt[rc.x] * l;
        }
    }
}

// Migration step of shots spanning the model and of shots with aperture windows.
template <int M, bool FS>
__global__ void __launch_bounds__(NTH, kAdjMinBlocks) k_adj2t(const __grid_constant__ Arg2D p)
{
    adj_body<M, false, FS>(p);
}
template <int M, bool FS>
__global__ void __launch_bounds__(NTH, kAdjMinBlocks) k_adj2d(const __grid_constant__ Arg2D p)
{
    adj_body<M, true, FS>(p);
}

// Start state of a reverse pass: (p, 0), (vx, 0), (vz, 0) from the saved
// background final state [p][vx][vz] of each shot of the batch.
__global__ void k_pack_adj(const GridDev g, const float *final_state, int shot0, int batch, float *st,
                           long long sstride)
{
    const long long plane = g.plane;
    const long long n = batch * plane;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const long long s = i / plane, c = i - s * plane;
        const float *fs = final_state + (shot0 + s) * 3 * plane;
        float2 *o = reinterpret_cast<float2 *>(st + s * sstride);
        o[(A_PL / 2) * plane + c] = make_float2(fs[c], 0.f);
        o[(A_VX / 2) * plane + c] = make_float2(fs[plane + c], 0.f);
        o[(A_VZ / 2) * plane + c] = make_float2(fs[2 * plane + c], 0.f);
    }
}

__global__ void k_window_model(const GridDev gm, const GridDev g, const int *win_x0, const int *win_nx, int shot0,
                               int batch, const float *kdt, const float *binv, const float2 *kd2,
                               const float2 *br2, float *st0, float *st1, long long sstride)
{
    const long long plane = g.plane;
    const long long n = (long long)batch * plane;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const int slot = (int)(i / plane);
        const long long c = i - (long long)slot * plane;
        const int z = (int)(c / g.pitch), x = (int)(c - (long long)z * g.pitch);
        const int shot = shot0 + slot;
        const int nxw = win_nx[shot], Nxw = nxw + 2 * g.x0;
        float k = 0.f, b = 0.f;
        float2 k2 = make_float2(0.f, 0.f), b2 = make_float2(0.f, 0.f);
        if (x < Nxw) {
            const int xi = min(max(x - g.x0, 0), nxw - 1);
            const long long cm = (long long)z * gm.pitch + gm.x0 + win_x0[shot] + xi;
            const bool inner = x >= g.x0 && x < g.x0 + nxw;
            k = kdt[cm];
            b = binv[cm];
            if (kd2) {
                k2 = kd2[cm];
                b2 = br2[cm];
                if (!inner) {
                    k2.y = 0.f;
                    b2.y = 0.f;
                }
            }
        }
        for (int q = 0; q < 2; ++q) {
            float *o = (q ? st1 : st0) + slot * sstride;
            o[W_KDT * plane + c] = k;
            o[W_BINV * plane + c] = b;
            if (kd2) {
                reinterpret_cast<float2 *>(o + W_KD2 * plane)[c] = k2;
                reinterpret_cast<float2 *>(o + W_BR2 * plane)[c] = b2;
            }
        }
    }
}


template <class K>
cudaError_t set_smem(K k, unsigned bytes)
{
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

// Calls f(WIN, FS) as compile-time constants.
template <class F>
cudaError_t with_flags(bool win, bool fs, F &&f)
{
    using T = std::true_type;
    using N = std::false_type;
    if (win) return fs ? f(T{}, T{}) : f(T{}, N{});
    return fs ? f(N{}, T{}) : f(N{}, N{});
}

template <int M, bool BANDS, bool HESS>
cudaError_t launch_bg(const Arg2D &p, dim3 grid, cudaStream_t s)
{
    return with_flags(p.a.win_nx != nullptr, p.a.g.fs != 0, [&](auto w, auto f) {
        k_fwd2d<M, BANDS, HESS, decltype(w)::value, decltype(f)::value><<<grid, NTH, FwdLay<M, false, HESS>::SMEM, s>>>(p);
        return cudaGetLastError();
    });
}

template <int M>
cudaError_t launch_fwd_M(const Arg2D &p, int batch, bool born, bool bands, bool hess, cudaStream_t s)
{
    const Step2D &a = p.a;
    const dim3 grid((a.g.Nx + Cols<M>::TXO - 1) / Cols<M>::TXO, (a.g.Nz + a.tzc - 1) / a.tzc, batch);
    if (born)
        return with_flags(a.win_nx != nullptr, a.g.fs != 0, [&](auto w, auto f) {
            if constexpr (decltype(w)::value) k_fwd2w<M, decltype(f)::value><<<grid, NTH, FwdLay<M, true, false>::SMEM, s>>>(p);
            else k_fwd2t<M, decltype(f)::value><<<grid, NTH, FwdLay<M, true, false>::SMEM, s>>>(p);
            return cudaGetLastError();
        });
    if (bands && hess) return launch_bg<M, true, true>(p, grid, s);
    if (bands) return launch_bg<M, true, false>(p, grid, s);
    if (hess) return launch_bg<M, false, true>(p, grid, s);
    return launch_bg<M, false, false>(p, grid, s);
}

template <int M>
cudaError_t launch_adj_M(const Arg2D &p, int batch, cudaStream_t s)
{
    const Step2D &a = p.a;
    const dim3 grid((a.g.Nx + Cols<M>::TXO - 1) / Cols<M>::TXO, (a.g.Nz + a.tzc - 1) / a.tzc, batch);
    return with_flags(a.win_nx != nullptr, a.g.fs != 0, [&](auto w, auto f) {
        if constexpr (decltype(w)::value) k_adj2d<M, decltype(f)::value><<<grid, NTH, AdjLayM<M>::SMEM, s>>>(p);
        else k_adj2t<M, decltype(f)::value><<<grid, NTH, AdjLayM<M>::SMEM, s>>>(p);
        return cudaGetLastError();
    });
}

template <int M>
cudaError_t attr_M()
{
    cudaError_t e = cudaSuccess;
    auto set = [&](auto k, unsigned bytes) {
        if (e == cudaSuccess) e = set_smem(k, bytes);
    };
    for (int i = 0; i < 4; ++i)
        with_flags(i & 1, i & 2, [&](auto w, auto f) {
            constexpr bool WIN = decltype(w)::value, FS = decltype(f)::value;
            set(k_fwd2d<M, true, true, WIN, FS>, FwdLay<M, false, true>::SMEM);
            set(k_fwd2d<M, true, false, WIN, FS>, FwdLay<M, false, false>::SMEM);
            set(k_fwd2d<M, false, true, WIN, FS>, FwdLay<M, false, true>::SMEM);
            set(k_fwd2d<M, false, false, WIN, FS>, FwdLay<M, false, false>::SMEM);
            if constexpr (WIN) {
                set(k_fwd2w<M, FS>, FwdLay<M, true, false>::SMEM);
                set(k_adj2d<M, FS>, AdjLayM<M>::SMEM);
            } else {
                set(k_fwd2t<M, FS>, FwdLay<M, true, false>::SMEM);
                set(k_adj2t<M, FS>, AdjLayM<M>::SMEM);
            }
            return cudaSuccess;
        });
    return e;
}

}  // namespace

int march2d_txo(int M) { return M == 2 ? Cols<2>::TXO : Cols<4>::TXO; }

// A chunk of t rows costs its CTA t + 2M rows (the warm-up ones included) and a
// start of about 7 rows' time (barriers, first copies, the ring's prologue).
// Up to three CTAs share an SM almost for free (a CTA alone waits for its own
// latencies most of the time: 1.1x its time with two on the SM, 1.25x with
// three), so a small batch is split until every SM has one to three CTAs: 1
// shot of 141 x 141 (order 4) 258 us a Born and migration step in one chunk, 23
// in chunks of 4; 16 shots of 240 x 240 209 -> 46 (10 rows); 12 shots of 227 x
// 451 (order 8) 284 -> 77 (12 rows). Past three, the starts hide behind other
// CTAs and what counts is the work repeated and the last wave (0.7 of one on
// average): 96 shots of 424 x 1192 take 1483 us in chunks of 106 rows, 1453 in
// 72, 1484 in 40, 1763 in 14.
int march2d_rows(int M, int Nz, long long ctas)
{
    constexpr double sms = 152.0, three = 1.25;
    double best = 1e300;
    int rows = Nz;
    for (int nc = 1; nc <= std::max(1, Nz / 2); ++nc) {
        int t = (Nz + nc - 1) / nc;
        t += t & 1;   // whole groups of two rows
        const double n = (double)ctas * ((Nz + t - 1) / t), q = std::ceil(n / sms);
        const double c = q <= 3.0 ? (t + 2 * M + 7) * (q <= 1.0 ? 1.0 : (q <= 2.0 ? 1.1 : three))
                                  : (t + M + 3) * three * (n / (3.0 * sms) + 0.7);
        if (c < best) {
            best = c;
            rows = t;
        }
    }
    return rows;
}

cudaError_t configure_2d_kernels()
{
    cudaError_t e = attr_M<2>();
    if (e != cudaSuccess) return e;
    return attr_M<4>();
}

// Kernel attributes are per device: a flag per device index, set under a
// mutex the first time a thread with that device current asks.
cudaError_t ensure_kernels_configured()
{
    constexpr int kMaxDev = 64;
    static bool done[kMaxDev] = {};
    static std::mutex mu;
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDev) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    if (done[dev]) return cudaSuccess;
    if ((e = configure_2d_kernels()) != cudaSuccess) return e;
    if ((e = configure_3d_kernels()) != cudaSuccess) return e;
    done[dev] = true;
    return cudaSuccess;
}

cudaError_t launch_fwd2d(const Step2D &a, const Maps2D &maps, int batch, bool born, bool save_bands, bool hess, cudaStream_t s)
{
    if (!a.err) return cudaErrorInvalidValue;
    const Arg2D p{a, maps};
    if (a.g.M == 2) return launch_fwd_M<2>(p, batch, born, save_bands, hess, s);
    return launch_fwd_M<4>(p, batch, born, save_bands, hess, s);
}

cudaError_t launch_adj2d(const Step2D &a, const Maps2D &maps, int batch, cudaStream_t s)
{
    if (!a.err) return cudaErrorInvalidValue;
    const Arg2D p{a, maps};
    if (a.g.M == 2) return launch_adj_M<2>(p, batch, s);
    return launch_adj_M<4>(p, batch, s);
}

cudaError_t maps2d(Maps2D *m, const GridDev &gm, const GridDev &g, const float *st, long long sstride, int planes,
                   const float *kdt, const float *binv, const float2 *kd2, const float2 *br2, const float2 *img,
                   const float *psiv, long long vstride, int batch)
{
    // the two model arrays of each kind are one map: their planes must be adjacent
    if (binv != kdt + gm.plane || br2 != kd2 + gm.plane) return cudaErrorInvalidValue;
    // (the pair map of a slot with an odd number of planes, a background-only
    // state, is never read)
    m->pps = (int)(sstride / (2 * g.plane));
    m->fps = (int)(sstride / g.plane);
    const auto u64 = CU_TENSOR_MAP_DATA_TYPE_UINT64, f32 = CU_TENSOR_MAP_DATA_TYPE_FLOAT32;
    const cuuint64_t s8[2] = {(cuuint64_t)g.pitch * 8, (cuuint64_t)g.plane * 8};
    const cuuint64_t s4[2] = {(cuuint64_t)g.pitch * 4, (cuuint64_t)g.plane * 4};
    const cuuint64_t nx = (cuuint64_t)g.Nx, nz = (cuuint64_t)g.Nz;
    const cuuint64_t dpr[3] = {nx, nz, (cuuint64_t)((batch - 1LL) * m->pps + planes / 2)};
    const cuuint64_t dfl[3] = {nx, nz, (cuuint64_t)((batch - 1LL) * m->fps + planes)};
    const cuuint64_t dim[3] = {nx, nz, (cuuint64_t)batch};
    // the model grid (without aperture windows the slots' own grid)
    const cuuint64_t dmd[3] = {(cuuint64_t)gm.Nx, (cuuint64_t)gm.Nz, 2};
    const cuuint64_t m8[2] = {(cuuint64_t)gm.pitch * 8, (cuuint64_t)gm.plane * 8};
    const cuuint64_t m4[2] = {(cuuint64_t)gm.pitch * 4, (cuuint64_t)gm.plane * 4};
    for (int r = 0; r < 2; ++r) {
        const cuuint32_t box[3] = {(cuuint32_t)NTH, (cuuint32_t)(r + 1), 1};
        cudaError_t e;
        if ((e = encode_tmap(&m->pr[r], u64, 3, st, dpr, s8, box)) != cudaSuccess) return e;
        if ((e = encode_tmap(&m->fl[r], f32, 3, st, dfl, s4, box)) != cudaSuccess) return e;
        if ((e = encode_tmap(&m->md[r], f32, 3, kdt, dmd, m4, box)) != cudaSuccess) return e;
        if ((e = encode_tmap(&m->mb[r], u64, 3, kd2, dmd, m8, box)) != cudaSuccess) return e;
        // two-row boxes over its floats and its pairs
        const cuuint64_t spv[2] = {(cuuint64_t)g.pitch * (r ? 8 : 4), (cuuint64_t)vstride * 4};
        const cuuint32_t box2[3] = {(cuuint32_t)NTH, 2, 1};
        if ((e = encode_tmap(&m->pv[r], r ? u64 : f32, 3, psiv, dim, spv, box2)) != cudaSuccess) return e;
        if (img && (e = encode_tmap(&m->im[r], u64, 3, img, dim, s8, box)) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_window_model(const GridDev &gm, const GridDev &g, const int *win_x0, const int *win_nx,
                                int shot0, int batch, const float *kdt, const float *binv, const float2 *kd2,
                                const float2 *br2, float *st0, float *st1, long long sstride, cudaStream_t s)
{
    long long n = batch * g.plane;
    int blocks = (int)std::min<long long>((n + 255) / 256, 152 * 16);
    k_window_model<<<blocks, 256, 0, s>>>(gm, g, win_x0, win_nx, shot0, batch, kdt, binv, kd2, br2, st0, st1,
                                          sstride);
    return cudaGetLastError();
}

cudaError_t launch_pack_adjoint(const GridDev &g, const float *final_state, int shot0, int batch, float *st,
                                long long sstride, cudaStream_t s)
{
    long long n = batch * g.plane;
    int blocks = (int)std::min<long long>((n + 255) / 256, 152 * 16);
    k_pack_adj<<<blocks, 256, 0, s>>>(g, final_state, shot0, batch, st, sstride);
    return cudaGetLastError();
}

}  // namespace lsrtm
