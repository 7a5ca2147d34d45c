// flr_fused.cu -- the whole FLR forward pass in one kernel (sm_103a): windowed moments,
// per-pixel centred ridge solve, coefficient averaging and apply.
//
// What it computes (arXiv 2410.11625, Sec. 3.1-3.2 and the Appendix): for every pixel k, the
// box sums over the clipped radius-r window of the linear moments and of the outer products
// x x^T, x y^T (box-filtering the outer products gives X_k^T X_k and X_k^T Y_k exactly), the
// centred ridge model a_k = (W_k + eps I)^{-1} (X^T Y / n - mu_X mu_Y^T), b_k = mu_Y - a_k^T mu_X
// (the Appendix's decomposition with eps on the diagonal of W), then the mean of the models
// over the clipped radius-rc window around each output pixel i, applied to its map-guide
// vector: I_i = mean_k b_k + (mean_k a_k)^T z_i.  With rc = 0 the pixel's own model is
// applied (Sec. 3.1, I_k = x_k A_k).
//
// Work layout.  One CTA owns a strip of TW output columns and a segment of output rows and
// walks down it kB rows per batch.  It solves TS = TW + 2 rc columns (the models its averaging
// window needs) over the rows [y0 - rc, y1 + rc), and sums moments over TM = TS + 2 r columns.
// Three teams of warps work on different batches at a time, handing over through named barriers:
//   1. V-pass (walkers): one thread per (pair of adjacent columns, quarter of the channels) keeps
//      vertical window sums of its channels in registers, as two accumulators per channel: E,
//      the products of the rows entered since the last block start, and Dn, the products of the
//      rows left since then minus the previous block's total.  A block is 2r + 1 rows, so
//      V = E - Dn is always a sum of at most 2(2r + 1) rounded terms: the error does not grow
//      along the strip.  Products are recomputed from TMA-staged entering and leaving rows.
//   2. H-pass (walkers; without averaging summers): the horizontal radius-r sums of every channel
//      row, in place, two runs per row, each re-seeded by a direct (2r + 1)-term sum.
//   3. Solve (solvers): one thread per two pixels, packed: centred, unnormalised moments
//      (n M = S - L mu^T + n eps I), Cholesky in registers, three right-hand sides.  A pixel
//      whose pivot ratio falls to tau or below is listed for an FP64 re-solve and left out of the
//      average (its FP64 model is added by flr_fused_fix_kernel).
//   4. Coefficient H-pass (summers): horizontal radius-rc sums of the 3(Q+1) model coefficients.
//   5. Coefficient V-pass and apply (summers): one thread per (pair of output columns, colour)
//      keeps the vertical radius-rc sums of its Q + 1 coefficients with the same block
//      accumulators; the rows that leave its window come from a ring of 2rc + 1 rows kept in tensor
//      memory.
// What bounds it.  At 1920x1080, r = rc = 8: 0.290 ms a launch (0.347 ms as one team of 12 warps
// going through the phases between CTA barriers, at 53% issue with every phase waiting for its own
// latency; 160 M against 207 M warp instructions), shared memory 57% and issue 48% busy, the rest
// the teams' waits for one another: walkers alone 234 us, solvers alone 150.  Packed FP32
// (fma.rn.f32x2) is used throughout for its halved issue slots.  Also measured: scalar walkers and
// solvers in two teams 347 us; the H-pass by 128 threads beside the apply 338 and in half rows by
// twice the threads 364; 4 walker warps of 36 channels 364; the coefficient H-pass by the solvers
// 435; prefetching rows into L2 no change.
// Values are shifted by the mean of a 16 x 16 sample grid of the CTA's input region before
// any product (the centred form is shift-invariant), and the models are applied in the same
// shifted coordinates, so no frame-wide reference is needed.
#include <cstring>
#include <mutex>
#include <utility>

#include "flr_device.cuh"
#include "flr_fp64_model.cuh"
#include "flr_internal.cuh"
#include "flr_tmem.cuh"
#include "pdl.cuh"
#include "tma.cuh"

namespace flr {
namespace fused {

constexpr int kB = 2;                     // rows per batch
constexpr int kTS = 96;                   // solve columns
constexpr int kStages = 3;                // buffers of staged input rows
// Teams: 8 warps of walkers, 3 of solvers (one thread per two pixels of a batch) and a helper warp,
// 4 of summers; and the registers a thread of each is given (setmaxnreg by groups of four warps:
// 256 x 120 + 128 x 168 + 128 x 104 = the 512 x 128 of the launch)
constexpr int kWalkers = 256, kSolvers = 96, kSummers = 128;
constexpr int kThreads = kWalkers + kSolvers + 32 + kSummers;
constexpr int kWalkRegs = 120, kSolveRegs = 168, kSumRegs = 104;
static_assert(kWalkers * kWalkRegs + (kSolvers + 32) * kSolveRegs + kSummers * kSumRegs <= 512 * 128, "register file");
static_assert(kB * kTS / 2 <= kSolvers, "one solver thread per pair of pixels");
constexpr unsigned long long kTimeoutNs = 1000000000ull;  // 1 s per bounded wait

__host__ __device__ constexpr int tile_width(int rc) { return (kTS - 2 * rc) & ~3; }

// ---- walker groups -------------------------------------------------------------------
// The NCH moment channels (numbered as in Chan) fall into rows that share their left factor:
// the linear moments (left factor 1: x_0..x_{Q-1}, y_0..y_2) and, for each guide u, the
// products x_u x_v (v = u..Q-1) and x_u y_c, whose right factors are the input slots u..Q+2.
// A walker thread keeps the vertical sums of one group of rows for a pair of adjacent columns, in
// registers: the packed FMAs (fma.rn.f32x2) take their operands straight from 8-byte shared loads.
// Four groups of two warps: the linear row and row 4 (18 channels of 11 slots), rows {0, 5} (17 of
// 11), {1, 3} (18 of 10) and {2, 6, 7} (18 of 9).
template <int Q>
struct Groups {
    static_assert(Q == 8, "the walker groups are laid out for eight guides");
    static constexpr int NG = 4, MAXG = 18;
    // the k-th left factor of group g (-1: the linear row; -2: none)
    __host__ __device__ static constexpr int row(int g, int k)
    {
        return g == 0 ? (k == 0 ? -1 : k == 1 ? 4 : -2) : g == 1 ? (k == 0 ? 0 : k == 1 ? 5 : -2) : g == 2 ? (k == 0 ? 1 : k == 1 ? 3 : -2)
                                                                                                     : (k == 0 ? 2 : k == 1 ? 6 : k == 2 ? 7 : -2);
    }
    __host__ __device__ static constexpr int row_len(int u) { return u < 0 ? Q + 3 : Q + 3 - u; }
    __host__ __device__ static constexpr int size(int g)
    {
        int n = 0;
        for (int k = 0; row(g, k) != -2; ++k) n += row_len(row(g, k));
        return n;
    }
    // the i-th channel of group g
    __host__ __device__ static constexpr int ch(int g, int i)
    {
        int k = 0;
        while (i >= row_len(row(g, k))) i -= row_len(row(g, k++));
        const int u = row(g, k);
        if (u < 0) return i < Q ? Chan<Q>::X0 + i : Chan<Q>::Y0 + (i - Q);
        const int v = u + i;
        return v < Q ? Chan<Q>::xx(u, v) : Chan<Q>::xy(u, v - Q);
    }
    __host__ __device__ static constexpr int s0(int g) { return g == 0 ? 0 : row(g, 0); }  // lowest slot read
};

// Compile-time geometry of one instantiation.
template <int Q, int R, int RC>
struct Geo {
    static constexpr int NS = Q + 3;
    static constexpr int NCH = Chan<Q>::NCH;
    static constexpr int NCF = 3 * (Q + 1);       // model coefficients per pixel
    static constexpr int TW = tile_width(RC);     // output columns
    static constexpr int TS = TW + 2 * RC;        // solve columns
    static constexpr int TM = TS + 2 * R;         // walker columns
    static constexpr int NCP = TM / 2;            // walker column pairs
    static constexpr int RA = (R + RC + 3) & ~3;  // staged rows start at column x0 - RA
    // staged row length: covers TW + 2 RA columns, and kB rows of it are a multiple of 128
    // bytes, so every TMA box of the staging buffer starts 128-byte aligned
    static constexpr int WSt = (TW + 2 * RA + 7) & ~7;
    static constexpr int SOFF = RA - R - RC;      // staged column of walker column 0
    static constexpr int VS = TM + ((12 - TM % 8) % 8);  // row stride >= TM, = 4 (mod 8)
    static constexpr int WR = 2 * R + 1, WC = 2 * RC + 1;
    // H-pass runs [0, CH), [CH, 2 CH) and coefficient H-pass runs [0, CL), [CL, 2 CL): equal, so
    // that one copy of the code serves both (the sums past TS and TW are of stale columns inside
    // the buffer rows, and nothing reads them)
    static constexpr int CH = (TS / 2 + 3) & ~3;
    // horizontally summed coefficient rows, in a buffer of their own so that a batch's apply runs
    // beside the next batch's V-pass; row stride 4 (mod 8)
    static constexpr int CL = (TW / 2 + 3) & ~3;
    static constexpr int CS = 2 * CL + ((12 - 2 * CL % 8) % 8);
    static constexpr size_t CBUF_FLOATS = RC > 0 ? ((size_t)kB * NCF * CS + 31) / 32 * 32 : 0;
    static constexpr size_t VBUF_FLOATS = ((size_t)kB * NCH * VS + 31) / 32 * 32;
    static constexpr size_t STAGE_FLOATS = (size_t)2 * NS * kB * WSt;
    // map-guide rows of a batch's output rows (the apply reads them)
    static constexpr size_t ZBUF_FLOATS = RC > 0 ? ((size_t)Q * kB * TW + 31) / 32 * 32 : 0;
    static constexpr unsigned ZBYTES = (unsigned)(Q * kB * TW * 4);
    static constexpr size_t SMEM = 128 + 4 * (2 * VBUF_FLOATS + kStages * STAGE_FLOATS + 3 * ZBUF_FLOATS + CBUF_FLOATS) + (kStages + 3) * 8 + 16;
    static_assert(SMEM <= 227 * 1024, "shared memory of one CTA");
    static_assert(TS <= kTS && TM <= 112 && WSt <= 112, "strip geometry");
    static_assert((kB * WSt * 4) % 128 == 0 && (VBUF_FLOATS * 4) % 128 == 0, "TMA boxes 128-byte aligned");
    static_assert(SOFF + TM <= WSt, "walker columns inside the staged rows");
    static_assert((R + RC) % 2 == 0 && SOFF % 2 == 0 && TM % 2 == 0 && TS % 2 == 0 && TW % 2 == 0, "column pairs at even columns");
    static_assert(NCP <= 64, "two warps of walkers per group");
    static_assert(kB * NCH <= kSummers + 32, "H-pass rows");
    static_assert(CH > 2 * R && CH < TS && CL < TW, "H-pass runs");
    static_assert(2 * CH >= TS && 2 * CL >= TW && 2 * CH + 2 * R <= VS && 2 * CL + 2 * RC <= VS, "runs inside the rows");
    static_assert(RC == 0 || 2 * CL <= CS, "runs inside the coefficient rows");
    static_assert(RC == 0 || (WC <= 17 && 3 * (TW / 2) <= kSummers), "coefficient ring");
    static_assert(Q + 1 == 9, "ring slots of 18 and a state of 36 tensor-memory columns");
};

// Tensor-memory columns of an applier thread (its lane of 512; every access aligned to its width):
// ring slot s at 16 s (x16) and 272 + 2 s (x2), the 36 accumulators at 320 (x32) and 352 (x4).
constexpr uint32_t kTmemCols = 512, kColRing2 = 272, kColState = 320;

__device__ __forceinline__ float2 ld2(const float *p) { return *reinterpret_cast<const float2 *>(p); }
__device__ __forceinline__ void st2(float *p, float2 v) { *reinterpret_cast<float2 *>(p) = v; }
__device__ __forceinline__ float2 neg2(float2 v) { return make_float2(-v.x, -v.y); }

// ---- V-pass: one group of channels, two columns ---------------------------------------
// E += left(e) * right(e), Dn += left(l) * right(l), V = E - Dn for every channel of group G;
// e and l: the shifted values of the entering and the leaving row at the two columns.
template <int Q, int G, int I>
__device__ __forceinline__ void walk_add(float2 (&E)[Groups<Q>::MAXG], const float2 (&e)[Q + 3])
{
    constexpr int c = Groups<Q>::ch(G, I);
    constexpr int u = Chan<Q>::slot_u(c), v = Chan<Q>::slot_v(c);
    if constexpr (v < 0) E[I] = __fadd2_rn(E[I], e[u]);
    else E[I] = __ffma2_rn(e[u], e[v], E[I]);
}
// se: the staged entering row of this batch row at the walker's first column; planes are
// kB * WST floats apart, the leaving rows NS planes further on.
template <int Q, int G, int WST, int... I>
__device__ __forceinline__ void walk_rows(float2 (&E)[Groups<Q>::MAXG], float2 (&Dn)[Groups<Q>::MAXG], float *vcol, int VS,
                                         const float *se, const float (&nsh)[Q + 3], bool ein, bool lout, bool store,
                                         std::integer_sequence<int, I...>)
{
    constexpr int NS = Q + 3, S0 = Groups<Q>::s0(G);
    constexpr size_t PL = (size_t)kB * WST;
    float2 e[NS];
    if (ein) {
#pragma unroll
        for (int k = S0; k < NS; ++k) e[k] = __fadd2_rn(ld2(se + k * PL), make_float2(nsh[k], nsh[k]));
        (walk_add<Q, G, I>(E, e), ...);
    }
    if (lout) {
        const float *sl = se + NS * PL;
#pragma unroll
        for (int k = S0; k < NS; ++k) e[k] = __fadd2_rn(ld2(sl + k * PL), make_float2(nsh[k], nsh[k]));
        (walk_add<Q, G, I>(Dn, e), ...);
    }
    if (store) (st2(vcol + (size_t)Groups<Q>::ch(G, I) * VS, __ffma2_rn(Dn[I], make_float2(-1.f, -1.f), E[I])), ...);
}

// ---- solve ---------------------------------------------------------------------------------
// Centred ridge models of two neighbouring pixels from their window sums S(ch) = col[ch * VS], [+ 1]
// (moment channels, Chan order), packed (fma.rn.f32x2): the solve is bound by instruction issue and
// latency, and a packed instruction does both pixels.  Unnormalised form n M = S - L mu^T + n eps I,
// n D = XY - L_y mu^T (the same a as M^{-1} D).  model_factor centres and factors n M, column by
// column with the trailing matrix updated at once, so that consecutive instructions are
// independent; low0/low1: whether a Cholesky pivot ratio d_j / (n M)_jj fell to tau or below.
// model_rhs solves for the three colours side by side.
template <int Q>
struct Factor {
    float2 nmu[Q], L[Q * (Q - 1) / 2], inv_d[Q];  // minus the guide means, strict lower triangle, 1 / L_jj
};
__device__ __forceinline__ constexpr int low_tri(int i, int j) { return i * (i - 1) / 2 + j; }  // i > j
template <int Q, int VS>
__device__ __forceinline__ void model_factor(const float *col, float2 n, float2 inv_n, float eps, float tau, Factor<Q> &f,
                                             bool &low0, bool &low1)
{
    using C = Chan<Q>;
    float2 sx[Q], D[Q];  // D: the diagonal
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        sx[i] = ld2(col + (C::X0 + i) * VS);
        f.nmu[i] = __fmul2_rn(sx[i], make_float2(-inv_n.x, -inv_n.y));
    }
    const float2 ne = make_float2(n.x * eps, n.y * eps);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        D[i] = __fadd2_rn(__ffma2_rn(f.nmu[i], sx[i], ld2(col + C::xx(i, i) * VS)), ne);
#pragma unroll
        for (int j = 0; j < Q; ++j)
            if (j < i) f.L[low_tri(i, j)] = __ffma2_rn(f.nmu[i], sx[j], ld2(col + C::xx(j, i) * VS));
    }
    low0 = low1 = false;
    const float dmin0 = ne.x > 0.f ? ne.x : 1e-30f, dmin1 = ne.y > 0.f ? ne.y : 1e-30f;  // every exact pivot is >= n eps
    float2 thr[Q];
#pragma unroll
    for (int j = 0; j < Q; ++j) thr[j] = make_float2(tau * D[j].x, tau * D[j].y);
#pragma unroll
    for (int j = 0; j < Q; ++j) {
        low0 |= !(D[j].x > thr[j].x);
        low1 |= !(D[j].y > thr[j].y);
        const float2 il = make_float2(rsqrtf(fmaxf(D[j].x, dmin0)), rsqrtf(fmaxf(D[j].y, dmin1)));
        f.inv_d[j] = il;
#pragma unroll
        for (int i = 0; i < Q; ++i)
            if (i > j) f.L[low_tri(i, j)] = __fmul2_rn(f.L[low_tri(i, j)], il);
#pragma unroll
        for (int i = 0; i < Q; ++i)
            if (i > j) {
                const float2 nl = neg2(f.L[low_tri(i, j)]);
                D[i] = __ffma2_rn(nl, f.L[low_tri(i, j)], D[i]);
#pragma unroll
                for (int k = 0; k < Q; ++k)
                    if (k > j && k < i) f.L[low_tri(i, k)] = __ffma2_rn(nl, f.L[low_tri(k, j)], f.L[low_tri(i, k)]);
            }
    }
}
// a and b of the three colours side by side: ys the radiance sums, xy the guide-radiance sums
template <int Q, int VS>
__device__ __forceinline__ void model_rhs(const Factor<Q> &f, const float2 (&ys)[3], const float *xy, float2 inv_n,
                                          float2 (&A)[3][Q], float2 (&b)[3])
{
#pragma unroll
    for (int i = 0; i < Q; ++i)
#pragma unroll
        for (int c = 0; c < 3; ++c) A[c][i] = __ffma2_rn(f.nmu[i], ys[c], ld2(xy + (3 * i + c) * VS));
#pragma unroll
    for (int j = 0; j < Q; ++j) {  // L z = n D
        float2 nz[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            A[c][j] = __fmul2_rn(A[c][j], f.inv_d[j]);
            nz[c] = neg2(A[c][j]);
        }
#pragma unroll
        for (int i = 0; i < Q; ++i)
#pragma unroll
            for (int c = 0; c < 3; ++c)
                if (i > j) A[c][i] = __ffma2_rn(f.L[low_tri(i, j)], nz[c], A[c][i]);
    }
#pragma unroll
    for (int jj = 0; jj < Q; ++jj) {  // L^T a = z
        const int j = Q - 1 - jj;
        float2 na[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            A[c][j] = __fmul2_rn(A[c][j], f.inv_d[j]);
            na[c] = neg2(A[c][j]);
        }
#pragma unroll
        for (int i = 0; i < Q; ++i)
#pragma unroll
            for (int c = 0; c < 3; ++c)
                if (i < j) A[c][i] = __ffma2_rn(f.L[low_tri(j, i)], na[c], A[c][i]);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        b[c] = __fmul2_rn(ys[c], inv_n);
#pragma unroll
        for (int i = 0; i < Q; ++i) b[c] = __ffma2_rn(A[c][i], f.nmu[i], b[c]);
    }
}

// ---- team barriers ---------------------------------------------------------------------
// Named barriers (0 is __syncthreads).  A signal is arrived at by one team and waited for by
// another; index k & 1 alternates with the buffer slot.
enum Bar { kBarWalk = 1, kBarSolve = 2, kBarSum = 3, kBarWalked = 4, kBarFull = 6, kBarModels = 8, kBarFree = 10 };
// With averaging the walkers do the H-pass themselves and the summers the coefficient passes;
// without it the summers (and the solvers' fourth warp: a batch has 142 rows) do the H-pass.  At
// 1920x1080, rc = 8 the H-pass takes 296 us a frame with the walkers and 338 with the summers, whose
// next coefficient sums then come late; at 3840x2160, rc = 0 802 and 750.
template <int RC>
struct Roles {
    static constexpr bool kWalkersSum = RC > 0;
    static constexpr int kWalked = kWalkers + kSummers + 32;                                    // walkers -> summers, helper
    static constexpr int kFull = (kWalkersSum ? kWalkers : kSummers + 32) + kSolvers;           // those -> solvers
    static constexpr int kModels = kSolvers + kSummers;                                         // solvers -> summers
    static constexpr int kFree = (RC > 0 ? kSummers : kSolvers) + kWalkers;                     // slot free -> walkers
};
__device__ __forceinline__ void bar_sync(int id, int n) { asm volatile("barrier.cta.sync %0, %1;\n" ::"r"(id), "r"(n) : "memory"); }
__device__ __forceinline__ void bar_arrive(int id, int n) { asm volatile("barrier.cta.arrive %0, %1;\n" ::"r"(id), "r"(n) : "memory"); }
__device__ __forceinline__ bool bar_or(int id, int n, bool p)
{
    uint32_t r;
    asm volatile("{\n.reg .pred p, q;\nsetp.ne.u32 q, %3, 0;\nbarrier.cta.red.or.pred p, %1, %2, q;\nselp.u32 %0, 1, 0, p;\n}\n"
                 : "=r"(r)
                 : "r"(id), "r"(n), "r"((uint32_t)p)
                 : "memory");
    return r != 0;
}

// Kernel parameters: TMA maps of the guide [Q][H][W] and radiance [3][H][W] planes (boxes of
// WSt columns x kB rows x all planes) and the arguments.
struct alignas(128) KArgs {
    CUtensorMap tg, tr, tz;  // tz: the map guide, boxes of TW columns x kB rows x Q planes
    FusedArgs a;
};

template <int Q, int R, int RC>
__global__ void __launch_bounds__(kThreads, 1) flr_fused_kernel(const __grid_constant__ KArgs ka)
{
    using G = Geo<Q, R, RC>;
    using C = Chan<Q>;
    using T = Roles<RC>;
    constexpr int NS = G::NS, NCH = G::NCH, NCF = G::NCF;
    constexpr int TW = G::TW, TS = G::TS, WSt = G::WSt, VS = G::VS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ float s_sh[NS];
    __shared__ int s_abort, s_nlist, s_wcnt[kSolvers / 32];
    __shared__ uint32_t s_tmem;
    const FusedArgs &a = ka.a;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int H = a.H, W = a.W;
    const size_t plane = (size_t)H * W;
    const int x0 = blockIdx.x * TW;
    const int row_hi = a.row_hi < 0 ? H : min(a.row_hi, H);
    const int y0 = a.row_lo + blockIdx.y * a.TH;
    const int y1 = min(y0 + a.TH, row_hi);
    const int cta = blockIdx.y * gridDim.x + blockIdx.x;
    if (y0 >= y1) {  // a segment past the last row (not produced by the host plan)
        pdl::wait();
        if (tid == 0) a.list_count[cta] = 0;
        return;
    }
    const int m_lo = y0 - RC, m_hi = y1 + RC;  // solve rows
    const int v0 = m_lo - 2 * R;               // first walker row: the window starts empty
    const int nlive = (m_hi - m_lo + kB - 1) / kB, nbatch = R + nlive;  // batches; the first R only fill the window

    unsigned char *base = smem_raw + ((128 - (tma::smem_addr(smem_raw) & 127)) & 127);
    float *Vbuf = reinterpret_cast<float *>(base);  // [2][kB][NCH][VS]: channel rows
    float *stage = Vbuf + 2 * G::VBUF_FLOATS;        // [kStages][2][NS][kB][WSt]: entering, leaving rows
    float *zbuf = stage + kStages * G::STAGE_FLOATS;  // [3][Q][kB][TW]: map-guide rows of the outputs
    float *cbuf = zbuf + 3 * G::ZBUF_FLOATS;         // [kB][NCF][CS]: summed coefficient rows
    uint64_t *bar = reinterpret_cast<uint64_t *>(cbuf + G::CBUF_FLOATS);  // [kStages] staged rows, [3] map guide
    uint64_t *zbar = bar + kStages;

    if (RC > 0 && warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(tma::smem_addr(&s_tmem)),
                     "r"(kTmemCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
    }
    if (tid == 0) {
        s_abort = 0x7fffffff;
        s_nlist = 0;
        for (int i = 0; i < kStages + 3; ++i) tma::mbar_init(bar + i, 1);
        tma::mbar_init_fence();
    }
    pdl::wait();  // the inputs and the zeroed counters
    // the CTA's reference shift: mean of a 16 x 16 sample grid of its input region
    if (warp == 1)
        dev::sample_mean<Q>(s_sh, a.guide, a.rad, H, W, max(0, m_lo - R), min(H, m_hi + R), max(0, x0 - RC - R),
                            min(W, x0 + TW + RC + R), lane);
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    unsigned bad = 0;  // non-finite outputs written by this thread
    // 2. H-pass of live batch k: row r of its (batch row, channel) rows, in place, seeded at 0 and CH
    auto sum_row = [&](int k, int r) {
        const int hb = r / NCH, hch = r % NCH;
        if (hb < kB && m_lo + kB * k + hb < m_hi) {
            float *row = Vbuf + (k & 1) * G::VBUF_FLOATS + ((size_t)hb * NCH + hch) * VS;
#pragma unroll 1
            for (int h = 0; h < 2; ++h) dev::hsum_run<R, G::CH>(row, row, h * G::CH);
        }
    };

    if (warp < kWalkers / 32) {
        // ================= walkers: V-pass and the copies of the input rows ====================
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;\n" ::"n"(kWalkRegs));
        // batch n: rows v0 + kB n ..; the entering (+ R) and leaving (- R - 1) input rows
        auto stage_batch = [&](int n) {
            const int v = v0 + kB * n;
            float *s = stage + (n % kStages) * G::STAGE_FLOATS;
            uint64_t *b = bar + n % kStages;
            tma::mbar_expect_tx(b, (unsigned)(2 * NS * kB * WSt * 4));
            const size_t box = (size_t)kB * WSt;
            tma::load_3d(s, &ka.tg, x0 - G::RA, v + R, 0, b);
            tma::load_3d(s + Q * box, &ka.tr, x0 - G::RA, v + R, 0, b);
            tma::load_3d(s + NS * box, &ka.tg, x0 - G::RA, v - R - 1, 0, b);
            tma::load_3d(s + (NS + Q) * box, &ka.tr, x0 - G::RA, v - R - 1, 0, b);
        };
        int issued = min(kStages, nbatch), waited = 0;
        bool aborted = false;
        if (tid == 0)
            for (int n = 0; n < issued; ++n) stage_batch(n);
        // walker column pair wcp: global columns x0 - RC - R + 2 wcp, + 1, staged columns 2 wcp + SOFF
        const int group = warp >> 1, wcp = ((warp & 1) << 5) + lane;
        const bool walker = wcp < G::NCP;
        const int gxw = x0 - RC - R + 2 * wcp;
        const bool wcol_in = gxw >= 0 && gxw < W;  // W and gxw are even: both columns or neither
        constexpr int MG = Groups<Q>::MAXG;
        float2 E[MG], Dn[MG];
        float nsh[NS];  // minus the shift (zero outside the image)
#pragma unroll
        for (int i = 0; i < MG; ++i) E[i] = Dn[i] = make_float2(0.f, 0.f);
#pragma unroll
        for (int k = 0; k < NS; ++k) nsh[k] = wcol_in ? -s_sh[k] : 0.f;
        int tb = 0, sn = 0, par = 0;  // rows since the block start; stage buffer and its phase

        for (int n = 0; n < nbatch; ++n) {
            const int v = v0 + kB * n, k = n - R;  // live batch k (the window is full from k = 0 on)
            const bool ok = tma::wait_warp(bar + sn, (uint32_t)par, kTimeoutNs);
            if (ok) waited = n + 1;
            else if (lane == 0 && a.status) atomicExch(a.status, 1);
            if (k >= 2) bar_sync(kBarFree + (k & 1), T::kFree);  // slot of batch k - 2
            // 1. V-pass
            if (walker) {
                const float *st = stage + sn * G::STAGE_FLOATS + 2 * wcp + G::SOFF;
                float *vcol = Vbuf + (k & 1) * G::VBUF_FLOATS + 2 * wcp;
#pragma unroll 1
                for (int b = 0; b < kB; ++b) {
                    const int vb = v + b;
                    if (vb >= m_hi) break;
                    if (tb == 0) {  // block start: Dn = -(previous block total), E = 0
#pragma unroll
                        for (int i = 0; i < MG; ++i) {
                            Dn[i] = make_float2(-E[i].x, -E[i].y);
                            E[i] = make_float2(0.f, 0.f);
                        }
                    }
                    tb = tb + 1 == G::WR ? 0 : tb + 1;
                    const bool ein = vb + R >= 0 && vb + R < H;
                    const bool lout = vb - v0 >= G::WR && vb - R - 1 >= 0 && vb - R - 1 < H;
                    const float *se = st + (size_t)b * WSt;
                    float *vc = vcol + (size_t)b * NCH * VS;
                    switch (group) {
                    case 0: walk_rows<Q, 0, WSt>(E, Dn, vc, VS, se, nsh, ein, lout, k >= 0, std::make_integer_sequence<int, Groups<Q>::size(0)>{}); break;
                    case 1: walk_rows<Q, 1, WSt>(E, Dn, vc, VS, se, nsh, ein, lout, k >= 0, std::make_integer_sequence<int, Groups<Q>::size(1)>{}); break;
                    case 2: walk_rows<Q, 2, WSt>(E, Dn, vc, VS, se, nsh, ein, lout, k >= 0, std::make_integer_sequence<int, Groups<Q>::size(2)>{}); break;
                    default: walk_rows<Q, 3, WSt>(E, Dn, vc, VS, se, nsh, ein, lout, k >= 0, std::make_integer_sequence<int, Groups<Q>::size(3)>{}); break;
                    }
                }
            }
            // the staged rows are read, the vertical sums complete; or a wait ran out in some warp
            if (bar_or(kBarWalk, kWalkers, !ok)) {
                aborted = true;
                if (tid == 0) s_abort = max(k, 0);
                // the team that waits for this batch
                if (T::kWalkersSum) bar_arrive(kBarFull + (max(k, 0) & 1), T::kFull);
                else bar_arrive(kBarWalked + (max(k, 0) & 1), T::kWalked);
                break;
            }
            if (issued < nbatch) {  // the next batch into the buffer just read
                if (tid == 0) {
                    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
                    stage_batch(n + kStages);
                }
                ++issued;
            }
            if (++sn == kStages) {
                sn = 0;
                par ^= 1;
            }
            if (k < 0) continue;
            if constexpr (T::kWalkersSum) {
                sum_row(k, tid);
                bar_arrive(kBarFull + (k & 1), T::kFull);
            } else {
                bar_arrive(kBarWalked + (k & 1), T::kWalked);
            }
        }
        if (aborted && warp == 0) {
            // after a wait ran out: give the copies in flight one more bounded wait to land before
            // the CTA exits (no further copy was issued)
            for (int n = waited; n < issued; ++n) tma::wait_warp(bar + n % kStages, (uint32_t)((n / kStages) & 1), kTimeoutNs);
        }
        if (!aborted)
            for (int k = max(nlive - 2, 0); k < nlive; ++k) bar_sync(kBarFree + (k & 1), T::kFree);
    } else if (warp < kWalkers / 32 + 4) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;\n" ::"n"(kSolveRegs));
        if (warp == kWalkers / 32 + 3) {
            // the fourth warp of this group helps the summers: a batch has 142 rows to sum
            for (int k = 0; !T::kWalkersSum && k < nlive; ++k) {
                bar_sync(kBarWalked + (k & 1), T::kWalked);
                const bool aborted = s_abort <= k;
                if (!aborted) sum_row(k, kSummers + lane);
                bar_arrive(kBarFull + (k & 1), T::kFull);
                if (aborted) break;
            }
        } else {
        // ================= solvers: two neighbouring pixels per thread =========================
        const int st = tid - kWalkers, swarp = warp - kWalkers / 32;
        const int sb = st / (TS / 2), sxs = 2 * (st % (TS / 2));  // batch row, first column
        const int sgx = x0 - RC + sxs;
        const float *zg = a.map_guide ? a.map_guide : a.guide;
        const float tau = a.tau, eps = a.eps;
        int *list = a.list + (size_t)cta * a.list_cap;
        const bool in0 = sgx >= 0 && sgx < W, in1 = sgx + 1 >= 0 && sgx + 1 < W;
        const float nx0 = in0 ? (float)(min(sgx + R, W - 1) - max(sgx - R, 0) + 1) : 1.f;
        const float nx1 = in1 ? (float)(min(sgx + 1 + R, W - 1) - max(sgx + 1 - R, 0) + 1) : 1.f;
        for (int k = 0; k < nlive; ++k) {
            bar_sync(kBarFull + (k & 1), T::kFull);
            if (s_abort <= k) {  // the walkers gave up at this batch
                if (RC > 0) bar_arrive(kBarModels + (k & 1), T::kModels);
                break;
            }
            // 3. solve
            bool flag0 = false, flag1 = false;
            const int m = m_lo + kB * k + sb;
            if (st < kB * (TS / 2) && m < m_hi) {
                const bool row_in = m >= 0 && m < H, live0 = row_in && in0, live1 = row_in && in1;
                float *col = Vbuf + (k & 1) * G::VBUF_FLOATS + (size_t)sb * NCH * VS + sxs;
                const float ny = row_in ? (float)(min(m + R, H - 1) - max(m - R, 0) + 1) : 1.f;
                const float2 n = make_float2(ny * nx0, ny * nx1), inv_n = make_float2(1.0f / n.x, 1.0f / n.y);
                Factor<Q> f;
                bool low0, low1;
                model_factor<Q, VS>(col, n, inv_n, eps, tau, f, low0, low1);
                flag0 = live0 && low0 && tau > 0.f;
                flag1 = live1 && low1 && tau > 0.f;
                const bool keep0 = live0 && !flag0, keep1 = live1 && !flag1;
                float2 ys[3], z[Q];
#pragma unroll
                for (int c = 0; c < 3; ++c) ys[c] = ld2(col + (C::Y0 + c) * VS);
                if constexpr (RC == 0) {
#pragma unroll
                    for (int i = 0; i < Q; ++i) {
                        const float *zp = zg + i * plane + (size_t)m * W + sgx;
                        z[i] = make_float2(keep0 ? __ldg(zp) - s_sh[i] : 0.f, keep1 ? __ldg(zp + 1) - s_sh[i] : 0.f);
                    }
                }
                float2 A[3][Q], bv[3];
                model_rhs<Q, VS>(f, ys, col + C::XY0 * VS, inv_n, A, bv);
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    if constexpr (RC > 0) {
                        // model coefficients (relative to the CTA shift) into channel rows [0, NCF)
                        // of these pixels, colour-major (the sums they replace are in registers); a
                        // flagged pixel contributes zero here and its FP64 model later
                        if (!(keep0 && keep1)) {
                            bv[c] = make_float2(keep0 ? bv[c].x : 0.f, keep1 ? bv[c].y : 0.f);
#pragma unroll
                            for (int i = 0; i < Q; ++i) A[c][i] = make_float2(keep0 ? A[c][i].x : 0.f, keep1 ? A[c][i].y : 0.f);
                        }
                        float *cc0 = col + (size_t)(c * (Q + 1)) * VS;
                        st2(cc0, bv[c]);
#pragma unroll
                        for (int i = 0; i < Q; ++i) st2(cc0 + (1 + i) * VS, A[c][i]);
                    } else {
                        float2 o = bv[c];
#pragma unroll
                        for (int i = 0; i < Q; ++i) o = __ffma2_rn(A[c][i], z[i], o);
                        o = make_float2(o.x + s_sh[Q + c], o.y + s_sh[Q + c]);
                        float *op = a.out + c * plane + (size_t)m * W + sgx;
                        if (keep0) op[0] = o.x, bad += !isfinite(o.x);
                        if (keep1) op[1] = o.y, bad += !isfinite(o.y);
                    }
                }
            }
            if constexpr (RC > 0) bar_arrive(kBarModels + (k & 1), T::kModels);
            else bar_arrive(kBarFree + (k & 1), T::kFree);
            if (bar_or(kBarSolve, kSolvers, flag0 || flag1)) {  // append the flagged pixels in (row, column) order
                const unsigned bal0 = __ballot_sync(0xffffffffu, flag0), bal1 = __ballot_sync(0xffffffffu, flag1);
                if (lane == 0) s_wcnt[swarp] = __popc(bal0) + __popc(bal1);
                bar_sync(kBarSolve, kSolvers);
                int at = s_nlist;
                for (int w = 0; w < swarp; ++w) at += s_wcnt[w];
                const unsigned below = (1u << lane) - 1u;
                at += __popc(bal0 & below) + __popc(bal1 & below);
                if (flag0) list[at++] = m * W + sgx;
                if (flag1) list[at] = m * W + sgx + 1;
                bar_sync(kBarSolve, kSolvers);
                if (st == 0) {
                    int tot = 0;
                    for (int w = 0; w < kSolvers / 32; ++w) tot += s_wcnt[w];
                    s_nlist += tot;
                }
                bar_sync(kBarSolve, kSolvers);
            }
        }
        }
    } else {
        // ================= summers: H-pass, coefficient H-pass, V-pass and apply ===============
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;\n" ::"n"(kSumRegs));
        const int st = tid - kThreads + kSummers;
        const uint32_t tmem = s_tmem + ((uint32_t)(32 * (warp & 3)) << 16);  // this warp's lane quarter
        const int cc = st / (TW / 2), cx = 2 * (st % (TW / 2));  // colour, first output column
        const bool colour = st < 3 * (TW / 2);
        const int cgx = x0 + cx;
        const bool cin = colour && cgx < W;  // W and cgx are even: both columns or neither
        const float mx0 = (float)(min(cgx + RC, W - 1) - max(cgx - RC, 0) + 1);
        const float mx1 = (float)(min(cgx + 1 + RC, W - 1) - max(cgx + 1 - RC, 0) + 1);
        const float inv_mx0 = 1.0f / mx0, inv_mx1 = 1.0f / mx1;
        auto stage_z = [&](int k) {
            uint64_t *b = zbar + k % 3;
            tma::mbar_expect_tx(b, G::ZBYTES);
            tma::load_3d(zbuf + (k % 3) * G::ZBUF_FLOATS, &ka.tz, x0, y0 - 2 * RC + kB * k, 0, b);
        };
        int zissued = RC > 0 ? min(2, nlive) : 0, zdone = 0, slot = 0;  // slot: ring slot of the next row
        if (RC > 0 && st == 0)
            for (int i = 0; i < zissued; ++i) stage_z(i);
        int k = 0;
        for (; k < nlive; ++k) {
            if constexpr (!T::kWalkersSum) {
                bar_sync(kBarWalked + (k & 1), T::kWalked);
                const bool aborted = s_abort <= k;
                if (!aborted) sum_row(k, st);
                bar_arrive(kBarFull + (k & 1), T::kFull);
                if (aborted) break;
            }
            if constexpr (RC > 0) {
            bar_sync(kBarModels + (k & 1), T::kModels);
            if (s_abort <= k) break;
            // 4. coefficient H-pass: unit (row b, coefficient, half) -> the coefficient buffer
            const int uk = st % NCF, uh = (st / NCF) & 1, ub = st / (2 * NCF);
            if (st < kB * NCF * 2 && m_lo + kB * k + ub < m_hi)
                dev::hsum_run<RC, G::CL>(Vbuf + (k & 1) * G::VBUF_FLOATS + ((size_t)ub * NCH + uk) * VS,
                                         cbuf + ((size_t)ub * NCF + uk) * G::CS, uh * G::CL);
            bar_arrive(kBarFree + (k & 1), T::kFree);
            const bool zok = tma::wait_warp(zbar + k % 3, (uint32_t)((k / 3) & 1), kTimeoutNs);
            if (!zok && lane == 0 && a.status) atomicExch(a.status, 1);
            zdone = k + 1;
            bar_sync(kBarSum, kSummers);
            // 5. coefficient V-pass and apply: thread (colour, pair of output columns).  A warp whose
            // map-guide wait ran out leaves its outputs of the batch unwritten.
            float2 Ec[Q + 1], Dc[Q + 1];
            if (k == 0) {
#pragma unroll
                for (int j = 0; j <= Q; ++j) Ec[j] = Dc[j] = make_float2(0.f, 0.f);
            } else {
                uint32_t s[36];
                tm_ld32(tmem + kColState, s);
                tm_ld4(tmem + kColState + 32, s + 32);
                tm_wait_ld();
#pragma unroll
                for (int j = 0; j <= Q; ++j) {
                    Ec[j] = make_float2(__uint_as_float(s[2 * j]), __uint_as_float(s[2 * j + 1]));
                    Dc[j] = make_float2(__uint_as_float(s[18 + 2 * j]), __uint_as_float(s[19 + 2 * j]));
                }
            }
            const float *zb = zbuf + (k % 3) * G::ZBUF_FLOATS + (colour ? cx : 0);
            const float *hcol = cbuf + (size_t)((colour ? cc : 0) * (Q + 1)) * G::CS + (colour ? cx : 0);
#pragma unroll 1
            for (int b = 0; b < kB; ++b) {
                const int m = m_lo + kB * k + b;
                if (m >= m_hi) break;
                const bool leaves = m - m_lo >= G::WC;
                uint32_t lv[18];
                if (leaves) {  // the row leaving the window, from the ring
                    tm_ld16(tmem + 16u * slot, lv);
                    tm_ld2(tmem + kColRing2 + 2u * slot, lv + 16);
                }
                float2 hv[Q + 1];
#pragma unroll
                for (int j = 0; j <= Q; ++j) hv[j] = ld2(hcol + (size_t)(b * NCF + j) * G::CS);
                tm_wait_ld();
                if (slot == 0) {
#pragma unroll
                    for (int j = 0; j <= Q; ++j) {
                        Dc[j] = make_float2(-Ec[j].x, -Ec[j].y);
                        Ec[j] = make_float2(0.f, 0.f);
                    }
                }
                if (leaves) {
#pragma unroll
                    for (int j = 0; j <= Q; ++j)
                        Dc[j] = __fadd2_rn(Dc[j], make_float2(__uint_as_float(lv[2 * j]), __uint_as_float(lv[2 * j + 1])));
                }
                uint32_t ent[18];
#pragma unroll
                for (int j = 0; j <= Q; ++j) {
                    Ec[j] = __fadd2_rn(Ec[j], hv[j]);
                    ent[2 * j] = __float_as_uint(hv[j].x);
                    ent[2 * j + 1] = __float_as_uint(hv[j].y);
                }
                __syncwarp();
                tm_st16(tmem + 16u * slot, ent);
                tm_st2(tmem + kColRing2 + 2u * slot, ent + 16);
                if (++slot == G::WC) slot = 0;
                const int y = m - RC;
                if (cin && zok && y >= y0 && y < y1) {
                    const float my = (float)(min(y + RC, H - 1) - max(y - RC, 0) + 1);
                    const float2 mone = make_float2(-1.f, -1.f);
                    float2 o = __ffma2_rn(Dc[0], mone, Ec[0]);
#pragma unroll
                    for (int i = 0; i < Q; ++i) {
                        const float2 zz = ld2(zb + (i * kB + b) * TW);
                        o = __ffma2_rn(__ffma2_rn(Dc[1 + i], mone, Ec[1 + i]), make_float2(zz.x - s_sh[i], zz.y - s_sh[i]), o);
                    }
                    const float sy = s_sh[Q + cc];
                    o = make_float2(fmaf(o.x, inv_mx0 / my, sy), fmaf(o.y, inv_mx1 / my, sy));
                    *reinterpret_cast<float2 *>(a.out + cc * plane + (size_t)y * W + cgx) = o;
                    bad += !isfinite(o.x) + !isfinite(o.y);
                }
                __syncwarp();
            }
            uint32_t s[36];
#pragma unroll
            for (int j = 0; j <= Q; ++j) {
                s[2 * j] = __float_as_uint(Ec[j].x);
                s[2 * j + 1] = __float_as_uint(Ec[j].y);
                s[18 + 2 * j] = __float_as_uint(Dc[j].x);
                s[19 + 2 * j] = __float_as_uint(Dc[j].y);
            }
            tm_st32(tmem + kColState, s);
            tm_st4(tmem + kColState + 32, s + 32);
            tm_wait_st();
            bar_sync(kBarSum, kSummers);  // the coefficient rows and the map-guide rows are read
            if (zissued < nlive) {
                if (st == 0) {
                    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
                    stage_z(k + 2);
                }
                ++zissued;
            }
            }
        }
        // after an abort: let the map-guide copies in flight land
        if (st < 32)
            for (; zdone < zissued; ++zdone) tma::wait_warp(zbar + zdone % 3, (uint32_t)((zdone / 3) & 1), kTimeoutNs);
    }
    if (bad && a.nonfinite) atomicAdd(a.nonfinite, (unsigned long long)bad);
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (RC > 0 && warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(s_tmem), "r"(kTmemCols));
    }
    if (tid == 0) a.list_count[cta] = s_nlist;
    if (tid < NS) a.cta_shift[(size_t)cta * NS + tid] = s_sh[tid];
}

// ---- FP64 correction of flagged pixels ----------------------------------------------------
// One CTA per CTA of the fused launch.  Its flagged pixels (in row, column order) get FP64
// models (one warp each, window sums recomputed in FP64 from the inputs), relative to the
// fused CTA's shift.  With rc = 0 the model's result is written to the pixel; with rc > 0 each
// model's share, (b + a^T (z_i - s)) / m_i, is added to every output i of this CTA whose
// averaging window holds the pixel, one flagged pixel after the other (a fixed order, so the
// result is deterministic).  Adds the number of flagged pixels that this CTA owns (outputs of
// its strip segment) to flag_count.
constexpr int kFixThreads = 256, kFixWarps = kFixThreads / 32;

template <int Q>
__global__ void __launch_bounds__(kFixThreads) flr_fused_fix_kernel(const FusedArgs a)
{
    constexpr int NS = Q + 3, NCF = 3 * (Q + 1);
    __shared__ double s_model[kFixWarps][NCF];
    __shared__ float s_sh[NS];
    __shared__ unsigned long long s_cnt[2];
    const int cta = blockIdx.y * gridDim.x + blockIdx.x;
    pdl::wait();
    const int n = a.list_count[cta];
    if (n == 0) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int H = a.H, W = a.W, rc = a.rc;
    const size_t plane = (size_t)H * W;
    const int TW = tile_width(rc);
    const int x0 = blockIdx.x * TW;
    const int row_hi = a.row_hi < 0 ? H : min(a.row_hi, H);
    const int y0 = a.row_lo + blockIdx.y * a.TH;
    const int y1 = min(y0 + a.TH, row_hi);
    const int x1 = min(x0 + TW, W);
    const int *list = a.list + (size_t)cta * a.list_cap;
    const float *zg = a.map_guide ? a.map_guide : a.guide;
    if (tid < NS) s_sh[tid] = a.cta_shift[(size_t)cta * NS + tid];
    if (tid < 2) s_cnt[tid] = 0ull;
    __syncthreads();
    unsigned own = 0;
    for (int e = tid; e < n; e += kFixThreads) {
        const int idx = list[e], py = idx / W, px = idx % W;
        own += py >= y0 && py < y1 && px >= x0 && px < x1;
    }
    long long dbad = 0;  // change in the number of non-finite output values
    for (int e0 = 0; e0 < n; e0 += kFixWarps) {
        if (e0 + warp < n) {
            double A[Q][3], bv[3];
            dev::fp64_model<Q>(a.guide, a.rad, H, W, a.r, (double)a.eps, list[e0 + warp], lane, s_sh, A, bv);
            if (lane == 0) {
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    s_model[warp][c * (Q + 1)] = bv[c];
#pragma unroll
                    for (int i = 0; i < Q; ++i) s_model[warp][c * (Q + 1) + 1 + i] = A[i][c];
                }
            }
        }
        __syncthreads();
        const int ne = min(kFixWarps, n - e0);
        for (int k = 0; k < ne; ++k) {
            const int idx = list[e0 + k], py = idx / W, px = idx % W;
            const double *md = s_model[k];
            if (rc == 0) {
                if (tid < 3 && py >= y0 && py < y1 && px >= x0 && px < x1) {
                    double o = md[tid * (Q + 1)];
                    for (int i = 0; i < Q; ++i) o += md[tid * (Q + 1) + 1 + i] * ((double)zg[i * plane + idx] - (double)s_sh[i]);
                    const float of = (float)(o + (double)s_sh[Q + tid]);
                    a.out[tid * plane + idx] = of;
                    dbad += !isfinite(of);
                }
            } else {
                const int wd = 2 * rc + 1;
                for (int t = tid; t < wd * wd; t += kFixThreads) {
                    const int yy = py - rc + t / wd, xx = px - rc + t % wd;
                    if (yy < y0 || yy >= y1 || xx < x0 || xx >= x1) continue;
                    const size_t off = (size_t)yy * W + xx;
                    const float my = (float)(min(yy + rc, H - 1) - max(yy - rc, 0) + 1);
                    const float mx = (float)(min(xx + rc, W - 1) - max(xx - rc, 0) + 1);
                    double zz[Q];
                    for (int i = 0; i < Q; ++i) zz[i] = (double)__ldg(zg + i * plane + off) - (double)s_sh[i];
                    for (int c = 0; c < 3; ++c) {
                        double o = md[c * (Q + 1)];
                        for (int i = 0; i < Q; ++i) o += md[c * (Q + 1) + 1 + i] * zz[i];
                        const float old = a.out[c * plane + off];
                        const float nw = (float)((double)old + o / ((double)my * (double)mx));
                        a.out[c * plane + off] = nw;
                        dbad += (long long)!isfinite(nw) - (long long)!isfinite(old);
                    }
                }
            }
            __syncthreads();
        }
    }
    atomicAdd(&s_cnt[0], (unsigned long long)own);
    if (dbad != 0) atomicAdd(&s_cnt[1], (unsigned long long)dbad);  // two's complement sum
    __syncthreads();
    if (tid == 0) {
        if (a.flag_count) atomicAdd(a.flag_count, s_cnt[0]);
        if (a.nonfinite && s_cnt[1]) atomicAdd(a.nonfinite, s_cnt[1]);
    }
}

// ---- host side -------------------------------------------------------------------------
template <int Q, int R, int RC>
cudaError_t prepare_qr()
{
    return cudaFuncSetAttribute(flr_fused_kernel<Q, R, RC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)Geo<Q, R, RC>::SMEM);
}

template <int Q, int R, int RC>
cudaError_t launch_qr(const FusedArgs &a, dim3 grid, cudaStream_t st)
{
    using G = Geo<Q, R, RC>;
    static std::mutex mu;
    static bool ready[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    {
        std::lock_guard<std::mutex> lock(mu);
        if (!ready[dev]) {  // this kernel instance always asks for the same shared memory
            e = prepare_qr<Q, R, RC>();
            if (e != cudaSuccess) return e;
            ready[dev] = true;
        }
    }
    KArgs ka;
    std::memset(&ka, 0, sizeof(ka));
    ka.a = a;
    if (tma::encode_planes_f32(&ka.tg, a.guide, a.W, a.H, Q, G::WSt, kB, Q) != cudaSuccess ||
        tma::encode_planes_f32(&ka.tr, a.rad, a.W, a.H, 3, G::WSt, kB, 3) != cudaSuccess ||
        tma::encode_planes_f32(&ka.tz, a.map_guide ? a.map_guide : a.guide, a.W, a.H, Q, G::TW, kB, Q) !=
            cudaSuccess)
        return cudaErrorInvalidValue;
    // dependent launches here and below, with no early trigger (a waiting CTA of the successor would
    // take an SM from another stream's fused kernel): 256 x 256 41.0 -> 38.7 us, 1920x1080 299.2 -> 296.5
    return pdl::launch(flr_fused_kernel<Q, R, RC>, grid, kThreads, G::SMEM, st, ka);
}

}  // namespace fused

// Radii of the fused kernel (compile-time instances): the 1080p workload (r = rc = 8), the
// 256 x 256 workload (r = rc = 5) and r = 8 without averaging; Q = 8.
bool fused_supported(int q, int r, int rc)
{
    return q == 8 && ((r == 8 && (rc == 8 || rc == 0)) || (r == 5 && rc == 5));
}

int fused_tile_width(int rc) { return fused::tile_width(rc); }

cudaError_t launch_fused(int q, const FusedArgs &a, dim3 grid, cudaStream_t st)
{
    if (q == 8) {
        if (a.r == 8 && a.rc == 8) return fused::launch_qr<8, 8, 8>(a, grid, st);
        if (a.r == 8 && a.rc == 0) return fused::launch_qr<8, 8, 0>(a, grid, st);
        if (a.r == 5 && a.rc == 5) return fused::launch_qr<8, 5, 5>(a, grid, st);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_fused_fix(int q, const FusedArgs &a, dim3 grid, cudaStream_t st)
{
    if (q != 8) return cudaErrorInvalidValue;
    return pdl::launch(fused::flr_fused_fix_kernel<8>, grid, fused::kFixThreads, 0, st, a);
}

}  // namespace flr
