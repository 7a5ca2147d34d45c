// flnr.cu -- the FLNR guide network (Sec. 3.3) on sm_103a: BF16 implicit-GEMM convolutions
// with FP32 accumulation on the fifth-generation tensor cores (tcgen05, accumulators in
// tensor memory) for the forward pass and for training -- input gradients as convolutions
// with rotated, transposed weights on the forward's TMA-staged kernel, weight gradients as
// one GEMM over pixels per layer with the operands transposed on chip -- Adam on FP32
// master weights, and the flnr_* entry points of include/flr.h.
//
// Network (weights and order as oracle/flnr_ref.py): 11 inputs (8 guides + noisy RGB)
//   in0 3x3 11->16 ReLU, in1 1x1 16->16 ReLU                                   f0 (H)
//   e1a 3x3 16->32 ReLU, e1b 3x3 32->32 stride 2 ReLU                          f1 (H/2)
//   e2a 3x3 32->64 ReLU, e2b 3x3 64->64 stride 2 ReLU                          f2 (H/4)
//   up(f2) ++ f1, d1a 3x3 96->32 ReLU, d1b 3x3 32->32 ReLU                     d1 (H/2)
//   up(d1) ++ f0, d0a 3x3 48->16 ReLU, d0b 3x3 16->16 ReLU                     d0 (H)
//   o0 3x3 16->16 ReLU, o1 1x1 16->8, sigmoid                                  X' (8 ch)
// Activations are BF16 in planes of eight channels, [N][C/8][H][W][8] (the 11 inputs padded
// to 16 channels, the 8 outputs of o1 computed as 16 with zero weights): a row of a plane is
// contiguous, so a tile with its halo arrives in rows of 8 (NT + 1/4) x 16 bytes per TMA request
// instead of 16 bytes (the eight channels of one pixel of an NHWC map; a 3x3 16->16 layer of a
// 1920x1080 frame: 49 us with NHWC tiles, 32 us with plane tiles).  The outputs of e1a and
// e2a, which stride-2 convolutions read, are additionally split by row and column parity,
// [N][C/8][2][2][H/2][W/2][8].  flnr_layer's tensors are NHWC; the kernels take either.  The
// enhanced guides leave as planar FP32 for FLR.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>

#include <cmath>
#include <cstdint>
#include <cstring>
#include <new>
#include <utility>
#include <vector>

#include "flr.h"
#include "pdl.cuh"
#include "tma.cuh"

namespace flnr {
namespace {

typedef __nv_bfloat16 bf16;

constexpr int kNL = 12;
struct LayerDef {
    int cin, cout, k, relu;  // true sizes (o1's cout is 8)
};
constexpr LayerDef kLayers[kNL] = {
    {11, 16, 3, 1}, {16, 16, 1, 1}, {16, 32, 3, 1}, {32, 32, 3, 1}, {32, 64, 3, 1}, {64, 64, 3, 1},
    {96, 32, 3, 1}, {32, 32, 3, 1}, {48, 16, 3, 1}, {16, 16, 3, 1}, {16, 16, 3, 1}, {16, 8, 1, 0}};
__host__ __device__ constexpr int pad16(int c) { return (c + 15) / 16 * 16; }

// ---------------------------------------------------------------------------------------
// Every launch of the passes is a programmatic dependent one (pdl.cuh); the weights' conversion, Adam
// and the losses are ordinary.  The network is a chain of short
// kernels, each reading what the one before wrote, and at 16 x 128^2 a training pass lost 120 us
// of 690 between them.  A kernel that allocates tensor memory triggers after its allocation: its
// successor's CTAs, which may be resident beside it and hold columns while they wait, then cannot
// keep it from allocating.

// ---------------------------------------------------------------------------------------
// Asynchronous 16-byte global -> shared copies (zero fill when !valid).
__device__ __forceinline__ void cp_async16(void *dst, const void *src, bool valid)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(valid ? 16 : 0));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N)); }

// Arguments of the convolution kernels (stride 1, zero padding KS/2, implicit GEMM on the
// tensor cores).  x: CIN channels, w [taps][COUT][CIN] bf16, bias [COUT] fp32.  The kernels'
// template parameters select the epilogue:
//   OUTM 0 -> y: COUT channels bf16 (ACT 1 = ReLU);
//   OUTM 1 -> yf planar fp32 [N][nbias][H][W] (may be NULL), sigmoid of the true outputs;
//   OUTM 2 -> y: the gradient g s (1 - s) at the sigmoid's input, s the sigmoid of the result
//             and g planar fp32 [N][nbias][H][W] (zero for the padding channels);
//   MASK   -> the result times (mask > 0), mask: COUT channels bf16 (the ReLU of the layer
//             input, for input gradients);
// The decoder kernel reads x as the half-resolution map (CA channels) and x2 as the skip
// (CIN - CA channels) of the concatenated input up2(x) ++ x2.  Every bf16 tensor has one of
// these layouts:
enum Layout {
    kNHWC = 0,    // [N][H][W][C]
    kPlanes = 1,  // [N][C/8][H][W][8]
    kParity = 2   // [N][C/8][2][2][H/2][W/2][8]: planes split by row and column parity, H and W even
};
struct ConvArgs {
    const bf16 *x, *w, *mask;
    const float *bias;
    bf16 *y;
    float *yf;
    const float *g;
    int N, H, W;
    int lx, ly, lm;  // layouts of x and x2, y, mask
    int nbias;       // valid bias entries (the true output channels); 0 without bias
    const bf16 *x2;
    int *status;  // tensor-core path: set to FLNR_STATUS_TIMEOUT if a completion wait ran out
};

// Address of pixel (n, y, x)'s first eight channels in a C-channel tensor of an H x W map;
// the further channel groups are *chunk elements apart.
__device__ __forceinline__ size_t pixel_at(int layout, int C, int H, int W, int n, int y, int x, size_t *chunk)
{
    const size_t hw = (size_t)H * W;
    if (layout == kNHWC) {
        *chunk = 8;
        return ((size_t)n * hw + (size_t)y * W + x) * C;
    }
    *chunk = hw * 8;
    const size_t q = layout == kPlanes ? (size_t)y * W + x
                                       : ((size_t)(2 * (y & 1) + (x & 1)) * (H / 2) + (y >> 1)) * (W / 2) + (x >> 1);
    return ((size_t)n * (C / 8) * hw + q) * 8;
}

// ---------------------------------------------------------------------------------------
// The same convolution on the fifth-generation tensor cores (tcgen05): BF16 operands in shared
// memory, FP32 accumulators in tensor memory (TMEM).
//
// A tile is 16 rows x 8 pixels = the M = 128 rows of one UMMA.  The input tile (with halo) is
// staged as [channel chunk c8][row][col][8 channels], so 8 consecutive pixels of one row and
// one 8-channel chunk form a contiguous 128-byte core matrix.  For tap (ky, kx) the operand A
// (128 output pixels x 16 channels) is then the no-swizzle K-major layout starting at pixel
// (ky, kx) of chunk 2kk: 8-row groups (output rows) SW * 16 bytes apart, the two K halves
// (chunks 2kk, 2kk + 1) SH * SW * 16 bytes apart.  No im2col copy is made.  The weights are
// staged once per CTA as [tap][c8][COUT][8]: operand B (COUT x 16, K-major) has 8-row groups
// 128 bytes apart and K halves COUT * 16 bytes apart.  One thread issues the taps x CIN/16
// MMAs of a tile and commits them to an mbarrier; four warps then read the accumulator rows of
// their TMEM lane quarter (one output pixel per thread) and run the epilogue, while the next
// tiles' inputs are already loading.  Every wait is bounded by the global timer.
#define FLNR_STATUS_TIMEOUT 1
constexpr unsigned long long kTcTimeoutNs = 1000000000ull;  // 1 s per wait

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// shared-memory matrix descriptor: no swizzle, K-major; LBO = distance between the two K
// halves of a core-matrix pair, SBO = distance between 8-row groups
__device__ __forceinline__ uint64_t umma_sdesc(uint32_t saddr, uint32_t lbo, uint32_t sbo)
{
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

// instruction descriptor, kind::f16: D FP32, A and B BF16, both K-major, M = 128, N = n
__host__ __device__ constexpr uint32_t umma_idesc(int n)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}

__device__ __forceinline__ void umma_bf16(uint32_t tmem_d, uint64_t ad, uint64_t bd, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
        "l"(ad), "l"(bd), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16])
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// bounded wait for the mbarrier phase with the given parity, polled by lane 0 of the warp
// (try_wait suspends the thread for up to 20 us per call); false if it ran out
__device__ __forceinline__ bool mbar_wait_warp(uint32_t mbar, uint32_t parity)
{
    uint32_t ok = 1;
    if ((threadIdx.x & 31) == 0) {
        const unsigned long long t0 = global_ns();
        for (;;) {
            uint32_t done;
            asm volatile(
                "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, 20000;\nselp.u32 %0, 1, 0, p;\n}\n"
                : "=r"(done)
                : "r"(mbar), "r"(parity)
                : "memory");
            if (done) break;
            if (global_ns() - t0 > kTcTimeoutNs) {
                ok = 0;
                break;
            }
        }
    }
    return __shfl_sync(0xffffffffu, ok, 0) != 0;
}

template <int N>
constexpr int tmem_cols()
{
    static_assert(N <= 512, "tensor memory has 512 columns");
    return N <= 32 ? 32 : N <= 64 ? 64 : N <= 128 ? 128 : N <= 256 ? 256 : 512;
}

// Kernel parameters: the tensor map (4-D: channels, W, H, N) of the operand that TMA stages
// (x, or the skip x2 of a decoder layer) and the convolution arguments.
struct alignas(128) TcArgs {
    CUtensorMap tm;
    ConvArgs c;
};

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap *tm, int c0, int c1, int c2, int c3,
                                            uint32_t mbar)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];\n" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(tm)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(mbar)
        : "memory");
}

// single-thread bounded wait on an mbarrier phase (the TMA issuer)
__device__ __forceinline__ bool mbar_wait_thread(uint32_t mbar, uint32_t parity)
{
    const unsigned long long t0 = global_ns();
    for (;;) {
        uint32_t done;
        asm volatile(
            "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, 20000;\nselp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(mbar), "r"(parity)
            : "memory");
        if (done) return true;
        if (global_ns() - t0 > kTcTimeoutNs) return false;
    }
}

// bounded wait of a whole warp, every lane polling and the branches decided by votes: the code after
// it stays one path
__device__ __forceinline__ bool mbar_wait_vote(uint32_t mbar, uint32_t parity)
{
    const unsigned long long t0 = global_ns();
    for (;;) {
        uint32_t done;
        asm volatile(
            "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, 20000;\nselp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(mbar), "r"(parity)
            : "memory");
        if (__all_sync(0xffffffffu, done != 0)) return true;
        if (__any_sync(0xffffffffu, global_ns() - t0 > kTcTimeoutNs)) return false;
    }
}

// Epilogue pieces shared by the tensor-core kernels.  tc_load_acc: one accumulator row (an
// output pixel) from the warp's TMEM lane quarter, COUT columns from `taddr` on.
template <int COUT>
__device__ __forceinline__ void tc_load_acc(uint32_t taddr, float (&v)[COUT])
{
#pragma unroll
    for (int c0 = 0; c0 < COUT; c0 += 16) {
        float q[16];
        tmem_ld16(taddr + (uint32_t)c0, q);
#pragma unroll
        for (int i = 0; i < 16; ++i) v[c0 + i] = q[i];
    }
    asm volatile("tcgen05.wait::ld.sync.aligned;\n");
    asm volatile("tcgen05.fence::before_thread_sync;\n");
}

// tc_store: bias, activation, optional ReLU mask, then bf16 stores, or sigmoid into planar
// fp32 (OUTM 1).  (n, yy, xx): the output pixel of an [N][a.H][a.W] map.
template <int COUT, int ACT, int OUTM, bool MASK>
__device__ __forceinline__ void tc_store(const ConvArgs &a, float (&v)[COUT], const float (&bias)[COUT], int n,
                                         int yy, int xx)
{
    const bool in = yy < a.H && xx < a.W;
#pragma unroll
    for (int c = 0; c < COUT; ++c) {
        v[c] += bias[c];
        if (ACT == 1) v[c] = fmaxf(v[c], 0.f);
    }
    if (MASK && in) {
        size_t mc;
        const bf16 *mp = a.mask + pixel_at(a.lm, COUT, a.H, a.W, n, yy, xx, &mc);
#pragma unroll
        for (int c8 = 0; c8 < COUT / 8; ++c8) {
            const uint4 m = *reinterpret_cast<const uint4 *>(mp + c8 * mc);
            const __nv_bfloat162 *mh = reinterpret_cast<const __nv_bfloat162 *>(&m);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (!(__bfloat162float(mh[i].x) > 0.f)) v[c8 * 8 + 2 * i] = 0.f;
                if (!(__bfloat162float(mh[i].y) > 0.f)) v[c8 * 8 + 2 * i + 1] = 0.f;
            }
        }
    }
    const size_t hw = (size_t)a.H * a.W, off = (size_t)yy * a.W + xx;  // planar fp32 (OUTM 1, 2)
    if (OUTM == 1) {
        // a.nbias planes: the head's true outputs, eight at a time, so that their exponentials and
        // divisions are not one behind the other (o0 + o1 at
        // 1920x1080: 81 us one by one, 63 us so)
        if (in && a.yf) {
            float *yo = a.yf + (size_t)n * a.nbias * hw + off;
#pragma unroll
            for (int c8 = 0; c8 < COUT / 8; ++c8) {
                if (8 * c8 >= a.nbias) break;
                float sv[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) sv[i] = expf(-v[8 * c8 + i]);
#pragma unroll
                for (int i = 0; i < 8; ++i) sv[i] = 1.f / (1.f + sv[i]);
#pragma unroll
                for (int i = 0; i < 8; ++i, yo += hw)
                    if (8 * c8 + i < a.nbias) *yo = sv[i];
            }
        }
        return;
    }
    if (OUTM == 2 && in) {
#pragma unroll
        for (int c = 0; c < COUT; ++c) {
            const float sv = 1.f / (1.f + expf(-v[c]));
            v[c] = c < a.nbias ? a.g[((size_t)n * a.nbias + c) * hw + off] * sv * (1.f - sv) : 0.f;
        }
    }
    size_t yc;
    bf16 *yp = a.y + pixel_at(a.ly, COUT, a.H, a.W, n, yy, xx, &yc);
#pragma unroll
    for (int c8 = 0; c8 < COUT / 8; ++c8) {
        uint4 o;
        __nv_bfloat162 *oh = reinterpret_cast<__nv_bfloat162 *>(&o);
#pragma unroll
        for (int i = 0; i < 4; ++i) oh[i] = __floats2bfloat162_rn(v[c8 * 8 + 2 * i], v[c8 * 8 + 2 * i + 1]);
        if (in) *reinterpret_cast<uint4 *>(yp + c8 * yc) = o;
    }
}

// ---------------------------------------------------------------------------------------
// Warp-specialised tensor-core convolution (layers whose input is one tensor): no CTA-wide
// barrier in the main loop.  The next warp (one lane) is the producer: it loads tile j into ring
// stage j % NBUF with one TMA box copy per channel chunk once the MMAs of tile j - NBUF have
// released the stage.  The last warp (one lane) issues tile j's MMAs into accumulator j & 1 once the
// stage has landed and the epilogue has drained that accumulator, then commits them to the
// stage's "empty" barrier and the accumulator's "full" barrier.  The epilogue warps read the
// accumulator rows of their TMEM lane quarter, release the accumulator, and run the epilogue
// (with several tiles per stage eight warps: the sigmoid of the head keeps four busy longer than
// the MMAs take; o0 + o1 at 1920x1080 101 us with four, 81 us with eight).
// A stage covers NT row phases of 8 columns (16 NT rows x 8 pixels, issue_phases; a 1x1 layer NT
// tiles of 16 rows x 8 pixels side by side): one halo and one hand-over of the barriers for NT accumulators, which pays where there are enough stages to
// go round (conv_ws_launch).  Every wait is bounded.
template <int CIN, int COUT, int KS, int NT>
struct WsGeom {
    // NT row phases of 8 columns, or (1x1: no row is read twice, and long rows cost TMA fewer
    // requests; 16 -> 16 at 16 x 128^2 19.4 us against 21.1) NT tiles side by side
    static constexpr bool PHASES = KS > 1;
    static constexpr int STEP = PHASES ? NT : 1;  // rows between an accumulator's 8-row groups
    static constexpr int TH = PHASES ? 16 * NT : 16, TW = PHASES ? 8 : 8 * NT;
    static constexpr int P = KS / 2, SH = TH + 2 * P, SW = TW + 2 * P, C8 = CIN / 8;
    // one MMA for the up to KS row phases that read a staged row (N <= 256)
    static constexpr bool MERGE = PHASES && NT > 1 && KS * COUT <= 256;
    static constexpr int NBUF = NT == 1 ? 4 : (C8 <= 2 ? 3 : 2);
    static constexpr int PS = (SH * SW * 16 + 127) / 128 * 128;
    static constexpr int XBYTES = C8 * PS;
    static constexpr int WBYTES = (KS * KS * C8 * COUT * 16 + 127) / 128 * 128;
    static constexpr int TMA_BYTES = C8 * SH * SW * 16;
    static constexpr int EW = NT == 1 ? 4 : 8;  // epilogue warps: warp w takes tiles w / 4, + EW / 4, ...
    static constexpr int THREADS = 32 * (EW + 2);
    static constexpr int NBAR = 2 * NBUF + 4;  // full[NBUF], empty[NBUF], accf[2], acce[2]
    static constexpr int SMEM = 128 + WBYTES + NBUF * XBYTES + NBAR * 8 + 16;
    static constexpr int COLS = tmem_cols<2 * NT * COUT>();
};
constexpr int kWsThreads = 192;

// One stage's input planes: channel chunk k of columns x.., rows y.. of image n
template <int C8, int PS>
__device__ __forceinline__ void load_planes(uint32_t dst, const CUtensorMap *tm, int layout, int x, int y, int n, uint32_t bar)
{
#pragma unroll
    for (int k = 0; k < C8; ++k) {
        if (layout == kNHWC) tma_load_4d(dst + k * PS, tm, k * 8, x, y, n, bar);
        else tma_load_4d(dst + k * PS, tm, 4 * x, y, k, n, bar);  // 32-bit elements: four per pixel
    }
}

// The MMAs of one stage.  Row phase t of a stage is its output rows t, t + NT, t + 2 NT, ...: 16
// rows x 8 pixels, the M = 128 rows of an operand whose 8-row groups lie NT staged rows apart.  Staged
// row rho + NT g is then read by phase t = rho - ky for tap row ky, so the same operand A serves up to
// KS phases, whose accumulators and weights ([kx][chunk][KS - 1 - ky][COUT]) lie side by side: one
// MMA of N = KS COUT instead of KS of N = COUT.  An MMA costs about 50 clocks whatever N is up to
// 64 and little more up to 200 (operand A is read from shared memory at 128 bytes per clock), and
// a 16 -> 16 layer spent 36 of them on 512 pixels (tiles side by side), now 21.  Each accumulator
// still takes its taps in the order (ky, kx, channels).  1920x1080 forward pass 428 us before, 417
// us so; gradients of 16 x 128^2 562 and 549 us.
template <class G, int CIN, int COUT, int KS, int NT>
__device__ __forceinline__ void issue_phases(uint32_t d0, uint64_t ab, uint64_t bdesc0)
{
    constexpr int C8 = G::C8, SW = G::SW, PS = G::PS;
    if constexpr (!G::PHASES) {
#pragma unroll
        for (int t = 0; t < NT; ++t)
#pragma unroll
            for (int kk = 0; kk < C8 / 2; ++kk)
                umma_bf16(d0 + (uint32_t)(t * COUT), ab + (uint32_t)((2 * kk * PS + 8 * t * 16) >> 4),
                          bdesc0 + (uint32_t)((2 * kk * COUT * 16) >> 4), umma_idesc(COUT), kk ? 1u : 0u);
        return;
    }
#pragma unroll
    for (int rho = 0; rho < NT + KS - 1; ++rho) {
        const int lo = rho - KS + 1 > 0 ? rho - KS + 1 : 0, hi = rho < NT - 1 ? rho : NT - 1;  // phases that read rho
#pragma unroll
        for (int kx = 0; kx < KS; ++kx) {
#pragma unroll
            for (int kk = 0; kk < C8 / 2; ++kk) {
                const uint64_t a = ab + (uint32_t)((2 * kk * PS + (rho * SW + kx) * 16) >> 4);
                // weights of phase t: tap row rho - t
                auto b = [&](int t) { return bdesc0 + (uint32_t)((((kx * C8 + 2 * kk) * KS + KS - 1 - (rho - t)) * COUT * 16) >> 4); };
                auto d = [&](int t) { return d0 + (uint32_t)(t * COUT); };
                const bool starts = rho < NT && (kx | kk) == 0;  // phase rho begins here
                if constexpr (G::MERGE) {
                    const int n = hi - lo + (starts ? 0 : 1);
                    if (n > 0) umma_bf16(d(lo), a, b(lo), umma_idesc(n * COUT), 1u);
                    if (starts) umma_bf16(d(rho), a, b(rho), umma_idesc(COUT), 0u);
                } else {
#pragma unroll
                    for (int t = lo; t <= hi; ++t) umma_bf16(d(t), a, b(t), umma_idesc(COUT), starts && t == rho ? 0u : 1u);
                }
            }
        }
    }
}

template <int CIN, int COUT, int KS, int ACT, int OUTM, bool MASK, int NT>
__global__ void __launch_bounds__(WsGeom<CIN, COUT, KS, NT>::THREADS) conv_ws_kernel(const __grid_constant__ TcArgs args)
{
    using G = WsGeom<CIN, COUT, KS, NT>;
    constexpr int TH = G::TH, TW = G::TW, P = G::P, SW = G::SW, C8 = G::C8, NBUF = G::NBUF, PS = G::PS;
    static_assert(CIN % 16 == 0 && COUT % 16 == 0 && COUT <= 256, "UMMA shape");
    const ConvArgs &a = args.c;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned char *base = smem_raw + ((128 - (smem_u32(smem_raw) & 127)) & 127);
    unsigned char *sw = base;
    unsigned char *sx0 = base + G::WBYTES;
    uint64_t *full = reinterpret_cast<uint64_t *>(sx0 + NBUF * G::XBYTES);
    uint64_t *empty = full + NBUF, *accf = empty + NBUF, *acce = accf + 2;
    uint32_t *tslot = reinterpret_cast<uint32_t *>(acce + 2);
    __shared__ int s_issued, s_consumed;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tiles_x = (a.W + TW - 1) / TW, tiles_y = (a.H + TH - 1) / TH;
    const int per_img = tiles_x * tiles_y, ntiles = a.N * per_img;
    const int mine = blockIdx.x < ntiles ? (ntiles - 1 - blockIdx.x) / gridDim.x + 1 : 0;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tslot)),
                     "r"(G::COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
    }
    if (tid == 0) {
        for (int i = 0; i < NBUF; ++i) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(full + i)));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(empty + i)));
        }
        for (int i = 0; i < 2; ++i) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(accf + i)));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(acce + i)), "r"(G::EW));
        }
        asm volatile("fence.mbarrier_init.release.cluster;\n");
        asm volatile("prefetch.tensormap [%0];\n" ::"l"(reinterpret_cast<uint64_t>(&args.tm)) : "memory");
        s_issued = 0;
        s_consumed = 0;
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n");
    __syncthreads();  // tensor memory allocated
    pdl::trigger();
    pdl::wait();
    for (int i = tid; i < KS * KS * COUT * C8; i += G::THREADS) {
        const int c8 = i % C8, row = i / C8, tap = row / COUT, co = row % COUT;
        cp_async16(sw + (((tap % KS * C8 + c8) * KS + KS - 1 - tap / KS) * COUT + co) * 16, a.w + (size_t)row * CIN + c8 * 8, true);
    }
    cp_async_commit();
    cp_async_wait<0>();
    asm volatile("fence.proxy.async.shared::cta;\n");  // weights visible to the tensor core
    asm volatile("tcgen05.fence::before_thread_sync;\n");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n");
    const uint32_t tmem = *tslot;
    auto fail = [&]() {
        if (a.status) atomicExch(a.status, FLNR_STATUS_TIMEOUT);
    };
    auto origin = [&](int j, int &n, int &ty0, int &tx0) {
        const int t = blockIdx.x + j * gridDim.x;
        n = t / per_img;
        const int r = t % per_img;
        ty0 = (r / tiles_x) * TH;
        tx0 = (r % tiles_x) * TW;
    };

    if (warp == G::EW) {
        if (lane == 0) {  // producer
            for (int j = 0; j < mine; ++j) {
                const int st = j % NBUF;
                if (j >= NBUF && !mbar_wait_thread(smem_u32(empty + st), (uint32_t)((j / NBUF - 1) & 1))) {
                    fail();
                    break;
                }
                int n, ty0, tx0;
                origin(j, n, ty0, tx0);
                const uint32_t bar = smem_u32(full + st);
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(G::TMA_BYTES) : "memory");
                const uint32_t dst = smem_u32(sx0 + st * G::XBYTES);
                load_planes<C8, PS>(dst, &args.tm, a.lx, tx0 - P, ty0 - P, n, bar);
                s_issued = j + 1;
            }
        }
    } else if (warp == G::EW + 1) {
        if (lane == 0) {  // MMA issuer
            const uint64_t adesc0 = umma_sdesc(smem_u32(sx0), PS, G::STEP * SW * 16);
            const uint64_t bdesc0 = umma_sdesc(smem_u32(sw), KS * COUT * 16, 128);
            for (int j = 0; j < mine; ++j) {
                const int st = j % NBUF, acc = j & 1;
                if (!mbar_wait_thread(smem_u32(full + st), (uint32_t)((j / NBUF) & 1))) {
                    fail();
                    break;
                }
                s_consumed = j + 1;
                if (j >= 2 && !mbar_wait_thread(smem_u32(acce + acc), (uint32_t)((j / 2 - 1) & 1))) {
                    fail();
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;\n");
                const uint64_t ab = adesc0 + (uint64_t)((st * G::XBYTES) >> 4);
                issue_phases<G, CIN, COUT, KS, NT>(tmem + (uint32_t)(acc * NT * COUT), ab, bdesc0);
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                    smem_u32(empty + st)));
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                    smem_u32(accf + acc)));
            }
        }
    } else {  // epilogue warps: TMEM lane quarter = warp % 4
        float bias[COUT];
#pragma unroll
        for (int c = 0; c < COUT; ++c) bias[c] = c < a.nbias ? a.bias[c] : 0.f;
        for (int j = 0; j < mine; ++j) {
            const int acc = j & 1;
            if (!mbar_wait_warp(smem_u32(accf + acc), (uint32_t)((j / 2) & 1))) {
                if (lane == 0) fail();
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;\n");
            int n, ty0, tx0;
            origin(j, n, ty0, tx0);
#pragma unroll 1
            for (int t = warp / 4; t < NT; t += G::EW / 4) {
                float v[COUT];
                tc_load_acc<COUT>(tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)((acc * NT + t) * COUT), v);
                if (t + G::EW / 4 >= NT) {
                    __syncwarp();
                    if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(acce + acc)) : "memory");
                }
                tc_store<COUT, ACT, OUTM, MASK>(a, v, bias, n, ty0 + G::STEP * (4 * (warp & 3) + (lane >> 3)) + (G::PHASES ? t : 0),
                         tx0 + (G::PHASES ? 0 : 8 * t) + (lane & 7));
            }
        }
    }
    __syncwarp();  // the single-lane roles rejoin their warps before the CTA barrier
    asm volatile("tcgen05.fence::before_thread_sync;\n");
    __syncthreads();
    if (tid == G::EW * 32) {  // after a failure: let copies still in flight land before the CTA exits
        for (int j = s_consumed; j < s_issued; ++j) mbar_wait_thread(smem_u32(full + j % NBUF), (uint32_t)((j / NBUF) & 1));
    }
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;\n");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(G::COLS));
    }
}

// ---------------------------------------------------------------------------------------
// Two layers in one pass: a KS x KS convolution (ReLU) followed by a 1x1 convolution of its
// output (in1 after in0, o1 after o0).  The first layer's tile never reaches HBM: the
// epilogue warps write its bias + ReLU + bfloat16 values into shared memory as the K-major
// A operand of the 1x1 MMA ([chunk][128 pixels][8 channels]), the MMA lane issues that one
// MMA into a second pair of accumulators, and the epilogue warps finish the tile from it
// (ReLU and BF16 for in1, sigmoid into planar FP32 for o1).  Roles as
// conv_ws_kernel; the MMA lane issues stage j's convolution, then stage j - 1's 1x1, and the
// epilogue warps write stage j's A operands before they finish stage j - 1, so that neither
// waits for the other's round trip.
// Barriers: full/empty per input stage, accf/acce per first accumulator set, a2full (the A
// operands of the 1x1 written, four epilogue warps), acc2f (1x1 committed) and acc2e (its
// accumulators drained, four warps), all per accumulator slot j & 1.
struct alignas(128) TailArgs {
    CUtensorMap tm;
    ConvArgs c;   // first layer: x, w, bias, nbias, N, H, W, status; y (may be NULL)
    ConvArgs c2;  // 1x1 layer: w, bias, nbias, N, H, W and the outputs (y / yf)
    bf16 *w2_kept;   // when given: a copy of the 1x1 layer's weights and biases as this pass used
    float *b2_kept;  // them (the backward pass forms the sigmoid again from the stored a5)
};

template <int CIN, int COUT, int KS, int COUT2, int NT>
struct TailGeom {
    using G1 = WsGeom<CIN, COUT, KS, NT>;
    static constexpr int NBUF = G1::NBUF;
    static constexpr int A2BYTES = (COUT / 8) * 128 * 16;             // one tile's 1x1 A operand
    static constexpr int W2BYTES = ((COUT / 8) * COUT2 * 16 + 127) / 128 * 128;
    static constexpr int NBAR = 2 * NBUF + 10;  // full, empty, accf, acce, a2full, acc2f, acc2e
    static constexpr int SMEM = 128 + G1::WBYTES + W2BYTES + NBUF * G1::XBYTES + 2 * NT * A2BYTES + NBAR * 8 + 16;
    static constexpr int COLS = tmem_cols<2 * NT * (COUT + COUT2)>();
};

template <int CIN, int COUT, int KS, int COUT2, int ACT2, int OUTM2, int NT>
__global__ void __launch_bounds__(WsGeom<CIN, COUT, KS, NT>::THREADS) conv_tail_kernel(const __grid_constant__ TailArgs args)
{
    using T = TailGeom<CIN, COUT, KS, COUT2, NT>;
    using G = typename T::G1;
    constexpr int TH = G::TH, TW = G::TW, P = G::P, SW = G::SW, C8 = G::C8, NBUF = G::NBUF, PS = G::PS;
    static_assert(CIN % 16 == 0 && COUT % 16 == 0 && COUT2 % 16 == 0, "UMMA shape");
    const ConvArgs &a = args.c;
    const ConvArgs &a2 = args.c2;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned char *base = smem_raw + ((128 - (smem_u32(smem_raw) & 127)) & 127);
    unsigned char *sw = base;
    unsigned char *sw2 = sw + G::WBYTES;
    unsigned char *sa2 = sw2 + T::W2BYTES;                   // [2][NT][COUT/8][128][8] 1x1 A operands
    unsigned char *sx0 = sa2 + 2 * NT * T::A2BYTES;
    uint64_t *full = reinterpret_cast<uint64_t *>(sx0 + NBUF * G::XBYTES);
    uint64_t *empty = full + NBUF, *accf = empty + NBUF, *acce = accf + 2;
    uint64_t *a2full = acce + 2, *acc2f = a2full + 2, *acc2e = acc2f + 2;
    uint32_t *tslot = reinterpret_cast<uint32_t *>(acc2e + 2);
    __shared__ int s_issued, s_consumed;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tiles_x = (a.W + TW - 1) / TW, tiles_y = (a.H + TH - 1) / TH;
    const int per_img = tiles_x * tiles_y, ntiles = a.N * per_img;
    const int mine = blockIdx.x < ntiles ? (ntiles - 1 - blockIdx.x) / gridDim.x + 1 : 0;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tslot)),
                     "r"(T::COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
    }
    if (tid == 0) {
        for (int i = 0; i < NBUF; ++i) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(full + i)));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(empty + i)));
        }
        for (int i = 0; i < 2; ++i) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(accf + i)));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(acce + i)), "r"(G::EW));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(a2full + i)), "r"(G::EW));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(acc2f + i)));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(acc2e + i)), "r"(G::EW));
        }
        asm volatile("fence.mbarrier_init.release.cluster;\n");
        asm volatile("prefetch.tensormap [%0];\n" ::"l"(reinterpret_cast<uint64_t>(&args.tm)) : "memory");
        s_issued = 0;
        s_consumed = 0;
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n");
    __syncthreads();  // tensor memory allocated
    pdl::trigger();
    pdl::wait();
    for (int i = tid; i < KS * KS * COUT * C8; i += G::THREADS) {
        const int c8 = i % C8, row = i / C8, tap = row / COUT, co = row % COUT;
        cp_async16(sw + (((tap % KS * C8 + c8) * KS + KS - 1 - tap / KS) * COUT + co) * 16, a.w + (size_t)row * CIN + c8 * 8, true);
    }
    if (args.w2_kept && blockIdx.x == 0) {
        for (int i = tid; i < COUT2 * COUT; i += G::THREADS) args.w2_kept[i] = a2.w[i];
        if (tid < a2.nbias) args.b2_kept[tid] = a2.bias[tid];
    }
    for (int i = tid; i < COUT2 * (COUT / 8); i += G::THREADS) {  // 1x1 weights [COUT2][COUT] -> [c8][COUT2][8]
        const int c8 = i % (COUT / 8), co = i / (COUT / 8);
        cp_async16(sw2 + (c8 * COUT2 + co) * 16, a2.w + (size_t)co * COUT + c8 * 8, true);
    }
    cp_async_commit();
    cp_async_wait<0>();
    asm volatile("fence.proxy.async.shared::cta;\n");  // weights visible to the tensor core
    asm volatile("tcgen05.fence::before_thread_sync;\n");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n");
    const uint32_t tmem = *tslot;
    const uint32_t tmem2 = tmem + (uint32_t)(2 * NT * COUT);  // the 1x1 accumulators
    auto fail = [&]() {
        if (a.status) atomicExch(a.status, FLNR_STATUS_TIMEOUT);
    };
    auto origin = [&](int j, int &n, int &ty0, int &tx0) {
        const int t = blockIdx.x + j * gridDim.x;
        n = t / per_img;
        const int r = t % per_img;
        ty0 = (r / tiles_x) * TH;
        tx0 = (r % tiles_x) * TW;
    };

    if (warp == G::EW) {
        if (lane == 0) {  // producer
            for (int j = 0; j < mine; ++j) {
                const int st = j % NBUF;
                if (j >= NBUF && !mbar_wait_thread(smem_u32(empty + st), (uint32_t)((j / NBUF - 1) & 1))) {
                    fail();
                    break;
                }
                int n, ty0, tx0;
                origin(j, n, ty0, tx0);
                const uint32_t bar = smem_u32(full + st);
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(G::TMA_BYTES) : "memory");
                const uint32_t dst = smem_u32(sx0 + st * G::XBYTES);
                load_planes<C8, PS>(dst, &args.tm, a.lx, tx0 - P, ty0 - P, n, bar);
                s_issued = j + 1;
            }
        }
    } else if (warp == G::EW + 1) {
        if (lane == 0) {  // MMA issuer
            constexpr uint32_t idesc2 = umma_idesc(COUT2);
            const uint64_t adesc0 = umma_sdesc(smem_u32(sx0), PS, G::STEP * SW * 16);
            const uint64_t bdesc0 = umma_sdesc(smem_u32(sw), KS * COUT * 16, 128);
            const uint64_t a2desc0 = umma_sdesc(smem_u32(sa2), 128 * 16, 128);
            const uint64_t b2desc0 = umma_sdesc(smem_u32(sw2), COUT2 * 16, 128);
            // the 1x1 of tile t: its A operand written, its accumulator slot drained
            auto tail = [&](int t) -> bool {
                const int sl = t & 1;
                if (!mbar_wait_thread(smem_u32(a2full + sl), (uint32_t)((t >> 1) & 1))) return false;
                if (t >= 2 && !mbar_wait_thread(smem_u32(acc2e + sl), (uint32_t)(((t >> 1) - 1) & 1))) return false;
                asm volatile("tcgen05.fence::after_thread_sync;\n");
#pragma unroll
                for (int i = 0; i < NT; ++i) {
                    const uint32_t d = tmem2 + (uint32_t)((sl * NT + i) * COUT2);
                    const uint64_t ab = a2desc0 + (uint64_t)(((sl * NT + i) * T::A2BYTES) >> 4);
#pragma unroll
                    for (int kk = 0; kk < COUT / 16; ++kk)
                        umma_bf16(d, ab + (uint64_t)((2 * kk * 128 * 16) >> 4), b2desc0 + (uint64_t)((2 * kk * COUT2 * 16) >> 4),
                                  idesc2, kk ? 1u : 0u);
                }
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                    smem_u32(acc2f + sl)));
                return true;
            };
            bool ok = true;
            for (int j = 0; j < mine && ok; ++j) {
                const int st = j % NBUF, acc = j & 1;
                if (!mbar_wait_thread(smem_u32(full + st), (uint32_t)((j / NBUF) & 1))) {
                    ok = false;
                    break;
                }
                s_consumed = j + 1;
                if (j >= 2 && !mbar_wait_thread(smem_u32(acce + acc), (uint32_t)((j / 2 - 1) & 1))) {
                    ok = false;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;\n");
                const uint64_t ab = adesc0 + (uint64_t)((st * G::XBYTES) >> 4);
                issue_phases<G, CIN, COUT, KS, NT>(tmem + (uint32_t)(acc * NT * COUT), ab, bdesc0);
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                    smem_u32(empty + st)));
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                    smem_u32(accf + acc)));
                if (j >= 1) ok = tail(j - 1);
            }
            if (ok && mine > 0) ok = tail(mine - 1);
            if (!ok) fail();
        }
    } else {  // epilogue warps: TMEM lane quarter q = warp % 4; row 32q + l = pixel (4q + l/8, l%8)
        float bias[COUT], bias2[COUT2];
#pragma unroll
        for (int c = 0; c < COUT; ++c) bias[c] = c < a.nbias ? a.bias[c] : 0.f;
#pragma unroll
        for (int c = 0; c < COUT2; ++c) bias2[c] = c < a2.nbias ? a2.bias[c] : 0.f;
        const int m = 32 * (warp & 3) + lane;
        // the 1x1's accumulators of stage t: false if the wait ran out
        auto finish = [&](int t) -> bool {
            const int sl = t & 1;
            if (!mbar_wait_warp(smem_u32(acc2f + sl), (uint32_t)((t / 2) & 1))) return false;
            asm volatile("tcgen05.fence::after_thread_sync;\n");
            int n, ty0, tx0;
            origin(t, n, ty0, tx0);
#pragma unroll 1
            for (int i = warp / 4; i < NT; i += G::EW / 4) {
                float v2[COUT2];
                tc_load_acc<COUT2>(tmem2 + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)((sl * NT + i) * COUT2), v2);
                if (i + G::EW / 4 >= NT) {
                    __syncwarp();
                    if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(acc2e + sl)) : "memory");
                }
                tc_store<COUT2, ACT2, OUTM2, false>(a2, v2, bias2, n, ty0 + G::STEP * (4 * (warp & 3) + (lane >> 3)) + (G::PHASES ? i : 0),
                         tx0 + (G::PHASES ? 0 : 8 * i) + (lane & 7));
            }
            return true;
        };
        bool ok = true;
        for (int j = 0; j < mine && ok; ++j) {
            const int acc = j & 1;
            if (!mbar_wait_warp(smem_u32(accf + acc), (uint32_t)((j / 2) & 1))) {
                ok = false;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;\n");
            int n, ty0, tx0;
            origin(j, n, ty0, tx0);
#pragma unroll 1
            for (int t = warp / 4; t < NT; t += G::EW / 4) {
                float v[COUT];
                tc_load_acc<COUT>(tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)((acc * NT + t) * COUT), v);
                if (t + G::EW / 4 >= NT) {
                    __syncwarp();
                    if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(acce + acc)) : "memory");
                }
                const int yy = ty0 + G::STEP * (4 * (warp & 3) + (lane >> 3)) + (G::PHASES ? t : 0);
                const int xx = tx0 + (G::PHASES ? 0 : 8 * t) + (lane & 7);
                const bool in = yy < a.H && xx < a.W;
                size_t yc = 0;
                bf16 *yp = a.y ? a.y + pixel_at(a.ly, COUT, a.H, a.W, n, yy, xx, &yc) : nullptr;
                // first layer's bias + ReLU, rounded to bfloat16: the 1x1's A operand row m, and
                // (when a.y is set) the first layer's stored output, which the backward pass reads
                unsigned char *arow = sa2 + (acc * NT + t) * T::A2BYTES + m * 16;
#pragma unroll
                for (int c8 = 0; c8 < COUT / 8; ++c8) {
                    uint4 o;
                    __nv_bfloat162 *oh = reinterpret_cast<__nv_bfloat162 *>(&o);
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        oh[i] = __floats2bfloat162_rn(fmaxf(v[c8 * 8 + 2 * i] + bias[c8 * 8 + 2 * i], 0.f),
                                                      fmaxf(v[c8 * 8 + 2 * i + 1] + bias[c8 * 8 + 2 * i + 1], 0.f));
                    *reinterpret_cast<uint4 *>(arow + c8 * 128 * 16) = o;
                    if (a.y && in) *reinterpret_cast<uint4 *>(yp + c8 * yc) = o;
                }
            }
            asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");  // visible to the tensor core
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(a2full + acc)) : "memory");
            if (j >= 1) ok = finish(j - 1);
        }
        if (ok && mine > 0) ok = finish(mine - 1);
        if (!ok && lane == 0) fail();
    }
    __syncwarp();  // the single-lane roles rejoin their warps before the CTA barrier
    asm volatile("tcgen05.fence::before_thread_sync;\n");
    __syncthreads();
    if (tid == G::EW * 32) {  // after a failure: let copies still in flight land before the CTA exits
        for (int j = s_consumed; j < s_issued; ++j) mbar_wait_thread(smem_u32(full + j % NBUF), (uint32_t)((j / NBUF) & 1));
    }
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;\n");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(T::COLS));
    }
}

// ---------------------------------------------------------------------------------------
// Decoder convolution (3x3, ReLU) on up2(lo) ++ skip without forming the upsampled map.
// A stage covers 32 x 16 output pixels: a 16 x 8 block of low-resolution positions (i0 + g,
// j0 + r) and its four parity classes (a, b), output pixel (2(i0 + g) + a, 2(j0 + r) + b),
// one 128-row accumulator per class (row 8g + r).  For tap (dy, dx), t = a + dy - 1 and
// u = b + dx - 1, every pixel of class (a, b) reads the low-resolution map at
// (i0 + g + t/2, j0 + r + u/2) (floor division) and the skip at full-resolution pixel
// (2(i0 + g + t/2) + (t mod 2), 2(j0 + r + u/2) + (u mod 2)).  Rows of a class step by one
// low-resolution position in both operands, so both are plain K-major tiles:
//   lo    CA/8 planes [18][10][8] (rows i0 - 1 .. i0 + 16, columns j0 - 1 .. j0 + 8), one TMA
//         box copy each;
//   skip  its four parity planes (a', b') x CB/8 chunks [18][10][8] (rows i0 - 1 .. i0 + 16
//         of row parity a', columns j0 - 1 .. j0 + 8 of column parity b'), one TMA box copy
//         each from a 5-D view (a column pair's channels, column pairs, row parity, row
//         pairs, images or chunk planes) in which the start channel selects the column parity.
// The products are those of the convolution on the concatenated map; only their order of
// accumulation differs.  Roles and waits as conv_ws_kernel; the MMA lane issues the four
// classes of a stage into one of two accumulator sets (4 * COUT columns each).
// Bound by the number of MMAs: reading the 128 x 16 operand A costs about 50 clocks whatever N is
// up to 64, and the four classes' 36 taps x (CA + CB)/16 of them took 71 us for d0a and 54 us for
// d1a of a 1920x1080 pass.  The two classes (a, 0) and (a, 1) read position (t, u) for taps
// dx = u + 1 and dx = u, whose weights lie side by side in shared memory ([dy][chunk][2 - dx]), so
// one MMA of N = 2 COUT serves both: 24 instead of 36 per channel step, in the same order for
// each class.
template <int CA, int CB, int COUT, int NBUF>
struct UpGeom {
    static constexpr int SH = 18, SW = 10;                       // staged rows and columns
    static constexpr int PS = (SH * SW * 16 + 127) / 128 * 128;  // one chunk plane [SH][SW][8]
    static constexpr int CA8 = CA / 8, CB8 = CB / 8, C8 = CA8 + CB8;
    static constexpr int PLANES = CA8 + 4 * CB8;                 // lo chunks, then skip (a', b', chunk)
    static constexpr int XBYTES = PLANES * PS;
    static constexpr int TMA_BYTES = PLANES * SH * SW * 16;
    static constexpr int WBYTES = (9 * C8 * COUT * 16 + 127) / 128 * 128;
    static constexpr int NBAR = 2 * NBUF + 4;
    static constexpr int SMEM = 128 + WBYTES + NBUF * XBYTES + NBAR * 8 + 16;
    static constexpr int COLS = tmem_cols<8 * COUT>();          // two sets of four class accumulators
};

struct alignas(128) UpArgs {
    CUtensorMap tlo, tskip;
    ConvArgs c;  // x = lo (CA channels, H/2 x W/2), x2 = skip (CB channels, H x W), H and W even
};

__device__ __forceinline__ void tma_load_5d(uint32_t dst, const CUtensorMap *tm, int c0, int c1, int c2, int c3,
                                            int c4, uint32_t mbar)
{
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, %6}], [%7];\n" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(tm)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(mbar)
        : "memory");
}

template <int CA, int CB, int COUT, int NBUF>
__global__ void __launch_bounds__(kWsThreads) conv_up_kernel(const __grid_constant__ UpArgs args)
{
    using G = UpGeom<CA, CB, COUT, NBUF>;
    constexpr int PS = G::PS, SW = G::SW, CA8 = G::CA8, CB8 = G::CB8, C8 = G::C8;
    static_assert(CA % 16 == 0 && CB % 16 == 0 && COUT % 16 == 0 && 8 * COUT <= 256, "UMMA shape");
    const ConvArgs &a = args.c;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned char *base = smem_raw + ((128 - (smem_u32(smem_raw) & 127)) & 127);
    unsigned char *sw = base;
    unsigned char *sx0 = base + G::WBYTES;
    uint64_t *full = reinterpret_cast<uint64_t *>(sx0 + NBUF * G::XBYTES);
    uint64_t *empty = full + NBUF, *accf = empty + NBUF, *acce = accf + 2;
    uint32_t *tslot = reinterpret_cast<uint32_t *>(acce + 2);
    __shared__ int s_issued, s_consumed;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int HL = a.H / 2, WL = a.W / 2;
    const int tiles_x = (WL + 7) / 8, tiles_y = (HL + 15) / 16;
    const int per_img = tiles_x * tiles_y, ntiles = a.N * per_img;
    const int mine = blockIdx.x < ntiles ? (ntiles - 1 - blockIdx.x) / gridDim.x + 1 : 0;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tslot)),
                     "r"(G::COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
    }
    if (tid == 0) {
        for (int i = 0; i < NBUF; ++i) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(full + i)));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(empty + i)));
        }
        for (int i = 0; i < 2; ++i) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(accf + i)));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 4;\n" ::"r"(smem_u32(acce + i)));  // 4 epilogue warps
        }
        asm volatile("fence.mbarrier_init.release.cluster;\n");
        asm volatile("prefetch.tensormap [%0];\n" ::"l"(reinterpret_cast<uint64_t>(&args.tlo)) : "memory");
        asm volatile("prefetch.tensormap [%0];\n" ::"l"(reinterpret_cast<uint64_t>(&args.tskip)) : "memory");
        s_issued = 0;
        s_consumed = 0;
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n");
    __syncthreads();  // tensor memory allocated
    pdl::trigger();
    pdl::wait();
    // weights: global [tap][COUT][CA + CB] -> shared [dy][c8][2 - dx][COUT][8] (lo chunks first)
    for (int i = tid; i < 9 * COUT * C8; i += kWsThreads) {
        const int c8 = i % C8, row = i / C8, tap = row / COUT, co = row % COUT;
        cp_async16(sw + ((((tap / 3) * C8 + c8) * 3 + 2 - tap % 3) * COUT + co) * 16, a.w + (size_t)row * (CA + CB) + c8 * 8, true);
    }
    cp_async_commit();
    cp_async_wait<0>();
    asm volatile("fence.proxy.async.shared::cta;\n");  // weights visible to the tensor core
    asm volatile("tcgen05.fence::before_thread_sync;\n");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n");
    const uint32_t tmem = *tslot;
    auto fail = [&]() {
        if (a.status) atomicExch(a.status, FLNR_STATUS_TIMEOUT);
    };
    auto origin = [&](int j, int &n, int &i0, int &j0) {
        const int t = blockIdx.x + j * gridDim.x;
        n = t / per_img;
        const int r = t % per_img;
        i0 = (r / tiles_x) * 16;
        j0 = (r % tiles_x) * 8;
    };

    if (warp == 4) {
        if (lane == 0) {  // producer
            for (int j = 0; j < mine; ++j) {
                const int st = j % NBUF;
                if (j >= NBUF && !mbar_wait_thread(smem_u32(empty + st), (uint32_t)((j / NBUF - 1) & 1))) {
                    fail();
                    break;
                }
                int n, i0, j0;
                origin(j, n, i0, j0);
                const uint32_t bar = smem_u32(full + st);
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(G::TMA_BYTES) : "memory");
                const uint32_t dst = smem_u32(sx0 + st * G::XBYTES);
                load_planes<CA8, PS>(dst, &args.tlo, a.lx, j0 - 1, i0 - 1, n, bar);
                const bool nhwc = a.lx == kNHWC;
#pragma unroll
                for (int pp = 0; pp < 4; ++pp) {
#pragma unroll
                    for (int k = 0; k < CB8; ++k)
                        tma_load_5d(dst + (CA8 + pp * CB8 + k) * PS, &args.tskip, (pp & 1) * (nhwc ? CB : 8) + (nhwc ? 8 * k : 0),
                                    j0 - 1, pp >> 1, i0 - 1, nhwc ? n : n * CB8 + k, bar);
                }
                s_issued = j + 1;
            }
        }
    } else if (warp == 5) {
        if (lane == 0) {  // MMA issuer
            constexpr uint32_t idesc1 = umma_idesc(COUT), idesc2 = umma_idesc(2 * COUT);
            const uint64_t adesc0 = umma_sdesc(smem_u32(sx0), PS, SW * 16);
            const uint64_t bdesc0 = umma_sdesc(smem_u32(sw), 3 * COUT * 16, 128);
            for (int j = 0; j < mine; ++j) {
                const int st = j % NBUF, acc = j & 1;
                if (!mbar_wait_thread(smem_u32(full + st), (uint32_t)((j / NBUF) & 1))) {
                    fail();
                    break;
                }
                s_consumed = j + 1;
                if (j >= 2 && !mbar_wait_thread(smem_u32(acce + acc), (uint32_t)((j / 2 - 1) & 1))) {
                    fail();
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;\n");
                const uint64_t ab = adesc0 + (uint64_t)((st * G::XBYTES) >> 4);
#pragma unroll
                for (int ca = 0; ca < 2; ++ca) {
                    const uint32_t d0 = tmem + (uint32_t)((acc * 4 + 2 * ca) * COUT);
#pragma unroll
                    for (int pos = 0; pos < 12; ++pos) {
                        const int dy = pos / 4, t = ca + dy - 1, u = pos % 4 - 1;  // t, u: -1 .. 2
                        const int oy = t >> 1, ox = u >> 1, pp = (t & 1) * 2 + (u & 1);
                        const int at = ((oy + 1) * SW + (ox + 1)) * 16;
                        const bool both = u == 0 || u == 1;  // classes b = 0 (dx = u + 1) and 1 (dx = u)
                        const uint32_t d = d0 + (u == 2 ? COUT : 0);
                        const int tap0 = u == -1 ? 2 : u == 0 ? 1 : 0;  // 2 - dx of the first class
#pragma unroll
                        for (int kk = 0; kk < C8 / 2; ++kk) {
                            const uint32_t aoff = (uint32_t)(((kk < CA8 / 2 ? 2 * kk : CA8 + pp * CB8 + 2 * kk - CA8) * PS + at) >> 4);
                            const uint64_t b = bdesc0 + (uint32_t)((((dy * C8 + 2 * kk) * 3 + tap0) * COUT * 16) >> 4);
                            if (dy == 0 && u == 0 && kk == 0) {  // class b = 1 starts here
                                umma_bf16(d, ab + aoff, b, idesc1, 1u);
                                umma_bf16(d + COUT, ab + aoff, b + (uint32_t)(COUT * 16 >> 4), idesc1, 0u);
                            } else {
                                umma_bf16(d, ab + aoff, b, both ? idesc2 : idesc1, (pos | kk) ? 1u : 0u);
                            }
                        }
                    }
                }
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                    smem_u32(empty + st)));
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                    smem_u32(accf + acc)));
            }
        }
    } else {  // epilogue warps 0-3: TMEM lane quarter = warp; row 32w + l = position (4w + l/8, l%8)
        float bias[COUT];
#pragma unroll
        for (int c = 0; c < COUT; ++c) bias[c] = c < a.nbias ? a.bias[c] : 0.f;
        const int g = 4 * warp + (lane >> 3), r = lane & 7;
        for (int j = 0; j < mine; ++j) {
            const int acc = j & 1;
            if (!mbar_wait_warp(smem_u32(accf + acc), (uint32_t)((j / 2) & 1))) {
                if (lane == 0) fail();
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;\n");
            int n, i0, j0;
            origin(j, n, i0, j0);
#pragma unroll 1
            for (int cls = 0; cls < 4; ++cls) {
                float v[COUT];
                tc_load_acc<COUT>(tmem + ((uint32_t)(32 * warp) << 16) + (uint32_t)((acc * 4 + cls) * COUT), v);
                if (cls == 3) {
                    __syncwarp();
                    if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(acce + acc)) : "memory");
                }
                tc_store<COUT, 1, 0, false>(a, v, bias, n, 2 * (i0 + g) + (cls >> 1), 2 * (j0 + r) + (cls & 1));
            }
        }
    }
    __syncwarp();  // the single-lane roles rejoin their warps before the CTA barrier
    asm volatile("tcgen05.fence::before_thread_sync;\n");
    __syncthreads();
    if (tid == 4 * 32) {  // after a failure: let copies still in flight land before the CTA exits
        for (int j = s_consumed; j < s_issued; ++j) mbar_wait_thread(smem_u32(full + j % NBUF), (uint32_t)((j / NBUF) & 1));
    }
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;\n");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(G::COLS));
    }
}

// ---------------------------------------------------------------------------------------
// Stride-2 3x3 convolution (the second convolution of an encoder block, Sec. 3.3; ReLU):
// output pixel (oy, ox) of the [N][H/2][W/2] map reads input pixels (2oy + u - 1,
// 2ox + v - 1) of the [N][H][W] input (H, W even), so only the kept outputs are computed.
// A tile is 16 x 8 output pixels (oy0 + g, ox0 + r), accumulator row 8g + r.  Its input is
// staged per 8-channel chunk as four parity planes: rows 2i + pr for row pairs
// i = oy0 - 1 .. oy0 + 15, and columns 2j + pc for column pairs j = ox0 .. ox0 + 7 (even
// columns, pc = 0, planes [17][8][8]) or j = ox0 - 1 .. ox0 + 7 (odd columns, pc = 1, planes
// [17][9][8]).  Tap u reads row parity pr = (u != 1) at row offset (u != 0); tap v reads
// column parity pc = (v != 1) at column offset (v == 2) of its plane.  Consecutive output
// pixels step by one pair, so every tap's operand is a plain K-major tile of the staged
// planes: 9 taps x CIN/16 MMAs per tile, no products for the dropped positions.  The planes
// are those of a kParity input (boxes 8 and 9 columns wide of its parity planes: contiguous
// rows), or come from two 5-D views of an NHWC input (channels of a column pair, column pairs,
// row parity, row pairs, images) whose start channel pc * CIN + 8k selects the column parity.
// Roles, waits and epilogue as conv_ws_kernel.
template <int CIN, int COUT, int NBUF_>
struct S2Geom {
    static constexpr int TH = 16, TW = 8, SH = TH + 1, WE = TW, WO = TW + 1, C8 = CIN / 8, NBUF = NBUF_;
    static constexpr int PSE = (SH * WE * 16 + 127) / 128 * 128;  // even-column plane [SH][WE][8]
    static constexpr int PSO = (SH * WO * 16 + 127) / 128 * 128;  // odd-column plane [SH][WO][8]
    static constexpr int ROWP = C8 * (PSE + PSO);                  // one row parity: even chunks, odd chunks
    static constexpr int XBYTES = 2 * ROWP;
    static constexpr int TMA_BYTES = 2 * C8 * SH * (WE + WO) * 16;
    static constexpr int WBYTES = (9 * C8 * COUT * 16 + 127) / 128 * 128;
    static constexpr int NBAR = 2 * NBUF + 4;
    static constexpr int SMEM = 128 + WBYTES + NBUF * XBYTES + NBAR * 8 + 16;
    static constexpr int COLS = tmem_cols<2 * COUT>();
    static_assert(PSE % 128 == 0 && PSO % 128 == 0, "TMA destinations 128-byte aligned");
};

struct alignas(128) S2Args {
    CUtensorMap te, to;  // even-column and odd-column views of the input
    ConvArgs c;          // x: CIN channels (H, W: the input's size), kNHWC or kParity; y at H/2 x W/2
};

template <int CIN, int COUT, int NBUF>
__global__ void __launch_bounds__(kWsThreads) conv_s2_kernel(const __grid_constant__ S2Args args)
{
    using G = S2Geom<CIN, COUT, NBUF>;
    constexpr int TH = G::TH, TW = G::TW, C8 = G::C8, PSE = G::PSE, PSO = G::PSO, ROWP = G::ROWP;
    static_assert(CIN % 16 == 0 && COUT % 16 == 0 && 2 * COUT <= 256, "UMMA shape");
    const ConvArgs &a = args.c;
    ConvArgs ao = a;  // the output map
    ao.H = a.H / 2;
    ao.W = a.W / 2;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned char *base = smem_raw + ((128 - (smem_u32(smem_raw) & 127)) & 127);
    unsigned char *sw = base;
    unsigned char *sx0 = base + G::WBYTES;
    uint64_t *full = reinterpret_cast<uint64_t *>(sx0 + NBUF * G::XBYTES);
    uint64_t *empty = full + NBUF, *accf = empty + NBUF, *acce = accf + 2;
    uint32_t *tslot = reinterpret_cast<uint32_t *>(acce + 2);
    __shared__ int s_issued, s_consumed;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tiles_x = (ao.W + TW - 1) / TW, tiles_y = (ao.H + TH - 1) / TH;
    const int per_img = tiles_x * tiles_y, ntiles = a.N * per_img;
    const int mine = blockIdx.x < ntiles ? (ntiles - 1 - blockIdx.x) / gridDim.x + 1 : 0;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tslot)),
                     "r"(G::COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
    }
    if (tid == 0) {
        for (int i = 0; i < NBUF; ++i) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(full + i)));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(empty + i)));
        }
        for (int i = 0; i < 2; ++i) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(accf + i)));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 4;\n" ::"r"(smem_u32(acce + i)));  // 4 epilogue warps
        }
        asm volatile("fence.mbarrier_init.release.cluster;\n");
        asm volatile("prefetch.tensormap [%0];\n" ::"l"(reinterpret_cast<uint64_t>(&args.te)) : "memory");
        asm volatile("prefetch.tensormap [%0];\n" ::"l"(reinterpret_cast<uint64_t>(&args.to)) : "memory");
        s_issued = 0;
        s_consumed = 0;
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n");
    __syncthreads();  // tensor memory allocated
    pdl::trigger();
    pdl::wait();
    for (int i = tid; i < 9 * COUT * C8; i += kWsThreads) {
        const int c8 = i % C8, row = i / C8, tap = row / COUT, co = row % COUT;
        cp_async16(sw + ((tap * C8 + c8) * COUT + co) * 16, a.w + (size_t)row * CIN + c8 * 8, true);
    }
    cp_async_commit();
    cp_async_wait<0>();
    asm volatile("fence.proxy.async.shared::cta;\n");  // weights visible to the tensor core
    asm volatile("tcgen05.fence::before_thread_sync;\n");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n");
    const uint32_t tmem = *tslot;
    auto fail = [&]() {
        if (a.status) atomicExch(a.status, FLNR_STATUS_TIMEOUT);
    };
    auto origin = [&](int j, int &n, int &oy0, int &ox0) {
        const int t = blockIdx.x + j * gridDim.x;
        n = t / per_img;
        const int r = t % per_img;
        oy0 = (r / tiles_x) * TH;
        ox0 = (r % tiles_x) * TW;
    };

    if (warp == 4) {
        if (lane == 0) {  // producer
            for (int j = 0; j < mine; ++j) {
                const int st = j % NBUF;
                if (j >= NBUF && !mbar_wait_thread(smem_u32(empty + st), (uint32_t)((j / NBUF - 1) & 1))) {
                    fail();
                    break;
                }
                int n, oy0, ox0;
                origin(j, n, oy0, ox0);
                const uint32_t bar = smem_u32(full + st);
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(G::TMA_BYTES) : "memory");
                const uint32_t dst = smem_u32(sx0 + st * G::XBYTES);
#pragma unroll
                for (int pr = 0; pr < 2; ++pr) {
#pragma unroll
                    for (int k = 0; k < C8; ++k) {
                        const uint32_t de = dst + pr * ROWP + k * PSE, dd = dst + pr * ROWP + C8 * PSE + k * PSO;
                        if (a.lx == kNHWC) {
                            tma_load_5d(de, &args.te, 8 * k, ox0, pr, oy0 - 1, n, bar);
                            tma_load_5d(dd, &args.to, CIN + 8 * k, ox0 - 1, pr, oy0 - 1, n, bar);
                        } else {
                            tma_load_4d(de, &args.te, 4 * ox0, oy0 - 1, 4 * k + 2 * pr, n, bar);
                            tma_load_4d(dd, &args.to, 4 * (ox0 - 1), oy0 - 1, 4 * k + 2 * pr + 1, n, bar);
                        }
                    }
                }
                s_issued = j + 1;
            }
        }
    } else if (warp == 5) {
        if (lane == 0) {  // MMA issuer
            constexpr uint32_t idesc = umma_idesc(COUT);
            const uint64_t adesc_e = umma_sdesc(smem_u32(sx0), PSE, G::WE * 16);
            const uint64_t adesc_o = umma_sdesc(smem_u32(sx0), PSO, G::WO * 16);
            const uint64_t bdesc0 = umma_sdesc(smem_u32(sw), COUT * 16, 128);
            for (int j = 0; j < mine; ++j) {
                const int st = j % NBUF, acc = j & 1;
                if (!mbar_wait_thread(smem_u32(full + st), (uint32_t)((j / NBUF) & 1))) {
                    fail();
                    break;
                }
                s_consumed = j + 1;
                if (j >= 2 && !mbar_wait_thread(smem_u32(acce + acc), (uint32_t)((j / 2 - 1) & 1))) {
                    fail();
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;\n");
                const uint32_t sbase = (uint32_t)(st * G::XBYTES);
                const uint32_t d = tmem + (uint32_t)(acc * COUT);
#pragma unroll
                for (int tap = 0; tap < 9; ++tap) {
                    const int u = tap / 3, v = tap % 3;
                    const int pr = u != 1, pc = v != 1, ro = u != 0, co = v == 2;
#pragma unroll
                    for (int kk = 0; kk < C8 / 2; ++kk) {
                        const uint32_t off = pc ? sbase + pr * ROWP + C8 * PSE + 2 * kk * PSO + (ro * G::WO + co) * 16
                                                : sbase + pr * ROWP + 2 * kk * PSE + ro * G::WE * 16;
                        const uint64_t ad = (pc ? adesc_o : adesc_e) + (uint64_t)(off >> 4);
                        const uint32_t boff = (uint32_t)(((tap * C8 + 2 * kk) * COUT * 16) >> 4);
                        umma_bf16(d, ad, bdesc0 + boff, idesc, (tap | kk) ? 1u : 0u);
                    }
                }
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                    smem_u32(empty + st)));
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                    smem_u32(accf + acc)));
            }
        }
    } else {  // epilogue warps 0-3: TMEM lane quarter = warp
        float bias[COUT];
#pragma unroll
        for (int c = 0; c < COUT; ++c) bias[c] = c < a.nbias ? a.bias[c] : 0.f;
        for (int j = 0; j < mine; ++j) {
            const int acc = j & 1;
            if (!mbar_wait_warp(smem_u32(accf + acc), (uint32_t)((j / 2) & 1))) {
                if (lane == 0) fail();
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;\n");
            float v[COUT];
            tc_load_acc<COUT>(tmem + ((uint32_t)(32 * warp) << 16) + (uint32_t)(acc * COUT), v);
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(acce + acc)) : "memory");
            int n, oy0, ox0;
            origin(j, n, oy0, ox0);
            tc_store<COUT, 1, 0, false>(ao, v, bias, n, oy0 + 4 * warp + (lane >> 3), ox0 + (lane & 7));
        }
    }
    __syncwarp();  // the single-lane roles rejoin their warps before the CTA barrier
    asm volatile("tcgen05.fence::before_thread_sync;\n");
    __syncthreads();
    if (tid == 4 * 32) {  // after a failure: let copies still in flight land before the CTA exits
        for (int j = s_consumed; j < s_issued; ++j) mbar_wait_thread(smem_u32(full + j % NBUF), (uint32_t)((j / NBUF) & 1));
    }
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;\n");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(G::COLS));
    }
}

// ---------------------------------------------------------------------------------------
// Weight and bias gradients (tcgen05):
//   dW[o][i][tap] = sum_p dz[p][o] x[p + off(tap)][i],   db[o] = sum_p dz[p][o],
// as D[o][(tap, i)] += A[o][p] B[(tap, i)][p] with the pixels as K.  Eight pixels of a row by
// eight channels, 128 bytes, are a core matrix of an MN-major operand as they lie (channels
// contiguous, pixels 16 bytes apart), so neither x nor dz is transposed or copied.  x is staged
// row by row, [row][chunk][col][8]: the channel chunks of consecutive rows are then one sequence
// of N groups, XW * 16 bytes apart, and one MMA takes three taps of a column kx (ky = 0, 1, 2)
// at N = 3 CIN.  An MMA costs about 60 clocks whatever its N up to there, so that is three times
// fewer clocks than a tap each (16 -> 16 channels on a 16 x 128^2 batch: 28.8 us, now 13.6).
// M = 64 rows of A are read: COUT of dz, the rest whatever the shared memory after it holds, rows
// of D that nothing reads.
// A tile is 16 rows x 8 pixels, K = 128.  A CTA walks tiles blockIdx.x, + gridDim.x, ...: one lane
// loads them by TMA into a ring, one lane issues a tile's MMAs, warp 3 adds up the bias gradient
// from the staged dz.  The tensor cores do not round their accumulations to nearest: a chain of n of
// them is off by up to n units in the last place, all in one direction.  So the accumulators start
// again every CHAIN tiles, and summing warps, one per 16 rows of D, add a chain's sums to
// FP32 sums of their own in registers (the 16 rows over all 32 lanes, as C fragments), unit by unit
// (WgGeom) while the MMAs of the next units run.  Operands of one sign, error over the sum, 16 -> 16
// channels: one chain per CTA 3.4e-6 on a 16 x 128^2 batch and 6.5e-5 at 1920x1080, two tiles 2.5e-7
// on both, one tile 1.1e-7.  Backward pass of 16 x 128^2: 373 us with one chain, 378 with two tiles.  Where nine taps do
// not fit (CIN = 64, 96), blockIdx.y takes a column of taps each.  MODE 1 is the stride-2 layer:
// dz at the output's size and x as parity planes (conv_s2_kernel's taps: rows ky = 0 and 2 of
// parity 1, ky = 1 of parity 0), so that no product is spent on dropped positions.  Every CTA
// writes its accumulators to its slice of the layer's partials and wgrad_reduce_kernel adds the
// slices in a fixed order.
// The form before built both operands with ldmatrix and shared stores from NHWC pixels and took
// its bias sums in kernels of their own: the backward pass of a 16 x 128^2 batch spent 343 us in
// weight gradients, 158 us in bias gradients and 110 us in twelve reductions; now about 150 us with the
// bias and one reduction of 27 us.
struct alignas(128) WgradArgs {
    CUtensorMap tx, tdz;
    float *part;  // [gridDim.x][COUT][KS^2 CIN + 8]
    int N, H, W;  // the size of dz
    int layout;   // of dz (and, MODE 0, of x): kNHWC or kPlanes
    int *status;
};

// Groups of tap columns that a layer's gradient is split into: the accumulators of one fit in tensor memory
__host__ __device__ constexpr int wgrad_groups(int cin, int ks) { return ks * ks * cin > 512 ? ks : 1; }
// Slices of a layer's partials: one CTA per SM and tap group
constexpr int wgrad_slots(int n_sm, int groups) { return n_sm / groups > 0 ? n_sm / groups : 1; }

template <int CIN, int COUT, int KS, int MODE>
struct WgGeom {
    static constexpr int P = KS / 2, C8 = CIN / 8, O8 = COUT / 8, TAPS = KS * KS;
    static constexpr int NG = wgrad_groups(CIN, KS);      // tap columns split over blockIdx.y
    static constexpr int KXN = KS / NG;                   // tap columns per CTA
    static constexpr int XH = MODE ? 17 : 16 + 2 * P, XW = MODE ? 9 : 8 + 2 * P;  // staged rows and columns
    static constexpr int RP = C8 * XW * 16;                                       // one row, all chunks
    static constexpr int XP = (XH * RP + 127) / 128 * 128;                        // x (MODE 1: one parity plane)
    static constexpr int NXP = MODE ? 4 : 1;
    static constexpr int DP = 16 * 8 * 16;                                        // one dz plane
    static constexpr int STAGE = NXP * XP + O8 * DP;
    static constexpr int NBUF = 4 * STAGE <= 150 * 1024 ? 4 : 2;
    static constexpr int TMA_BYTES = NXP * XH * RP + O8 * DP;
    static constexpr int PAD = (8 - O8) * DP;  // the 64 rows of A reach past the last stage
    static constexpr int CTOT = TAPS * CIN + 8;  // columns of a partial: (kx, ky, channel), then the bias
    // tap rows of one MMA: MODE 0 as many as N = 256 holds; MODE 1 rows 0 and 2, then row 1
    static constexpr int KYN = KS == 1 ? 1 : MODE ? 2 : (3 * CIN <= 256 ? 3 : 2);
    // units: the accumulators of one MMA (tap column, group of tap rows), each handed over by itself
    static constexpr int NSG = (KS + KYN - 1) / KYN, U = KXN * NSG;
    static constexpr int DCOLS = KXN * KS * CIN;   // accumulator columns of a tile
    static constexpr int SETS = U == 1 ? 2 : 1;    // a lone unit has two sets, so that the MMAs need not wait
    static constexpr int CHAIN = NG > 1 ? 1 : 2;   // tiles that the tensor cores accumulate
    static constexpr int COLS = tmem_cols<SETS * DCOLS>();
    __host__ __device__ static constexpr int unit_col(int u) { return ((u / NSG) * KS + (u % NSG) * KYN) * CIN; }
    __host__ __device__ static constexpr int unit_len(int u) { return (KS - (u % NSG) * KYN < KYN ? KS - (u % NSG) * KYN : KYN) * CIN; }
    // summing warps: one per 16 rows of D, two where one's half of the columns fills its registers
    static constexpr int EW = COUT / 16, EH = DCOLS > 288 ? 2 : 1;
    static constexpr int THREADS = 32 * (EH == 1 ? 4 + EW : 12);
    static constexpr int SMEM = 128 + NBUF * STAGE + PAD + (2 * NBUF + 2 * U * SETS) * 8 + 16;
};

// instruction descriptor, kind::f16: D FP32, A and B BF16, both MN-major, M = 64, N = n
__host__ __device__ constexpr uint32_t umma_idesc_mn64(int n)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(64 >> 4) << 24);
}

// The MMAs of unit u of one staged tile (tap columns from kx0 on) into the accumulators at `set`
template <int CIN, int COUT, int KS, int MODE>
__device__ __forceinline__ void wgrad_mmas(const int u, uint32_t stage, uint32_t set, int kx0, bool first)
{
    using G = WgGeom<CIN, COUT, KS, MODE>;
    // MN-major, no swizzle: LBO between K groups (8 pixels), SBO between groups of 8 channels
    const uint64_t ad0 = umma_sdesc(stage + G::NXP * G::XP, 128, G::DP);
    const uint64_t bd0 = umma_sdesc(stage, G::RP, G::XW * 16);
    const int s = u % G::NSG * G::KYN;  // first slot of the column (MODE 1: ky = 0, 2, 1)
    const int kx = kx0 + u / G::NSG;
    uint32_t off;
    if (MODE) off = (uint32_t)((2 * (s == 0) + (kx != 1)) * G::XP + (s != 0) * G::RP + (kx != 0) * 16);
    else off = (uint32_t)(s * G::RP + kx * 16);
    const uint32_t idesc = umma_idesc_mn64(G::unit_len(u));
#pragma unroll
    for (int ks = 0; ks < 8; ++ks)
        umma_bf16(set + G::unit_col(u), ad0 + (uint64_t)((ks * 256) >> 4), bd0 + (uint64_t)((off + 2 * ks * G::RP) >> 4), idesc,
                  first && ks == 0 ? 0u : 1u);
}

// 16 lanes x 8 N columns of the warp's TMEM lane quarter, as C fragments: of block b (8 columns)
// v[4 b], v[4 b + 1] are row lane / 4, columns 2 (lane % 4) and + 1, v[4 b + 2], v[4 b + 3] row lane / 4 + 8
template <int N>
__device__ __forceinline__ void tmem_ld_frag(uint32_t taddr, uint32_t *r)
{
    if constexpr (N >= 4) {
        asm volatile(
            "tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
              "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
            : "r"(taddr));
        if constexpr (N > 4) tmem_ld_frag<N - 4>(taddr + 32, r + 16);
    } else if constexpr (N >= 2) {
        asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                     : "r"(taddr));
        if constexpr (N > 2) tmem_ld_frag<N - 2>(taddr + 16, r + 8);
    } else {
        asm volatile("tcgen05.ld.sync.aligned.16x256b.x1.b32 {%0,%1,%2,%3}, [%4];\n"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                     : "r"(taddr));
    }
}

// acc += the LEN columns at taddr (16 lanes), up to 48 columns in flight
template <int LEN>
__device__ __forceinline__ void add_frags(float *acc, uint32_t taddr)
{
    constexpr int B = LEN % 48 == 0 ? 48 : LEN % 32 == 0 ? 32 : LEN % 24 == 0 ? 24 : 16;
    static_assert(LEN % B == 0 && B % 8 == 0, "columns in blocks of eight");
#pragma unroll
    for (int c = 0; c < LEN; c += B) {
        uint32_t r[B / 2];
        tmem_ld_frag<B / 8>(taddr + (uint32_t)c, r);
        asm volatile("tcgen05.wait::ld.sync.aligned;\n");
#pragma unroll
        for (int i = 0; i < B / 2; ++i) acc[c / 2 + i] += __uint_as_float(r[i]);
    }
}

template <int CIN, int COUT, int KS, int MODE, int... UN>
__device__ __forceinline__ void wgrad_body(const WgradArgs &a, std::integer_sequence<int, UN...>)
{
    using G = WgGeom<CIN, COUT, KS, MODE>;
    static_assert(CIN % 16 == 0 && COUT % 16 == 0 && COUT <= 64 && (MODE == 0 || KS == 3), "UMMA shape");
    constexpr int NBUF = G::NBUF, SETS = G::SETS, CHAIN = G::CHAIN;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned char *base = smem_raw + ((128 - (smem_u32(smem_raw) & 127)) & 127);
    uint64_t *full = reinterpret_cast<uint64_t *>(base + NBUF * G::STAGE + G::PAD);
    uint64_t *empty = full + NBUF, *ufull = empty + NBUF, *uempty = ufull + G::U * SETS;  // [U][SETS]
    __shared__ uint32_t s_tmem;
    __shared__ int s_issued, s_consumed, s_fail;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tiles_x = (a.W + 7) / 8, tiles_y = (a.H + 15) / 16;
    const int per_img = tiles_x * tiles_y, ntiles = a.N * per_img;
    const int mine = blockIdx.x < ntiles ? (ntiles - 1 - blockIdx.x) / gridDim.x + 1 : 0;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&s_tmem)),
                     "r"(G::COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
    }
    if (tid == 0) {
        for (int i = 0; i < NBUF; ++i) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(full + i)));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 2;\n" ::"r"(smem_u32(empty + i)));  // MMAs, bias warp
        }
        for (int i = 0; i < G::U * SETS; ++i) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(ufull + i)));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(uempty + i)), "r"(G::EW * G::EH));
        }
        asm volatile("fence.mbarrier_init.release.cluster;\n");
        s_issued = s_consumed = s_fail = 0;
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n");
    const uint32_t tmem = s_tmem;
    pdl::trigger();
    pdl::wait();

    // summing warps: quarter and half of the columns; acc: the sums over this CTA's tiles
    const int quarter = warp & 3, half = (warp - 4) >> 2;
    const bool sums = warp >= 4 && quarter < G::EW && half < G::EH;
    float acc[G::DCOLS / G::EH / 2];
    if (warp == 1 && lane == 0) {  // producer
        for (int j = 0; j < mine; ++j) {
            const int st = j % NBUF;
            if (j >= NBUF && !mbar_wait_thread(smem_u32(empty + st), (uint32_t)((j / NBUF - 1) & 1))) {
                s_fail = 1;
                break;
            }
            const int t = blockIdx.x + j * gridDim.x, n = t / per_img, r = t % per_img;
            const int ty0 = (r / tiles_x) * 16, tx0 = (r % tiles_x) * 8;
            const uint32_t bar = smem_u32(full + st), dst = smem_u32(base + st * G::STAGE);
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(G::TMA_BYTES) : "memory");
            if (MODE) {
#pragma unroll
                for (int pp = 0; pp < 4; ++pp) tma_load_5d(dst + pp * G::XP, &a.tx, 4 * (tx0 - 1), 0, ty0 - 1, pp, n, bar);
            } else if (a.layout == kNHWC) {
                tma_load_5d(dst, &a.tx, 0, tx0 - G::P, 0, ty0 - G::P, n, bar);
            } else {
                tma_load_4d(dst, &a.tx, 4 * (tx0 - G::P), 0, ty0 - G::P, n, bar);
            }
            load_planes<G::O8, G::DP>(dst + G::NXP * G::XP, &a.tdz, a.layout, tx0, ty0, n, bar);
            s_issued = j + 1;
        }
    } else if (warp == 2 && lane == 0) {  // MMA issuer
        int j = 0;
        for (; j < mine; ++j) {
            const int st = j % NBUF, chain = j / CHAIN, set = chain % SETS;
            const bool first = j % CHAIN == 0, last = (j + 1) % CHAIN == 0 || j + 1 == mine;
            if (!mbar_wait_thread(smem_u32(full + st), (uint32_t)((j / NBUF) & 1))) {
                s_fail = 1;
                break;
            }
            s_consumed = j + 1;
            asm volatile("tcgen05.fence::after_thread_sync;\n");
            bool ok = true;
            const uint32_t stage = smem_u32(base + st * G::STAGE), d = tmem + set * G::DCOLS;
            const int kx0 = G::NG > 1 ? (int)blockIdx.y : 0;
            if (first) {
#pragma unroll
                for (int u = 0; u < G::U; ++u) {
                    if (chain >= SETS) {
                        ok &= mbar_wait_thread(smem_u32(uempty + u * SETS + set), (uint32_t)((chain / SETS - 1) & 1));
                        asm volatile("tcgen05.fence::after_thread_sync;\n");
                    }
                    wgrad_mmas<CIN, COUT, KS, MODE>(u, stage, d, kx0, true);
                    if (last) asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                        smem_u32(ufull + u * SETS + set)));
                }
            } else {
#pragma unroll
                for (int u = 0; u < G::U; ++u) {
                    wgrad_mmas<CIN, COUT, KS, MODE>(u, stage, d, kx0, false);
                    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                        smem_u32(ufull + u * SETS + set)));
                }
            }
            if (!ok) {
                s_fail = 1;
                break;
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                smem_u32(empty + st)));
        }
        // the last stages' commits have arrived before the CTA exits
        for (int i = mine > NBUF ? mine - NBUF : 0; j == mine && i < mine; ++i)
            if (!mbar_wait_thread(smem_u32(empty + i % NBUF), (uint32_t)((i / NBUF) & 1))) s_fail = 1;
    } else if (warp == 3) {  // bias gradient: LP lanes per 8-channel chunk of dz, every LP-th pixel each
        constexpr int LP = 32 / G::O8;
        const int o8 = lane / LP, l = lane % LP;
        float bsum[8] = {};  // over the tiles; a tile's own sums in two, even and odd steps
        for (int j = 0; j < mine; ++j) {
            const int st = j % NBUF;
            if (!mbar_wait_vote(smem_u32(full + st), (uint32_t)((j / NBUF) & 1))) {
                if (lane == 0) s_fail = 1;
                break;
            }
            if (blockIdx.y == 0) {
                const uint4 *dz = reinterpret_cast<const uint4 *>(base + st * G::STAGE + G::NXP * G::XP + o8 * G::DP) + l;
                float2 t[2][4] = {};
#pragma unroll
                for (int p0 = 0; p0 < 128 / LP; p0 += 8) {
                    uint4 v[8];  // eight loads in flight
#pragma unroll
                    for (int p = 0; p < 8; ++p) v[p] = dz[(p0 + p) * LP];
#pragma unroll
                    for (int p = 0; p < 8; ++p) {
                        const __nv_bfloat162 *h = reinterpret_cast<const __nv_bfloat162 *>(&v[p]);
#pragma unroll
                        for (int i = 0; i < 4; ++i) t[p & 1][i] = __fadd2_rn(t[p & 1][i], __bfloat1622float2(h[i]));
                    }
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float2 u = __fadd2_rn(t[0][i], t[1][i]);
                    bsum[2 * i] += u.x;
                    bsum[2 * i + 1] += u.y;
                }
            }
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(empty + st)) : "memory");
        }
        if (blockIdx.y == 0) {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
#pragma unroll
                for (int o = LP / 2; o > 0; o >>= 1) bsum[i] += __shfl_xor_sync(0xffffffffu, bsum[i], o);
                if (l == 0) a.part[((size_t)blockIdx.x * COUT + o8 * 8 + i) * G::CTOT + G::TAPS * CIN] = bsum[i];
            }
        }
    } else if (sums) {
#pragma unroll
        for (int i = 0; i < G::DCOLS / G::EH / 2; ++i) acc[i] = 0.f;
        bool ok = true;
        for (int j = 0; j < (mine + CHAIN - 1) / CHAIN && ok; ++j) {
            const int set = j % SETS;
            auto unit = [&](auto un) {
                constexpr int u = decltype(un)::value, len = G::unit_len(u) / G::EH;
                if (!ok) return;
                if (!mbar_wait_vote(smem_u32(ufull + u * SETS + set), (uint32_t)((j / SETS) & 1))) {
                    ok = false;
                    return;
                }
                asm volatile("tcgen05.fence::after_thread_sync;\n");
                add_frags<len>(acc + G::unit_col(u) / G::EH / 2,
                               tmem + ((uint32_t)(32 * quarter) << 16) + (uint32_t)(set * G::DCOLS + G::unit_col(u) + half * len));
                asm volatile("tcgen05.fence::before_thread_sync;\n");
                __syncwarp();
                if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(uempty + u * SETS + set)) : "memory");
            };
            (unit(std::integral_constant<int, UN>{}), ...);
        }
        if (!ok && lane == 0) s_fail = 1;
    }
    __syncwarp();
    __syncthreads();  // every role is through: the sums hold every tile, or a wait ran out
    if (s_fail) {
        if (tid == 0 && a.status) atomicExch(a.status, FLNR_STATUS_TIMEOUT);
        if (tid == 32)  // let copies still in flight land before the CTA exits
            for (int j = s_consumed; j < s_issued; ++j) mbar_wait_thread(smem_u32(full + j % NBUF), (uint32_t)((j / NBUF) & 1));
    } else if (sums) {
        // M = 64: rows 16 w .. 16 w + 15 in lanes 0-15 of lane quarter w
        float *dst = a.part + ((size_t)blockIdx.x * COUT + 16 * quarter + lane / 4) * G::CTOT + blockIdx.y * G::DCOLS + 2 * (lane & 3);
        auto unit = [&](auto un) {
            constexpr int u = decltype(un)::value, len = G::unit_len(u) / G::EH;
            const float *v = acc + G::unit_col(u) / G::EH / 2;
            float *d = dst + G::unit_col(u) + half * len;
#pragma unroll
            for (int b = 0; b < len / 8; ++b) {
                *reinterpret_cast<float2 *>(d + 8 * b) = make_float2(v[4 * b], v[4 * b + 1]);
                *reinterpret_cast<float2 *>(d + 8 * b + 8 * G::CTOT) = make_float2(v[4 * b + 2], v[4 * b + 3]);
            }
        };
        (unit(std::integral_constant<int, UN>{}), ...);
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;\n");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(G::COLS));
    }
}

template <int CIN, int COUT, int KS, int MODE>
__global__ void __launch_bounds__(WgGeom<CIN, COUT, KS, MODE>::THREADS) wgrad_tc_kernel(const __grid_constant__ WgradArgs a)
{
    wgrad_body<CIN, COUT, KS, MODE>(a, std::make_integer_sequence<int, WgGeom<CIN, COUT, KS, MODE>::U>{});
}

// The layers' partials into the FP32 master gradients, one launch for all of them: element f of
// a layer is (o, column) of its slices [slices][COUT][CTOT]; 32 consecutive elements per CTA
// (coalesced), sixteen warps take slices w, w + 16, ... and their sums are added, in a fixed order, so
// the result is the same every run.  Padding channels are skipped.
struct RedLayer {
    const float *part;
    float *gw, *gb;
    int slices, cout, cin, ks, s2, cin_true, cout_true, first_block;
};
struct RedArgs {
    RedLayer l[kNL];
    int n = 0, blocks = 0;
};
constexpr int kRedWarps = 16;

__global__ void __launch_bounds__(32 * kRedWarps) wgrad_reduce_kernel(const __grid_constant__ RedArgs a)
{
    pdl::trigger();
    pdl::wait();
    int k = 0;
    while (k + 1 < a.n && (int)blockIdx.x >= a.l[k + 1].first_block) ++k;
    const RedLayer &l = a.l[k];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int taps = l.ks * l.ks, ctot = taps * l.cin + 8, total = l.cout * ctot;
    const int f = (blockIdx.x - l.first_block) * 32 + lane;
    __shared__ float s_sum[kRedWarps][32];
    float s = 0.f;
    if (f < total) {
        const float *p = l.part + f;
        constexpr int NB = 10;  // loads in flight: all of a warp's slices on 152 SMs
        for (int j = w; j < l.slices; j += NB * kRedWarps) {
            float v[NB];
#pragma unroll
            for (int u = 0; u < NB; ++u) {
                const int jj = j + u * kRedWarps;
                v[u] = jj < l.slices ? __ldg(p + (size_t)jj * total) : 0.f;
            }
            // in pairs, here and below: half the rounding of a chain
            s += (((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]))) + (v[8] + v[9]);
        }
    }
    s_sum[w][lane] = s;
    __syncthreads();
    if (w != 0 || f >= total) return;
    float v[kRedWarps];
#pragma unroll
    for (int u = 0; u < kRedWarps; ++u) v[u] = s_sum[u][lane];
#pragma unroll
    for (int n = kRedWarps / 2; n > 0; n /= 2)
#pragma unroll
        for (int u = 0; u < n; ++u) v[u] += v[u + n];
    s = v[0];
    const int o = f / ctot, c = f % ctot;
    if (o >= l.cout_true) return;
    if (c == taps * l.cin) {
        l.gb[o] += s;
    } else if (c < taps * l.cin) {
        const int i = c % l.cin, slot = c / l.cin % l.ks, kx = c / (l.cin * l.ks);
        const int ky = l.s2 ? (slot == 1 ? 2 : slot == 2 ? 1 : 0) : slot;
        if (i < l.cin_true) l.gw[((size_t)o * l.cin_true + i) * taps + ky * l.ks + kx] += s;
    }
}

// ---------------------------------------------------------------------------------------
// Elementwise and layout kernels
// planar fp32 [N][11][H][W] -> bf16 planes with 16 channels (11 used); the radiance channels
// enter the network as log(1 + max(Y, 0)), which keeps fireflies from dominating the features
__global__ void pack_input_kernel(const float *in, bf16 *x, int N, int H, int W)
{
    pdl::trigger();
    pdl::wait();
    const size_t hw = (size_t)H * W, total = (size_t)N * hw;
    for (size_t p = (size_t)blockIdx.x * blockDim.x + threadIdx.x; p < total; p += (size_t)gridDim.x * blockDim.x) {
        const size_t n = p / hw, o = p % hw;
        alignas(16) bf16 v[16];
#pragma unroll
        for (int c = 0; c < 16; ++c) {
            float u = 0.f;
            if (c < 8) u = in[(n * 11 + c) * hw + o];
            else if (c < 11) u = log1pf(fmaxf(in[(n * 11 + c) * hw + o], 0.f));  // radiance: log(1 + max(Y, 0))
            v[c] = __float2bfloat16(u);
        }
        *reinterpret_cast<uint4 *>(x + (2 * n * hw + o) * 8) = *reinterpret_cast<uint4 *>(v);
        *reinterpret_cast<uint4 *>(x + ((2 * n + 1) * hw + o) * 8) = *reinterpret_cast<uint4 *>(v + 8);
    }
}

// gradient with respect to the network's planar input [N][11][H][W] from the gradient dx (bf16
// planes, 16 channels) with respect to the packed input x: the guides pass through; a radiance
// channel was read as L = log(1 + max(Y, 0)), whose derivative is 1 / (1 + Y) = exp(-L) for
// Y > 0 and 0 for Y < 0 (L is the stored bfloat16 value, so Y > 0 exactly when L > 0)
__global__ void unpack_grad_kernel(const bf16 *dx, const bf16 *x, float *g, int N, int H, int W)
{
    pdl::trigger();
    pdl::wait();
    const size_t hw = (size_t)H * W, total = (size_t)N * hw;
    for (size_t p = (size_t)blockIdx.x * blockDim.x + threadIdx.x; p < total; p += (size_t)gridDim.x * blockDim.x) {
        const size_t n = p / hw, o = p % hw;
#pragma unroll
        for (int c = 0; c < 11; ++c) {
            const size_t e = ((2 * n + c / 8) * hw + o) * 8 + c % 8;
            float d = __bfloat162float(dx[e]);
            if (c >= 8) {
                const float L = __bfloat162float(x[e]);
                d = L > 0.f ? d * expf(-L) : 0.f;
            }
            g[(n * 11 + c) * hw + o] = d;
        }
    }
}

// nearest 2x upsampling of lo (Ca channels, H/2 x W/2) concatenated with skip (Cb channels,
// H x W), all bf16 planes (the input of a decoder level, materialised for its weight gradient)
__global__ void upcat_kernel(const bf16 *lo, const bf16 *skip, bf16 *y, int N, int H, int W, int Ca, int Cb)
{
    pdl::trigger();
    pdl::wait();
    // one thread per pixel of a chunk plane of y: 16-byte copies
    const int C8 = (Ca + Cb) / 8, A8 = Ca / 8, B8 = Cb / 8, hw = H * W;
    const size_t total = (size_t)N * C8 * hw;
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
        const int q = (int)(e / hw), p = (int)(e % hw), n = q / C8, c8 = q % C8;
        const uint4 *src;
        if (c8 < A8)
            src = reinterpret_cast<const uint4 *>(lo) + (size_t)(n * A8 + c8) * (hw / 4) + (size_t)(p / W / 2) * (W / 2) + p % W / 2;
        else
            src = reinterpret_cast<const uint4 *>(skip) + (size_t)(n * B8 + c8 - A8) * hw + p;
        reinterpret_cast<uint4 *>(y)[e] = *src;
    }
}

// backward of up ++ skip (bf16 planes): g_lo[q][c] = mask(lo) * sum_{2x2} gy[p][c] (c < Ca);
// g_skip[p][c] = gy[p][Ca + c] in fp32 planes (unmasked, the caller masks where the skip is
// consumed)
__global__ void upcat_bwd_kernel(const bf16 *gy, const bf16 *lo, bf16 *g_lo, float *g_skip, int N, int H, int W,
                                 int Ca, int Cb)
{
    pdl::trigger();
    pdl::wait();
    // eight channels of one pixel per thread: 16-byte loads and stores
    const int A8 = Ca / 8, B8 = Cb / 8, C8 = A8 + B8, hw = H * W, hl = hw / 4, Wl = W / 2;
    const size_t tl = (size_t)N * A8 * hl, ts = (size_t)N * B8 * hw;
    const uint4 *g4 = reinterpret_cast<const uint4 *>(gy);
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < tl + ts; e += (size_t)gridDim.x * blockDim.x) {
        if (e < tl) {
            const int q = (int)(e / hl), pl = (int)(e % hl), n = q / A8, c8 = q % A8;
            const size_t b = (size_t)(n * C8 + c8) * hw + (size_t)(2 * (pl / Wl)) * W + 2 * (pl % Wl);
            const uint4 r0 = g4[b], r1 = g4[b + 1], r2 = g4[b + W], r3 = g4[b + W + 1];
            const uint4 l = reinterpret_cast<const uint4 *>(lo)[e];
            const bf16 *g0 = reinterpret_cast<const bf16 *>(&r0), *g1 = reinterpret_cast<const bf16 *>(&r1);
            const bf16 *g2 = reinterpret_cast<const bf16 *>(&r2), *g3 = reinterpret_cast<const bf16 *>(&r3);
            const bf16 *lv = reinterpret_cast<const bf16 *>(&l);
            uint4 o;
            bf16 *ov = reinterpret_cast<bf16 *>(&o);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const float sum = __bfloat162float(g0[i]) + __bfloat162float(g1[i]) + __bfloat162float(g2[i]) +
                                  __bfloat162float(g3[i]);
                ov[i] = __float2bfloat16(__bfloat162float(lv[i]) > 0.f ? sum : 0.f);
            }
            reinterpret_cast<uint4 *>(g_lo)[e] = o;
        } else {
            const size_t f = e - tl;
            const int q = (int)(f / hw), p = (int)(f % hw), n = q / B8, c8 = q % B8;
            const uint4 r = g4[(size_t)(n * C8 + A8 + c8) * hw + p];
            const bf16 *rv = reinterpret_cast<const bf16 *>(&r);
            float4 v0, v1;
            v0.x = __bfloat162float(rv[0]); v0.y = __bfloat162float(rv[1]);
            v0.z = __bfloat162float(rv[2]); v0.w = __bfloat162float(rv[3]);
            v1.x = __bfloat162float(rv[4]); v1.y = __bfloat162float(rv[5]);
            v1.z = __bfloat162float(rv[6]); v1.w = __bfloat162float(rv[7]);
            *reinterpret_cast<float4 *>(g_skip + 8 * f) = v0;
            *reinterpret_cast<float4 *>(g_skip + 8 * f + 4) = v1;
        }
    }
}

// Gradient with respect to the pre-activation of a layer whose ReLU output f (C channels,
// Ho x Wo) feeds the next encoder convolution (gradient g_path, bf16 planes) and, when g_skip is
// given, a decoder skip (fp32 planes): dz = mask(f) * (g_skip + g_path); no mask when f is NULL.
// S = 2 (the layer strides by 2): dz is written zero-upsampled onto the layer's input grid
// 2Ho x 2Wo, nonzero only at even rows and columns, so that the stride-1 input-gradient kernel
// gives the stride-2 layer's gradient, and, when dlo is given, at its own size too (for the
// weight gradient).
template <int S>
__global__ void join_bwd_kernel(const float *g_skip, const bf16 *g_path, const bf16 *f, bf16 *dz, bf16 *dlo, int N,
                                int Ho, int Wo, int C)
{
    pdl::trigger();
    pdl::wait();
    // eight channels of one pixel per thread: 16-byte loads and stores
    const int hw = S * Ho * S * Wo, W = S * Wo;
    const size_t total = (size_t)N * (C / 8) * hw;
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
        const int k = (int)(e / hw), p = (int)(e % hw), x = p % W, y = p / W;
        uint4 o = make_uint4(0u, 0u, 0u, 0u);  // bfloat16 +0
        if (S == 1 || ((x | y) & 1) == 0) {
            const size_t q = (size_t)k * Ho * Wo + (size_t)(y / S) * Wo + x / S;
            const uint4 gp = reinterpret_cast<const uint4 *>(g_path)[q];
            const bf16 *gv = reinterpret_cast<const bf16 *>(&gp);
            float sk[8];
            if (g_skip) {
                const float4 s0 = *reinterpret_cast<const float4 *>(g_skip + 8 * q);
                const float4 s1 = *reinterpret_cast<const float4 *>(g_skip + 8 * q + 4);
                sk[0] = s0.x; sk[1] = s0.y; sk[2] = s0.z; sk[3] = s0.w;
                sk[4] = s1.x; sk[5] = s1.y; sk[6] = s1.z; sk[7] = s1.w;
            }
            uint4 fm = make_uint4(0u, 0u, 0u, 0u);
            if (f) fm = reinterpret_cast<const uint4 *>(f)[q];
            const bf16 *fv = reinterpret_cast<const bf16 *>(&fm);
            bf16 *ov = reinterpret_cast<bf16 *>(&o);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                float v = __bfloat162float(gv[i]) + (g_skip ? sk[i] : 0.f);
                if (f && !(__bfloat162float(fv[i]) > 0.f)) v = 0.f;
                ov[i] = __float2bfloat16(v);
            }
            if (S == 2 && dlo) reinterpret_cast<uint4 *>(dlo)[q] = o;
        }
        reinterpret_cast<uint4 *>(dz)[e] = o;
    }
}

// zero-upsampling of an NHWC gradient [N][Ho][Wo][C] onto [N][2Ho][2Wo][C] (flnr_layer)
__global__ void spread_nhwc_kernel(const bf16 *g, bf16 *dz, int N, int Ho, int Wo, int C)
{
    pdl::trigger();
    pdl::wait();
    const int C8 = C / 8, W = 2 * Wo, H = 2 * Ho;
    const size_t total = (size_t)N * H * W * C8;
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
        const size_t p = e / C8;
        const int c8 = (int)(e % C8), x = (int)(p % W), y = (int)(p / W % H);
        const size_t n = p / ((size_t)W * H);
        uint4 o = make_uint4(0u, 0u, 0u, 0u);
        if (((x | y) & 1) == 0) o = reinterpret_cast<const uint4 *>(g)[((n * Ho + y / 2) * Wo + x / 2) * C8 + c8];
        reinterpret_cast<uint4 *>(dz)[e] = o;
    }
}

// Every layer's master fp32 [Cout][Cin][k][k] -> forward bf16 [tap][CoutP][CinP] and dgrad bf16
// [tap'][CinP][CoutP] with tap' = taps - 1 - tap (rotated by 180 degrees), zero pads; blockIdx.y
// is the layer (one launch for the twelve: 21 us of twelve launches per training step before).
struct WeightsArgs {
    const float *w[kNL];
    bf16 *wf[kNL], *wd[kNL];
    int cin[kNL], cout[kNL], k[kNL];
};
__global__ void weights_kernel(const __grid_constant__ WeightsArgs a)
{
    const int l = blockIdx.y, cin = a.cin[l], cout = a.cout[l], cinp = pad16(cin), coutp = pad16(cout);
    const int taps = a.k[l] * a.k[l], total = taps * coutp * cinp;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
        const int i = e % cinp, o = (e / cinp) % coutp, tap = e / (cinp * coutp);
        const float v = (i < cin && o < cout) ? a.w[l][((size_t)o * cin + i) * taps + tap] : 0.f;
        a.wf[l][e] = __float2bfloat16(v);
        a.wd[l][((size_t)(taps - 1 - tap) * cinp + i) * coutp + o] = __float2bfloat16(v);
    }
}

__global__ void adam_kernel(float *w, const float *g, float *m, float *v, size_t n, float lr, float b1, float b2,
                            float eps, float c1, float c2)
{
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
        const float gr = g[e];
        const float mm = b1 * m[e] + (1.f - b1) * gr;
        const float vv = b2 * v[e] + (1.f - b2) * gr * gr;
        m[e] = mm;
        v[e] = vv;
        w[e] -= lr * (mm / c1) / (sqrtf(vv / c2) + eps);
    }
}

// L1 loss between prediction and reference (planar fp32, n values): writes d/dpred = sign / n
// and accumulates the mean absolute error into *loss
// SMAPE of pred against ref (Sec. 3.3 trains FLNR on it): loss += mean |p - r| / D with
// D = |p| + |r| + eps, and d/dp = (sign(p - r) / D - |p - r| sign(p) / D^2) / n
__global__ void smape_kernel(const float *pred, const float *ref, float *grad, float *loss, size_t n, float eps)
{
    __shared__ float part[256];
    float s = 0.f;
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
        const float p = pred[e], d = p - ref[e], a = fabsf(d);
        const float inv = 1.f / (fabsf(p) + fabsf(ref[e]) + eps);
        const float sd = d > 0.f ? 1.f : (d < 0.f ? -1.f : 0.f), sp = p > 0.f ? 1.f : (p < 0.f ? -1.f : 0.f);
        grad[e] = (sd - a * sp * inv) * inv / (float)n;
        s += a * inv;
    }
    part[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) part[threadIdx.x] += part[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) atomicAdd(loss, part[0] / (float)n);
}

__global__ void l1_kernel(const float *pred, const float *ref, float *grad, float *loss, size_t n)
{
    __shared__ float part[256];
    float s = 0.f;
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
        const float d = pred[e] - ref[e];
        grad[e] = (d > 0.f ? 1.f : (d < 0.f ? -1.f : 0.f)) / (float)n;
        s += fabsf(d);
    }
    part[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) part[threadIdx.x] += part[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) atomicAdd(loss, part[0] / (float)n);
}

int egrid(size_t n) { return (int)((n + 255) / 256 < 8192 ? (n + 255) / 256 : 8192); }

// ---------------------------------------------------------------------------------------
// Launch helpers for the template instantiations the network uses.
// 4-D map of an NHWC bf16 tensor [N][H][W][C]: box (8 channels, bw, bh, 1), zero fill outside
cudaError_t make_tmap(CUtensorMap *m, const void *base, int C, int W, int H, int N, int bw, int bh)
{
    PFN_cuTensorMapEncodeTiled_v12000 fn = tma::encoder();
    if (!fn) return cudaErrorNotSupported;
    const cuuint64_t dims[4] = {(cuuint64_t)C, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)N};
    const cuuint64_t strides[3] = {(cuuint64_t)C * 2, (cuuint64_t)W * C * 2, (cuuint64_t)H * W * C * 2};
    const cuuint32_t box[4] = {8, (cuuint32_t)bw, (cuuint32_t)bh, 1};
    const cuuint32_t es[4] = {1, 1, 1, 1};
    const CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(base), dims, strides, box, es,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// 5-D map of an NHWC bf16 tensor [N][H][W][C] (H, W even) that stages one parity plane per
// box: dims (2C channels of a column pair, W/2 column pairs, 2 row parities, H/2 row pairs,
// N); box (8, bw, 1, bh, 1).  The start channel b * C + 8k selects column parity b, chunk k.
cudaError_t make_tmap_parity(CUtensorMap *m, const void *base, int C, int W, int H, int N, int bw, int bh)
{
    PFN_cuTensorMapEncodeTiled_v12000 fn = tma::encoder();
    if (!fn) return cudaErrorNotSupported;
    const cuuint64_t dims[5] = {(cuuint64_t)2 * C, (cuuint64_t)W / 2, 2, (cuuint64_t)H / 2, (cuuint64_t)N};
    const cuuint64_t strides[4] = {(cuuint64_t)C * 4, (cuuint64_t)W * C * 2, (cuuint64_t)W * C * 4,
                                   (cuuint64_t)H * W * C * 2};
    const cuuint32_t box[5] = {8, (cuuint32_t)bw, 1, (cuuint32_t)bh, 1};
    const cuuint32_t es[5] = {1, 1, 1, 1, 1};
    const CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void *>(base), dims, strides, box, es,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// 4-D map of planes of 16-byte pixels [N][P][H][W] (32-bit elements, four per pixel): box bw
// columns x bh rows of one plane, zero fill outside
cudaError_t make_tmap_planes(CUtensorMap *m, const void *base, int P, int W, int H, int N, int bw, int bh)
{
    PFN_cuTensorMapEncodeTiled_v12000 fn = tma::encoder();
    if (!fn) return cudaErrorNotSupported;
    const cuuint64_t row = (cuuint64_t)W * 16;
    const cuuint64_t dims[4] = {(cuuint64_t)4 * W, (cuuint64_t)H, (cuuint64_t)P, (cuuint64_t)N};
    const cuuint64_t strides[3] = {row, row * H, row * H * P};
    const cuuint32_t box[4] = {(cuuint32_t)(4 * bw), (cuuint32_t)bh, 1, 1};
    const cuuint32_t es[4] = {1, 1, 1, 1};
    const CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_UINT32, 4, const_cast<void *>(base), dims, strides, box, es,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// 5-D map of a kPlanes tensor (H, W even) that stages one parity plane per box: dims (16 values
// of a column pair, W/2 column pairs, 2 row parities, H/2 row pairs, C/8 * N chunk planes); box
// (8, bw, 1, bh, 1).  The start value 8 b selects column parity b.
cudaError_t make_tmap_pairs(CUtensorMap *m, const void *base, int C, int W, int H, int N, int bw, int bh)
{
    PFN_cuTensorMapEncodeTiled_v12000 fn = tma::encoder();
    if (!fn) return cudaErrorNotSupported;
    const cuuint64_t row = (cuuint64_t)W * 16;
    const cuuint64_t dims[5] = {16, (cuuint64_t)W / 2, 2, (cuuint64_t)H / 2, (cuuint64_t)(C / 8) * N};
    const cuuint64_t strides[4] = {32, row, 2 * row, row * H};
    const cuuint32_t box[5] = {8, (cuuint32_t)bw, 1, (cuuint32_t)bh, 1};
    const cuuint32_t es[5] = {1, 1, 1, 1, 1};
    const CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void *>(base), dims, strides, box, es,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// Map of x for the weight gradients, boxes in the order [row][chunk][col][8]: a kNHWC or kPlanes
// tensor (box bw columns x all chunks x bh rows), or one parity plane of a kParity tensor
// (W, H: the plane's size).
cudaError_t make_tmap_rows(CUtensorMap *m, int layout, const void *base, int C, int W, int H, int N, int bw, int bh)
{
    PFN_cuTensorMapEncodeTiled_v12000 fn = tma::encoder();
    if (!fn) return cudaErrorNotSupported;
    const cuuint64_t w = W, h = H, n = N, c8 = C / 8, row = w * 16;
    const cuuint32_t es[5] = {1, 1, 1, 1, 1}, b4 = 4 * bw, bb = bw, hh = bh, cc = C / 8;
    CUresult r;
    if (layout == kNHWC) {
        const cuuint64_t dims[5] = {8, w, c8, h, n}, st[4] = {c8 * 16, 16, c8 * row, c8 * row * h};
        const cuuint32_t box[5] = {8, bb, cc, hh, 1};
        r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void *>(base), dims, st, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    } else if (layout == kPlanes) {
        const cuuint64_t dims[4] = {4 * w, c8, h, n}, st[3] = {row * h, row, row * h * c8};
        const cuuint32_t box[4] = {b4, cc, hh, 1};
        r = fn(m, CU_TENSOR_MAP_DATA_TYPE_UINT32, 4, const_cast<void *>(base), dims, st, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    } else {
        const cuuint64_t dims[5] = {4 * w, c8, h, 4, n}, st[4] = {4 * row * h, row, row * h, 4 * row * h * c8};
        const cuuint32_t box[5] = {b4, cc, hh, 1, 1};
        r = fn(m, CU_TENSOR_MAP_DATA_TYPE_UINT32, 5, const_cast<void *>(base), dims, st, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    }
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// the map of a tensor in layout kNHWC or kPlanes, for load_planes
cudaError_t make_tmap_tile(CUtensorMap *m, int layout, const void *base, int C, int W, int H, int N, int bw, int bh)
{
    return layout == kNHWC ? make_tmap(m, base, C, W, H, N, bw, bh) : make_tmap_planes(m, base, C / 8, W, H, N, bw, bh);
}

// Resident CTAs per SM of a kernel that allocates tensor memory.  The occupancy API reports one
// CTA per SM for such kernels, so the count is computed here from the kernel's registers,
// shared memory and threads, and capped at 512 / (tensor-memory columns per CTA); where threads
// alone would allow more CTAs than tensor memory can hold, the shared-memory request is raised
// (tc_smem) so that no more can be resident (an allocation never has to wait for another CTA).
constexpr int kSmemPerSm = 228 * 1024, kReservedPerCta = 1024, kThreadsPerSm = 2048;
constexpr size_t tc_smem(int smem, int cols, int threads)
{
    const int cap = 512 / cols;
    const int least = cap < kThreadsPerSm / threads ? kSmemPerSm / cap - kReservedPerCta - 256 : 0;
    return (size_t)(smem > least ? smem : least);
}
struct Resident {
    int per_sm = 0, n_sm = 0;
};
// known: the kernel's own, so that it is asked once per device.
template <class K>
cudaError_t resident(PerDevice<Resident> &known, K kern, int threads, size_t smem, int cols, Resident &out)
{
    int dev = 0;
    const cudaError_t ed = cudaGetDevice(&dev);
    if (ed != cudaSuccess) return ed;
    return known.get(dev, [&](Resident &v) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
        if (e != cudaSuccess) return e;
        cudaFuncAttributes fa;
        if ((e = cudaFuncGetAttributes(&fa, kern)) != cudaSuccess) return e;
        int n_sm = 0;
        if ((e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
        // registers are split over the SM's four sub-partitions: warps per sub-partition first
        const int regs_per_warp = (fa.numRegs * 32 + 255) / 256 * 256;
        const int by_regs = (4 * (16384 / regs_per_warp)) / (threads / 32);
        const int by_smem = kSmemPerSm / ((int)smem + (int)fa.sharedSizeBytes + kReservedPerCta);
        int r = kThreadsPerSm / threads;
        r = r < by_regs ? r : by_regs;
        r = r < by_smem ? r : by_smem;
        r = r < 512 / cols ? r : 512 / cols;
        if (r < 1) return cudaErrorInvalidConfiguration;
        v.n_sm = n_sm;
        v.per_sm = r;
        return cudaSuccess;
    }, out);
}

// Stages of a map of N images.  NT tiles per stage share a halo, a hand-over of the barriers and
// eight epilogue warps; they are taken as soon as half the SMs get a stage (a 1920x1080 forward
// pass took 472 us with several tiles per stage and 516 us with one, forward and backward over
// 16 x 128^2 572 and 621 us, both before the row phases); smaller maps would leave the chip idle.
long long stages(int N, int H, int W, int th, int tw) { return (long long)N * ((H + th - 1) / th) * ((W + tw - 1) / tw); }

// Launch of the warp-specialised convolution with NT tiles per stage; when only asked, *fits
// reports whether that many per stage is the better choice.
template <int CIN, int COUT, int KS, int ACT, int OUTM, bool MASK, int NT>
cudaError_t conv_ws_launch_nt(const ConvArgs &a, bool ask, bool *fits, cudaStream_t st)
{
    using G = WsGeom<CIN, COUT, KS, NT>;
    constexpr size_t smem = tc_smem(G::SMEM, G::COLS, G::THREADS);
    static_assert(smem <= 227 * 1024, "warp-specialised conv tile does not fit in shared memory");
    auto kern = conv_ws_kernel<CIN, COUT, KS, ACT, OUTM, MASK, NT>;
    static PerDevice<Resident> known;
    Resident res;
    cudaError_t e = resident(known, kern, G::THREADS, smem, G::COLS, res);
    if (e != cudaSuccess) return e;
    const long long ntiles = stages(a.N, a.H, a.W, G::TH, G::TW), cap = (long long)res.per_sm * res.n_sm;
    if (ask) {
        *fits = 2 * ntiles >= res.n_sm;
        return cudaSuccess;
    }
    if (ntiles <= 0) return cudaSuccess;
    TcArgs ta;
    std::memset(&ta, 0, sizeof(ta));
    ta.c = a;
    if ((e = make_tmap_tile(&ta.tm, a.lx, a.x, CIN, a.W, a.H, a.N, G::SW, G::SH)) != cudaSuccess) return e;
    return pdl::launch(kern, (int)(ntiles < cap ? ntiles : cap), G::THREADS, smem, st, ta);
}
template <int CIN, int COUT, int KS, int ACT, int OUTM, bool MASK>
cudaError_t conv_ws_launch(const ConvArgs &a, cudaStream_t st)
{
    constexpr int NT = CIN <= 32 && COUT <= 32 ? 4 : 2;
    bool wide = false;
    cudaError_t e = conv_ws_launch_nt<CIN, COUT, KS, ACT, OUTM, MASK, NT>(a, true, &wide, st);
    if (e != cudaSuccess) return e;
    if (wide) return conv_ws_launch_nt<CIN, COUT, KS, ACT, OUTM, MASK, NT>(a, false, nullptr, st);
    return conv_ws_launch_nt<CIN, COUT, KS, ACT, OUTM, MASK, 1>(a, false, nullptr, st);
}

// Input gradient of a layer on the tensor cores: the stride-1 convolution of dz with the
// layer's weights rotated by 180 degrees and transposed ([tap][CinP][CoutP]), no bias, no
// activation, times (mask > 0) when MASK (the ReLU of the layer input, in layout lm).
template <int CIN, int COUT, int KS, bool MASK>
cudaError_t dgrad_launch(const bf16 *dz, const bf16 *wd, const bf16 *mask, bf16 *dx, int N, int H, int W, int *status,
                         cudaStream_t st, int lm = kPlanes)
{
    ConvArgs a{};
    a.x = dz;
    a.w = wd;
    a.mask = mask;
    a.y = dx;
    a.N = N;
    a.H = H;
    a.W = W;
    a.lx = a.ly = kPlanes;
    a.lm = lm;
    a.status = status;
    return conv_ws_launch<CIN, COUT, KS, 0, 0, MASK>(a, st);
}

// Launch of the fused KS x KS + 1x1 pair (c: first layer, c2: the 1x1 layer); NT as for
// conv_ws_launch.
template <int CIN, int COUT, int KS, int COUT2, int ACT2, int OUTM2, int NT>
cudaError_t conv_tail_launch_nt(const ConvArgs &c, const ConvArgs &c2, bf16 *w2_kept, float *b2_kept, bool ask, bool *fits,
                                cudaStream_t st)
{
    using T = TailGeom<CIN, COUT, KS, COUT2, NT>;
    using G = typename T::G1;
    constexpr size_t smem = tc_smem(T::SMEM, T::COLS, G::THREADS);
    static_assert(smem <= 227 * 1024, "fused conv stage does not fit in shared memory");
    auto kern = conv_tail_kernel<CIN, COUT, KS, COUT2, ACT2, OUTM2, NT>;
    static PerDevice<Resident> known;
    Resident res;
    cudaError_t e = resident(known, kern, G::THREADS, smem, T::COLS, res);
    if (e != cudaSuccess) return e;
    const long long ntiles = stages(c.N, c.H, c.W, G::TH, G::TW), cap = (long long)res.per_sm * res.n_sm;
    if (ask) {
        *fits = 2 * ntiles >= res.n_sm;
        return cudaSuccess;
    }
    if (ntiles <= 0) return cudaSuccess;
    TailArgs ta;
    std::memset(&ta, 0, sizeof(ta));
    ta.c = c;
    ta.c2 = c2;
    ta.w2_kept = w2_kept;
    ta.b2_kept = b2_kept;
    if ((e = make_tmap_tile(&ta.tm, c.lx, c.x, CIN, c.W, c.H, c.N, G::SW, G::SH)) != cudaSuccess) return e;
    return pdl::launch(kern, (int)(ntiles < cap ? ntiles : cap), G::THREADS, smem, st, ta);
}
template <int CIN, int COUT, int KS, int COUT2, int ACT2, int OUTM2>
cudaError_t conv_tail_launch(const ConvArgs &c, const ConvArgs &c2, cudaStream_t st, bf16 *w2_kept = nullptr,
                             float *b2_kept = nullptr)
{
    bool wide = false;
    cudaError_t e = conv_tail_launch_nt<CIN, COUT, KS, COUT2, ACT2, OUTM2, 4>(c, c2, w2_kept, b2_kept, true, &wide, st);
    if (e != cudaSuccess) return e;
    if (wide) return conv_tail_launch_nt<CIN, COUT, KS, COUT2, ACT2, OUTM2, 4>(c, c2, w2_kept, b2_kept, false, nullptr, st);
    return conv_tail_launch_nt<CIN, COUT, KS, COUT2, ACT2, OUTM2, 1>(c, c2, w2_kept, b2_kept, false, nullptr, st);
}

// Launch of the parity-class decoder convolution (a.x = lo, a.x2 = skip, both in layout a.lx;
// H, W even).
template <int CA, int CB, int COUT, int NBUF>
cudaError_t conv_up_launch(const ConvArgs &a, cudaStream_t st)
{
    using G = UpGeom<CA, CB, COUT, NBUF>;
    constexpr size_t smem = tc_smem(G::SMEM, G::COLS, kWsThreads);
    static_assert(smem <= 227 * 1024, "decoder conv stage does not fit in shared memory");
    auto kern = conv_up_kernel<CA, CB, COUT, NBUF>;
    static PerDevice<Resident> known;
    Resident res;
    cudaError_t e = resident(known, kern, kWsThreads, smem, G::COLS, res);
    if (e != cudaSuccess) return e;
    if ((a.H | a.W) & 1) return cudaErrorInvalidValue;
    const long long ntiles = stages(a.N, a.H / 2, a.W / 2, 16, 8), cap = (long long)res.per_sm * res.n_sm;
    if (ntiles <= 0) return cudaSuccess;
    UpArgs ua;
    std::memset(&ua, 0, sizeof(ua));
    ua.c = a;
    if ((e = make_tmap_tile(&ua.tlo, a.lx, a.x, CA, a.W / 2, a.H / 2, a.N, G::SW, G::SH)) != cudaSuccess) return e;
    e = a.lx == kNHWC ? make_tmap_parity(&ua.tskip, a.x2, CB, a.W, a.H, a.N, G::SW, G::SH)
                      : make_tmap_pairs(&ua.tskip, a.x2, CB, a.W, a.H, a.N, G::SW, G::SH);
    if (e != cudaSuccess) return e;
    return pdl::launch(kern, (int)(ntiles < cap ? ntiles : cap), kWsThreads, smem, st, ua);
}

// Launch of the stride-2 convolution (a.H, a.W: the input's size, both even; output at half
// size).
template <int CIN, int COUT, int NBUF>
cudaError_t conv_s2_launch(const ConvArgs &a, cudaStream_t st)
{
    using G = S2Geom<CIN, COUT, NBUF>;
    constexpr size_t smem = tc_smem(G::SMEM, G::COLS, kWsThreads);
    static_assert(smem <= 227 * 1024, "stride-2 conv stage does not fit in shared memory");
    auto kern = conv_s2_kernel<CIN, COUT, NBUF>;
    static PerDevice<Resident> known;
    Resident res;
    cudaError_t e = resident(known, kern, kWsThreads, smem, G::COLS, res);
    if (e != cudaSuccess) return e;
    if ((a.H | a.W) & 1) return cudaErrorInvalidValue;
    const long long ntiles = stages(a.N, a.H / 2, a.W / 2, 16, G::TW), cap = (long long)res.per_sm * res.n_sm;
    if (ntiles <= 0) return cudaSuccess;
    S2Args sa;
    std::memset(&sa, 0, sizeof(sa));
    sa.c = a;
    if (a.lx == kNHWC) {
        if ((e = make_tmap_parity(&sa.te, a.x, CIN, a.W, a.H, a.N, G::WE, G::SH)) != cudaSuccess) return e;
        if ((e = make_tmap_parity(&sa.to, a.x, CIN, a.W, a.H, a.N, G::WO, G::SH)) != cudaSuccess) return e;
    } else {
        if ((e = make_tmap_planes(&sa.te, a.x, CIN / 2, a.W / 2, a.H / 2, a.N, G::WE, G::SH)) != cudaSuccess) return e;
        if ((e = make_tmap_planes(&sa.to, a.x, CIN / 2, a.W / 2, a.H / 2, a.N, G::WO, G::SH)) != cudaSuccess) return e;
    }
    return pdl::launch(kern, (int)(ntiles < cap ? ntiles : cap), kWsThreads, smem, st, sa);
}

// Where a layer's gradients go: its partials (n_sm slices), master weight and bias gradients
struct WgradDest {
    float *part, *gw, *gb;
    int cin_true, cout_true;
};

// Launch of a layer's weight and bias gradient over dz [N][H][W] (MODE 1: x is the kParity input
// of twice that size): one CTA per SM (and tap group), and the layer's entry for the reduction.
template <int CIN, int COUT, int KS, int MODE>
cudaError_t wgrad_launch(const bf16 *x, const bf16 *dz, int layout, int N, int H, int W, const WgradDest &d, RedArgs &ra,
                         int n_sm, int *status, cudaStream_t st)
{
    using G = WgGeom<CIN, COUT, KS, MODE>;
    constexpr size_t smem = tc_smem(G::SMEM, G::COLS, G::THREADS);
    static_assert(smem <= 227 * 1024, "weight-gradient tile does not fit in shared memory");
    auto kern = wgrad_tc_kernel<CIN, COUT, KS, MODE>;
    static PerDevice<Resident> known;
    Resident res;
    cudaError_t e = resident(known, kern, G::THREADS, smem, G::COLS, res);
    if (e != cudaSuccess) return e;
    const long long ntiles = stages(N, H, W, 16, 8);
    const int slots = wgrad_slots(n_sm, G::NG);
    const int slices = (int)(ntiles < slots ? ntiles : slots);
    WgradArgs a;
    std::memset(&a, 0, sizeof(a));
    a.part = d.part;
    a.N = N;
    a.H = H;
    a.W = W;
    a.layout = layout;
    a.status = status;
    if ((e = make_tmap_rows(&a.tx, MODE ? kParity : layout, x, CIN, W, H, N, G::XW, G::XH)) != cudaSuccess) return e;
    if ((e = make_tmap_tile(&a.tdz, layout, dz, COUT, W, H, N, 8, 16)) != cudaSuccess) return e;
    ra.l[ra.n++] = RedLayer{d.part, d.gw, d.gb, slices, COUT, CIN, KS, MODE, d.cin_true, d.cout_true, ra.blocks};
    ra.blocks += (COUT * G::CTOT + 31) / 32;
    return pdl::launch(kern, dim3(slices, G::NG), G::THREADS, smem, st, a);
}

cudaError_t wgrad_reduce(const RedArgs &ra, cudaStream_t st)
{
    return pdl::launch(wgrad_reduce_kernel, ra.blocks, 32 * kRedWarps, 0, st, ra);
}

}  // namespace
}  // namespace flnr

// =========================================================================================
// The network object behind flnr_*.

struct flnr_net {
    int max_pix = 0;  // N * H * W the activation buffers hold
    int n_sm = 0;
    int nout = 8;     // output channels of the head o1: 8, or 16 (model and map guide sets)
    size_t nparam = 0;
    size_t poff[flnr::kNL][2];  // offsets of each layer's weights and bias in the flat arrays
    float *w = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;  // master fp32, grads, Adam moments
    __nv_bfloat16 *wf[flnr::kNL] = {}, *wd[flnr::kNL] = {};          // bf16 forward / dgrad weights
    std::vector<void *> bufs;
    // activations (bf16 NHWC) and gradients
    __nv_bfloat16 *x0, *a0, *f0, *a1, *f1, *a2, *f2, *c1, *a3, *d1, *c0, *a4, *d0, *a5;
    __nv_bfloat16 *gA, *gB, *gC, *gLo, *gLo2;  // gradient scratch (largest: 48 channels at full res)
    float *gskip0, *gskip1;             // skip gradients (fp32)
    float *wpart = nullptr;             // partial weight and bias gradients of every layer
    size_t wpart_off[flnr::kNL] = {};   // (fixed-order reduction), layer l's from wpart_off[l] on
    __nv_bfloat16 *head_w = nullptr;    // the head's weights and biases of the last forward pass
    float *head_b = nullptr;
    int *status = nullptr;              // device status word of the tensor-core kernels
    int N = 0, H = 0, W = 0;            // shape of the last forward
    bool weights_fresh = false;
};

namespace {

template <typename T>
int nalloc(flnr_net *n, T **p, size_t count)
{
    void *q = nullptr;
    if (cudaMalloc(&q, count * sizeof(T)) != cudaSuccess) return FLR_ERR_NOMEM;
    n->bufs.push_back(q);
    *p = (T *)q;
    return FLR_OK;
}

// layer l's true sizes in a network with `nout` head outputs
flnr::LayerDef layer_def(int nout, int l)
{
    flnr::LayerDef d = flnr::kLayers[l];
    if (l == flnr::kNL - 1) d.cout = nout;
    return d;
}

flnr::WgradDest wgrad_dest(flnr_net *n, int l)
{
    const auto d = layer_def(n->nout, l);
    return {n->wpart + n->wpart_off[l], n->g + n->poff[l][0], n->g + n->poff[l][1], d.cin, d.cout};
}

cudaError_t refresh_weights(flnr_net *n, cudaStream_t st)
{
    flnr::WeightsArgs wa;
    for (int l = 0; l < flnr::kNL; ++l) {
        const auto d = layer_def(n->nout, l);
        wa.w[l] = n->w + n->poff[l][0];
        wa.wf[l] = n->wf[l];
        wa.wd[l] = n->wd[l];
        wa.cin[l] = d.cin;
        wa.cout[l] = d.cout;
        wa.k[l] = d.k;
    }
    flnr::weights_kernel<<<dim3(64, flnr::kNL), 256, 0, st>>>(wa);
    n->weights_fresh = true;
    return cudaGetLastError();
}

}  // namespace

extern "C" {

size_t flnr_param_count(int outputs)
{
    if (outputs != 8 && outputs != 16) return 0;
    size_t s = 0;
    for (int l = 0; l < flnr::kNL; ++l) {
        const auto d = layer_def(outputs, l);
        s += (size_t)d.cout * d.cin * d.k * d.k + d.cout;
    }
    return s;
}

int flnr_create(int max_pixels, int outputs, flnr_net **out)
{
    if (!out || max_pixels <= 0 || (outputs != 8 && outputs != 16)) return FLR_ERR_ARG;
    *out = nullptr;
    flnr_net *n = new (std::nothrow) flnr_net();
    if (!n) return FLR_ERR_NOMEM;
    n->max_pix = max_pixels;
    n->nout = outputs;
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n->n_sm, cudaDevAttrMultiProcessorCount, dev);
    size_t off = 0;
    for (int l = 0; l < flnr::kNL; ++l) {
        const auto d = layer_def(outputs, l);
        n->poff[l][0] = off;
        off += (size_t)d.cout * d.cin * d.k * d.k;
        n->poff[l][1] = off;
        off += d.cout;
    }
    n->nparam = off;
    const size_t P = (size_t)max_pixels, P2 = P / 4 + 1, P4 = P / 16 + 1;
    int st = FLR_OK;
    st |= nalloc(n, &n->w, off) | nalloc(n, &n->g, off) | nalloc(n, &n->m, off) | nalloc(n, &n->v, off);
    for (int l = 0; l < flnr::kNL && st == FLR_OK; ++l) {
        const auto &d = flnr::kLayers[l];
        const size_t e = (size_t)d.k * d.k * flnr::pad16(d.cin) * flnr::pad16(d.cout);
        st |= nalloc(n, &n->wf[l], e) | nalloc(n, &n->wd[l], e);
    }
    st |= nalloc(n, &n->x0, P * 16) | nalloc(n, &n->a0, P * 16) | nalloc(n, &n->f0, P * 16);
    st |= nalloc(n, &n->a1, P * 32) | nalloc(n, &n->f1, P2 * 32);
    st |= nalloc(n, &n->a2, P2 * 64) | nalloc(n, &n->f2, P4 * 64) | nalloc(n, &n->c1, P2 * 96);
    st |= nalloc(n, &n->a3, P2 * 32) | nalloc(n, &n->d1, P2 * 32) | nalloc(n, &n->c0, P * 48);
    st |= nalloc(n, &n->a4, P * 16) | nalloc(n, &n->d0, P * 16) | nalloc(n, &n->a5, P * 16);
    st |= nalloc(n, &n->gA, P * 48) | nalloc(n, &n->gB, P * 48) | nalloc(n, &n->gC, P * 48) | nalloc(n, &n->gLo, P * 16);
    st |= nalloc(n, &n->gLo2, P2 * 32);
    st |= nalloc(n, &n->gskip0, P * 16) | nalloc(n, &n->gskip1, P2 * 32);
    st |= nalloc(n, &n->head_w, 16 * 16) | nalloc(n, &n->head_b, 16);
    st |= nalloc(n, &n->status, 1);
    // partial gradients: the slices of each layer's [Cout][k k Cin + 8] sums (47 MB on 152 SMs)
    size_t wp = 0;
    for (int l = 0; l < flnr::kNL; ++l) {
        const auto &d = flnr::kLayers[l];
        const int cin = flnr::pad16(d.cin), slots = flnr::wgrad_slots(n->n_sm, flnr::wgrad_groups(cin, d.k));
        n->wpart_off[l] = wp;
        wp += (size_t)slots * flnr::pad16(d.cout) * (d.k * d.k * cin + 8);
    }
    st |= nalloc(n, &n->wpart, wp);
    if (st != FLR_OK) {
        flnr_destroy(n);
        return FLR_ERR_NOMEM;
    }
    cudaMemset(n->status, 0, sizeof(int));
    cudaMemset(n->g, 0, off * sizeof(float));
    cudaMemset(n->m, 0, off * sizeof(float));
    cudaMemset(n->v, 0, off * sizeof(float));
    *out = n;
    return FLR_OK;
}

int flnr_destroy(flnr_net *n)
{
    if (!n) return FLR_OK;
    cudaDeviceSynchronize();
    for (void *p : n->bufs) cudaFree(p);
    delete n;
    return FLR_OK;
}

int flnr_set_weights(flnr_net *n, const float *host, size_t count)
{
    if (!n || !host || count != n->nparam) return FLR_ERR_ARG;
    if (cudaMemcpy(n->w, host, count * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess) return FLR_ERR_CUDA;
    if (cudaMemset(n->m, 0, count * sizeof(float)) != cudaSuccess || cudaMemset(n->v, 0, count * sizeof(float)) != cudaSuccess)
        return FLR_ERR_CUDA;
    if (refresh_weights(n, nullptr) != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess) return FLR_ERR_CUDA;
    return FLR_OK;
}

int flnr_get_weights(flnr_net *n, float *host, size_t count)
{
    if (!n || !host || count != n->nparam) return FLR_ERR_ARG;
    return cudaMemcpy(host, n->w, count * sizeof(float), cudaMemcpyDeviceToHost) == cudaSuccess ? FLR_OK : FLR_ERR_CUDA;
}

int flnr_get_state(flnr_net *n, float *host, size_t count)
{
    if (!n || !host || count != 3 * n->nparam) return FLR_ERR_ARG;
    const size_t b = n->nparam * sizeof(float);
    if (cudaMemcpy(host, n->w, b, cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemcpy(host + n->nparam, n->m, b, cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemcpy(host + 2 * n->nparam, n->v, b, cudaMemcpyDeviceToHost) != cudaSuccess)
        return FLR_ERR_CUDA;
    return FLR_OK;
}

int flnr_set_state(flnr_net *n, const float *host, size_t count)
{
    if (!n || !host || count != 3 * n->nparam) return FLR_ERR_ARG;
    const size_t b = n->nparam * sizeof(float);
    if (cudaMemcpy(n->w, host, b, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(n->m, host + n->nparam, b, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(n->v, host + 2 * n->nparam, b, cudaMemcpyHostToDevice) != cudaSuccess)
        return FLR_ERR_CUDA;
    if (refresh_weights(n, nullptr) != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess) return FLR_ERR_CUDA;
    return FLR_OK;
}

int flnr_get_grads(flnr_net *n, float *host, size_t count)
{
    if (!n || !host || count != n->nparam) return FLR_ERR_ARG;
    return cudaMemcpy(host, n->g, count * sizeof(float), cudaMemcpyDeviceToHost) == cudaSuccess ? FLR_OK : FLR_ERR_CUDA;
}

int flnr_zero_grads(flnr_net *n, void *stream)
{
    if (!n) return FLR_ERR_ARG;
    return cudaMemsetAsync(n->g, 0, n->nparam * sizeof(float), (cudaStream_t)stream) == cudaSuccess ? FLR_OK : FLR_ERR_CUDA;
}

#define FLNR_TRY(x)                                 \
    do {                                            \
        if ((x) != cudaSuccess) return FLR_ERR_CUDA; \
    } while (0)

int flnr_guide_forward(flnr_net *n, const float *in, float *guide_out, int N, int H, int W, void *stream)
{
    using namespace flnr;
    if (!n || !in || N <= 0 || H <= 0 || W <= 0 || (H % 4) || (W % 4)) return FLR_ERR_ARG;
    if ((long long)N * H * W > n->max_pix) return FLR_ERR_UNSUPPORTED;
    if (!n->weights_fresh) return FLR_ERR_ARG;  // flnr_set_weights first
    cudaStream_t st = (cudaStream_t)stream;
    n->N = N;
    n->H = H;
    n->W = W;
    const size_t P = (size_t)N * H * W;
    const int H2 = H / 2, W2 = W / 2;
    auto bias = [&](int l) { return n->w + n->poff[l][1]; };
    FLNR_TRY(pdl::launch(pack_input_kernel, egrid(P), 256, 0, st, in, n->x0, N, H, W));
    const ConvArgs z{};
    auto conv = [&](const __nv_bfloat16 *x, int l, __nv_bfloat16 *y, int h, int w, int ly = kPlanes) {
        ConvArgs c = z;
        c.x = x; c.w = n->wf[l]; c.bias = bias(l); c.y = y; c.N = N; c.H = h; c.W = w;
        c.lx = kPlanes; c.ly = ly; c.nbias = layer_def(n->nout, l).cout; c.status = n->status;
        return c;
    };
    ConvArgs c;
    // in0 and in1 in one pass (a0, which the backward pass reads, is still stored)
    FLNR_TRY((conv_tail_launch<16, 16, 3, 16, 1, 0>(conv(n->x0, 0, n->a0, H, W), conv(n->a0, 1, n->f0, H, W), st)));
    // encoder blocks: a 3x3 convolution, then a stride-2 one (sizes passed: the input's)
    FLNR_TRY((conv_ws_launch<16, 32, 3, 1, 0, false>(conv(n->f0, 2, n->a1, H, W, kParity), st)));
    c = conv(n->a1, 3, n->f1, H, W);
    c.lx = kParity;
    FLNR_TRY((conv_s2_launch<32, 32, 2>(c, st)));
    FLNR_TRY((conv_ws_launch<32, 64, 3, 1, 0, false>(conv(n->f1, 4, n->a2, H2, W2, kParity), st)));
    c = conv(n->a2, 5, n->f2, H2, W2);
    c.lx = kParity;
    FLNR_TRY((conv_s2_launch<64, 64, 2>(c, st)));
    c = conv(n->f2, 6, n->a3, H2, W2);  // input up(f2) ++ f1, formed while staging
    c.x2 = n->f1;
    FLNR_TRY((conv_up_launch<64, 32, 32, 2>(c, st)));
    FLNR_TRY((conv_ws_launch<32, 32, 3, 1, 0, false>(conv(n->a3, 7, n->d1, H2, W2), st)));
    c = conv(n->d1, 8, n->a4, H, W);  // input up(d1) ++ f0
    c.x2 = n->f0;
    FLNR_TRY((conv_up_launch<32, 16, 16, 2>(c, st)));
    FLNR_TRY((conv_ws_launch<16, 16, 3, 1, 0, false>(conv(n->a4, 9, n->d0, H, W), st)));
    c = conv(n->a5, 11, nullptr, H, W);
    c.yf = guide_out;
    // o0 and the head o1 (sigmoid into planar FP32) in one pass; a5 is still stored, and the
    // backward pass forms the guides again from it (a copy of the guides cost 133 MB of traffic,
    // 21 us, per 1920x1080 frame)
    FLNR_TRY((conv_tail_launch<16, 16, 3, 16, 2, 1>(conv(n->d0, 10, n->a5, H, W), c, st, n->head_w, n->head_b)));
    return FLR_OK;
}

int flnr_guide_backward(flnr_net *n, const float *grad_out, float *grad_in, void *stream)
{
    using namespace flnr;
    if (!n || !grad_out || n->N <= 0) return FLR_ERR_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    const int N = n->N, H = n->H, W = n->W, H2 = H / 2, W2 = W / 2, H4 = H / 4, W4 = W / 4;
    const size_t P = (size_t)N * H * W;
    // every layer's weight and bias gradient goes to its partials; one reduction at the end
    RedArgs ra;
#define FLNR_WGRAD(ci, co, ks, mode, l, x, dz, h, w) \
    FLNR_TRY((wgrad_launch<ci, co, ks, mode>(x, dz, kPlanes, N, h, w, wgrad_dest(n, l), ra, n->n_sm, n->status, st)))
    // output head: sigmoid of o1 (1x1, 16 -> 8 padded to 16; the forward pass's products and
    // weights again) and its gradient, then o1 and o0
    ConvArgs hc{};
    hc.x = n->a5; hc.w = n->head_w; hc.bias = n->head_b; hc.y = n->gA; hc.g = grad_out; hc.N = N; hc.H = H; hc.W = W;
    hc.lx = hc.ly = kPlanes; hc.nbias = n->nout; hc.status = n->status;
    FLNR_TRY((conv_ws_launch<16, 16, 1, 2, 2, false>(hc, st)));
    FLNR_WGRAD(16, 16, 1, 0, 11, n->a5, n->gA, H, W);
    FLNR_TRY((dgrad_launch<16, 16, 1, true>(n->gA, n->wd[11], n->a5, n->gB, N, H, W, n->status, st)));
    FLNR_WGRAD(16, 16, 3, 0, 10, n->d0, n->gB, H, W);
    FLNR_TRY((dgrad_launch<16, 16, 3, true>(n->gB, n->wd[10], n->d0, n->gA, N, H, W, n->status, st)));
    // decoder level 0
    FLNR_WGRAD(16, 16, 3, 0, 9, n->a4, n->gA, H, W);
    FLNR_TRY((dgrad_launch<16, 16, 3, true>(n->gA, n->wd[9], n->a4, n->gB, N, H, W, n->status, st)));
    FLNR_TRY(pdl::launch(upcat_kernel, egrid(P * 6), 256, 0, st, n->d1, n->f0, n->c0, N, H, W, 32, 16));  // d0a's input
    FLNR_WGRAD(48, 16, 3, 0, 8, n->c0, n->gB, H, W);
    FLNR_TRY((dgrad_launch<16, 48, 3, false>(n->gB, n->wd[8], nullptr, n->gC, N, H, W, n->status, st)));
    FLNR_TRY(pdl::launch(upcat_bwd_kernel, egrid(P * 48 / 8), 256, 0, st, n->gC, n->d1, n->gLo, n->gskip0, N, H, W, 32, 16));  // gLo = dz(d1b)
    // decoder level 1 (H/2)
    const size_t P2 = P / 4;
    FLNR_WGRAD(32, 32, 3, 0, 7, n->a3, n->gLo, H2, W2);
    FLNR_TRY((dgrad_launch<32, 32, 3, true>(n->gLo, n->wd[7], n->a3, n->gA, N, H2, W2, n->status, st)));
    FLNR_TRY(pdl::launch(upcat_kernel, egrid(P2 * 12), 256, 0, st, n->f2, n->f1, n->c1, N, H2, W2, 64, 32));  // d1a's input
    FLNR_WGRAD(96, 32, 3, 0, 6, n->c1, n->gA, H2, W2);
    FLNR_TRY((dgrad_launch<32, 96, 3, false>(n->gA, n->wd[6], nullptr, n->gC, N, H2, W2, n->status, st)));
    FLNR_TRY(pdl::launch(upcat_bwd_kernel, egrid(P2 * 96 / 8), 256, 0, st, n->gC, n->f2, n->gLo, n->gskip1, N, H2, W2, 64, 32));  // gLo = dz(e2b)
    // encoder level 2: e2b (stride 2, H/2 -> H/4), then e2a (H/2).  A stride-2 layer's input
    // gradient is that of the stride-1 kernel at its input's size on dz zero-upsampled onto
    // that grid; its weight gradient takes dz as it is.
    FLNR_WGRAD(64, 64, 3, 1, 5, n->a2, n->gLo, H4, W4);
    FLNR_TRY(pdl::launch(join_bwd_kernel<2>, egrid(P2 * 64 / 8), 256, 0, st, nullptr, n->gLo, nullptr, n->gB, nullptr, N, H4, W4, 64));
    FLNR_TRY((dgrad_launch<64, 64, 3, true>(n->gB, n->wd[5], n->a2, n->gA, N, H2, W2, n->status, st, kParity)));
    FLNR_WGRAD(32, 64, 3, 0, 4, n->f1, n->gA, H2, W2);
    FLNR_TRY((dgrad_launch<64, 32, 3, false>(n->gA, n->wd[4], nullptr, n->gB, N, H2, W2, n->status, st)));
    // encoder level 1: e1b (stride 2, H -> H/2; f1 also feeds the d1a skip), then e1a (H)
    FLNR_TRY(pdl::launch(join_bwd_kernel<2>, egrid(P * 32 / 8), 256, 0, st, n->gskip1, n->gB, n->f1, n->gC, n->gLo2, N, H2, W2, 32));
    FLNR_WGRAD(32, 32, 3, 1, 3, n->a1, n->gLo2, H2, W2);
    FLNR_TRY((dgrad_launch<32, 32, 3, true>(n->gC, n->wd[3], n->a1, n->gA, N, H, W, n->status, st, kParity)));
    FLNR_WGRAD(16, 32, 3, 0, 2, n->f0, n->gA, H, W);
    FLNR_TRY((dgrad_launch<32, 16, 3, false>(n->gA, n->wd[2], nullptr, n->gB, N, H, W, n->status, st)));
    FLNR_TRY(pdl::launch(join_bwd_kernel<1>, egrid(P * 16 / 8), 256, 0, st, n->gskip0, n->gB, n->f0, n->gLo, nullptr, N, H, W, 16));  // dz(in1)
    // input projection (H)
    FLNR_WGRAD(16, 16, 1, 0, 1, n->a0, n->gLo, H, W);
    FLNR_TRY((dgrad_launch<16, 16, 1, true>(n->gLo, n->wd[1], n->a0, n->gA, N, H, W, n->status, st)));
    FLNR_WGRAD(16, 16, 3, 0, 0, n->x0, n->gA, H, W);
#undef FLNR_WGRAD
    if (grad_in) {  // through in0 to the packed input, then through the input transform
        FLNR_TRY((dgrad_launch<16, 16, 3, false>(n->gA, n->wd[0], nullptr, n->gB, N, H, W, n->status, st)));
        FLNR_TRY(pdl::launch(unpack_grad_kernel, egrid(P), 256, 0, st, n->gB, n->x0, grad_in, N, H, W));
    }
    FLNR_TRY(cudaGetLastError());
    FLNR_TRY(wgrad_reduce(ra, st));
    return FLR_OK;
}

}  // extern "C"

namespace {

// One layer's kernels by themselves (flnr_layer): CI / CO are the padded channel counts, CA
// the upsampled part of a decoder input, S2 whether the layer strides by 2 (N, H, W: the
// layer's input size).
template <int CI, int CO, int KS, int CA, bool S2, bool HEAD = false>
int layer_ops(flnr_net *n, int l, int op, const void *a, const void *b, const void *mask, void *out, int N, int H,
              int W, cudaStream_t st)
{
    using namespace flnr;
    using bf = __nv_bfloat16;
    const auto d = layer_def(n->nout, l);
    const long long P = (long long)N * H * W;
    if (op == FLNR_OP_FORWARD) {
        ConvArgs c{};
        c.x = (const bf *)a;
        c.w = n->wf[l];
        c.bias = n->w + n->poff[l][1];
        c.N = N;
        c.H = H;
        c.W = W;
        c.nbias = d.cout;  // lx, ly: NHWC
        c.status = n->status;
        if constexpr (HEAD) {
            c.yf = (float *)out;
            FLNR_TRY((conv_ws_launch<CI, CO, KS, 2, 1, false>(c, st)));
        } else {
            c.y = (bf *)out;
            if constexpr (CA > 0) {
                if (b) {
                    if ((H | W) & 1) return FLR_ERR_ARG;
                    c.x2 = (const bf *)b;
                    FLNR_TRY((conv_up_launch<CA, CI - CA, CO, 2>(c, st)));
                    return FLR_OK;
                }
            }
            if constexpr (S2) {
                if ((H | W) & 1) return FLR_ERR_ARG;
                FLNR_TRY((conv_s2_launch<CI, CO, 2>(c, st)));
            } else {
                FLNR_TRY((conv_ws_launch<CI, CO, KS, 1, 0, false>(c, st)));
            }
        }
        return FLR_OK;
    }
    const bf *dz = (const bf *)(op == FLNR_OP_DGRAD ? a : b);
    if constexpr (S2) {  // dz [N][H/2][W/2][CO], zero-upsampled onto the input grid in scratch
        if ((H | W) & 1) return FLR_ERR_ARG;
        if (P * CO > (long long)n->max_pix * 48) return FLR_ERR_UNSUPPORTED;
        FLNR_TRY(pdl::launch(spread_nhwc_kernel, egrid((size_t)P * CO / 8), 256, 0, st, dz, n->gC, N, H / 2, W / 2, CO));
        dz = n->gC;
    }
    if (op == FLNR_OP_DGRAD) {
        ConvArgs c{};  // NHWC
        c.x = dz;
        c.w = n->wd[l];
        c.mask = (const bf *)mask;
        c.y = (bf *)out;
        c.N = N;
        c.H = H;
        c.W = W;
        c.status = n->status;
        if (mask) FLNR_TRY((conv_ws_launch<CO, CI, KS, 0, 0, true>(c, st)));
        else FLNR_TRY((conv_ws_launch<CO, CI, KS, 0, 0, false>(c, st)));
    } else {
        RedArgs ra;
        FLNR_TRY((wgrad_launch<CI, CO, KS, 0>((const bf *)a, dz, kNHWC, N, H, W, wgrad_dest(n, l), ra, n->n_sm, n->status, st)));
        FLNR_TRY(wgrad_reduce(ra, st));
    }
    return FLR_OK;
}

}  // namespace

extern "C" {

int flnr_layer(flnr_net *n, int layer, int op, const void *a, const void *b, const void *mask, void *out, int N,
               int H, int W, void *stream)
{
    if (!n || layer < 0 || layer >= flnr::kNL || op < FLNR_OP_FORWARD || op > FLNR_OP_WGRAD || !a || N <= 0 ||
        H <= 0 || W <= 0)
        return FLR_ERR_ARG;
    if ((op == FLNR_OP_WGRAD && !b) || (op != FLNR_OP_WGRAD && !out)) return FLR_ERR_ARG;
    if ((long long)N * H * W > 0x7fffffffLL) return FLR_ERR_ARG;
    if (!n->weights_fresh) return FLR_ERR_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    switch (layer) {
    case 0: return layer_ops<16, 16, 3, 0, false>(n, 0, op, a, b, mask, out, N, H, W, st);
    case 1: return layer_ops<16, 16, 1, 0, false>(n, 1, op, a, b, mask, out, N, H, W, st);
    case 2: return layer_ops<16, 32, 3, 0, false>(n, 2, op, a, b, mask, out, N, H, W, st);
    case 3: return layer_ops<32, 32, 3, 0, true>(n, 3, op, a, b, mask, out, N, H, W, st);
    case 4: return layer_ops<32, 64, 3, 0, false>(n, 4, op, a, b, mask, out, N, H, W, st);
    case 5: return layer_ops<64, 64, 3, 0, true>(n, 5, op, a, b, mask, out, N, H, W, st);
    case 6: return layer_ops<96, 32, 3, 64, false>(n, 6, op, a, b, mask, out, N, H, W, st);
    case 7: return layer_ops<32, 32, 3, 0, false>(n, 7, op, a, b, mask, out, N, H, W, st);
    case 8: return layer_ops<48, 16, 3, 32, false>(n, 8, op, a, b, mask, out, N, H, W, st);
    case 9: return layer_ops<16, 16, 3, 0, false>(n, 9, op, a, b, mask, out, N, H, W, st);
    case 10: return layer_ops<16, 16, 3, 0, false>(n, 10, op, a, b, mask, out, N, H, W, st);
    default: return layer_ops<16, 16, 1, 0, false, true>(n, 11, op, a, b, mask, out, N, H, W, st);
    }
}

int flnr_status(flnr_net *n)
{
    if (!n) return FLR_ERR_ARG;
    int h = 0;
    if (cudaDeviceSynchronize() != cudaSuccess) return FLR_ERR_CUDA;
    if (cudaMemcpy(&h, n->status, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return FLR_ERR_CUDA;
    if (h != 0 && cudaMemset(n->status, 0, sizeof(int)) != cudaSuccess) return FLR_ERR_CUDA;
    return h ? FLR_ERR_TIMEOUT : FLR_OK;
}

int flnr_adam_step(flnr_net *n, float lr, float beta1, float beta2, float eps, int step, void *stream)
{
    if (!n || step < 1 || !(lr >= 0.f)) return FLR_ERR_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    const float c1 = 1.f - powf(beta1, (float)step), c2 = 1.f - powf(beta2, (float)step);
    flnr::adam_kernel<<<flnr::egrid(n->nparam), 256, 0, st>>>(n->w, n->g, n->m, n->v, n->nparam, lr, beta1, beta2, eps, c1, c2);
    FLNR_TRY(cudaGetLastError());
    FLNR_TRY(refresh_weights(n, st));
    return FLR_OK;
}

int flnr_l1_loss(const float *pred, const float *ref, float *grad, float *loss, size_t count, void *stream)
{
    if (!pred || !ref || !grad || !loss || count == 0) return FLR_ERR_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    FLNR_TRY(cudaMemsetAsync(loss, 0, sizeof(float), st));
    flnr::l1_kernel<<<flnr::egrid(count) < 1024 ? flnr::egrid(count) : 1024, 256, 0, st>>>(pred, ref, grad, loss, count);
    return cudaGetLastError() == cudaSuccess ? FLR_OK : FLR_ERR_CUDA;
}

int flnr_smape_loss(const float *pred, const float *ref, float *grad, float *loss, size_t count, float eps, void *stream)
{
    if (!pred || !ref || !grad || !loss || count == 0 || !(eps > 0.f)) return FLR_ERR_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    FLNR_TRY(cudaMemsetAsync(loss, 0, sizeof(float), st));
    flnr::smape_kernel<<<flnr::egrid(count) < 1024 ? flnr::egrid(count) : 1024, 256, 0, st>>>(pred, ref, grad, loss, count,
                                                                                                 eps);
    return cudaGetLastError() == cudaSuccess ? FLR_OK : FLR_ERR_CUDA;
}

}  // extern "C"
