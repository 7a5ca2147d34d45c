// flr_fast.cu -- the paper's fast FLR (Sec. 3.2) and its joint denoising and upsampling
// (Sec. 3.2.1) on sm_103a, behind the flr_fast_* entry points of include/flr.h.
//
// The paper's four steps, as four kernels over all the frames of a call:
//   1. block_moments: outer products of the shifted inputs summed over F x F blocks of the
//      input grid (the strided box filter);  one thread per pair of input columns walks the
//      F rows of its block row, fed by its own ring of asynchronous copies, then the F / 2 lanes
//      of a block fold their sums;
//   2. blur_h:  horizontal Gaussian over the block grid (one thread per block);
//   3. blur_v_solve: vertical Gaussian, then the centred ridge model of every block in
//      registers (the window sums staged per thread in shared memory); a block whose
//      Cholesky pivot ratio falls to tau or below is re-solved in FP64 from the same sums;
//   4. apply: bilinear interpolation of the block models at every output pixel (output
//      grid s times finer than the input grid) and application to the map guide.
// Only step 1 and step 4 touch full-resolution data: the input is read once (44 B per
// input pixel for Q = 8), the map guide once and the output written once (32 + 12 B per
// output pixel); everything in between lives in (F^2)-times smaller planes that stay in L2.
// At 1920x1080, F = 8, without overlap: 21 + 9 + 10 + 14 us (26.5 + 9 + 11.6 + 19 before the ring,
// the block-major models and the packed apply), 57 us in all (77); the bytes alone take 17 us.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <new>
#include <utility>
#include <vector>

#include "flr.h"
#include "flr_fast_stages.cuh"
#include "pdl.cuh"
#include "tma.cuh"

namespace flr {
namespace {

using fast::FastArgs;
using fast::kMaxTaps;

// The blurs are bound by the latency of their loads, 82 per tap: two CTAs of 128 threads per SM
// with up to 255 registers let the compiler keep more of them in flight than it does by itself
// (146 registers): 63.7 -> 57.4 us for the whole frame at 1920x1080.  CTAs of 64 threads: 74.9 us.
constexpr int kBlurThreads = 128;

// The frames of one call: one (N = 1), or up to FLR_MAX_BATCH of mixed sizes (N = FLR_MAX_BATCH).
// Stage s of frame i covers CTAs (stages 1 to 3) or work items (stage 4) off[s][i] .. off[s][i + 1].
// A batch is the four stages over all its frames, not four launches per frame: 8 frames fill the
// chip's last wave of each stage once instead of eight times.  (One persistent kernel over the
// stages with grid barriers between them, the form before this, ran every stage at the occupancy
// of the most demanding one, 8 warps per SM: 488 us for 3 frames each of 1280x720 and 1920x1080
// and 2 of 2560x1440 outputs.)
template <int N>
struct FrameTable {
    FastArgs f[N];
    int n;
    unsigned off[4][N + 1];
    unsigned long long *count;  // zeroed by stage 1, counted by stage 3
    int *status;                // zeroed by stage 1 if not NULL (the batch's status word)
};

template <int N>
__device__ __forceinline__ int frame_of(const FrameTable<N> &t, int stage, unsigned item)
{
    int f = 0;
    if (N > 1)
        while (f + 1 < t.n && item >= t.off[stage][f + 1]) ++f;
    return f;
}

template <int Q, int F, int N>
__global__ void __launch_bounds__(fast::kMomThreads, 512 / fast::kMomThreads) block_moments_kernel(const __grid_constant__ FrameTable<N> t)
{
    extern __shared__ __align__(16) float ring[];
    pdl::trigger();
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *t.count = 0ull;
        if (t.status) *t.status = 0;
    }
    const int f = frame_of(t, 0, blockIdx.x);
    const FastArgs &a = t.f[f];
    const int item = (int)(blockIdx.x - t.off[0][f]), chunks = fast::moment_chunks(a.Wi);
    fast::stage_moments<Q, F>(a, item / chunks, item % chunks, ring);
}

template <int Q, int N>
__global__ void __launch_bounds__(kBlurThreads, 2) blur_h_kernel(const __grid_constant__ FrameTable<N> t)
{
    pdl::trigger();
    const int f = frame_of(t, 1, blockIdx.x);
    pdl::wait();
    fast::stage_blur_h<Q>(t.f[f], (size_t)(blockIdx.x - t.off[1][f]) * kBlurThreads + threadIdx.x);
}

template <int Q, int N>
__global__ void __launch_bounds__(kBlurThreads, 2) blur_v_solve_kernel(const __grid_constant__ FrameTable<N> t)
{
    extern __shared__ float sS[];  // [NCH][kBlurThreads]
    pdl::trigger();
    const int f = frame_of(t, 2, blockIdx.x);
    pdl::wait();
    fast::stage_blur_v_solve<Q>(t.f[f], (size_t)(blockIdx.x - t.off[2][f]) * kBlurThreads + threadIdx.x, sS + threadIdx.x,
                                kBlurThreads);
}

// Stage 4 for frames whose rows do not start on 16-byte boundaries, cells of more than 8 rows and
// the parameter gradients: as apply_tma_kernel below, with plain loads of the map guide.  One item
// per CTA: kFW output columns of up to kApplyRows rows of a cell row (a cell has up to 64).
// Coalesced in every access, four CTAs per SM, the loads of two rows in flight per thread.  With one
// thread per run of P pixels of a row (each reading its four block-major models for that row
// alone) four 1080x1919 frames took 470 us, so 250; 16 frames of 540x960 from 270x480, F = 8, 348
// and 144; one 1080x1919 frame 119 and 72.
constexpr int kFW = 128, kApplyRows = 8;

__host__ __device__ inline int apply_parts(int P) { return (P + kApplyRows - 1) / kApplyRows; }

template <int Q, int N>
__global__ void __launch_bounds__(kFW, 4) fast_apply_kernel(const __grid_constant__ FrameTable<N> t)
{
    using M = fast::Model<Q>;
    const int f = frame_of(t, 3, blockIdx.x);
    const FastArgs &a = t.f[f];
    const int P = a.F * a.s, ncx = (a.Wo + kFW - 1) / kFW, parts = apply_parts(P);
    const int local = (int)(blockIdx.x - t.off[3][f]), cx = local % ncx, part = local / ncx % parts, ci = local / ncx / parts;
    const int x = cx * kFW + (int)threadIdx.x, ya = P * ci - P / 2;
    const int t0 = max(kApplyRows * part, -ya), t1 = min(min(kApplyRows * (part + 1), P), a.Ho - ya);
    pdl::wait();
    if (x >= a.Wo || t0 >= t1) return;
    float2 top[M::CS / 2], dtb[M::CS / 2], nsh[M::QE / 2];
    float shr[3];
    const size_t oplane = (size_t)a.Ho * a.Wo, off = (size_t)(ya + t0) * a.Wo + x;
    const float *zp = a.map_guide + off;
    float *out = a.out + off;
    const int i0 = fast::column_models<Q>(a, P, x, ya, top, dtb);
    fast::load_reference<Q>(a, nsh, shr);
    for (int r = t0; r < t1; r += 2, zp += 2 * (size_t)a.Wo, out += 2 * (size_t)a.Wo) {
        const bool two = r + 1 < t1;
        float z0[Q], z1[Q];
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            z0[i] = __ldg(zp + i * oplane);
            z1[i] = two ? __ldg(zp + i * oplane + a.Wo) : 0.f;
        }
        fast::apply_pixel<Q>(a, P, ya + r, i0, top, dtb, nsh, shr, [&](int i) { return z0[i]; }, out, oplane);
        if (two)
            fast::apply_pixel<Q>(a, P, ya + r + 1, i0, top, dtb, nsh, shr, [&](int i) { return z1[i]; }, out + a.Wo, oplane);
    }
}

// ---- parameter gradients (sigma and the regularisation terms) ---------------------------
template <int Q>
__global__ void __launch_bounds__(128) blur_v_tangent_kernel(const FastArgs a)
{
    extern __shared__ float sS[];  // [2][NCH][blockDim.x]: blurred sums, their sigma-derivative
    fast::stage_blur_v_tangent<Q>(a, (size_t)blockIdx.x * blockDim.x + threadIdx.x, sS + threadIdx.x,
                                  sS + Chan<Q>::NCH * blockDim.x + threadIdx.x, blockDim.x);
}

// Deterministic dot product: kDotBlocks partial sums in double (each thread strides through
// the data in a fixed order, then a fixed tree per CTA), summed by one CTA in a fixed tree.
constexpr int kDotBlocks = 256;
__global__ void __launch_bounds__(256) dot_partial_kernel(const float *x, const float *y, size_t n, double *part)
{
    __shared__ double sp[256];
    double acc = 0.0;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        acc += (double)x[i] * (double)y[i];
    sp[threadIdx.x] = acc;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) sp[threadIdx.x] += sp[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = sp[0];
}

__global__ void __launch_bounds__(256) dot_final_kernel(const double *part, double *out)
{
    __shared__ double sp[kDotBlocks];
    sp[threadIdx.x] = part[threadIdx.x];
    __syncthreads();
    for (int o = kDotBlocks / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) sp[threadIdx.x] += sp[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = sp[0];
}

// ---- TMA version of the apply stage (rows 16-byte aligned) ------------------------------
//
// Persistent CTAs walk work items of kFW output columns; each item's map-guide rows arrive
// by one TMA box copy into a two-stage ring (the next item loads while the current one is
// computed), so the bytes in flight do not depend on registers per thread.  The copy
// engine zero-fills outside the image.  Waits are bounded (1 s) and report through the
// status word.
constexpr unsigned long long kFastTimeoutNs = 1000000000ull;

template <int N>
struct alignas(128) FastKArgs {
    CUtensorMap t0[N];  // map-guide planes [Q][Ho][Wo], box (kFW, P, Q)
    FrameTable<N> t;
    unsigned long long wait_ns;  // limit of a wait for a copy (0: gives up at once, the self-test)
};

__device__ __forceinline__ float *align128(float *p)
{
    return p + (((128 - (tma::smem_addr(p) & 127)) & 127) >> 2);
}

// Stage 4 with TMA: item (cell row i, column chunk cx), the P rows of the Q map-guide planes.  The
// corner models are interpolated horizontally while the item's rows are still on their way.  PC: P
// known at compile time (the weights' divisions become products), or 0.
template <int Q, int N, int PC>
__global__ void __launch_bounds__(kFW, 3) apply_tma_kernel(const __grid_constant__ FastKArgs<N> k)
{
    using M = fast::Model<Q>;
    constexpr int PMAX = 8, STAGE = Q * PMAX * kFW;
    extern __shared__ __align__(16) float smem[];
    float *base = align128(smem);
    uint64_t *bar = reinterpret_cast<uint64_t *>(base + 2 * STAGE);
    __shared__ int s_abort;
    const int tid = threadIdx.x, lane = tid & 31;
    const unsigned nitems = k.t.off[3][k.t.n];
    const int P = PC ? PC : k.t.f[0].F * k.t.f[0].s;  // the handle's: the same for every frame
    int *status = k.t.f[0].status;
    if (tid == 0) {
        s_abort = 0;
        tma::mbar_init(bar, 1);
        tma::mbar_init(bar + 1, 1);
        tma::mbar_init_fence();
    }
    __syncthreads();
    auto issue = [&](unsigned item, int st) {
        const int f = frame_of(k.t, 3, item);
        const int local = (int)(item - k.t.off[3][f]), ncx = (k.t.f[f].Wo + kFW - 1) / kFW;
        const int ci = local / ncx, cx = local % ncx;
        tma::mbar_expect_tx(bar + st, (unsigned)(Q * P * kFW * 4));
        tma::load_3d_hint(base + st * STAGE, &k.t0[f], cx * kFW, P * ci - P / 2, 0, bar + st, fast::l2_policy_stream());
    };
    // the map guide is the caller's, complete before stage 1 began: its first rows come ahead of
    // the block models
    if (tid == 0 && blockIdx.x < nitems) issue(blockIdx.x, 0);
    pdl::wait();
    int it = 0;
    for (unsigned item = blockIdx.x; item < nitems; item += gridDim.x, ++it) {
        const int st = it & 1;
        const int f = frame_of(k.t, 3, item);
        const FastArgs &a = k.t.f[f];
        const int ncx = (a.Wo + kFW - 1) / kFW, local = (int)(item - k.t.off[3][f]);
        if (tid == 0 && item + gridDim.x < nitems) {
            asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
            issue(item + gridDim.x, st ^ 1);
        }
        const int ci = local / ncx, cx = local % ncx;
        const int x = min(cx * kFW + tid, a.Wo - 1);
        const int ya = P * ci - P / 2;       // first output row of the cell (may be < 0)
        float2 top[M::CS / 2], dtb[M::CS / 2], nsh[M::QE / 2];
        float shr[3];
        const int i0 = fast::column_models<Q>(a, P, x, ya, top, dtb);
        fast::load_reference<Q>(a, nsh, shr);
        if (!(k.wait_ns && tma::wait_warp(bar + st, (uint32_t)((it >> 1) & 1), k.wait_ns)) && lane == 0) {
            s_abort = 1;
            if (status) atomicExch(status, 1);
        }
        __syncthreads();
        if (s_abort) {  // let the copies in flight, this item's and the next one's, land before the CTA exits
            if (tid < 32) {
                tma::wait_warp(bar + st, (uint32_t)((it >> 1) & 1), kFastTimeoutNs);
                if (item + gridDim.x < nitems) tma::wait_warp(bar + (st ^ 1), (uint32_t)(((it + 1) >> 1) & 1), kFastTimeoutNs);
            }
            break;
        }
        const float *T = base + st * STAGE + tid;  // [Q][P][kFW]
        if (cx * kFW + tid < a.Wo) {
            const size_t oplane = (size_t)a.Ho * a.Wo;
            const int t0 = max(-ya, 0), t1 = min(P, a.Ho - ya);
            float *out = a.out + (size_t)(ya + t0) * a.Wo + x;
#pragma unroll 2
            for (int t = t0; t < t1; ++t, out += a.Wo)
                fast::apply_pixel<Q>(a, P, ya + t, i0, top, dtb, nsh, shr, [&](int i) { return T[(i * P + t) * kFW]; }, out, oplane);
        }
        __syncthreads();  // stage st is read; the next iteration may refill it
    }
}

template <int Q>
size_t apply_tma_smem()
{
    return 128 + sizeof(float) * 2 * (size_t)Q * 8 * kFW + 16;
}

// Table of the frames f[0..n) with the CTAs of stages 1 to 3; stage 4's items are its launch's.
template <int N>
void fill_table(FrameTable<N> &t, int n, const FastArgs *f, unsigned long long *count, int *status)
{
    t.n = n;
    t.count = count;
    t.status = status;
    for (int s = 0; s < 4; ++s) t.off[s][0] = 0;
    for (int i = 0; i < n; ++i) {
        t.f[i] = f[i];
        const size_t nb = (size_t)f[i].Hb * f[i].Wb;
        t.off[0][i + 1] = t.off[0][i] + (unsigned)f[i].Hb * fast::moment_chunks(f[i].Wi);
        t.off[1][i + 1] = t.off[1][i] + (unsigned)((nb + kBlurThreads - 1) / kBlurThreads);
        t.off[2][i + 1] = t.off[1][i + 1];
        t.off[3][i + 1] = t.off[3][i];
    }
}

// Names a kernel instance for pdl::allow_smem
template <int KIND, int... I>
struct KernelTag {};

template <int Q, int F, int N>
cudaError_t launch_moments(const FrameTable<N> &t, cudaStream_t st)
{
    constexpr size_t smem = fast::moments_smem<Q>();
    const cudaError_t e = pdl::allow_smem<KernelTag<0, Q, F, N>>(block_moments_kernel<Q, F, N>, smem, false);
    if (e != cudaSuccess) return e;
    // an ordinary launch, not a dependent one: apply_tma_kernel reads the map guide before its wait
    block_moments_kernel<Q, F, N><<<t.off[0][t.n], fast::kMomThreads, smem, st>>>(t);
    return cudaGetLastError();
}

template <int Q, int N>
cudaError_t launch_moments_f(const FrameTable<N> &t, cudaStream_t st)
{
    switch (t.f[0].F) {
    case 2: return launch_moments<Q, 2>(t, st);
    case 4: return launch_moments<Q, 4>(t, st);
    case 8: return launch_moments<Q, 8>(t, st);
    default: return cudaErrorInvalidValue;
    }
}

// Any row alignment and any P: the frames of t, whose stage-4 items are counted here.
template <int Q, int N>
cudaError_t launch_apply_plain(FrameTable<N> &t, cudaStream_t st)
{
    for (int i = 0; i < t.n; ++i) {
        const FastArgs &a = t.f[i];
        t.off[3][i + 1] = t.off[3][i] + (unsigned)(a.Hb + 1) * apply_parts(a.F * a.s) * ((a.Wo + kFW - 1) / kFW);
    }
    return pdl::launch(fast_apply_kernel<Q, N>, dim3(t.off[3][t.n]), kFW, 0, st, t);
}

// Stage 4.  Frames whose rows start on 16-byte boundaries, with P <= 8, take the TMA kernel; the
// others (and frames whose tensor map is refused) the one above.
template <int Q, int N>
cudaError_t launch_apply_fast(const FrameTable<N> &all, cudaStream_t st)
{
    FastKArgs<N> k;
    FrameTable<N> rest;
    FastArgs tma_f[N], run_f[N];
    int nt = 0, nr = 0;
    std::memset(&k, 0, sizeof(k));
    k.wait_ns = kFastTimeoutNs;
    for (int i = 0; i < all.n; ++i) {
        const FastArgs &a = all.f[i];
        const int P = a.F * a.s;
        const bool aligned = (a.Wo & 3) == 0 && ((uintptr_t)a.map_guide & 15) == 0 && P <= 8;
        if (aligned && tma::encode_planes_f32(&k.t0[nt], a.map_guide, a.Wo, a.Ho, Q, kFW, P, Q) == cudaSuccess)
            tma_f[nt++] = a;
        else
            run_f[nr++] = a;
    }
    if (nt > 0) {
        fill_table(k.t, nt, tma_f, all.count, all.status);
        for (int i = 0; i < nt; ++i)
            k.t.off[3][i + 1] = k.t.off[3][i] + (unsigned)((tma_f[i].Hb + 1) * ((tma_f[i].Wo + kFW - 1) / kFW));
        const size_t smem = apply_tma_smem<Q>();
        const bool cell8 = tma_f[0].F * tma_f[0].s == 8;
        auto kern = cell8 ? apply_tma_kernel<Q, N, 8> : apply_tma_kernel<Q, N, 0>;
        // three CTAs per SM need the whole unified L1 / shared array as shared memory
        cudaError_t e = cell8 ? pdl::allow_smem<KernelTag<1, Q, N, 8>>(kern, smem, true) : pdl::allow_smem<KernelTag<1, Q, N, 0>>(kern, smem, true);
        if (e != cudaSuccess) return e;
        const unsigned nitems = k.t.off[3][nt], most = 3 * (unsigned)pdl::sm_count();  // three CTAs per SM
        e = pdl::launch(kern, dim3(nitems < most ? nitems : most), kFW, smem, st, k);
        if (e != cudaSuccess || nr == 0) return e;
    }
    fill_table(rest, nr, run_f, all.count, all.status);
    return launch_apply_plain<Q>(rest, st);
}

// The four stages over n frames: each launch may start while its predecessor drains (pdl.cuh),
// which hides three launch gaps of about 2.5 us each.
template <int Q, int N>
cudaError_t launch_fast_q(int n, const FastArgs *f, unsigned long long *count, int *status, cudaStream_t st)
{
    FrameTable<N> t;
    fill_table(t, n, f, count, status);
    cudaError_t e = launch_moments_f<Q>(t, st);
    if (e != cudaSuccess) return e;
    if ((e = pdl::launch(blur_h_kernel<Q, N>, dim3(t.off[1][n]), kBlurThreads, 0, st, t)) != cudaSuccess) return e;
    e = pdl::launch(blur_v_solve_kernel<Q, N>, dim3(t.off[2][n]), kBlurThreads,
                    sizeof(float) * Chan<Q>::NCH * kBlurThreads, st, t);
    if (e != cudaSuccess) return e;
    return launch_apply_fast<Q>(t, st);
}

// Parameter gradients of one frame: the forward's moments and horizontal blur, the
// horizontal blur with the weights' sigma-derivative, the tangent solve, then per parameter
// the apply of its model tangents (frame reference without the radiance offset, tshift) and
// the dot product with grad_out into grad[t].  dout: [3][Ho][Wo] scratch; part: kDotBlocks
// doubles.
template <int Q>
cudaError_t launch_param_grad_q(const FastArgs &a, unsigned long long *count, float *tshift, const float *grad_out,
                                float *dout, double *part, double *grad, cudaStream_t st)
{
    FrameTable<1> t;
    fill_table(t, 1, &a, count, (int *)nullptr);
    cudaError_t e = launch_moments_f<Q>(t, st);
    if (e != cudaSuccess) return e;
    const size_t nb = (size_t)a.Hb * a.Wb;
    const unsigned gb = (unsigned)((nb + 127) / 128);
    if ((e = pdl::launch(blur_h_kernel<Q, 1>, dim3(t.off[1][1]), kBlurThreads, 0, st, t)) != cudaSuccess) return e;
    FrameTable<1> td = t;  // the horizontal blur with w' = dw/dsigma into tmp2
    td.f[0].tmp = a.tmp2;
    std::memcpy(td.f[0].w, a.wd, sizeof(a.wd));
    if ((e = pdl::launch(blur_h_kernel<Q, 1>, dim3(t.off[1][1]), kBlurThreads, 0, st, td)) != cudaSuccess) return e;
    const size_t smem = sizeof(float) * 2 * Chan<Q>::NCH * 128;
    if ((e = pdl::allow_smem<KernelTag<2, Q>>(blur_v_tangent_kernel<Q>, smem, false)) != cudaSuccess) return e;
    blur_v_tangent_kernel<Q><<<gb, 128, smem, st>>>(a);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    // the frame reference the moments wrote, with the radiance offset zero: a tangent of the
    // output carries no constant
    if ((e = cudaMemcpyAsync(tshift, a.shift, sizeof(float) * Q, cudaMemcpyDeviceToDevice, st)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(tshift + Q, 0, sizeof(float) * 3, st)) != cudaSuccess) return e;
    const size_t npx = 3 * (size_t)a.Ho * a.Wo;
    for (int p = 0; p < 3; ++p) {
        FrameTable<1> tp = t;
        tp.f[0].coef = a.dcoef + (size_t)p * nb * fast::Model<Q>::CS;
        tp.f[0].shift = tshift;
        tp.f[0].out = dout;
        if ((e = launch_apply_plain<Q>(tp, st)) != cudaSuccess) return e;
        dot_partial_kernel<<<kDotBlocks, 256, 0, st>>>(dout, grad_out, npx, part);
        dot_final_kernel<<<1, kDotBlocks, 0, st>>>(part, grad + p);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_param_grad(int q, const FastArgs &a, unsigned long long *count, float *tshift, const float *grad_out,
                              float *dout, double *part, double *grad, cudaStream_t st)
{
    switch (q) {
    case 1: return launch_param_grad_q<1>(a, count, tshift, grad_out, dout, part, grad, st);
    case 2: return launch_param_grad_q<2>(a, count, tshift, grad_out, dout, part, grad, st);
    case 3: return launch_param_grad_q<3>(a, count, tshift, grad_out, dout, part, grad, st);
    case 4: return launch_param_grad_q<4>(a, count, tshift, grad_out, dout, part, grad, st);
    case 5: return launch_param_grad_q<5>(a, count, tshift, grad_out, dout, part, grad, st);
    case 6: return launch_param_grad_q<6>(a, count, tshift, grad_out, dout, part, grad, st);
    case 7: return launch_param_grad_q<7>(a, count, tshift, grad_out, dout, part, grad, st);
    case 8: return launch_param_grad_q<8>(a, count, tshift, grad_out, dout, part, grad, st);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_fast(int q, const FastArgs &a, unsigned long long *count, cudaStream_t st)
{
    switch (q) {
    case 1: return launch_fast_q<1, 1>(1, &a, count, nullptr, st);
    case 2: return launch_fast_q<2, 1>(1, &a, count, nullptr, st);
    case 3: return launch_fast_q<3, 1>(1, &a, count, nullptr, st);
    case 4: return launch_fast_q<4, 1>(1, &a, count, nullptr, st);
    case 5: return launch_fast_q<5, 1>(1, &a, count, nullptr, st);
    case 6: return launch_fast_q<6, 1>(1, &a, count, nullptr, st);
    case 7: return launch_fast_q<7, 1>(1, &a, count, nullptr, st);
    case 8: return launch_fast_q<8, 1>(1, &a, count, nullptr, st);
    default: return cudaErrorInvalidValue;
    }
}

bool batch_supported(int q, int F) { return (q == 1 || q == 4 || q == 8) && (F == 2 || F == 4 || F == 8); }

cudaError_t launch_fast_batch(int q, int n, const FastArgs *f, unsigned long long *count, int *status, cudaStream_t st)
{
    switch (q) {
    case 1: return launch_fast_q<1, FLR_MAX_BATCH>(n, f, count, status, st);
    case 4: return launch_fast_q<4, FLR_MAX_BATCH>(n, f, count, status, st);
    case 8: return launch_fast_q<8, FLR_MAX_BATCH>(n, f, count, status, st);
    default: return cudaErrorInvalidValue;
    }
}

// Self-test of the bounded mbarrier wait the TMA and tensor-core kernels use: barrier 0
// expects two arrivals and receives one, so its phase never completes and every warp's wait
// must run out (status bit 0); barrier 1 expects one arrival and receives it, so the wait
// must succeed (a timeout there sets bit 1).
__global__ void mbarrier_selftest_kernel(int *status, unsigned long long timeout_ns)
{
    __shared__ uint64_t bar[2];
    if (threadIdx.x == 0) {
        tma::mbar_init(&bar[0], 2);
        tma::mbar_init(&bar[1], 1);
        tma::mbar_init_fence();
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(tma::smem_addr(&bar[0])) : "memory");
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(tma::smem_addr(&bar[1])) : "memory");
    }
    __syncthreads();
    const bool done0 = tma::wait_warp(&bar[0], 0, timeout_ns);
    const bool done1 = tma::wait_warp(&bar[1], 0, timeout_ns);
    if ((threadIdx.x & 31) == 0) {
        if (!done0) atomicOr(status, 1);
        if (!done1) atomicOr(status, 2);
    }
}

// Self-test of apply_tma_kernel's way out: a frame of zero models on four CTAs of nine items each,
// once with waits that give up at once, so that every CTA leaves with two copies in flight, and
// once with the ordinary limit into an output of NaNs.
cudaError_t abort_selftest(int *result)
{
    constexpr int Q = 8, F = 8, H = 64, W = 512, Hb = H / F, Wb = W / F, CS = fast::Model<Q>::CS;
    constexpr size_t px = (size_t)H * W, nz = Q * px, nc = (size_t)Hb * Wb * CS, total = nz + nc + 32 + 3 * px;
    float *buf = nullptr;
    cudaError_t e = cudaMalloc(&buf, total * sizeof(float));
    if (e != cudaSuccess) return e;
    FastKArgs<1> k;
    std::memset(&k, 0, sizeof(k));
    FastArgs a = {};
    a.map_guide = buf;
    a.coef = buf + nz;
    a.shift = a.coef + nc;
    a.status = (int *)(a.shift + 16);
    a.out = a.shift + 32;
    a.Hi = a.Ho = H;
    a.Wi = a.Wo = W;
    a.Hb = Hb;
    a.Wb = Wb;
    a.F = F;
    a.s = 1;
    fill_table(k.t, 1, &a, (unsigned long long *)nullptr, (int *)nullptr);
    k.t.off[3][1] = (Hb + 1) * (W / kFW);
    const size_t smem = apply_tma_smem<Q>();
    e = tma::encode_planes_f32(&k.t0[0], a.map_guide, W, H, Q, kFW, F, Q);
    if (e == cudaSuccess)
        e = pdl::allow_smem<KernelTag<1, Q, 1, 8>>(apply_tma_kernel<Q, 1, 8>, smem, true);
    std::vector<float> out(3 * px);
    *result = 0;
    for (int pass = 0; pass < 2 && e == cudaSuccess; ++pass) {
        int status = 0;
        k.wait_ns = pass ? kFastTimeoutNs : 0;
        e = cudaMemset(buf, 0, (nz + nc + 32) * sizeof(float));
        if (e == cudaSuccess) e = cudaMemset(a.out, 0xff, 3 * px * sizeof(float));
        if (e == cudaSuccess) e = pdl::launch(apply_tma_kernel<Q, 1, 8>, dim3(4), kFW, smem, (cudaStream_t)0, k);
        if (e == cudaSuccess) e = cudaMemcpy(&status, a.status, sizeof(int), cudaMemcpyDeviceToHost);
        if (e == cudaSuccess) e = cudaMemcpy(out.data(), a.out, 3 * px * sizeof(float), cudaMemcpyDeviceToHost);
        bool zero = true;
        for (float v : out) zero &= v == 0.f;
        if (pass == 0 && status != 0) *result |= 1;
        if (pass == 1 && (status != 0 || !zero)) *result |= 2;
    }
    cudaFree(buf);
    return e;
}

thread_local char g_fast_err[256] = "no error";

}  // namespace
}  // namespace flr

struct flr_fast_handle {
    flr_fast_params p;
    float w[2 * flr::fast::kMaxTaps + 1];
    float *ws = nullptr;  // block moments, blur temporary, block models
    size_t ws_blocks = 0;
    float *shift = nullptr;
    unsigned long long *count = nullptr;
    int *status = nullptr;  // set by a kernel whose bounded wait ran out
    cudaStream_t last_stream = nullptr;
    // parameter gradients: sigma-derivative of the weights, workspace (second horizontal
    // blur, model tangents, frame reference without radiance offset, output tangent), partials
    float wd[2 * flr::fast::kMaxTaps + 1];
    float *gws = nullptr;
    size_t gws_floats = 0;
    double *gpart = nullptr;
    // batch path: per-frame workspace, status word
    float *bws = nullptr;
    size_t bws_floats = 0;
    int *bstatus = nullptr;
};

namespace {

int n_channels(int q) { return q + 3 + q * (q + 1) / 2 + 3 * q; }

// Workspace of a frame of nb blocks: block sums and references, blurred sums and count, models
// (16-byte aligned: up to 3 floats more)
size_t frame_floats(int q, size_t nb)
{
    return nb * (2 * (size_t)n_channels(q) + (size_t)(q + 3) + 1 + flr::fast::model_floats(q)) + 4;
}
float *align16(float *p) { return (float *)(((uintptr_t)p + 15) & ~(uintptr_t)15); }

// Fill one frame's arguments; ws points at its per-block workspace.
void frame_args(const flr_fast_handle *h, const flr_frame &fr, float *ws, flr::fast::FastArgs &a)
{
    const int q = h->p.q, F = h->p.factor, s = h->p.scale;
    const int Hb = (fr.H + F - 1) / F, Wb = (fr.W + F - 1) / F;
    const size_t nb = (size_t)Hb * Wb;
    const int nch = n_channels(q);
    a.guide = fr.guide;
    a.rad = fr.radiance;
    a.map_guide = fr.map_guide ? fr.map_guide : fr.guide;
    a.out = fr.out;
    a.blk = ws;
    a.tmp = ws + nb * (nch + q + 3);
    a.coef = align16(a.tmp + nb * (nch + 1));
    a.shift = h->shift;  // replaced per frame by the caller
    a.flag_count = h->count;
    a.Hi = fr.H;
    a.Wi = fr.W;
    a.Ho = fr.H * s;
    a.Wo = fr.W * s;
    a.Hb = Hb;
    a.Wb = Wb;
    a.F = F;
    a.s = s;
    a.taps = h->p.taps;
    a.eps = h->p.eps;
    a.tau = h->p.pivot_ratio;
    a.appendix = (h->p.flags & FLR_FAST_APPENDIX) ? 1 : 0;
    a.eps_mul = h->p.eps_mul;
    std::memcpy(a.w, h->w, sizeof(a.w));
}

int check_frames(const flr_fast_handle *h, int n, const flr_frame *frames, size_t *floats)
{
    if (!h || n <= 0 || n > FLR_MAX_BATCH || !frames) return FLR_ERR_ARG;
    if (!flr::batch_supported(h->p.q, h->p.factor)) return FLR_ERR_UNSUPPORTED;
    size_t total = 0;
    for (int i = 0; i < n; ++i) {
        const flr_frame &f = frames[i];
        if (!f.guide || !f.radiance || !f.out || f.H <= 0 || f.W <= 0) return FLR_ERR_ARG;
        if (h->p.scale > 1 && !f.map_guide) return FLR_ERR_ARG;
        if ((long long)f.H * h->p.scale * f.W * h->p.scale > 0x7fffffffLL) return FLR_ERR_ARG;
        if (((uintptr_t)f.guide | (uintptr_t)f.radiance | (uintptr_t)f.out | (uintptr_t)f.map_guide) & 15u)
            return FLR_ERR_ALIGN;
        const size_t nb = (size_t)((f.H + h->p.factor - 1) / h->p.factor) * ((f.W + h->p.factor - 1) / h->p.factor);
        total += frame_floats(h->p.q, nb) + 64;  // + room for the frame's reference shift
    }
    *floats = total;
    return FLR_OK;
}

}  // namespace

extern "C" {

int flr_fast_create(const flr_fast_params *p, flr_fast_handle **out)
{
    if (!out || !p) return FLR_ERR_ARG;
    *out = nullptr;
    if ((p->flags & ~FLR_FAST_APPENDIX) != 0u || !(p->eps >= 0.f) || !(p->sigma > 0.f) || p->taps < 0 ||
        p->scale < 1 || p->pivot_ratio != p->pivot_ratio || !(p->eps_mul >= 0.f && p->eps_mul <= 1.f) ||
        (!(p->flags & FLR_FAST_APPENDIX) && p->eps_mul != 0.f))
        return FLR_ERR_ARG;
    if (p->q < 1 || p->q > FLR_MAX_Q || p->taps > flr::fast::kMaxTaps || p->scale > 8 ||
        (p->factor != 2 && p->factor != 4 && p->factor != 8))
        return FLR_ERR_UNSUPPORTED;
    flr_fast_handle *h = new (std::nothrow) flr_fast_handle();
    if (!h) return FLR_ERR_NOMEM;
    h->p = *p;
    for (int d = -p->taps; d <= p->taps; ++d) {
        const double sg = (double)p->sigma, wv = std::exp(-(double)d * d / (2.0 * sg * sg));
        h->w[d + p->taps] = (float)wv;
        h->wd[d + p->taps] = (float)(wv * (double)d * d / (sg * sg * sg));  // d w / d sigma
    }
    if (cudaMalloc(&h->shift, sizeof(float) * (FLR_MAX_Q + 3)) != cudaSuccess ||
        cudaMalloc(&h->count, sizeof(unsigned long long)) != cudaSuccess ||
        cudaMalloc(&h->status, sizeof(int)) != cudaSuccess || cudaMemset(h->status, 0, sizeof(int)) != cudaSuccess) {
        flr_fast_destroy(h);
        return FLR_ERR_NOMEM;
    }
    *out = h;
    return FLR_OK;
}

int flr_fast_destroy(flr_fast_handle *h)
{
    if (!h) return FLR_OK;
    cudaDeviceSynchronize();
    cudaFree(h->ws);
    cudaFree(h->gws);
    cudaFree(h->gpart);
    cudaFree(h->bws);
    cudaFree(h->bstatus);
    cudaFree(h->shift);
    cudaFree(h->count);
    cudaFree(h->status);
    delete h;
    return FLR_OK;
}

int flr_fast_denoise(flr_fast_handle *h, const float *guide, const float *map_guide, const float *radiance,
                     float *out, int Hi, int Wi, void *stream)
{
    if (!h || !guide || !radiance || !out || Hi <= 0 || Wi <= 0) return FLR_ERR_ARG;
    const int s = h->p.scale, F = h->p.factor, q = h->p.q;
    if (s > 1 && !map_guide) return FLR_ERR_ARG;
    if ((long long)Hi * s * Wi * s > 0x7fffffffLL) return FLR_ERR_ARG;
    if (((uintptr_t)guide | (uintptr_t)radiance | (uintptr_t)out | (uintptr_t)map_guide) & 15u) return FLR_ERR_ALIGN;
    const int Hb = (Hi + F - 1) / F, Wb = (Wi + F - 1) / F;
    const size_t nb = (size_t)Hb * Wb;
    const int nch = n_channels(q);
    if (h->ws_blocks < nb || !h->ws) {
        cudaFree(h->ws);
        h->ws = nullptr;
        h->ws_blocks = 0;
        if (cudaMalloc(&h->ws, sizeof(float) * frame_floats(q, nb)) != cudaSuccess)
            return FLR_ERR_NOMEM;
        h->ws_blocks = nb;
    }
    flr::fast::FastArgs a;
    a.guide = guide;
    a.rad = radiance;
    a.map_guide = map_guide ? map_guide : guide;
    a.out = out;
    a.blk = h->ws;
    a.tmp = h->ws + nb * (nch + q + 3);
    a.coef = align16(a.tmp + nb * (nch + 1));
    a.shift = h->shift;
    a.flag_count = h->count;
    a.Hi = Hi;
    a.Wi = Wi;
    a.Ho = Hi * s;
    a.Wo = Wi * s;
    a.Hb = Hb;
    a.Wb = Wb;
    a.F = F;
    a.s = s;
    a.taps = h->p.taps;
    a.eps = h->p.eps;
    a.tau = h->p.pivot_ratio;
    a.appendix = (h->p.flags & FLR_FAST_APPENDIX) ? 1 : 0;
    a.eps_mul = h->p.eps_mul;
    a.status = h->status;
    std::memcpy(a.w, h->w, sizeof(a.w));
    cudaStream_t st = (cudaStream_t)stream;
    h->last_stream = st;
    const cudaError_t e = flr::launch_fast(q, a, h->count, st);
    if (e != cudaSuccess) {
        std::snprintf(flr::g_fast_err, sizeof(flr::g_fast_err), "%s", cudaGetErrorString(e));
        return FLR_ERR_CUDA;
    }
    return FLR_OK;
}

int flr_fast_reserve_batch(flr_fast_handle *h, int n, const flr_frame *frames)
{
    size_t floats = 0;
    int st = check_frames(h, n, frames, &floats);
    if (st != FLR_OK) return st;
    if (!h->bstatus && cudaMalloc(&h->bstatus, sizeof(int)) != cudaSuccess) return FLR_ERR_NOMEM;
    if (h->bws_floats < floats || !h->bws) {
        cudaFree(h->bws);
        h->bws = nullptr;
        h->bws_floats = 0;
        if (cudaMalloc(&h->bws, floats * sizeof(float)) != cudaSuccess) return FLR_ERR_NOMEM;
        h->bws_floats = floats;
    }
    return FLR_OK;
}

int flr_fast_denoise_batch(flr_fast_handle *h, int n, const flr_frame *frames, void *stream)
{
    size_t floats = 0;
    int st = check_frames(h, n, frames, &floats);
    if (st != FLR_OK) return st;
    if (h->bws_floats < floats || !h->bstatus) {
        st = flr_fast_reserve_batch(h, n, frames);
        if (st != FLR_OK) return st;
    }
    flr::fast::FastArgs fa[FLR_MAX_BATCH];
    float *ws = h->bws;
    for (int i = 0; i < n; ++i) {
        frame_args(h, frames[i], ws + 64, fa[i]);
        fa[i].shift = ws;  // this frame's reference shift
        fa[i].status = h->bstatus;
        const size_t nb = (size_t)fa[i].Hb * fa[i].Wb;
        ws += frame_floats(h->p.q, nb) + 64;
    }
    cudaStream_t s = (cudaStream_t)stream;
    h->last_stream = s;
    const cudaError_t e = flr::launch_fast_batch(h->p.q, n, fa, h->count, h->bstatus, s);
    if (e != cudaSuccess) {
        std::snprintf(flr::g_fast_err, sizeof(flr::g_fast_err), "%s", cudaGetErrorString(e));
        return FLR_ERR_CUDA;
    }
    return FLR_OK;
}

int flr_fast_batch_status(flr_fast_handle *h)
{
    if (!h || !h->bstatus) return FLR_ERR_ARG;
    int status = 0;
    if (cudaStreamSynchronize(h->last_stream) != cudaSuccess ||
        cudaMemcpy(&status, h->bstatus, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess)
        return FLR_ERR_CUDA;
    return status == 0 ? FLR_OK : FLR_ERR_TIMEOUT;
}

int flr_barrier_selftest(int ctas, unsigned long long timeout_ns, int *status)
{
    if (ctas <= 0 || ctas > 1024 || !status || timeout_ns > 10000000000ull) return FLR_ERR_ARG;
    unsigned *w = nullptr;
    if (cudaMalloc(&w, 4 * sizeof(unsigned)) != cudaSuccess) return FLR_ERR_NOMEM;
    cudaError_t e = cudaMemset(w, 0, 4 * sizeof(unsigned));
    if (e == cudaSuccess) e = flr::launch_barrier_selftest(w, w + 1, (unsigned)ctas + 1, (int *)(w + 2), timeout_ns, ctas, nullptr);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = cudaMemcpy(status, w + 2, sizeof(int), cudaMemcpyDeviceToHost);
    cudaFree(w);
    return e == cudaSuccess ? FLR_OK : FLR_ERR_CUDA;
}

int flr_mbarrier_selftest(int ctas, unsigned long long timeout_ns, int *status)
{
    if (ctas <= 0 || ctas > 1024 || !status || timeout_ns > 10000000000ull) return FLR_ERR_ARG;
    int *d = nullptr;
    if (cudaMalloc(&d, sizeof(int)) != cudaSuccess) return FLR_ERR_NOMEM;
    cudaError_t e = cudaMemset(d, 0, sizeof(int));
    if (e == cudaSuccess) {
        flr::mbarrier_selftest_kernel<<<ctas, 64>>>(d, timeout_ns);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = cudaMemcpy(status, d, sizeof(int), cudaMemcpyDeviceToHost);
    cudaFree(d);
    return e == cudaSuccess ? FLR_OK : FLR_ERR_CUDA;
}

int flr_fast_abort_selftest(int *status)
{
    if (!status) return FLR_ERR_ARG;
    const cudaError_t e = flr::abort_selftest(status);
    return e == cudaSuccess ? FLR_OK : e == cudaErrorMemoryAllocation ? FLR_ERR_NOMEM : FLR_ERR_CUDA;
}

int flr_fast_param_grad(flr_fast_handle *h, const float *guide, const float *map_guide, const float *radiance,
                        const float *grad_out, double *grad, int Hi, int Wi, void *stream)
{
    if (!h || !guide || !radiance || !grad_out || !grad || Hi <= 0 || Wi <= 0) return FLR_ERR_ARG;
    const int s = h->p.scale, F = h->p.factor, q = h->p.q;
    if (s > 1 && !map_guide) return FLR_ERR_ARG;
    if ((long long)Hi * s * Wi * s > 0x7fffffffLL) return FLR_ERR_ARG;
    if (((uintptr_t)guide | (uintptr_t)radiance | (uintptr_t)grad_out | (uintptr_t)map_guide) & 15u ||
        ((uintptr_t)grad & 7u))
        return FLR_ERR_ALIGN;
    const int Hb = (Hi + F - 1) / F, Wb = (Wi + F - 1) / F;
    const size_t nb = (size_t)Hb * Wb, npx = (size_t)Hi * s * Wi * s;
    const int nch = n_channels(q);
    if (h->ws_blocks < nb || !h->ws) {
        cudaFree(h->ws);
        h->ws = nullptr;
        h->ws_blocks = 0;
        if (cudaMalloc(&h->ws, sizeof(float) * frame_floats(q, nb)) != cudaSuccess)
            return FLR_ERR_NOMEM;
        h->ws_blocks = nb;
    }
    // gradient workspace: tmp2, dcoef, tshift (32 floats), dout
    const size_t off_dc = ((size_t)(nch + 1) * nb + 3) & ~(size_t)3, off_ts = off_dc + 3 * (size_t)flr::fast::model_floats(q) * nb;
    const size_t off_out = (off_ts + 32 + 3) & ~(size_t)3, need = off_out + 3 * npx;
    if (h->gws_floats < need || !h->gws) {
        cudaFree(h->gws);
        h->gws = nullptr;
        h->gws_floats = 0;
        if (cudaMalloc(&h->gws, need * sizeof(float)) != cudaSuccess) return FLR_ERR_NOMEM;
        h->gws_floats = need;
    }
    if (!h->gpart && cudaMalloc(&h->gpart, sizeof(double) * flr::kDotBlocks) != cudaSuccess) return FLR_ERR_NOMEM;
    flr::fast::FastArgs a;
    std::memset(&a, 0, sizeof(a));
    a.guide = guide;
    a.rad = radiance;
    a.map_guide = map_guide ? map_guide : guide;
    a.out = nullptr;
    a.blk = h->ws;
    a.tmp = h->ws + nb * (nch + q + 3);
    a.coef = align16(a.tmp + nb * (nch + 1));
    a.tmp2 = h->gws;
    a.dcoef = h->gws + off_dc;
    a.shift = h->shift;
    a.flag_count = h->count;
    a.Hi = Hi;
    a.Wi = Wi;
    a.Ho = Hi * s;
    a.Wo = Wi * s;
    a.Hb = Hb;
    a.Wb = Wb;
    a.F = F;
    a.s = s;
    a.taps = h->p.taps;
    a.eps = h->p.eps;
    a.tau = h->p.pivot_ratio;
    a.appendix = (h->p.flags & FLR_FAST_APPENDIX) ? 1 : 0;
    a.eps_mul = h->p.eps_mul;
    a.status = h->status;
    std::memcpy(a.w, h->w, sizeof(a.w));
    std::memcpy(a.wd, h->wd, sizeof(a.wd));
    cudaStream_t st = (cudaStream_t)stream;
    h->last_stream = st;
    const cudaError_t e =
        flr::launch_param_grad(q, a, h->count, h->gws + off_ts, grad_out, h->gws + off_out, h->gpart, grad, st);
    if (e != cudaSuccess) {
        std::snprintf(flr::g_fast_err, sizeof(flr::g_fast_err), "%s", cudaGetErrorString(e));
        return FLR_ERR_CUDA;
    }
    return FLR_OK;
}

int flr_fast_get_stats(flr_fast_handle *h, flr_stats *out)
{
    if (!h || !out) return FLR_ERR_ARG;
    unsigned long long n = 0;
    if (cudaStreamSynchronize(h->last_stream) != cudaSuccess ||
        cudaMemcpy(&n, h->count, sizeof(n), cudaMemcpyDeviceToHost) != cudaSuccess)
        return FLR_ERR_CUDA;
    out->flagged = n;
    out->resolved = h->p.pivot_ratio > 0.f ? n : 0ull;
    out->nonfinite = 0ull;  // not counted by the fast path
    int status = 0;
    if (cudaMemcpy(&status, h->status, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return FLR_ERR_CUDA;
    if (status != 0) {
        if (cudaMemset(h->status, 0, sizeof(int)) != cudaSuccess) return FLR_ERR_CUDA;
        return FLR_ERR_TIMEOUT;
    }
    return FLR_OK;
}

}  // extern "C"
