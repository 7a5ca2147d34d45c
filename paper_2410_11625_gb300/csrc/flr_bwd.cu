// flr_bwd.cu -- kernels of the FLR backward pass that are not the per-pixel adjoint solve
// (that one is the forward kernel in adjoint mode, flr_fwd_kernel.cuh).  sm_103a.
//
// The backward pass is the reverse-mode derivative of the forward's steps (the paper
// trains through FLR by backpropagation, Sec. 3.2-3.3; it prints no adjoint).  With
// g = dL/dI and m_i the size of the clipped averaging window T'_i:
//   fields    F_i = (1, z_i - s) g_i^T / m_i                       (adjoint of the apply)
//   G(A_k)    = sum_{i in T'_k} F_i                                (adjoint of the average)
//   adjoint   per pixel k: the moment gradients GS_k               (flr_fwd_kernel.cuh, ADJ = true)
//   BS_j      = sum_{k in T_j} GS_k                                (adjoint of the window sums)
//   contract  dx_j = BS_x + 2 BS_xx (x_j - s) + BS_xy (y_j - s_y)
//             dy_j = BS_y + BS_xy^T (x_j - s)
//             dz_j = Abar_j g_j                                    (the applied guide)
// j in T_k <=> k in T_j for clipped square windows of one radius, so every adjoint of a
// window sum is the same clipped box sum.
// Every launch here is a dependent one (pdl.cuh) without an early trigger, as those of the unfused
// forward path: backward 1920x1080 957 -> 946 us, 719 x 1277 forward, q = 6, 151 -> 146 us.
#include <algorithm>
#include <cstring>
#include <type_traits>

#include "flr.h"
#include "flr_internal.cuh"
#include "pdl.cuh"
#include "tma.cuh"

namespace flr {
namespace {

constexpr int kBW = 64, kBH = 32, kBThreads = 256;

template <int Q>
__global__ void bwd_fields_kernel(const float *__restrict__ g, const float *__restrict__ z,
                                  const float *__restrict__ shift, float *__restrict__ F, int H, int W, int pitch, int rc)
{
    pdl::wait();
    const size_t plane = (size_t)H * W;
    for (size_t p = (size_t)blockIdx.x * blockDim.x + threadIdx.x; p < plane; p += (size_t)gridDim.x * blockDim.x) {
        const int y = (int)(p / W), x = (int)(p % W);
        const size_t fplane = (size_t)H * pitch, fp = (size_t)y * pitch + x;
        float inv_m = 1.f;
        if (rc > 0) {
            const float ny = (float)(min(y + rc, H - 1) - max(y - rc, 0) + 1);
            const float nx = (float)(min(x + rc, W - 1) - max(x - rc, 0) + 1);
            inv_m = 1.0f / (ny * nx);
        }
        float gc[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            gc[c] = g[c * plane + p] * inv_m;
            F[c * fplane + fp] = gc[c];
        }
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const float zi = z[i * plane + p] - shift[i];
#pragma unroll
            for (int c = 0; c < 3; ++c) F[(3 * (i + 1) + c) * fplane + fp] = zi * gc[c];
        }
    }
}

// out[plane] = sum over the clipped radius-rad window of in[plane]; blockIdx.z = plane.
__global__ void __launch_bounds__(kBThreads) box_sum_kernel(const float *__restrict__ in, float *__restrict__ out,
                                                           int H, int W, int pitch, int rad)
{
    pdl::wait();
    extern __shared__ float sm[];
    const int TWh = kBW + 2 * rad, THh = kBH + 2 * rad;
    const int TS = TWh + 1, HS = kBW + 1;
    float *T = sm;
    float *Hb = T + THh * TS;
    const size_t plane = (size_t)H * pitch;
    const float *src = in + (size_t)blockIdx.z * plane;
    float *dst = out + (size_t)blockIdx.z * plane;
    const int tx0 = blockIdx.x * kBW, ty0 = blockIdx.y * kBH;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int row = warp; row < THh; row += kBThreads / 32) {
        const int sy = ty0 - rad + row;
        for (int col = lane; col < TWh; col += 32) {
            const int sx = tx0 - rad + col;
            T[row * TS + col] = (sy >= 0 && sy < H && sx >= 0 && sx < W) ? __ldg(src + (size_t)sy * pitch + sx) : 0.f;
        }
    }
    __syncthreads();
    for (int item = tid; item < THh * 4; item += kBThreads) {
        const int row = item % THh, xr = (item / THh) * 16;
        const float *q = T + row * TS + xr;
        float *h = Hb + row * HS + xr;
        float s = 0.f;
        for (int k = 0; k <= 2 * rad; ++k) s += q[k];
        h[0] = s;
#pragma unroll
        for (int t = 1; t < 16; ++t) {
            s += q[t + 2 * rad] - q[t - 1];
            h[t] = s;
        }
    }
    __syncthreads();
    const int x = tid % kBW, run = tid / kBW;
    const int gx = tx0 + x;
    const float *q = Hb + (run * 8) * HS + x;
    float s = 0.f;
    for (int k = 0; k <= 2 * rad; ++k) s += q[k * HS];
#pragma unroll
    for (int t = 0; t < 8; ++t) {
        if (t > 0) s += q[(t + 2 * rad) * HS] - q[(t - 1) * HS];
        const int gy = ty0 + run * 8 + t;
        if (gx < W && gy < H) dst[(size_t)gy * pitch + gx] = s;
    }
}

// The same clipped box sum over many planes with TMA staging (row pitch a multiple of 16 bytes): a CTA
// walks the planes [p0, p1) of one 64 x 64 output tile, p0 = blockIdx.z * per_cta; each plane's
// tile + halo arrives by one TMA box copy (the copy engine zero-fills outside the image) into
// a double-buffered ring, so the next plane loads while the current one is summed.  Waits are
// bounded (1 s).
//
// The planes' rows are padded to 16 bytes (coef_pitch), so that every width from 16 on comes this
// way: backward 1919 x 1080, r = rc = 8, 1827 us at first, 1089 us so (same bits).
//
// Bound by DRAM: the three calls of a 1080p backward pass (Q = 8) read and write 122 planes of
// 8.3 MB, 298 us at the measured copy rate; they take 324 us.  The form before this was bound by
// instruction issue (64 x 32 tiles, a second buffer for the horizontal sums, one column per
// thread: 38 instructions per value, 68% of the issue slots, 372 us).  Ten warps of
// eight rows each cover the 80 staged rows of radius 8 exactly; a warp's eight rows are its own,
// so the horizontal sums replace their operands in place after a warp-wide barrier (which also
// leaves room for three CTAs per SM); the vertical sums take two columns per thread, packed.
// Each sum adds the same values in the same order as that form did: a run of 16 columns (8 rows)
// from a multiple of 16 (8) on starts from its full window and slides.
constexpr int kTH = 64, kTThreads = 320;

struct alignas(128) BoxKArgs {
    CUtensorMap tm;  // [nplanes][H][W] float32, box (TS, THh, 1)
    float *out;
    int H, W, pitch, rad, nplanes, per_cta;
    int *status;
};

struct BoxGeom {
    int RCA, TWa, THh, TS;
    __host__ __device__ constexpr BoxGeom(int rad)
        : RCA((rad + 3) & ~3),        // staged columns start 16-byte aligned
          TWa(kBW + 2 * ((rad + 3) & ~3)),
          THh(kTH + 2 * rad),
          TS(kBW + 2 * ((rad + 3) & ~3) + 4)  // row stride = 4 (mod 8) floats: conflict-free 128-bit phases
    {
    }
    __host__ __device__ constexpr int tile_floats() const { return (THh * TS + 31) / 32 * 32; }
    __host__ __device__ constexpr size_t floats() const { return 32 + (size_t)2 * tile_floats() + 8; }
};

constexpr unsigned long long kBoxTimeoutNs = 1000000000ull;

__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }

// RT: the radius at compile time, or -1 (k.rad).  PARTS: a window's first horizontal sum in four
// interleaved parts (radius 8 at widths that are multiples of 4), else from left to right: each
// width keeps the order of additions it has always had, which the gradients follow.
template <int RT, bool PARTS>
__global__ void __launch_bounds__(kTThreads, 3) box_sum_tma_kernel(const __grid_constant__ BoxKArgs k)
{
    extern __shared__ __align__(16) float sm[];
    const int rad = RT >= 0 ? RT : k.rad;
    const BoxGeom g(rad);
    float *base = sm + (((128 - (tma::smem_addr(sm) & 127)) & 127) >> 2);
    uint64_t *bar = reinterpret_cast<uint64_t *>(base + 2 * g.tile_floats());
    __shared__ int s_abort;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tx0 = blockIdx.x * kBW, ty0 = blockIdx.y * kTH;
    const size_t plane = (size_t)k.H * k.pitch;
    const int p0 = blockIdx.z * k.per_cta, np = min(k.per_cta, k.nplanes - p0);  // p below counts from p0
    auto stage = [&](int p) {
        uint64_t *b = bar + (p & 1);
        tma::mbar_expect_tx(b, (unsigned)(g.THh * g.TS * 4));
        tma::load_3d(base + (p & 1) * g.tile_floats(), &k.tm, tx0 - g.RCA, ty0 - rad, p0 + p, b);
    };
    if (tid == 0) {
        s_abort = 0;
        tma::mbar_init(bar, 1);
        tma::mbar_init(bar + 1, 1);
        tma::mbar_init_fence();
    }
    pdl::wait();
    if (tid == 0) stage(0);
    __syncthreads();
    // vertical sums: a warp takes a run of 8 rows, a lane two columns
    const int gx = tx0 + 2 * lane, gy = ty0 + 8 * warp;
    const int vrows = warp < kTH / 8 && gx < k.W ? min(8, k.H - gy) : 0;
    float *dst = k.out + (size_t)p0 * plane + (size_t)gy * k.pitch + gx;
    for (int p = 0; p < np; ++p, dst += plane) {
        float *T = base + (p & 1) * g.tile_floats();
        if (tid == 0 && p + 1 < np) stage(p + 1);
        if (!tma::wait_warp(bar + (p & 1), (uint32_t)((p >> 1) & 1), kBoxTimeoutNs) && lane == 0) {
            s_abort = 1;
            if (k.status) atomicExch(k.status, 1);
        }
        // horizontal sums in place: 16 outputs per lane, eight rows per warp (lanes 0-7 take
        // consecutive rows: 16-byte accesses at row stride 4 mod 8 floats, distinct banks)
        for (int row = warp * 8 + (lane & 7); row - (lane & 7) < g.THh; row += kTThreads / 4) {
            const bool in = row < g.THh;
            float *q = T + row * g.TS + (lane >> 3) * 16;
            float o[16];
            if (in) {
                if constexpr (RT >= 0) {
                    constexpr int RCA = (RT + 3) & ~3, XO = RCA - RT, N = 16 + 2 * RCA;
                    float v[N];
#pragma unroll
                    for (int kk = 0; kk < N; kk += 4) {
                        const float4 f = *reinterpret_cast<const float4 *>(q + kk);
                        v[kk] = f.x;
                        v[kk + 1] = f.y;
                        v[kk + 2] = f.z;
                        v[kk + 3] = f.w;
                    }
                    float s;
                    if constexpr (PARTS) {
                        float s4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                        for (int kk = 0; kk <= 2 * RT; ++kk) s4[kk & 3] += v[XO + kk];
                        s = (s4[0] + s4[1]) + (s4[2] + s4[3]);
                    } else {
                        s = 0.f;
#pragma unroll
                        for (int kk = 0; kk <= 2 * RT; ++kk) s += v[XO + kk];
                    }
                    o[0] = s;
#pragma unroll
                    for (int t = 1; t < 16; ++t) {
                        s += v[XO + t + 2 * RT] - v[XO + t - 1];
                        o[t] = s;
                    }
                } else {
                    const float *qq = q + (g.RCA - rad);
                    float s = 0.f;
                    for (int kk = 0; kk <= 2 * rad; ++kk) s += qq[kk];
                    o[0] = s;
#pragma unroll
                    for (int t = 1; t < 16; ++t) {
                        s += qq[t + 2 * rad] - qq[t - 1];
                        o[t] = s;
                    }
                }
            }
            __syncwarp();  // the row's operands are read
            if (in) {
#pragma unroll
                for (int t = 0; t < 16; t += 4) *reinterpret_cast<float4 *>(q + t) = make_float4(o[t], o[t + 1], o[t + 2], o[t + 3]);
            }
        }
        __syncthreads();  // horizontal sums complete
        if (s_abort) {  // let a copy still in flight land before the CTA exits, then stop
            if (p + 1 < np && tid < 32)
                tma::wait_warp(bar + ((p + 1) & 1), (uint32_t)(((p + 1) >> 1) & 1), kBoxTimeoutNs);
            return;
        }
        if (vrows > 0) {
            const float2 *q = reinterpret_cast<const float2 *>(T + (warp * 8) * g.TS) + lane;
            const int st = g.TS / 2;
            float2 first[7], s = make_float2(0.f, 0.f);
            if constexpr (RT >= 4) {
#pragma unroll
                for (int kk = 0; kk <= 2 * RT; ++kk) {
                    const float2 f = q[kk * st];
                    if (kk < 7) first[kk < 7 ? kk : 0] = f;
                    s = __fadd2_rn(s, f);
                }
            } else {
                for (int kk = 0; kk <= 2 * rad; ++kk) s = __fadd2_rn(s, q[kk * st]);
            }
            float *d = dst;
#pragma unroll
            for (int t = 0; t < 8; ++t, d += k.pitch) {
                if (t > 0) {
                    const float2 old = RT >= 4 ? first[t - 1] : q[(t - 1) * st];
                    s = __fadd2_rn(s, sub2(q[(t + 2 * rad) * st], old));
                }
                if (t < vrows) *reinterpret_cast<float2 *>(d) = s;
            }
        }
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        __syncthreads();  // this buffer may be refilled from here on
    }
}

template <int Q>
__global__ void __launch_bounds__(256) bwd_contract_kernel(const BwdArgs a)
{
    using C = Chan<Q>;
    pdl::wait();
    const int H = a.H, W = a.W;
    const size_t plane = (size_t)H * W;
    for (size_t p = (size_t)blockIdx.x * blockDim.x + threadIdx.x; p < plane; p += (size_t)gridDim.x * blockDim.x) {
        const int y = (int)(p / W), x = (int)(p % W);
        const size_t bplane = (size_t)H * a.pitch, bp = (size_t)y * a.pitch + x;  // of BS and BA
        // every input of this pixel is read once, up front (the outputs may not alias them)
        float xs[Q], ys[3], gc[3];
#pragma unroll
        for (int i = 0; i < Q; ++i) xs[i] = __ldg(a.guide + i * plane + p) - a.shift[i];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            ys[c] = __ldg(a.rad + c * plane + p) - a.shift[Q + c];
            gc[c] = __ldg(a.g + c * plane + p);
        }
        float inv_m = 1.f;
        if (a.rc > 0) {
            const float ny = (float)(min(y + a.rc, H - 1) - max(y - a.rc, 0) + 1);
            const float nx = (float)(min(x + a.rc, W - 1) - max(x - a.rc, 0) + 1);
            inv_m = 1.0f / (ny * nx);
        }
        const float *BS = a.BS;
        float bxx[C::NXX];
#pragma unroll
        for (int t = 0; t < C::NXX; ++t) bxx[t] = __ldg(BS + (C::XX0 + t) * bplane + bp);
        float bxy[Q][3];
#pragma unroll
        for (int i = 0; i < Q; ++i)
#pragma unroll
            for (int c = 0; c < 3; ++c) bxy[i][c] = __ldg(BS + C::xy(i, c) * bplane + bp);
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            float d = __ldg(BS + (C::X0 + i) * bplane + bp);
#pragma unroll
            for (int j = 0; j < Q; ++j) {
                const int t = (i <= j ? C::xx(i, j) : C::xx(j, i)) - C::XX0;
                d = fmaf(2.f * bxx[t], xs[j], d);
            }
#pragma unroll
            for (int c = 0; c < 3; ++c) d = fmaf(bxy[i][c], ys[c], d);
            // the applied guide: dz_i = sum_c Abar[i][c] g_c
            float dz = 0.f;
#pragma unroll
            for (int c = 0; c < 3; ++c) dz = fmaf(__ldg(a.BA + (3 * (i + 1) + c) * bplane + bp), gc[c], dz);
            dz *= inv_m;
            if (a.separate_map) {
                a.grad_guide[i * plane + p] = d;
                if (a.grad_map) a.grad_map[i * plane + p] = dz;
            } else {
                a.grad_guide[i * plane + p] = d + dz;
            }
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            float d = __ldg(BS + (C::Y0 + c) * bplane + bp);
#pragma unroll
            for (int i = 0; i < Q; ++i) d = fmaf(bxy[i][c], xs[i], d);
            a.grad_rad[c * plane + p] = d;
        }
    }
}

// The same contraction for four consecutive pixels of a row per thread (workspace rows a multiple
// of 16 bytes; ALIGNED: the images' too): one 16-byte load per plane and four pixels instead of four
// 4-byte loads, and each output channel's gradient formed from its own planes in turn, so
// that a thread holds four pixels' inputs and one channel's operands at a time.  Every
// pixel's arithmetic (operands, order of the fused multiply-adds) is that of
// bwd_contract_kernel, so the results are the same bit for bit.  With gridDim.y = Q + 3 a
// thread forms only output channel blockIdx.y (guide channels, then radiance): a small frame
// has too few pixels to fill the chip, and its planes stay in L2 for the second reading.
__device__ __forceinline__ float4 ld4(const float *p) { return __ldg(reinterpret_cast<const float4 *>(p)); }
__device__ __forceinline__ void st4(float *p, float4 v) { *reinterpret_cast<float4 *>(p) = v; }
__device__ __forceinline__ float4 fma4(float4 a, float4 b, float4 c)
{
    return make_float4(fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y), fmaf(a.z, b.z, c.z), fmaf(a.w, b.w, c.w));
}

// The caller's images: 16-byte rows (ALIGNED), or row by row of any width, n of the four pixels inside
template <bool ALIGNED>
__device__ __forceinline__ float4 ld4u(const float *p, int n)
{
    if (ALIGNED) return ld4(p);
    return make_float4(__ldg(p), n > 1 ? __ldg(p + 1) : 0.f, n > 2 ? __ldg(p + 2) : 0.f, n > 3 ? __ldg(p + 3) : 0.f);
}
template <bool ALIGNED>
__device__ __forceinline__ void st4u(float *p, float4 v, int n)
{
    if (ALIGNED) {
        st4(p, v);
        return;
    }
    p[0] = v.x;
    if (n > 1) p[1] = v.y;
    if (n > 2) p[2] = v.z;
    if (n > 3) p[3] = v.w;
}

template <int Q, bool ALIGNED>
__global__ void __launch_bounds__(256) bwd_contract4_kernel(const BwdArgs a)
{
    using C = Chan<Q>;
    pdl::wait();
    const int H = a.H, W = a.W;
    const size_t plane = (size_t)H * W;
    // BS and BA have padded rows of a.pitch floats (a.pitch = W when ALIGNED)
    const int quads = a.pitch / 4;
    const size_t bplane = (size_t)H * a.pitch, nq = (size_t)H * quads;
    for (size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x; q < nq; q += (size_t)gridDim.x * blockDim.x) {
        const int y = (int)(q / quads), x0 = 4 * (int)(q % quads), n = W - x0;
        const size_t p = (size_t)y * W + x0, bp = 4 * q;
        float4 xs[Q], ys[3], gc[3];
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const float4 v = ld4u<ALIGNED>(a.guide + i * plane + p, n);
            const float s = a.shift[i];
            xs[i] = make_float4(v.x - s, v.y - s, v.z - s, v.w - s);
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float4 v = ld4u<ALIGNED>(a.rad + c * plane + p, n);
            const float s = a.shift[Q + c];
            ys[c] = make_float4(v.x - s, v.y - s, v.z - s, v.w - s);
            gc[c] = ld4u<ALIGNED>(a.g + c * plane + p, n);
        }
        float inv_m[4] = {1.f, 1.f, 1.f, 1.f};
        if (a.rc > 0) {
            const float ny = (float)(min(y + a.rc, H - 1) - max(y - a.rc, 0) + 1);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int x = x0 + k;
                const float nx = (float)(min(x + a.rc, W - 1) - max(x - a.rc, 0) + 1);
                inv_m[k] = 1.0f / (ny * nx);
            }
        }
        const float *BS = a.BS;
        const bool all = gridDim.y == 1;
        const int one = blockIdx.y;
#pragma unroll 1
        for (int i = all ? 0 : min(one, Q); i < (all ? Q : min(one + 1, Q)); ++i) {  // one channel's 15 planes in flight
            float4 d = ld4(BS + (C::X0 + i) * bplane + bp);
#pragma unroll
            for (int j = 0; j < Q; ++j) {
                const int t = (i <= j ? C::xx(i, j) : C::xx(j, i));
                const float4 b = ld4(BS + t * bplane + bp);
                d = fma4(make_float4(2.f * b.x, 2.f * b.y, 2.f * b.z, 2.f * b.w), xs[j], d);
            }
#pragma unroll
            for (int c = 0; c < 3; ++c) d = fma4(ld4(BS + C::xy(i, c) * bplane + bp), ys[c], d);
            float4 dz = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int c = 0; c < 3; ++c) dz = fma4(ld4(a.BA + (3 * (i + 1) + c) * bplane + bp), gc[c], dz);
            dz = make_float4(dz.x * inv_m[0], dz.y * inv_m[1], dz.z * inv_m[2], dz.w * inv_m[3]);
            if (a.separate_map) {
                st4u<ALIGNED>(a.grad_guide + i * plane + p, d, n);
                if (a.grad_map) st4u<ALIGNED>(a.grad_map + i * plane + p, dz, n);
            } else {
                st4u<ALIGNED>(a.grad_guide + i * plane + p, make_float4(d.x + dz.x, d.y + dz.y, d.z + dz.z, d.w + dz.w), n);
            }
        }
#pragma unroll 1
        for (int c = all ? 0 : max(one - Q, 0); c < (all ? 3 : one - Q + 1); ++c) {
            float4 d = ld4(BS + (C::Y0 + c) * bplane + bp);
#pragma unroll
            for (int i = 0; i < Q; ++i) d = fma4(ld4(BS + C::xy(i, c) * bplane + bp), xs[i], d);
            st4u<ALIGNED>(a.grad_rad + c * plane + p, d, n);
        }
    }
}

int elem_grid(size_t n) { return (int)((n + 255) / 256 < 4096 ? (n + 255) / 256 : 4096); }

}  // namespace

cudaError_t launch_bwd_fields(int q, const float *g, const float *z, const float *shift, float *F, int H, int W,
                              int pitch, int rc, cudaStream_t st)
{
    const int grid = elem_grid((size_t)H * W);
    switch (q) {
    case 1: return pdl::launch(bwd_fields_kernel<1>, dim3(grid), 256, 0, st, g, z, shift, F, H, W, pitch, rc);
    case 2: return pdl::launch(bwd_fields_kernel<2>, dim3(grid), 256, 0, st, g, z, shift, F, H, W, pitch, rc);
    case 3: return pdl::launch(bwd_fields_kernel<3>, dim3(grid), 256, 0, st, g, z, shift, F, H, W, pitch, rc);
    case 4: return pdl::launch(bwd_fields_kernel<4>, dim3(grid), 256, 0, st, g, z, shift, F, H, W, pitch, rc);
    case 5: return pdl::launch(bwd_fields_kernel<5>, dim3(grid), 256, 0, st, g, z, shift, F, H, W, pitch, rc);
    case 6: return pdl::launch(bwd_fields_kernel<6>, dim3(grid), 256, 0, st, g, z, shift, F, H, W, pitch, rc);
    case 7: return pdl::launch(bwd_fields_kernel<7>, dim3(grid), 256, 0, st, g, z, shift, F, H, W, pitch, rc);
    case 8: return pdl::launch(bwd_fields_kernel<8>, dim3(grid), 256, 0, st, g, z, shift, F, H, W, pitch, rc);
    default: return cudaErrorInvalidValue;
    }
}

template <int RT, bool PARTS>
cudaError_t launch_box_sum_tma(const BoxKArgs &k, cudaStream_t st)
{
    const BoxGeom g(k.rad);
    const size_t smem = sizeof(float) * g.floats();
    // three CTAs per SM need most of the unified L1 / shared array as shared memory
    const BoxGeom most(RT >= 0 ? RT : 16);
    static_assert(FLR_MAX_RADIUS == 16 && FLR_MAX_COEF_RADIUS == 16, "radii known at run time");
    cudaError_t e = pdl::allow_smem<std::integral_constant<int, 2 * RT + PARTS>>(box_sum_tma_kernel<RT, PARTS>, sizeof(float) * most.floats(), true);
    if (e != cudaSuccess) return e;
    dim3 grid((k.W + kBW - 1) / kBW, (k.H + kTH - 1) / kTH, (k.nplanes + k.per_cta - 1) / k.per_cta);
    return pdl::launch(box_sum_tma_kernel<RT, PARTS>, grid, kTThreads, smem, st, k);
}

cudaError_t launch_box_sum(const float *in, float *out, int nplanes, int H, int W, int pitch, int rad, cudaStream_t st,
                           int *status)
{
    if ((pitch & 3) == 0 && ((uintptr_t)in & 15) == 0 && nplanes > 0) {
        BoxKArgs k;
        std::memset(&k, 0, sizeof(k));
        const BoxGeom g(rad);
        if (tma::encode_planes_f32(&k.tm, in, W, H, nplanes, g.TS, g.THh, 1, pitch) == cudaSuccess) {
            k.out = out;
            k.H = H;
            k.W = W;
            k.pitch = pitch;
            k.rad = rad;
            k.nplanes = nplanes;
            k.status = status;
            // Planes per CTA: about eight waves of three CTAs per SM, so that the last wave
            // costs little, and one plane per CTA on frames with fewer tile-planes than that.
            // One CTA walking every plane of a tile left a 128 x 128 frame on 8 SMs (its three
            // box sums 105 us, split 10 us) and a 1080p frame with a second wave two thirds
            // full (the backward pass 1.066 ms, split 1.029 ms).
            const long long tiles = (long long)((W + kBW - 1) / kBW) * ((H + kTH - 1) / kTH);
            const long long target = 8LL * 3 * pdl::sm_count();
            k.per_cta = (int)std::min<long long>(nplanes, std::max<long long>(1, tiles * nplanes / target));
            if (rad == 8) return (W & 3) == 0 ? launch_box_sum_tma<8, true>(k, st) : launch_box_sum_tma<8, false>(k, st);
            return rad == 5 ? launch_box_sum_tma<5, false>(k, st) : launch_box_sum_tma<-1, false>(k, st);
        }
    }
    const size_t smem = sizeof(float) * ((size_t)(kBH + 2 * rad) * (kBW + 2 * rad + 1) + (size_t)(kBH + 2 * rad) * (kBW + 1));
    cudaError_t e = cudaFuncSetAttribute(box_sum_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    dim3 grid((W + kBW - 1) / kBW, (H + kBH - 1) / kBH, nplanes);
    return pdl::launch(box_sum_kernel, grid, kBThreads, smem, st, in, out, H, W, pitch, rad);
}

cudaError_t launch_bwd_contract(int q, const BwdArgs &a, cudaStream_t st)
{
    auto al = [](const void *p) { return ((uintptr_t)p & 15) == 0; };
    if ((a.pitch & 3) == 0 && al(a.BS) && al(a.BA)) {
        // one thread per four pixels; below two CTAs per SM (about 311k pixels, whose planes fit
        // in L2) also one output channel per thread: 128 x 128 takes 14.8 us without, 4.0 us with.
        // Images whose rows are not 16-byte aligned are read and written by single values beside the
        // workspace's 16-byte loads (backward 1919 x 1080: 1052 us, with one thread per pixel 1089).
        const bool aligned = (a.W & 3) == 0 && al(a.guide) && al(a.rad) && al(a.g) && al(a.grad_guide) && al(a.grad_map) &&
                             al(a.grad_rad);
        const int ctas = (int)(((size_t)a.H * (a.pitch / 4) + 255) / 256);
        const dim3 grid4(ctas, ctas < 2 * pdl::sm_count() ? q + 3 : 1);
        auto launch = [&](auto with, auto without) { return pdl::launch(aligned ? with : without, grid4, 256, 0, st, a); };
        switch (q) {
        case 1: return launch(bwd_contract4_kernel<1, true>, bwd_contract4_kernel<1, false>);
        case 2: return launch(bwd_contract4_kernel<2, true>, bwd_contract4_kernel<2, false>);
        case 3: return launch(bwd_contract4_kernel<3, true>, bwd_contract4_kernel<3, false>);
        case 4: return launch(bwd_contract4_kernel<4, true>, bwd_contract4_kernel<4, false>);
        case 5: return launch(bwd_contract4_kernel<5, true>, bwd_contract4_kernel<5, false>);
        case 6: return launch(bwd_contract4_kernel<6, true>, bwd_contract4_kernel<6, false>);
        case 7: return launch(bwd_contract4_kernel<7, true>, bwd_contract4_kernel<7, false>);
        case 8: return launch(bwd_contract4_kernel<8, true>, bwd_contract4_kernel<8, false>);
        default: return cudaErrorInvalidValue;
        }
    }
    const int grid = (int)(((size_t)a.H * a.W + 255) / 256);  // one thread per pixel
    switch (q) {
    case 1: return pdl::launch(bwd_contract_kernel<1>, dim3(grid), 256, 0, st, a);
    case 2: return pdl::launch(bwd_contract_kernel<2>, dim3(grid), 256, 0, st, a);
    case 3: return pdl::launch(bwd_contract_kernel<3>, dim3(grid), 256, 0, st, a);
    case 4: return pdl::launch(bwd_contract_kernel<4>, dim3(grid), 256, 0, st, a);
    case 5: return pdl::launch(bwd_contract_kernel<5>, dim3(grid), 256, 0, st, a);
    case 6: return pdl::launch(bwd_contract_kernel<6>, dim3(grid), 256, 0, st, a);
    case 7: return pdl::launch(bwd_contract_kernel<7>, dim3(grid), 256, 0, st, a);
    case 8: return pdl::launch(bwd_contract_kernel<8>, dim3(grid), 256, 0, st, a);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace flr
