// flr_apply.cu -- FLR coefficient averaging and model application (sm_103a).
//
// Input: the per-pixel models A_k = (b_k, a_k) written by the forward kernel, as
// (Q+1)*3 planes (plane 3*i + c holds row i, column c of A_k; row 0 is the bias), with
// the bias expressed relative to the frame reference shift s.  Output, per pixel i:
//     I_i = (1, z_i - s) * mean_{k in T'_i} A_k  + s_y,
// where T'_i is the clipped square window of radius rc and z the map guide (Sec. 3.1
// applies the model to the centre pixel, I_k = x_k A_k; the averaging over T'_i is the
// coefficient box-average of the guided-filter family that Sec. 3.2 contrasts FLR with).
//
// It reads (Q+1)*3 coefficient planes plus the Q map-guide planes (once per colour, from L2 after
// the first) and writes 3 planes.  The general form follows; eight guides with radii up to 12 have one
// of their own (below).  A CTA owns a 64 x 64 output tile; for each coefficient plane
// it stages the tile plus a radius-rc halo in shared memory, double-buffered so the next plane
// is in flight while this one is summed (zero outside the image, which is what clipping the
// window means for a sum), forms horizontal then vertical radius-rc sums, and accumulates
// sum_k A_k[i][c] * (z_i - s_i) in registers, one colour after the other.  Division by the
// window size happens once at the end, so the averaged coefficients are never materialised.
// Bound by instruction issue and the latency of a plane's three phases, so: the horizontal sums
// replace their operands in place, each warp on eight rows of its own; the vertical sums and the
// products take two columns per thread, packed; every radius is compiled, so that a run's
// operands are registers.  One thread stages each plane tile with a single TMA box copy
// completing on an mbarrier (the coefficient rows are padded to 16 bytes, coef_pitch); planes
// without the padding come by 4-byte asynchronous copies.  719 x 1277, q = 6, rc = 6: 43 us (123 us
// before: 64 x 32 tiles, one column per thread, sums of run-time radius, 4-byte copies).
#include <cstring>
#include <type_traits>

#include "flr.h"
#include "flr_internal.cuh"
#include "pdl.cuh"
#include "tma.cuh"

namespace flr {
namespace {

constexpr int kAW = 64, kAH = 64, kAThreads = 320, kARun = 8;

__device__ __forceinline__ void cp_async4(float *dst, const float *src, bool valid)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(d), "l"(src), "r"(valid ? 4 : 0));
}

// Tile geometry: the tile covers rows ty0 - rc .. ty0 + kAH + rc and columns starting at
// tx0 - RCA (RCA = rc rounded up to a multiple of 4, so rows start 16-byte aligned).
struct ApplyGeom {
    int RCA, TWa, THh, TS;
    __host__ __device__ constexpr ApplyGeom(int rc)
        : RCA((rc + 3) & ~3), TWa(kAW + 2 * ((rc + 3) & ~3)), THh(kAH + 2 * rc),
          TS(kAW + 2 * ((rc + 3) & ~3) + 4)  // 4 (mod 8) floats: conflict-free 16-byte accesses down the rows (the TMA box width)
    {
    }
    __host__ __device__ constexpr int tile_floats() const { return (THh * TS + 31) / 32 * 32; }  // 128-byte multiple
    __host__ __device__ constexpr size_t floats() const { return 32 + (size_t)2 * tile_floats() + 8; }  // slack, tiles, mbarriers
};

constexpr unsigned long long kApplyTimeoutNs = 1000000000ull;  // 1 s per wait

// Kernel parameters: the TMA map of the coefficient planes (valid when use_tma) and the
// apply arguments.
struct alignas(128) ApplyKArgs {
    CUtensorMap tm;
    ApplyArgs a;
    int q, use_tma;
};

// Copy the tile + halo of one coefficient plane into shared memory (zero outside the
// image), asynchronously: each warp copies whole rows, lanes along the row.
__device__ __forceinline__ void load_tile(float *T, const ApplyGeom &g, const float *src, int H, int W, int pitch,
                                          int ty0, int tx0, int rc, int warp, int lane)
{
    const int xs0 = tx0 - g.RCA;
    for (int row = warp; row < g.THh; row += kAThreads / 32) {
        const int sy = ty0 - rc + row;
        const bool row_ok = sy >= 0 && sy < H;
        const float *srow = src + (size_t)(row_ok ? sy : 0) * pitch;
        float *trow = T + row * g.TS;
        for (int col = lane; col < g.TWa; col += 32) {
            const int sx = xs0 + col;
            const bool ok = row_ok && sx >= 0 && sx < W;
            cp_async4(trow + col, ok ? srow + sx : src, ok);
        }
    }
    asm volatile("cp.async.commit_group;\n" ::);
}

// RC: the radius (every radius is compiled: the horizontal and vertical runs live in registers).
template <int RC>
__global__ void __launch_bounds__(kAThreads, 2) flr_apply_kernel(const __grid_constant__ ApplyKArgs ka)
{
    extern __shared__ __align__(16) float sm[];
    const ApplyArgs &a = ka.a;
    const bool use_tma = ka.use_tma != 0;
    const int H = a.H, W = a.W, Q = ka.q;
    constexpr ApplyGeom g(RC);
    float *base = sm + (((128 - (tma::smem_addr(sm) & 127)) & 127) >> 2);  // 128-byte aligned
    uint64_t *bar = reinterpret_cast<uint64_t *>(base + 2 * g.tile_floats());  // [2] TMA arrivals
    __shared__ int s_abort;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int row_hi = a.row_hi < 0 ? H : min(a.row_hi, H);
    const int tx0 = blockIdx.x * kAW, ty0 = a.row_lo + blockIdx.y * kAH;
    const size_t plane = (size_t)H * W;
    const int NP = 3 * (Q + 1);

    // step n takes plane 3 i + c, colour c = n / (Q + 1) outermost: one colour's accumulators at a time
    auto stage = [&](int n) {
        const int p = 3 * (n % (Q + 1)) + n / (Q + 1);
        float *T = base + (n & 1) * g.tile_floats();
        if (use_tma) {
            if (tid == 0) {
                uint64_t *b = bar + (n & 1);
                tma::mbar_expect_tx(b, (unsigned)(g.THh * g.TS * 4));
                tma::load_3d(T, &ka.tm, tx0 - g.RCA, ty0 - RC, p, b);
            }
        } else {
            load_tile(T, g, a.coef + (size_t)p * H * a.coef_pitch, H, W, a.coef_pitch, ty0, tx0, RC, warp, lane);
        }
    };
    if (tid == 0) {
        s_abort = 0;
        if (use_tma) {
            tma::mbar_init(bar, 1);
            tma::mbar_init(bar + 1, 1);
            tma::mbar_init_fence();
        }
    }
    __syncthreads();
    pdl::wait();
    stage(0);
    // vertical sums and accumulation: warps 0 to 7 take a run of 8 rows each, a lane two columns
    const int gx = tx0 + 2 * lane, gy = ty0 + kARun * warp;
    const int vrows = warp < kAH / kARun && gx < W ? min(kARun, row_hi - gy) : 0;
    const bool two = gx + 1 < W;
    float2 acc[kARun];
    int bad = 0, n = 0;
#pragma unroll 1
    for (int c = 0; c < 3; ++c) {
#pragma unroll
        for (int t = 0; t < kARun; ++t) acc[t] = make_float2(0.f, 0.f);
#pragma unroll 1
        for (int i = 0; i <= Q; ++i, ++n) {
            float *T = base + (n & 1) * g.tile_floats();
            if (n + 1 < NP) stage(n + 1);
            // the map guide's values of this plane's rows, on their way during the horizontal sums
            float2 z[kARun];
            const float *zp = a.map_guide + (size_t)(i > 0 ? i - 1 : 0) * plane + (size_t)gy * W + gx;
#pragma unroll
            for (int t = 0; t < kARun; ++t, zp += W) {
                z[t] = make_float2(1.f, 1.f);
                if (i > 0 && t < vrows) {
                    z[t].x = __ldg(zp);
                    if (two) z[t].y = __ldg(zp + 1);
                }
            }
            const float sz = i > 0 ? __ldg(a.shift + i - 1) : 0.f;
            if (use_tma) {
                if (!tma::wait_warp(bar + (n & 1), (uint32_t)((n >> 1) & 1), kApplyTimeoutNs) && lane == 0) {
                    s_abort = 1;
                    if (a.status) atomicExch(a.status, 1);
                }
            } else {
                if (n + 1 < NP) asm volatile("cp.async.wait_group 1;\n" ::: "memory");
                else asm volatile("cp.async.wait_group 0;\n" ::: "memory");
                __syncthreads();  // every thread's copies of this plane have landed
            }
            // horizontal sums in place: 16 outputs per lane, eight rows per warp (lanes 0-7 take
            // consecutive rows: 16-byte accesses at row stride 4 mod 8 floats, distinct banks)
#pragma unroll 1
            for (int row = warp * 8 + (lane & 7); row - (lane & 7) < g.THh; row += kAThreads / 4) {
                const bool in = row < g.THh;
                float *q = T + row * g.TS + (lane >> 3) * 16;
                float o[16];
                if (in) {
                    constexpr int XO = g.RCA - RC, N = 16 + 2 * g.RCA;
                    float v[N];
#pragma unroll
                    for (int k = 0; k < N; k += 4) {
                        const float4 f = *reinterpret_cast<const float4 *>(q + k);
                        v[k] = f.x;
                        v[k + 1] = f.y;
                        v[k + 2] = f.z;
                        v[k + 3] = f.w;
                    }
                    float s4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                    for (int k = 0; k <= 2 * RC; ++k) s4[k & 3] += v[XO + k];
                    float s = (s4[0] + s4[1]) + (s4[2] + s4[3]);
                    o[0] = s;
#pragma unroll
                    for (int t = 1; t < 16; ++t) {
                        s += v[XO + t + 2 * RC] - v[XO + t - 1];
                        o[t] = s;
                    }
                }
                __syncwarp();  // the rows' operands are read
                if (in) {
#pragma unroll
                    for (int t = 0; t < 16; t += 4) *reinterpret_cast<float4 *>(q + t) = make_float4(o[t], o[t + 1], o[t + 2], o[t + 3]);
                }
            }
            __syncthreads();  // horizontal sums complete
            if (s_abort) {  // let a copy still in flight land before the CTA exits, then stop
                if (use_tma && n + 1 < NP && warp == 0)
                    tma::wait_warp(bar + ((n + 1) & 1), (uint32_t)(((n + 1) >> 1) & 1), kApplyTimeoutNs);
                return;
            }
            if (vrows > 0) {
                const float2 *q = reinterpret_cast<const float2 *>(T + (warp * kARun) * g.TS) + lane;
                constexpr int st = g.TS / 2;
                const float2 minus = make_float2(-1.f, -1.f), nsz = make_float2(-sz, -sz);
                float2 first[kARun - 1], s2[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
                for (int k = 0; k <= 2 * RC; ++k) {
                    const float2 f = q[k * st];
                    if (k < kARun - 1) first[k < kARun - 1 ? k : 0] = f;
                    s2[k & 1] = __fadd2_rn(s2[k & 1], f);
                }
                float2 s = __fadd2_rn(s2[0], s2[1]);
#pragma unroll
                for (int t = 0; t < kARun; ++t) {
                    if (t > 0) {
                        const float2 old = t - 1 <= 2 * RC ? first[t - 1] : q[(t - 1) * st];
                        s = __fadd2_rn(s, __ffma2_rn(old, minus, q[(t + 2 * RC) * st]));
                    }
                    acc[t] = __ffma2_rn(s, __fadd2_rn(z[t], nsz), acc[t]);
                }
            }
            if (use_tma) asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
            __syncthreads();  // this buffer may be refilled from here on
        }
        if (vrows > 0) {
            const float sc = __ldg(a.shift + Q + c);
            const float n0 = (float)(min(gx + RC, W - 1) - max(gx - RC, 0) + 1);
            const float n1 = (float)(min(gx + 1 + RC, W - 1) - max(gx + 1 - RC, 0) + 1);
            float *out = a.out + c * plane + (size_t)gy * W + gx;
#pragma unroll
            for (int t = 0; t < kARun; ++t, out += W) {
                if (t < vrows) {
                    const float ny = (float)(min(gy + t + RC, H - 1) - max(gy + t - RC, 0) + 1);
                    const float o0 = fmaf(acc[t].x, 1.0f / (n0 * ny), sc);
                    out[0] = o0;
                    bad += !isfinite(o0);
                    if (two) {
                        const float o1 = fmaf(acc[t].y, 1.0f / (n1 * ny), sc);
                        out[1] = o1;
                        bad += !isfinite(o1);
                    }
                }
            }
        }
    }
    if (bad && a.nonfinite) atomicAdd(a.nonfinite, (unsigned long long)bad);
}

// ---- eight guides: the three colours of a guide together ----------------------------------------
// 64 x 32 output tiles, one column and eight rows per thread, a buffer of their own for the horizontal
// sums, every colour's accumulators live (24 registers): the map guide is read once instead of once per
// colour.  64 registers a thread and at most 56 KB leave four CTAs of eight warps per SM, where the
// form above has two of ten; bound, like it, by the latency of a plane's phases, which the others hide.
// q = 8, rc = 8: 94 us at 1080p and 29 us at 480 x 640 (above: 119 and 43).
constexpr int kPW = 64, kPH = 32, kPThreads = 256, kPRun = 8;

template <int RC>
struct PlanarGeom {
    static constexpr int RCA = (RC + 3) & ~3, THh = kPH + 2 * RC, TS = kPW + 2 * RCA + 4;
    static constexpr int HS = kPW + 1;  // odd: the column walks of the vertical pass are conflict-free
    static constexpr int TILE = (THh * TS + 31) / 32 * 32;
    static constexpr size_t SMEM = sizeof(float) * (32 + 2 * TILE + ((THh * HS + 1) & ~1) + 8);  // slack, tiles, sums, mbarriers
};

template <int Q, int RC>
__global__ void __launch_bounds__(kPThreads, 4) flr_apply_planar_kernel(const __grid_constant__ ApplyKArgs ka)
{
    using G = PlanarGeom<RC>;
    constexpr int NP = 3 * (Q + 1);
    extern __shared__ __align__(16) float sm[];
    const ApplyArgs &a = ka.a;
    const int H = a.H, W = a.W;
    float *base = sm + (((128 - (tma::smem_addr(sm) & 127)) & 127) >> 2);  // 128-byte aligned
    float *Hb = base + 2 * G::TILE;                                        // [THh][HS] horizontal sums
    uint64_t *bar = reinterpret_cast<uint64_t *>(Hb + ((G::THh * G::HS + 1) & ~1));
    __shared__ int s_abort;
    __shared__ float s_shift[Q + 3];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int row_hi = a.row_hi < 0 ? H : min(a.row_hi, H);
    const int tx0 = blockIdx.x * kPW, ty0 = a.row_lo + blockIdx.y * kPH;
    const int x = tid % kPW, run = tid / kPW, gx = tx0 + x, gy0 = ty0 + run * kPRun;
    const size_t plane = (size_t)H * W;
    const int vrows = gx < W ? min(kPRun, row_hi - gy0) : 0;
    auto stage = [&](int p) {
        uint64_t *b = bar + (p & 1);
        tma::mbar_expect_tx(b, (unsigned)(G::THh * G::TS * 4));
        tma::load_3d(base + (p & 1) * G::TILE, &ka.tm, tx0 - G::RCA, ty0 - RC, p, b);
    };
    if (tid == 0) {
        s_abort = 0;
        tma::mbar_init(bar, 1);
        tma::mbar_init(bar + 1, 1);
        tma::mbar_init_fence();
    }
    pdl::wait();
    if (tid == 0) stage(0);
    if (tid < Q + 3) s_shift[tid] = a.shift[tid];
    __syncthreads();
    // the map-guide values of guide i + 1 are on their way into L1 while guide i is summed
    const float *zp = a.map_guide + (size_t)gy0 * W + gx;
    auto prefetch_z = [&](int i) {
        if (i < 1 || i > Q) return;
#pragma unroll
        for (int t = 0; t < kPRun; ++t)
            if (t < vrows) asm volatile("prefetch.global.L1 [%0];\n" ::"l"(zp + (size_t)(i - 1) * plane + (size_t)t * W));
    };
    prefetch_z(1);
    float acc[3][kPRun];
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int t = 0; t < kPRun; ++t) acc[c][t] = 0.f;
#pragma unroll 1
    for (int i = 0; i <= Q; ++i) {
        float z[kPRun];
#pragma unroll
        for (int t = 0; t < kPRun; ++t)
            z[t] = i == 0 ? 1.f : t < vrows ? __ldg(zp + (size_t)(i - 1) * plane + (size_t)t * W) - s_shift[i - 1] : 0.f;
        prefetch_z(i + 1);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const int p = 3 * i + c;
            const float *T = base + (p & 1) * G::TILE;
            if (tid == 0 && p + 1 < NP) stage(p + 1);
            if (!tma::wait_warp(bar + (p & 1), (uint32_t)((p >> 1) & 1), kApplyTimeoutNs) && lane == 0) {
                s_abort = 1;
                if (a.status) atomicExch(a.status, 1);
            }
            __syncthreads();  // the sums of the plane before are read
            if (s_abort) {    // let a copy still in flight land before the CTA exits, then stop
                if (p + 1 < NP && warp == 0)
                    tma::wait_warp(bar + ((p + 1) & 1), (uint32_t)(((p + 1) >> 1) & 1), kApplyTimeoutNs);
                return;
            }
            // horizontal sums: 16 outputs per item, consecutive lanes on consecutive rows (16-byte loads
            // at row stride 4 mod 8 floats: distinct banks)
            for (int item = tid; item < G::THh * 4; item += kPThreads) {
                const int xr = (item / G::THh) * 16, row = item % G::THh;
                const float *q = T + row * G::TS + xr;
                float *h = Hb + row * G::HS + xr;
                constexpr int XO = G::RCA - RC, N = 16 + 2 * G::RCA;
                float v[N];
#pragma unroll
                for (int k = 0; k < N; k += 4) {
                    const float4 f = *reinterpret_cast<const float4 *>(q + k);
                    v[k] = f.x;
                    v[k + 1] = f.y;
                    v[k + 2] = f.z;
                    v[k + 3] = f.w;
                }
                float s4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int k = 0; k <= 2 * RC; ++k) s4[k & 3] += v[XO + k];
                float s = (s4[0] + s4[1]) + (s4[2] + s4[3]);
                h[0] = s;
#pragma unroll
                for (int t = 1; t < 16; ++t) {
                    s += v[XO + t + 2 * RC] - v[XO + t - 1];
                    h[t] = s;
                }
            }
            __syncthreads();  // horizontal sums complete; the tile may be refilled from here on
            if (tid == 0) asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
            const float *q = Hb + (run * kPRun) * G::HS + x;
            float v[kPRun + 2 * RC];
#pragma unroll
            for (int k = 0; k < kPRun + 2 * RC; ++k) v[k] = q[k * G::HS];
            float s2[2] = {0.f, 0.f};
#pragma unroll
            for (int k = 0; k <= 2 * RC; ++k) s2[k & 1] += v[k];
            float s = s2[0] + s2[1];
            acc[c][0] = fmaf(s, z[0], acc[c][0]);
#pragma unroll
            for (int t = 1; t < kPRun; ++t) {
                s += v[t + 2 * RC] - v[t - 1];
                acc[c][t] = fmaf(s, z[t], acc[c][t]);
            }
        }
    }
    if (vrows > 0) {
        const float nx = (float)(min(gx + RC, W - 1) - max(gx - RC, 0) + 1);
        int bad = 0;
        float *out = a.out + (size_t)gy0 * W + gx;
#pragma unroll
        for (int t = 0; t < kPRun; ++t, out += W) {
            if (t >= vrows) break;
            const float ny = (float)(min(gy0 + t + RC, H - 1) - max(gy0 + t - RC, 0) + 1);
            const float inv_m = 1.0f / (nx * ny);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const float o = fmaf(acc[c][t], inv_m, s_shift[Q + c]);
                out[c * plane] = o;
                bad += !isfinite(o);
            }
        }
        if (bad && a.nonfinite) atomicAdd(a.nonfinite, (unsigned long long)bad);
    }
}

// Eight guides and padded coefficient planes take the form of the three colours together while four of
// its CTAs fit an SM's shared memory, rc <= 12: 109 against 135 us at rc = 12, 84 against 95 at rc = 1
// (1080p), ahead at every radius between and at every size down to 256 x 256.  With three (rc = 13) it
// gains 5% at 1080p but loses 12% at 719 x 1277, a last wave that is nearly empty.
template <int RC>
constexpr bool kPlanar = 4 * (PlanarGeom<RC>::SMEM + 1024) <= 228 * 1024;
static_assert(kPlanar<12> && !kPlanar<13>, "four CTAs per SM up to a radius of 12");

template <int RC>
cudaError_t launch_apply_rc(int q, const ApplyArgs &a, cudaStream_t st)
{
    constexpr ApplyGeom g(RC);
    constexpr size_t smem = sizeof(float) * g.floats();
    // two CTAs per SM need most of the unified L1 / shared array
    cudaError_t e = pdl::allow_smem<std::integral_constant<int, RC>>(flr_apply_kernel<RC>, smem, true);
    if (e != cudaSuccess) return e;
    const int rows = (a.row_hi < 0 ? a.H : a.row_hi) - a.row_lo;
    if (rows <= 0) return cudaSuccess;
    dim3 grid((a.W + kAW - 1) / kAW, (rows + kAH - 1) / kAH);
    ApplyKArgs ka;
    std::memset(&ka, 0, sizeof(ka));
    ka.a = a;
    ka.q = q;
    if constexpr (kPlanar<RC>) {
        using P = PlanarGeom<RC>;
        if (q == 8 && (a.coef_pitch & 3) == 0 && ((uintptr_t)a.coef & 15) == 0 &&
            tma::encode_planes_f32(&ka.tm, a.coef, a.W, a.H, 3 * (q + 1), P::TS, P::THh, 1, a.coef_pitch) == cudaSuccess) {
            e = pdl::allow_smem<PlanarGeom<RC>>(flr_apply_planar_kernel<8, RC>, P::SMEM, true);
            if (e != cudaSuccess) return e;
            return pdl::launch(flr_apply_planar_kernel<8, RC>, dim3((a.W + kPW - 1) / kPW, (rows + kPH - 1) / kPH), kPThreads,
                               P::SMEM, st, ka);
        }
    }
    ka.use_tma = ((a.coef_pitch & 3) == 0 && ((uintptr_t)a.coef & 15) == 0 &&
                  tma::encode_planes_f32(&ka.tm, a.coef, a.W, a.H, 3 * (q + 1), g.TS, g.THh, 1, a.coef_pitch) == cudaSuccess)
                     ? 1
                     : 0;
    return pdl::launch(flr_apply_kernel<RC>, grid, kAThreads, smem, st, ka);
}

}  // namespace

cudaError_t launch_apply(int q, const ApplyArgs &a, cudaStream_t st)
{
    static_assert(FLR_MAX_COEF_RADIUS == 16, "every radius is compiled");
    switch (a.rc) {
    case 1: return launch_apply_rc<1>(q, a, st);
    case 2: return launch_apply_rc<2>(q, a, st);
    case 3: return launch_apply_rc<3>(q, a, st);
    case 4: return launch_apply_rc<4>(q, a, st);
    case 5: return launch_apply_rc<5>(q, a, st);
    case 6: return launch_apply_rc<6>(q, a, st);
    case 7: return launch_apply_rc<7>(q, a, st);
    case 8: return launch_apply_rc<8>(q, a, st);
    case 9: return launch_apply_rc<9>(q, a, st);
    case 10: return launch_apply_rc<10>(q, a, st);
    case 11: return launch_apply_rc<11>(q, a, st);
    case 12: return launch_apply_rc<12>(q, a, st);
    case 13: return launch_apply_rc<13>(q, a, st);
    case 14: return launch_apply_rc<14>(q, a, st);
    case 15: return launch_apply_rc<15>(q, a, st);
    case 16: return launch_apply_rc<16>(q, a, st);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace flr
