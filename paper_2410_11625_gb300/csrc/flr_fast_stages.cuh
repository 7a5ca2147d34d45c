// flr_fast_stages.cuh -- the four stages of the paper's fast FLR (Sec. 3.2, 3.2.1) as device
// functions (flr_fast.cu has the kernels).
#pragma once

#include <utility>

#include "flr_device.cuh"
#include "flr_internal.cuh"

namespace flr {
namespace fast {

constexpr int kMaxTaps = 8;

// acc += the product that defines moment channel CH (slots fixed at compile time)
template <int Q, int CH>
__device__ __forceinline__ void moment_one(float &acc, const float (&v)[Q + 3])
{
    constexpr int u = Chan<Q>::slot_u(CH), w = Chan<Q>::slot_v(CH);
    if constexpr (w < 0) acc += v[u];
    else acc = fmaf(v[u], v[w], acc);
}

template <int Q, int... I>
__device__ __forceinline__ void moments_all(float (&acc)[Chan<Q>::NCH], const float (&v)[Q + 3],
                                            std::integer_sequence<int, I...>)
{
    (moment_one<Q, I>(acc[I], v), ...);
}

// L2 eviction priorities for the full-resolution planes.  The moment stage reads the guide
// planes with evict_last so that they are still in L2 when the apply stage reads them again
// as the map guide (66 MB at 1080p, half of L2); the radiance, read once, and the apply's own
// reads take evict_first, so they do not push the guides out.
__device__ __forceinline__ uint64_t l2_policy_keep()
{
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;\n" : "=l"(p));
    return p;
}
__device__ __forceinline__ uint64_t l2_policy_stream()
{
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;\n" : "=l"(p));
    return p;
}
// Asynchronous 8- and 4-byte copies into shared memory, with an L2 eviction policy
__device__ __forceinline__ void copy8_hint(uint32_t dst, const float *src, uint64_t pol)
{
    asm volatile("cp.async.ca.shared.global.L2::cache_hint [%0], [%1], 8, %2;\n" ::"r"(dst), "l"(src), "l"(pol) : "memory");
}
__device__ __forceinline__ void copy4_hint(uint32_t dst, const float *src, uint64_t pol)
{
    asm volatile("cp.async.ca.shared.global.L2::cache_hint [%0], [%1], 4, %2;\n" ::"r"(dst), "l"(src), "l"(pol) : "memory");
}

// A block's model in memory: 16-byte aligned [biases of the 3 colours, 0][colour][QE], QE guide
// coefficients rounded up to an even count (the last one 0 for odd Q), so that the apply reads a
// corner with vector loads and works on pairs of guides.
template <int Q>
struct Model {
    static constexpr int QE = (Q + 1) / 2 * 2, CS = (4 + 3 * QE + 3) / 4 * 4;
    __host__ __device__ static constexpr int at(int c, int i) { return 4 + c * QE + i; }
};
__host__ __device__ constexpr int model_floats(int q) { return (4 + 3 * ((q + 1) / 2 * 2) + 3) / 4 * 4; }

struct FastArgs {
    const float *guide, *rad, *map_guide;  // model inputs [q|3][Hi][Wi], map guide [q][Ho][Wo]
    float *out;                            // [3][Ho][Wo]
    float *blk;   // [NCH + Q+3][Hb][Wb]: block sums relative to the block's reference, then that reference
    float *tmp;   // [NCH + 1][Hb][Wb]: horizontally blurred sums (same reference), weighted count
    float *coef;  // [Hb][Wb] block models (struct Model) relative to the frame reference
    float *tmp2;  // parameter gradients: [NCH + 1][Hb][Wb] horizontal blur with the weights' sigma-derivative
    float *dcoef; // parameter gradients: [3][Hb][Wb] model tangents (sigma, eps, eps_mul)
    float *shift;                          // frame reference shift, Q + 3 floats
    unsigned long long *flag_count;
    int Hi, Wi, Ho, Wo, Hb, Wb, F, s, taps;
    float eps, tau;
    int appendix;   // 1: the Appendix's regularised normalised solve (additive eps, multiplicative eps_mul)
    float eps_mul;
    float w[2 * kMaxTaps + 1];             // Gaussian weights
    float wd[2 * kMaxTaps + 1];            // their derivatives with respect to sigma (parameter gradients)
    int *status = nullptr;                 // set to 1 if a bounded device wait ran out (may be NULL)
};

// Sums over the LPB lanes of a block, O = 1, 2, .. LPB / 2 apart, by halving: in each step a lane
// sends the half of its channels that its partner keeps, so NCH channels take about NCH shuffles
// instead of NCH log2(LPB), and every lane stores its own share of the channels.  The sums are
// those of a butterfly, bit for bit.  cnt of a's N channels, from ch0 on, exist.
template <int N, int O, int LPB>
__device__ __forceinline__ void fold_store(const float (&a)[N], int lane, int ch0, int cnt, float *dst, size_t bplane)
{
    if constexpr (O == LPB) {
        float *p = dst + ch0 * bplane;
#pragma unroll
        for (int i = 0; i < N; ++i) {
            if (i < cnt) *p = a[i];
            p += bplane;
        }
    } else {
        constexpr int H = (N + 1) / 2;
        const bool up = (lane & O) != 0;
        float b[H];
#pragma unroll
        for (int i = 0; i < H; ++i) {
            const float hi = i + H < N ? a[i + H < N ? i + H : 0] : 0.f;
            b[i] = (up ? hi : a[i]) + __shfl_xor_sync(0xffffffffu, up ? a[i] : hi, O);
        }
        fold_store<H, 2 * O, LPB>(b, lane, up ? ch0 + H : ch0, up ? cnt - H : (cnt < H ? cnt : H), dst, bplane);
    }
}

// 1. block moments.  Block (i, j) covers input rows [iF, iF+F) and columns [jF, jF+F).
// Work item (by, cx): block row by, input columns [256 cx, 256 cx + 256); 128 threads, each
// summing two adjacent columns over the F rows, then fold_store over the F / 2 lanes of a block.
// The rows come through a ring of kMomStages asynchronous copies that each thread keeps for
// itself, without any barrier: a warp's 71 accumulators leave room for 16 warps per SM, too few to
// cover DRAM latency with loads into registers, where a row waits out its load (long_scoreboard
// 4.6 of 8.7 stall cycles per issue; 26.5 us at 1920x1080 against 21 us so).  One row's products are
// the loop body: the rows unrolled are 20 KB of instructions that every warp fetches once.
// Measured besides: the two columns' products as packed pairs (142 accumulators, 8 warps per SM)
// 22 us; persistent CTAs whose ring runs on from item to item 33 us; 4 stages 21 us (but 74 against
// 72 us for the whole 1280x720 -> 2560x1440 frame); 256 threads 22 us.
constexpr int kMomThreads = 128, kMomStages = 2;
template <int Q>
constexpr size_t moments_smem()
{
    return sizeof(float) * kMomStages * (Q + 3) * 2 * kMomThreads;
}

template <int Q, int F>
__device__ __forceinline__ void stage_moments(const FastArgs &a, int by, int cx, float *ring)
{
    using C = Chan<Q>;
    constexpr int NS = Q + 3, LPB = F / 2;  // lanes per block
    constexpr int D = F < kMomStages ? F : kMomStages;
    static_assert(F >= 2 && 32 % F == 0, "block width");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int x = cx * 2 * kMomThreads + 2 * tid;  // this thread's columns x, x + 1
    const size_t plane = (size_t)a.Hi * a.Wi;
    const int y0 = by * F, rows = min(F, a.Hi - y0);
    // with an even width, x + 1 < Wi and the 8-byte copies are aligned (x even, planes 16-byte
    // aligned)
    const bool in = x < a.Wi, vec = (a.Wi & 1) == 0, two = x + 1 < a.Wi;
    const uint64_t pol_keep = l2_policy_keep(), pol_stream = l2_policy_stream();
    float2 *mine = reinterpret_cast<float2 *>(ring) + tid;  // [stage][slot][thread]
    auto issue = [&](int row) {
        if (row < rows && in) {
            uint32_t dst = (uint32_t)__cvta_generic_to_shared(mine + (row % D) * NS * kMomThreads);
            const float *pg = a.guide + (size_t)(y0 + row) * a.Wi + x, *pr = a.rad + (size_t)(y0 + row) * a.Wi + x;
            if (vec) {
#pragma unroll
                for (int k = 0; k < Q; ++k, dst += 8 * kMomThreads, pg += plane) copy8_hint(dst, pg, pol_keep);
#pragma unroll
                for (int c = 0; c < 3; ++c, dst += 8 * kMomThreads, pr += plane) copy8_hint(dst, pr, pol_stream);
            } else {
#pragma unroll
                for (int k = 0; k < Q; ++k, dst += 8 * kMomThreads, pg += plane) {
                    copy4_hint(dst, pg, pol_keep);
                    if (two) copy4_hint(dst + 4, pg + 1, pol_keep);
                }
#pragma unroll
                for (int c = 0; c < 3; ++c, dst += 8 * kMomThreads, pr += plane) {
                    copy4_hint(dst, pr, pol_stream);
                    if (two) copy4_hint(dst + 4, pr + 1, pol_stream);
                }
            }
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
#pragma unroll
    for (int row = 0; row < D; ++row) issue(row);
    if (by == 0 && cx == 0 && warp == 0) {
        // the frame reference the models are expressed in (used by the solve and apply)
        __shared__ float s_ref[NS];
        dev::sample_mean<Q>(s_ref, a.guide, a.rad, a.Hi, a.Wi, 0, a.Hi, 0, a.Wi, lane);
        __syncwarp();
        if (lane < NS) a.shift[lane] = s_ref[lane];
    }
    // the block's reference: its top-left input pixel (column x of lane (lane & ~(LPB-1)))
    asm volatile("cp.async.wait_group %0;\n" ::"n"(D - 1) : "memory");
    float ref[NS], acc[C::NCH];
#pragma unroll
    for (int k = 0; k < NS; ++k) ref[k] = __shfl_sync(0xffffffffu, mine[k * kMomThreads].x, lane & ~(LPB - 1));
#pragma unroll
    for (int c = 0; c < C::NCH; ++c) acc[c] = 0.f;
#pragma unroll 1
    for (int row = 0; row < rows; ++row) {
        asm volatile("cp.async.wait_group %0;\n" ::"n"(D - 1) : "memory");
        const float2 *src = mine + (row % D) * NS * kMomThreads;
        float v0[NS], v1[NS];
#pragma unroll
        for (int k = 0; k < NS; ++k) {
            const float2 g = src[k * kMomThreads];
            v0[k] = g.x - ref[k];
            v1[k] = two ? g.y - ref[k] : 0.f;
        }
        issue(row + D);
        moments_all<Q>(acc, v0, std::make_integer_sequence<int, C::NCH>{});
        moments_all<Q>(acc, v1, std::make_integer_sequence<int, C::NCH>{});
    }
    if (!in) {  // columns past the image: lanes of a block that starts inside it add nothing
#pragma unroll
        for (int c = 0; c < C::NCH; ++c) acc[c] = 0.f;
    }
    // blocks never straddle a warp (32 % LPB == 0); a block's first column is that of its first lane
    const int sub = lane & (LPB - 1), bx = (x - 2 * sub) / F;
    const bool block_in = x - 2 * sub < a.Wi;
    const size_t bplane = (size_t)a.Hb * a.Wb;
    float *dst = a.blk + (size_t)by * a.Wb + bx;
    fold_store<C::NCH, 1, LPB>(acc, lane, 0, block_in ? C::NCH : 0, dst, bplane);
    if (block_in) {
#pragma unroll
        for (int k = 0; k < NS; ++k)
            if ((k & (LPB - 1)) == sub) dst[(C::NCH + k) * bplane] = ref[k];
    }
}

// Input pixels of block index b along an axis of n pixels split into blocks of F.
__device__ __forceinline__ float block_len(int b, int F, int n) { return (float)min(F, n - b * F); }

// acc += w * (sums of block b re-expressed relative to another reference), given
// d = ref_b - ref_target for the Q + 3 input slots and the block's pixel count nb:
//   G = sum (v + d) = L + nb d,   sum (v + d)(v' + d') = S + L' d + G d'.
// p: channel 0 of the block; the other channels follow stride apart, read in order.
template <int Q>
__device__ __forceinline__ void accumulate_shifted(float (&acc)[Chan<Q>::NCH], const float *p, size_t stride,
                                                   const float (&d)[Q + 3], float nb, float w)
{
    using C = Chan<Q>;
    static_assert(C::X0 == 0 && C::XX0 == Q + 3 && C::XY0 == C::XX0 + C::NXX, "channels in order");
    float L[Q + 3], G[Q + 3];
#pragma unroll
    for (int k = 0; k < Q + 3; ++k, p += stride) L[k] = *p;  // X0..Y0+2 are the linear sums
#pragma unroll
    for (int k = 0; k < Q + 3; ++k) {
        G[k] = fmaf(nb, d[k], L[k]);
        acc[C::X0 + k] = fmaf(w, G[k], acc[C::X0 + k]);
    }
#pragma unroll
    for (int i = 0; i < Q; ++i)
#pragma unroll
        for (int j = i; j < Q; ++j, p += stride) {
            const int ch = C::xx(i, j);
            acc[ch] = fmaf(w, fmaf(G[i], d[j], fmaf(d[i], L[j], *p)), acc[ch]);
        }
#pragma unroll
    for (int i = 0; i < Q; ++i)
#pragma unroll
        for (int c = 0; c < 3; ++c, p += stride) {
            const int ch = C::xy(i, c);
            acc[ch] = fmaf(w, fmaf(G[i], d[Q + c], fmaf(d[i], L[Q + c], *p)), acc[ch]);
        }
}

// 2. horizontal Gaussian over the block grid, clipped: every neighbour's sums re-expressed
// relative to the target block's reference before weighting; also the weighted count.
template <int Q>
__device__ __forceinline__ void stage_blur_h(const FastArgs &a, size_t k)
{
    using C = Chan<Q>;
    constexpr int NS = Q + 3;
    const size_t bplane = (size_t)a.Hb * a.Wb;
    if (k >= bplane) return;
    const int by = (int)(k / a.Wb), bx = (int)(k % a.Wb);
    float rk[NS];
#pragma unroll
    for (int q = 0; q < NS; ++q) rk[q] = a.blk[(C::NCH + q) * bplane + k];
    float acc[C::NCH];
#pragma unroll
    for (int c = 0; c < C::NCH; ++c) acc[c] = 0.f;
    float n = 0.f;
    const float rows = block_len(by, a.F, a.Hi);
    for (int dd = -a.taps; dd <= a.taps; ++dd) {
        const int xx = bx + dd;
        if (xx < 0 || xx >= a.Wb) continue;
        const size_t kb = (size_t)by * a.Wb + xx;
        float d[NS];
#pragma unroll
        for (int q = 0; q < NS; ++q) d[q] = a.blk[(C::NCH + q) * bplane + kb] - rk[q];
        const float nb = rows * block_len(xx, a.F, a.Wi);
        const float w = a.w[dd + a.taps];
        accumulate_shifted<Q>(acc, a.blk + kb, bplane, d, nb, w);
        n = fmaf(w, nb, n);
    }
#pragma unroll
    for (int c = 0; c < C::NCH; ++c) a.tmp[c * bplane + k] = acc[c];
    a.tmp[C::NCH * bplane + k] = n;
}

// The Appendix's regularised normalised solve of one block (additive term eps, multiplicative
// term eps_mul), in an equivalent un-normalised form.  With D_s = diag(sigma^),
// C^ + eps I = D_s^-1 (W^ + eps D_s^2) D_s^-1 and B^ = D_s^-1 D, so the model
// ((x - mu) / sigma^) A^ has guide coefficients a = A^ / sigma^ = (W^ + eps diag(W^))^-1 D:
// one Cholesky solve of W^ with its diagonal scaled by (1 + eps), no divisions by sigma^.
// W^ = W + eps_mul (mu mu^T + diag(mu^2)) + eps I takes the block's absolute guide means,
// ref + (mean of the sums taken relative to ref); W and D are shift-invariant.  Returns the
// model in the block-shifted coordinates, as solve_pixel, with the factor of M, and whether
// a pivot fell low.
template <int Q>
__device__ __forceinline__ bool solve_appendix(const float *Sp, int VS, float n, float eps, float eps_mul,
                                               float tau, const float *ref, float (&A)[Q][3], float (&bv)[3],
                                               float (&mu)[Q], float (&muy)[3], float (&L)[Q * (Q + 1) / 2],
                                               float (&inv_d)[Q])
{
    using C = Chan<Q>;
    // a one-pixel block: the guide moments drop out (a = 0, b = mu_y), as in solve_pixel
    const float inv_n = 1.0f / n;
    const float inv_nx = n > 1.5f ? inv_n : 0.f;
    float ma[Q], D[Q][3];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        mu[i] = Sp[(C::X0 + i) * VS] * inv_nx;
        ma[i] = ref[i] + mu[i];
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) muy[c] = Sp[(C::Y0 + c) * VS] * inv_n;
    const float grow = 1.f + eps;
#pragma unroll
    for (int i = 0; i < Q; ++i)
#pragma unroll
        for (int j = 0; j < Q; ++j) {
            if (j <= i) {
                float m = fmaf(-mu[i], mu[j], Sp[C::xx(j, i) * VS] * inv_nx);
                m = fmaf(eps_mul * ma[i], ma[j], m);
                if (i == j) m = (fmaf(eps_mul * ma[i], ma[i], m) + eps) * grow;
                L[dev::tri(i, j)] = m;
            }
        }
#pragma unroll
    for (int i = 0; i < Q; ++i)
#pragma unroll
        for (int c = 0; c < 3; ++c) D[i][c] = fmaf(-mu[i], muy[c], Sp[C::xy(i, c) * VS] * inv_nx);
    const bool low = dev::chol_factor<Q>(L, eps > 0.f ? eps : 1e-30f, tau, inv_d);  // every exact pivot is >= eps
    dev::chol_solve3<Q>(L, inv_d, D, A);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        float b = muy[c];
#pragma unroll
        for (int i = 0; i < Q; ++i) b = fmaf(-A[i][c], mu[i], b);
        bv[c] = b;
    }
    return low;
}

template <int Q>
__device__ __forceinline__ void store_model(float *dst, const float (&A)[Q][3], const float (&b)[3])
{
    using M = Model<Q>;
    float m[M::CS];
#pragma unroll
    for (int k = 0; k < M::CS; ++k) m[k] = 0.f;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        m[c] = b[c];
#pragma unroll
        for (int i = 0; i < Q; ++i) m[M::at(c, i)] = A[i][c];
    }
#pragma unroll
    for (int k = 0; k < M::CS; k += 4) *reinterpret_cast<float4 *>(dst + k) = make_float4(m[k], m[k + 1], m[k + 2], m[k + 3]);
}

// 3. vertical Gaussian + per-block solve; S: this thread's column of a [NCH][stride] buffer
template <int Q>
__device__ __forceinline__ void stage_blur_v_solve(const FastArgs &a, size_t k, float *S, int stride)
{
    using C = Chan<Q>;
    const size_t bplane = (size_t)a.Hb * a.Wb;
    if (k >= bplane) return;
    const int by = (int)(k / a.Wb), bx = (int)(k % a.Wb);
    constexpr int NS = Q + 3;
    float rk[NS];
#pragma unroll
    for (int q = 0; q < NS; ++q) rk[q] = a.blk[(C::NCH + q) * bplane + k];
    float n = 0.f;
    {
        float acc[C::NCH];
#pragma unroll
        for (int c = 0; c < C::NCH; ++c) acc[c] = 0.f;
        for (int dd = -a.taps; dd <= a.taps; ++dd) {
            const int yy = by + dd;
            if (yy < 0 || yy >= a.Hb) continue;
            const size_t kb = (size_t)yy * a.Wb + bx;
            float d[NS];
#pragma unroll
            for (int q = 0; q < NS; ++q) d[q] = a.blk[(C::NCH + q) * bplane + kb] - rk[q];
            const float nb = a.tmp[C::NCH * bplane + kb];  // weighted count of that row's sums
            const float w = a.w[dd + a.taps];
            accumulate_shifted<Q>(acc, a.tmp + kb, bplane, d, nb, w);
            n = fmaf(w, nb, n);
        }
#pragma unroll
        for (int c = 0; c < C::NCH; ++c) S[c * stride] = acc[c];
    }
    float A[Q][3], bv[3], mu[Q], muy[3];
    bool low;
    {
        float L[Q * (Q + 1) / 2], inv_d[Q];
        low = a.appendix ? solve_appendix<Q>(S, stride, n, a.eps, a.eps_mul, a.tau, rk, A, bv, mu, muy, L, inv_d)
                         : dev::solve_pixel<Q>(S, stride, n, a.eps, a.tau, A, bv, mu, muy, L, inv_d);
    }
    if (low && a.tau > 0.f) {
        // FP64 re-solve of this block from the same (FP32) window sums
        atomicAdd(a.flag_count, 1ull);
        const double inv_n = 1.0 / (double)n;
        double dmu[Q], dmuy[3], M[Q][Q], D[Q][3];
#pragma unroll
        for (int i = 0; i < Q; ++i) dmu[i] = (double)S[(C::X0 + i) * stride] * inv_n;
#pragma unroll
        for (int c = 0; c < 3; ++c) dmuy[c] = (double)S[(C::Y0 + c) * stride] * inv_n;
#pragma unroll
        for (int i = 0; i < Q; ++i) {
#pragma unroll
            for (int j = 0; j < Q; ++j)
                if (j <= i) {
                    M[i][j] = (double)S[C::xx(j, i) * stride] * inv_n - dmu[i] * dmu[j] + (i == j ? (double)a.eps : 0.0);
                    if (a.appendix) {  // W^ with its diagonal scaled by (1 + eps), as solve_appendix
                        const double mi = (double)rk[i] + dmu[i], mj = (double)rk[j] + dmu[j];
                        M[i][j] += (double)a.eps_mul * mi * mj;
                        if (i == j) M[i][j] = (M[i][j] + (double)a.eps_mul * mi * mi) * (1.0 + (double)a.eps);
                    }
                }
#pragma unroll
            for (int c = 0; c < 3; ++c) D[i][c] = (double)S[C::xy(i, c) * stride] * inv_n - dmu[i] * dmuy[c];
        }
#pragma unroll
        for (int j = 0; j < Q; ++j) {
            double d = M[j][j];
#pragma unroll
            for (int kk = 0; kk < Q; ++kk)
                if (kk < j) d -= M[j][kk] * M[j][kk];
            // every exact pivot is >= eps; rounding in the FP32 sums must not push it below
            d = sqrt(fmax(d, a.eps > 0.f ? (double)a.eps : 1e-300));
            M[j][j] = d;
#pragma unroll
            for (int i = 0; i < Q; ++i)
                if (i > j) {
                    double t = M[i][j];
#pragma unroll
                    for (int kk = 0; kk < Q; ++kk)
                        if (kk < j) t -= M[i][kk] * M[j][kk];
                    M[i][j] = t / d;
                }
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            double z[Q], x[Q];
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                double t = D[i][c];
#pragma unroll
                for (int kk = 0; kk < Q; ++kk)
                    if (kk < i) t -= M[i][kk] * z[kk];
                z[i] = t / M[i][i];
            }
#pragma unroll
            for (int ii = 0; ii < Q; ++ii) {
                const int i = Q - 1 - ii;
                double t = z[i];
#pragma unroll
                for (int kk = 0; kk < Q; ++kk)
                    if (kk > i) t -= M[kk][i] * x[kk];
                x[i] = t / M[i][i];
            }
            double b = dmuy[c];
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                A[i][c] = (float)x[i];
                b -= x[i] * dmu[i];
            }
            bv[c] = (float)b;
        }
    }
    // the model was fitted relative to this block's reference; re-express the bias
    // relative to the frame reference the apply step uses
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int i = 0; i < Q; ++i) bv[c] = fmaf(-A[i][c], rk[i] - a.shift[i], i == 0 ? bv[c] + (rk[Q + c] - a.shift[Q + c]) : bv[c]);
    store_model<Q>(a.coef + k * Model<Q>::CS, A, bv);
}

// 3'. Tangents of the block models with respect to the Gaussian's sigma and the
// regularisation terms, for their gradients (Sec. 3.2 learns them by backpropagation).  The
// vertical blur gives the blurred sums S from tmp (the horizontal blur, weights w) and
// dS/dsigma from tmp2 (the horizontal blur with w' = dw/dsigma) and tmp: with the separable
// weights w(dy) w(dx), dS = V H' B + V' H B.  The model solves M a = D (b = mu_y - a^T mu), so
// for each parameter theta
//   da = M^-1 (dD - dM a),   db = dmu_y - da^T mu - a^T dmu,
// using the block's Cholesky factor of M.  For sigma, dmu, dW and dD follow from dS and the
// blurred count's tangent dn; eps (the ridge or the Appendix's additive term) and eps_mul (its
// multiplicative term) enter M only:
//   ridge:    M = W + eps I                          dM/deps = I
//   Appendix: M = W^ + eps diag(W^),  W^ = W + eps_mul (m m^T + diag m^2) + eps I  (m: absolute
//             guide means)   dM/deps = I + diag(W^) + eps I,
//             dM/deps_mul = (m m^T + diag m^2) + 2 eps diag(m^2),
//             and for sigma dW^ = dW + eps_mul (dm m^T + m dm^T + 2 diag(m dm)), dM = dW^ + eps diag(dW^).
// Writes the three tangents of the block model in the coef layout, the bias re-expressed
// relative to the frame reference (db - da^T (ref - frame reference)).  Blocks whose Cholesky
// pivot fell low get tangents from the FP32 factor (no FP64 re-solve).  S, dS: this thread's
// columns of two [NCH][stride] buffers.
template <int Q>
__device__ __forceinline__ void stage_blur_v_tangent(const FastArgs &a, size_t k, float *S, float *dS, int stride)
{
    using C = Chan<Q>;
    constexpr int NS = Q + 3;
    const size_t bplane = (size_t)a.Hb * a.Wb;
    if (k >= bplane) return;
    const int by = (int)(k / a.Wb), bx = (int)(k % a.Wb);
    float rk[NS];
#pragma unroll
    for (int q = 0; q < NS; ++q) rk[q] = a.blk[(C::NCH + q) * bplane + k];
    float n = 0.f, dn = 0.f;
    for (int pass = 0; pass < 2; ++pass) {
        float acc[C::NCH];
#pragma unroll
        for (int c = 0; c < C::NCH; ++c) acc[c] = 0.f;
        for (int dd = -a.taps; dd <= a.taps; ++dd) {
            const int yy = by + dd;
            if (yy < 0 || yy >= a.Hb) continue;
            const size_t kb = (size_t)yy * a.Wb + bx;
            float d[NS];
#pragma unroll
            for (int q = 0; q < NS; ++q) d[q] = a.blk[(C::NCH + q) * bplane + kb] - rk[q];
            const float nb = a.tmp[C::NCH * bplane + kb];
            const float w = a.w[dd + a.taps];
            if (pass == 0) {
                accumulate_shifted<Q>(acc, a.tmp + kb, bplane, d, nb, w);
                n = fmaf(w, nb, n);
            } else {
                const float nb2 = a.tmp2[C::NCH * bplane + kb], wd = a.wd[dd + a.taps];
                accumulate_shifted<Q>(acc, a.tmp2 + kb, bplane, d, nb2, w);
                accumulate_shifted<Q>(acc, a.tmp + kb, bplane, d, nb, wd);
                dn = fmaf(w, nb2, fmaf(wd, nb, dn));
            }
        }
        float *dst = pass == 0 ? S : dS;
#pragma unroll
        for (int c = 0; c < C::NCH; ++c) dst[c * stride] = acc[c];
    }
    float A[Q][3], bv[3], mu[Q], muy[3], L[Q * (Q + 1) / 2], inv_d[Q];
    if (a.appendix)
        solve_appendix<Q>(S, stride, n, a.eps, a.eps_mul, a.tau, rk, A, bv, mu, muy, L, inv_d);
    else
        dev::solve_pixel<Q>(S, stride, n, a.eps, a.tau, A, bv, mu, muy, L, inv_d);
    const float inv_n = 1.0f / n;
    const bool one_px = !(n > 1.5f);  // one-pixel block: a = 0, b = mu_y (see solve_pixel)
    // the Appendix's absolute means and diag(W^)
    float m[Q], whd[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        m[i] = rk[i] + mu[i];
        whd[i] = fmaf(-mu[i], mu[i], S[C::xx(i, i) * stride] * inv_n) + 2.f * a.eps_mul * m[i] * m[i] + a.eps;
    }
    float dmu[Q], dmuy[3];
#pragma unroll
    for (int i = 0; i < Q; ++i) dmu[i] = one_px ? 0.f : (dS[(C::X0 + i) * stride] - mu[i] * dn) * inv_n;
#pragma unroll
    for (int c = 0; c < 3; ++c) dmuy[c] = (dS[(C::Y0 + c) * stride] - muy[c] * dn) * inv_n;
    for (int t = 0; t < 3; ++t) {
        // dM (packed lower triangle) and dD of parameter t: 0 sigma, 1 eps, 2 eps_mul
        float dM[Q * (Q + 1) / 2], R[Q][3], da[Q][3];
#pragma unroll
        for (int i = 0; i < Q; ++i)
#pragma unroll
            for (int j = 0; j < Q; ++j) {
                if (j > i) continue;
                float v = 0.f;
                if (t == 0 && !one_px) {
                    const float sxx = S[C::xx(j, i) * stride] * inv_n;
                    v = (dS[C::xx(j, i) * stride] - sxx * dn) * inv_n - dmu[i] * mu[j] - mu[i] * dmu[j];
                    if (a.appendix) v = fmaf(a.eps_mul, dmu[i] * m[j] + m[i] * dmu[j] + (i == j ? 2.f * m[i] * dmu[i] : 0.f), v);
                } else if (t == 1) {
                    v = i == j ? 1.f : 0.f;
                } else if (t == 2 && a.appendix) {
                    v = m[i] * m[j] + (i == j ? m[i] * m[i] : 0.f);
                }
                dM[dev::tri(i, j)] = v;
            }
        if (a.appendix) {  // M = W^ + eps diag(W^): add eps dW^_ii (and W^_ii for eps itself)
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                const int ii = dev::tri(i, i);
                dM[ii] = fmaf(a.eps, dM[ii], dM[ii]) + (t == 1 ? whd[i] : 0.f);
            }
        }
#pragma unroll
        for (int i = 0; i < Q; ++i)
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                float r = 0.f;
                if (t == 0 && !one_px) {
                    const float sxy = S[C::xy(i, c) * stride] * inv_n;
                    r = (dS[C::xy(i, c) * stride] - sxy * dn) * inv_n - dmu[i] * muy[c] - mu[i] * dmuy[c];
                }
#pragma unroll
                for (int j = 0; j < Q; ++j) r = fmaf(-dM[j <= i ? dev::tri(i, j) : dev::tri(j, i)], A[j][c], r);
                R[i][c] = r;
            }
        dev::chol_solve3<Q>(L, inv_d, R, da);
        float dbv[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            float db = t == 0 ? dmuy[c] : 0.f;
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                if (one_px) da[i][c] = 0.f;
                db = fmaf(-da[i][c], mu[i], db);
                if (t == 0) db = fmaf(-A[i][c], dmu[i], db);
                db = fmaf(-da[i][c], rk[i] - a.shift[i], db);  // re-expressed relative to the frame reference
            }
            dbv[c] = db;
        }
        store_model<Q>(a.dcoef + ((size_t)t * bplane + k) * Model<Q>::CS, da, dbv);
    }
}

// 4. bilinear interpolation of the block models + apply.  Block centres are P = F s output pixels
// apart, so the output rows [P i - P/2, P i + P/2) of cell row i interpolate between the same two
// block rows: a thread takes one output column of a cell row and interpolates its four corner
// models horizontally once, then each row's model vertically, two guides per instruction (packed
// FP32).
//
// column_models: the models of output column x, the cell row beginning at output row ya (< 0 for
// the first): the upper block row's, and lower minus upper.  Returns the upper block row.
template <int Q>
__device__ __forceinline__ int column_models(const FastArgs &a, int P, int x, int ya, float2 (&top)[Model<Q>::CS / 2],
                                             float2 (&dtb)[Model<Q>::CS / 2])
{
    constexpr int CS = Model<Q>::CS;
    const int den = 2 * P;
    // block rows of the cell (the same for all its rows)
    const int ny0 = min(max(2 * max(ya, 0) + 1 - P, 0), (a.Hb - 1) * den);
    const int i0 = min(ny0 / den, max(a.Hb - 2, 0)), i1 = min(i0 + 1, a.Hb - 1);
    // block columns and weight of this column (exact rational coordinate (2 x + 1 - P) / (2 P))
    const int r = (x + P / 2) / P;
    const int jl = min(max(r - 1, 0), a.Wb - 1), jr = min(max(r, 0), a.Wb - 1);
    const int nx = min(max(2 * x + 1 - P, 0), (a.Wb - 1) * den);
    const float fx = fminf(fmaxf((float)(nx - (r - 1) * den) / (float)den, 0.f), 1.f);
    const float4 *l0 = reinterpret_cast<const float4 *>(a.coef + ((size_t)i0 * a.Wb + jl) * CS);
    const float4 *l1 = reinterpret_cast<const float4 *>(a.coef + ((size_t)i1 * a.Wb + jl) * CS);
    const int step = (jr - jl) * (CS / 4);
    const float2 fx2 = make_float2(fx, fx), minus = make_float2(-1.f, -1.f);
#pragma unroll
    for (int c = 0; c < CS / 4; ++c) {
        const float4 tl = __ldg(l0 + c), tr = __ldg(l0 + step + c), bl = __ldg(l1 + c), br = __ldg(l1 + step + c);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float2 t0 = h ? make_float2(tl.z, tl.w) : make_float2(tl.x, tl.y);
            const float2 t1 = h ? make_float2(tr.z, tr.w) : make_float2(tr.x, tr.y);
            const float2 b0 = h ? make_float2(bl.z, bl.w) : make_float2(bl.x, bl.y);
            const float2 b1 = h ? make_float2(br.z, br.w) : make_float2(br.x, br.y);
            const float2 tp = __ffma2_rn(fx2, __ffma2_rn(t0, minus, t1), t0);
            top[2 * c + h] = tp;
            dtb[2 * c + h] = __ffma2_rn(tp, minus, __ffma2_rn(fx2, __ffma2_rn(b0, minus, b1), b0));
        }
    }
    return i0;
}

// The frame reference: minus the guides' in pairs, and the radiance's
template <int Q>
__device__ __forceinline__ void load_reference(const FastArgs &a, float2 (&nsh)[Model<Q>::QE / 2], float (&shr)[3])
{
#pragma unroll
    for (int i = 0; i < Model<Q>::QE; i += 2) nsh[i / 2] = make_float2(-a.shift[i], i + 1 < Q ? -a.shift[i + 1] : 0.f);
#pragma unroll
    for (int c = 0; c < 3; ++c) shr[c] = a.shift[Q + c];
}

// apply_pixel: the model of output row y of that column, applied to the map guide z(i), i < Q, into
// out[c * oplane]
template <int Q, class Z>
__device__ __forceinline__ void apply_pixel(const FastArgs &a, int P, int y, int i0, const float2 (&top)[Model<Q>::CS / 2],
                                            const float2 (&dtb)[Model<Q>::CS / 2], const float2 (&nsh)[Model<Q>::QE / 2],
                                            const float (&shr)[3], Z z, float *out, size_t oplane)
{
    using M = Model<Q>;
    const int den = 2 * P;
    const int ny = min(max(2 * y + 1 - P, 0), (a.Hb - 1) * den);
    const float fy = (float)(ny - i0 * den) / (float)den;
    const float2 fy2 = make_float2(fy, fy), one = make_float2(1.f, 1.f);
    float2 zs[M::QE / 2], o2[3];
#pragma unroll
    for (int i = 0; i < M::QE; i += 2)
        zs[i / 2] = __ffma2_rn(make_float2(z(i), i + 1 < Q ? z(i + 1) : 0.f), one, nsh[i / 2]);
    float bias[3] = {fmaf(fy, dtb[0].x, top[0].x), fmaf(fy, dtb[0].y, top[0].y), fmaf(fy, dtb[1].x, top[1].x)};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        o2[c] = make_float2(0.f, 0.f);
#pragma unroll
        for (int i = 0; i < M::QE; i += 2) {
            const int m = M::at(c, i) / 2;
            o2[c] = __ffma2_rn(__ffma2_rn(fy2, dtb[m], top[m]), zs[i / 2], o2[c]);
        }
        __stcs(out + c * oplane, (bias[c] + (o2[c].x + o2[c].y)) + shr[c]);  // streamed: not kept in L2
    }
}

// Input columns of a row are dealt to CTAs of stage 1 in chunks of two per thread.
__host__ __device__ inline int moment_chunks(int Wi) { return (Wi + 2 * kMomThreads - 1) / (2 * kMomThreads); }

}  // namespace fast
}  // namespace flr
