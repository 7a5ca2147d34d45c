// flr_fwd.cu -- the frame reference shift by itself, and the dispatch of the unfused forward and
// adjoint kernel (flr_fwd_kernel.cuh) over the guide count.
#include "flr_fwd.cuh"
#include "flr_internal.cuh"
#include "pdl.cuh"

namespace flr {
namespace {

// The frame reference shift alone (the forward kernel's s_ref: the same sample of rows
// [0, ref_rows)), for a pass that needs it before any forward-kernel launch.
// One warp per input channel: a channel's sum takes the samples in sample_mean's order (lane l
// adds samples l, l + 32, ..., then the shuffle tree), so the values are the same, while the
// Q + 3 chains of loads run side by side (128 x 128: one warp for all channels 3.6 us, this 1.9 us).
template <int Q>
__global__ void __launch_bounds__(32 * (Q + 3)) frame_shift_kernel(const float *guide, const float *rad, int H, int W,
                                                                    int ref_rows, float *shift_out)
{
    pdl::wait();
    constexpr int NS = kShiftSamples;
    const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int yb = ref_rows > 0 ? min(ref_rows, H) : H;
    const size_t plane = (size_t)H * W;
    const float *src = k < Q ? guide + k * plane : rad + (k - Q) * plane;
    float acc = 0.f;
#pragma unroll
    for (int it = 0; it < NS * NS / 32; ++it) {
        const int s = lane + 32 * it, iy = s / NS, ix = s % NS;
        const int y = (int)(((long long)(2 * iy + 1) * yb) / (2 * NS)), x = (int)(((long long)(2 * ix + 1) * W) / (2 * NS));
        acc += __ldg(src + (size_t)y * W + x);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) shift_out[k] = acc * (1.0f / (NS * NS));
}

}  // namespace

#define FLR_Q_DISPATCH(q, ...)  \
    switch (q) {                 \
    case 1: { constexpr int QQ = 1; __VA_ARGS__; } \
    case 2: { constexpr int QQ = 2; __VA_ARGS__; } \
    case 3: { constexpr int QQ = 3; __VA_ARGS__; } \
    case 4: { constexpr int QQ = 4; __VA_ARGS__; } \
    case 5: { constexpr int QQ = 5; __VA_ARGS__; } \
    case 6: { constexpr int QQ = 6; __VA_ARGS__; } \
    case 7: { constexpr int QQ = 7; __VA_ARGS__; } \
    case 8: { constexpr int QQ = 8; __VA_ARGS__; } \
    default: break;              \
    }

cudaError_t launch_fwd(int q, const FwdArgs &a, dim3 grid, size_t smem, cudaStream_t st)
{
    FLR_Q_DISPATCH(q, return FwdLaunch<QQ>::launch(false, a, grid, smem, st));
    return cudaErrorInvalidValue;
}

cudaError_t launch_adj(int q, const FwdArgs &a, dim3 grid, size_t smem, cudaStream_t st)
{
    FLR_Q_DISPATCH(q, return FwdLaunch<QQ>::launch(true, a, grid, smem, st));
    return cudaErrorInvalidValue;
}

cudaError_t launch_frame_shift(int q, const float *guide, const float *rad, int H, int W, int ref_rows, float *shift_out,
                               cudaStream_t st)
{
    FLR_Q_DISPATCH(q, return pdl::launch(frame_shift_kernel<QQ>, dim3(1), 32 * (QQ + 3), 0, st, guide, rad, H, W, ref_rows,
                                         shift_out));
    return cudaErrorInvalidValue;
}

size_t fwd_smem_bytes(int q, int r)
{
    FLR_Q_DISPATCH(q, return FwdLaunch<QQ>::smem(r, false));
    return 0;
}

size_t adj_smem_bytes(int q, int r)
{
    FLR_Q_DISPATCH(q, return FwdLaunch<QQ>::smem(r, true));
    return 0;
}

cudaError_t fwd_prepare(int q, int r, size_t smem)
{
    FLR_Q_DISPATCH(q, return FwdLaunch<QQ>::prepare(false, r, smem));
    return cudaErrorInvalidValue;
}

cudaError_t adj_prepare(int q, int r, size_t smem)
{
    FLR_Q_DISPATCH(q, return FwdLaunch<QQ>::prepare(true, r, smem));
    return cudaErrorInvalidValue;
}

}  // namespace flr
