// tma.cuh -- tensor-memory-access (TMA) helpers for sm_103a kernels: tensor-map encoding
// through the runtime's driver entry point, bulk tensor loads that complete on an mbarrier,
// and bounded mbarrier waits.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>
#include <stdint.h>

#include <atomic>

namespace tma {

// cuTensorMapEncodeTiled, looked up once (no link against libcuda)
inline PFN_cuTensorMapEncodeTiled_v12000 encoder()
{
    static std::atomic<PFN_cuTensorMapEncodeTiled_v12000> known{nullptr};
    PFN_cuTensorMapEncodeTiled_v12000 fn = known.load(std::memory_order_acquire);
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess) {
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
            known.store(fn, std::memory_order_release);
        }
    }
    return fn;
}

// 3-D map of float32 planes [P][H][W] (W innermost): box (bw, bh, bp) -- bw columns,
// bh rows, bp planes -- zero fill outside.  One copy of the box transfers bw * bh * bp * 4
// bytes.  Needs the row pitch in bytes and the base address to be multiples of 16.
// pitch: floats per row in memory (a multiple of 4; 0: W).
inline cudaError_t encode_planes_f32(CUtensorMap *m, const float *base, int W, int H, int P, int bw, int bh, int bp,
                                     int pitch = 0)
{
    PFN_cuTensorMapEncodeTiled_v12000 fn = encoder();
    if (!fn) return cudaErrorNotSupported;
    const cuuint64_t row = (cuuint64_t)(pitch ? pitch : W) * 4;
    const cuuint64_t dims[3] = {(cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)P};
    const cuuint64_t strides[2] = {row, row * H};
    const cuuint32_t box[3] = {(cuuint32_t)bw, (cuuint32_t)bh, (cuuint32_t)bp};
    const cuuint32_t es[3] = {1, 1, 1};
    const CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float *>(base), dims, strides, box, es,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ unsigned long long now_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_addr(bar)), "r"(count));
}

__device__ __forceinline__ void mbar_init_fence() { asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory"); }

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}

// 3-D tile load (x innermost) into shared memory, completing on `bar`
__device__ __forceinline__ void load_3d(void *dst, const CUtensorMap *tm, int x, int y, int z, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];\n" ::"r"(
            smem_addr(dst)),
        "l"(reinterpret_cast<uint64_t>(tm)), "r"(x), "r"(y), "r"(z), "r"(smem_addr(bar))
        : "memory");
}

// The same load with an L2 eviction policy (from createpolicy)
__device__ __forceinline__ void load_3d_hint(void *dst, const CUtensorMap *tm, int x, int y, int z, uint64_t *bar,
                                             uint64_t policy)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint"
        " [%0], [%1, {%2, %3, %4}], [%5], %6;\n" ::"r"(smem_addr(dst)),
        "l"(reinterpret_cast<uint64_t>(tm)), "r"(x), "r"(y), "r"(z), "r"(smem_addr(bar)), "l"(policy)
        : "memory");
}

// Bounded wait for the phase of `bar` with the given parity, polled by lane 0 of each warp
// (try_wait suspends up to 20 us per call).  Returns false if timeout_ns ran out.
__device__ __forceinline__ bool wait_warp(uint64_t *bar, uint32_t parity, unsigned long long timeout_ns)
{
    uint32_t ok = 1;
    if ((threadIdx.x & 31) == 0) {
        const uint32_t a = smem_addr(bar);
        const unsigned long long t0 = now_ns();
        for (;;) {
            uint32_t done;
            asm volatile(
                "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, 20000;\nselp.u32 %0, 1, 0, p;\n}\n"
                : "=r"(done)
                : "r"(a), "r"(parity)
                : "memory");
            if (done) break;
            if (now_ns() - t0 > timeout_ns) {
                ok = 0;
                break;
            }
        }
    }
    return __shfl_sync(0xffffffffu, ok, 0) != 0;
}

}  // namespace tma
