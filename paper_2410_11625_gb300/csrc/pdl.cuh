// pdl.cuh -- programmatic dependent launch.
//
// A kernel launched with pdl::launch may start when every CTA of its predecessor has called
// pdl::trigger (or exited); it must call pdl::wait, which returns when the predecessor has
// finished and its writes are visible, before it touches global memory.  Only set-up (barriers,
// tensor memory, index arithmetic) runs ahead.  Every CTA of a kernel that triggers calls wait
// itself, so a finished predecessor implies that its own predecessors have finished.
#pragma once

#include <cuda_runtime.h>

#include <atomic>
#include <utility>

namespace pdl {

__device__ __forceinline__ void trigger() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }
__device__ __forceinline__ void wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }

template <class... P, class... A>
cudaError_t launch(void (*kern)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st, A &&...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, std::forward<A>(args)...);
}

// Lets a kernel use `bytes` of dynamic shared memory (and, when asked, prefer the largest shared
// carveout).  A function's attributes belong to the device, so they are set once per device and
// kernel (Tag: one type per kernel), not on every launch: two calls of about 1 us each, which a
// small frame's nine launches wait for.  bytes is the same on every call of one Tag.
template <class Tag, class K>
cudaError_t allow_smem(K kern, size_t bytes, bool max_carveout)
{
    static std::atomic<bool> done[64];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64 && done[dev].load(std::memory_order_acquire)) return cudaSuccess;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess && max_carveout)
        e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
    if (e == cudaSuccess && dev >= 0 && dev < 64) done[dev].store(true, std::memory_order_release);
    return e;
}

}  // namespace pdl
