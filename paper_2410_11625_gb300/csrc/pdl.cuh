// pdl.cuh -- programmatic dependent launch.
//
// A kernel launched with pdl::launch may start when every CTA of its predecessor has called
// pdl::trigger (or exited); it must call pdl::wait, which returns when the predecessor has
// finished and its writes are visible, before it touches global memory.  Only set-up (barriers,
// tensor memory, index arithmetic) runs ahead.  Every CTA of a dependent kernel that triggers calls
// wait itself, so a finished predecessor implies that its own predecessors have finished.
// One chain differs: the first stage of fast FLR is an ordinary launch that triggers without
// waiting.  It starts when everything before the call is complete, so the last stage may read the
// caller's map guide ahead of its wait; were the first stage a dependent launch, that read would race
// with the map guide's producer.
#pragma once

#include <cuda_runtime.h>

#include <utility>

#include "device_cache.h"

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
    static PerDevice<bool> done;
    int dev = 0;
    bool set = false;
    const cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    return done.get(dev, [&](bool &d) {
        cudaError_t f = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        if (f == cudaSuccess && max_carveout)
            f = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
        d = f == cudaSuccess;
        return f;
    }, set);
}

// SMs of the current device (1 if the device cannot be asked)
inline int sm_count()
{
    static PerDevice<int> known;
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 1;
    const cudaError_t e = known.get(dev, [&](int &v) { return cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev); }, n);
    return e == cudaSuccess && n > 0 ? n : 1;
}

}  // namespace pdl
