// flr_batch.cu -- the bounded grid barrier's self-test (flr_barrier_selftest): a barrier for
// co-resident CTAs whose wait is bounded in time, launched so that it must run out.
#include <cuda_runtime.h>

#include "flr.h"
#include "flr_internal.cuh"

namespace flr {
namespace {

__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Grid-wide barrier for co-resident CTAs, bounded in time.  Returns false (and records the
// timeout in *status) if the other CTAs did not all arrive within timeout_ns.
__device__ bool grid_barrier(unsigned *count, unsigned *gen, unsigned nblocks, int *status,
                             unsigned long long timeout_ns)
{
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        ok = 1;
        const unsigned g = *(volatile unsigned *)gen;
        __threadfence();
        if (atomicAdd(count, 1u) == nblocks - 1) {
            atomicExch(count, 0u);
            __threadfence();
            atomicAdd(gen, 1u);
        } else {
            const unsigned long long t0 = global_ns();
            while (*(volatile unsigned *)gen == g) {
                if (global_ns() - t0 > timeout_ns) {
                    atomicExch(status, FLR_BATCH_TIMEOUT);
                    ok = 0;
                    break;
                }
                __nanosleep(256);
            }
        }
        __threadfence();
    }
    __syncthreads();
    return ok != 0;
}

// A barrier that waits for more CTAs than exist: every wait runs out.  Tests the bounded
// wait and the status path without any fault.
__global__ void barrier_selftest_kernel(unsigned *count, unsigned *gen, unsigned expected, int *status,
                                        unsigned long long timeout_ns)
{
    grid_barrier(count, gen, expected, status, timeout_ns);
}

}  // namespace

cudaError_t launch_barrier_selftest(unsigned *count, unsigned *gen, unsigned expected, int *status,
                                    unsigned long long timeout_ns, int grid, cudaStream_t st)
{
    barrier_selftest_kernel<<<grid, 32, 0, st>>>(count, gen, expected, status, timeout_ns);
    return cudaGetLastError();
}

}  // namespace flr
