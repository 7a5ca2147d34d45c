// flr_fwd.cuh -- launches of the unfused forward / adjoint kernel (flr_fwd_kernel.cuh).
#pragma once

#include "flr_internal.cuh"

namespace flr {

// The instances of guide count Q: each in one source file (flr_fwd_q*.cu), so that they compile side
// by side.
template <int Q>
struct FwdLaunch {
    static cudaError_t launch(bool adj, const FwdArgs &a, dim3 grid, size_t smem, cudaStream_t st);
    static cudaError_t prepare(bool adj, int r, size_t smem);
    static size_t smem(int r, bool adj);
};

}  // namespace flr
