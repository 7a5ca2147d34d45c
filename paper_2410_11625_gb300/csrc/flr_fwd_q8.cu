// flr_fwd_q8.cu -- instances of the unfused forward / adjoint kernel for guide count 8.
#include "flr_fwd_kernel.cuh"

namespace flr {

template struct FwdLaunch<8>;

}  // namespace flr
