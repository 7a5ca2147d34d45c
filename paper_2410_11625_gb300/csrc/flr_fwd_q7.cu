// flr_fwd_q7.cu -- instances of the unfused forward / adjoint kernel for guide count 7.
#include "flr_fwd_kernel.cuh"

namespace flr {

template struct FwdLaunch<7>;

}  // namespace flr
