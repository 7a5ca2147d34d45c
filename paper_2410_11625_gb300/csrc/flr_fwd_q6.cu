// flr_fwd_q6.cu -- instances of the unfused forward / adjoint kernel for guide count 6.
#include "flr_fwd_kernel.cuh"

namespace flr {

template struct FwdLaunch<6>;

}  // namespace flr
