// flr_fwd_q45.cu -- instances of the unfused forward / adjoint kernel for guide counts 4, 5.
#include "flr_fwd_kernel.cuh"

namespace flr {

template struct FwdLaunch<4>;
template struct FwdLaunch<5>;

}  // namespace flr
