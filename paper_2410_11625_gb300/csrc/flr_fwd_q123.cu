// flr_fwd_q123.cu -- instances of the unfused forward / adjoint kernel for guide counts 1, 2, 3.
#include "flr_fwd_kernel.cuh"

namespace flr {

template struct FwdLaunch<1>;
template struct FwdLaunch<2>;
template struct FwdLaunch<3>;

}  // namespace flr
