// dwt_pass_p19.cu -- the passes of p = 19 (see dwt_pass.cuh)
#include "dwt_pass.cuh"

namespace dwt {
DWT_INSTANTIATE_PRIME(19)
}  // namespace dwt
