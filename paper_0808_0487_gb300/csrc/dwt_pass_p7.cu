// dwt_pass_p7.cu -- the passes of p = 7 (see dwt_pass.cuh)
#include "dwt_pass.cuh"

namespace dwt {
DWT_INSTANTIATE_PRIME(7)
}  // namespace dwt
