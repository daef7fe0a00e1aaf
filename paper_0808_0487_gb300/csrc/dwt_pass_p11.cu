// dwt_pass_p11.cu -- the passes of p = 11 (see dwt_pass.cuh)
#include "dwt_pass.cuh"

namespace dwt {
DWT_INSTANTIATE_PRIME(11)
}  // namespace dwt
