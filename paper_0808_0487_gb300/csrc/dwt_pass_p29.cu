// dwt_pass_p29.cu -- the passes of p = 29 (see dwt_pass.cuh)
#include "dwt_pass.cuh"

namespace dwt {
DWT_INSTANTIATE_PRIME(29)
}  // namespace dwt
