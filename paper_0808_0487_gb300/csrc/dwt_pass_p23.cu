// dwt_pass_p23.cu -- the passes of p = 23 (see dwt_pass.cuh)
#include "dwt_pass.cuh"

namespace dwt {
DWT_INSTANTIATE_PRIME(23)
}  // namespace dwt
