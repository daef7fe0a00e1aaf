// dwt_pass_p13.cu -- the passes of p = 13 (see dwt_pass.cuh)
#include "dwt_pass.cuh"

namespace dwt {
DWT_INSTANTIATE_PRIME(13)
}  // namespace dwt
