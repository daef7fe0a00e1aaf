// dwt_pass_p17.cu -- the passes of p = 17 (see dwt_pass.cuh)
#include "dwt_pass.cuh"

namespace dwt {
DWT_INSTANTIATE_PRIME(17)
}  // namespace dwt
