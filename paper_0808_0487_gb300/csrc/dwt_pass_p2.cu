// dwt_pass_p2.cu -- the passes of p = 2 (see dwt_pass.cuh)
#include "dwt_pass.cuh"

namespace dwt {
DWT_INSTANTIATE_PRIME(2)
}  // namespace dwt
