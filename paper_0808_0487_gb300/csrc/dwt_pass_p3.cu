// dwt_pass_p3.cu -- the passes of p = 3 (see dwt_pass.cuh)
#include "dwt_pass.cuh"

namespace dwt {
DWT_INSTANTIATE_PRIME(3)
}  // namespace dwt
