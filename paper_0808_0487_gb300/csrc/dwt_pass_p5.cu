// dwt_pass_p5.cu -- the passes of p = 5 (see dwt_pass.cuh)
#include "dwt_pass.cuh"

namespace dwt {
DWT_INSTANTIATE_PRIME(5)
}  // namespace dwt
