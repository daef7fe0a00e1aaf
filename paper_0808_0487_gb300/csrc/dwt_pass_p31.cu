// dwt_pass_p31.cu -- the passes of p = 31 (see dwt_pass.cuh)
#include "dwt_pass.cuh"

namespace dwt {
DWT_INSTANTIATE_PRIME(31)
}  // namespace dwt
