// split_m1.cu -- instantiations of the two-warp run kernel for model 1 (overdamped washboard).
#include "split_kernels.cuh"

namespace sde {

SDE_SPLIT_UNIT(1)

}  // namespace sde
