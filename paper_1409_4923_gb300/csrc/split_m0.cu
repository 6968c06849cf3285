// split_m0.cu -- instantiations of the two-warp run kernel for model 0 (inertial washboard).
#include "split_kernels.cuh"

namespace sde {

SDE_SPLIT_UNIT(0)

}  // namespace sde
