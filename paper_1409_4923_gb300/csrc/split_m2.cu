// split_m2.cu -- instantiations of the two-warp run kernel for model 2 (piecewise-linear).
#include "split_kernels.cuh"

namespace sde {

SDE_SPLIT_UNIT(2)

}  // namespace sde
