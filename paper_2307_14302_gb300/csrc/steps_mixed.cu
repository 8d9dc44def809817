// steps_mixed.cu -- small-mesh kernel (steps.cuh), mixed precision: the generic instantiations and
// those of the feature sets that also have specialised tile kernels.
#include "steps_launch.cuh"

namespace dg {
DG_DEFINE_STEPS_LAUNCHERS(Mixed)
}  // namespace dg
