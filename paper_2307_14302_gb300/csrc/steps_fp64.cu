// steps_fp64.cu -- small-mesh kernel (steps.cuh), FP64.
#include "steps_launch.cuh"

namespace dg {
DG_DEFINE_STEPS_LAUNCHERS(Fp64)
}  // namespace dg
