// Fused (2+1)D kernels: uniform and Klein-step coefficients, no or constant links.
#include "fused2d.cuh"

namespace dirac {
namespace fused {

// (the plain kernels' resident warps stand for all; a restarted item costs about
// kT + 1 rows: its stages start one after another)
ChunkShape shape2d(const int N[3], int steps) {
  if (steps == 2)
    return {strips2d<2>(N[0]), N[1], workers2d<fused2d_kernel<F32, COEF_UNIFORM, LINK_NONE, 2, true>>(), 2, 3.0};
  return {strips2d<1>(N[0]), N[1], workers2d<fused2d_kernel<F32, COEF_UNIFORM, LINK_NONE, 1, true>>(), 2, 1.0};
}

#define STEPS_2D(COEF, LINK, T) template int launch2d<COEF, LINK, T>(FusedArgs<F32>, cudaStream_t);
#define ALL_2D(COEF, LINK) STEPS_2D(COEF, LINK, 1) STEPS_2D(COEF, LINK, 2)
ALL_2D(COEF_UNIFORM, LINK_NONE)
ALL_2D(COEF_STEP, LINK_NONE)
ALL_2D(COEF_STEP_X, LINK_NONE)
ALL_2D(COEF_UNIFORM, LINK_CONST)
ALL_2D(COEF_STEP, LINK_CONST)
ALL_2D(COEF_STEP_X, LINK_CONST)

}  // namespace fused
}  // namespace dirac
