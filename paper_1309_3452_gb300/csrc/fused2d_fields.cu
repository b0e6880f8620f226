// Fused (2+1)D kernels: tabulated and soft-core coefficients, tabulated links, and the
// per-site paths.
#include "fused2d.cuh"

namespace dirac {
namespace fused {

#define STEPS_2D(COEF, LINK, T) template int launch2d<COEF, LINK, T>(FusedArgs<F32>, cudaStream_t);
#define ALL_2D(COEF, LINK) STEPS_2D(COEF, LINK, 1) STEPS_2D(COEF, LINK, 2)
ALL_2D(COEF_TABLE, LINK_NONE)
ALL_2D(COEF_SOFTCORE, LINK_NONE)
ALL_2D(COEF_SOFTCORR, LINK_NONE)
ALL_2D(COEF_UNIFORM, LINK_TABLE)
ALL_2D(COEF_STEP, LINK_TABLE)
ALL_2D(COEF_STEP_X, LINK_TABLE)
ALL_2D(COEF_TABLE, LINK_TABLE)
ALL_2D(COEF_SOFTCORE, LINK_TABLE)
STEPS_2D(kAnyMode, kAnyMode, 1)

}  // namespace fused
}  // namespace dirac
