// Fused (2+1)D kernels: a plane wave across its polarisation.
#include "fused2d.cuh"

namespace dirac {
namespace fused {

#define STEPS_2D(COEF, LINK, T) template int launch2d<COEF, LINK, T>(FusedArgs<F32>, cudaStream_t);
#define ALL_2D(COEF, LINK) STEPS_2D(COEF, LINK, 1) STEPS_2D(COEF, LINK, 2)
ALL_2D(COEF_UNIFORM, LINK_PLANE)
ALL_2D(COEF_STEP, LINK_PLANE)
ALL_2D(COEF_STEP_X, LINK_PLANE)
ALL_2D(COEF_TABLE, LINK_PLANE)
ALL_2D(COEF_SOFTCORE, LINK_PLANE)
ALL_2D(COEF_SOFTCORR, LINK_PLANE)

}  // namespace fused
}  // namespace dirac
