// Fused (3+1)D kernels: tabulated and soft-core coefficients, and the per-site paths.
#include "fused3d.cuh"

namespace dirac {
namespace fused {

#define STEP_3D(COEF, LINK) template int launch3d<COEF, LINK>(FusedArgs<F32>, cudaStream_t);
STEP_3D(COEF_TABLE, LINK_NONE)
STEP_3D(COEF_SOFTCORE, LINK_NONE)
STEP_3D(COEF_SOFTCORR, LINK_NONE)
STEP_3D(kAnyMode, kAnyMode)

}  // namespace fused
}  // namespace dirac
