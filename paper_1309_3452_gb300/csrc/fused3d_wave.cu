// Fused (3+1)D kernels: a plane wave along z polarised along x.
#include "fused3d.cuh"

namespace dirac {
namespace fused {

#define STEP_3D(COEF, LINK) template int launch3d<COEF, LINK>(FusedArgs<F32>, cudaStream_t);
STEP_3D(COEF_UNIFORM, LINK_PLANE_ZX)
STEP_3D(COEF_STEP, LINK_PLANE_ZX)
STEP_3D(COEF_TABLE, LINK_PLANE_ZX)
STEP_3D(COEF_SOFTCORE, LINK_PLANE_ZX)
STEP_3D(COEF_SOFTCORR, LINK_PLANE_ZX)

}  // namespace fused
}  // namespace dirac
