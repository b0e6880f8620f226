// Fused (3+1)D kernels: constant and tabulated link factors.
#include "fused3d.cuh"

namespace dirac {
namespace fused {

#define STEP_3D(COEF, LINK) template int launch3d<COEF, LINK>(FusedArgs<F32>, cudaStream_t);
STEP_3D(COEF_UNIFORM, LINK_CONST)
STEP_3D(COEF_STEP, LINK_CONST)
STEP_3D(COEF_UNIFORM, LINK_TABLE)
STEP_3D(COEF_STEP, LINK_TABLE)
STEP_3D(COEF_TABLE, LINK_TABLE)
STEP_3D(COEF_SOFTCORE, LINK_TABLE)

}  // namespace fused
}  // namespace dirac
