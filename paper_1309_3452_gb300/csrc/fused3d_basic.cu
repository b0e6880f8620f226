// Fused (3+1)D kernels: uniform and Klein-step coefficients, no vector potential.
#include "fused3d.cuh"

namespace dirac {
namespace fused {

ChunkShape shape3d(const int N[3]) {
  const int n[3] = {N[0], N[1], N[2]};
  return {tiles3d<kBatchPairs>(n), N[2],
          workers3d<fused3d_kernel<F32, COEF_UNIFORM, LINK_NONE, false, kBatchPairs, true>, kBatchPairs>(), 4, 0.5};
}

#define STEP_3D(COEF, LINK) template int launch3d<COEF, LINK>(FusedArgs<F32>, cudaStream_t);
STEP_3D(COEF_UNIFORM, LINK_NONE)
STEP_3D(COEF_STEP, LINK_NONE)

}  // namespace fused
}  // namespace dirac
