// Fused (3+1)D kernels: several simulations per launch.
#include "fused3d.cuh"

namespace dirac {
namespace fused {

#define BATCH_3D(COEF, LINK)                                                               \
  template void launch3d_batch<COEF, LINK, true>(BatchArgs<F32>, long long, cudaStream_t); \
  template void launch3d_batch<COEF, LINK, false>(BatchArgs<F32>, long long, cudaStream_t);
BATCH_3D(COEF_UNIFORM, LINK_NONE)
BATCH_3D(COEF_STEP, LINK_NONE)
BATCH_3D(COEF_UNIFORM, LINK_CONST)
BATCH_3D(COEF_STEP, LINK_CONST)

}  // namespace fused
}  // namespace dirac
