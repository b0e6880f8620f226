// Fused (2+1)D kernels: several simulations per launch.
#include "fused2d.cuh"

namespace dirac {
namespace fused {

#define BATCH_2D(COEF, LINK, T)                                                               \
  template void launch2d_batch<COEF, LINK, T, true>(BatchArgs<F32>, long long, cudaStream_t); \
  template void launch2d_batch<COEF, LINK, T, false>(BatchArgs<F32>, long long, cudaStream_t);
#define ALL_2D(COEF, LINK) BATCH_2D(COEF, LINK, 1) BATCH_2D(COEF, LINK, 2)
ALL_2D(COEF_UNIFORM, LINK_NONE)
ALL_2D(COEF_STEP, LINK_NONE)
ALL_2D(COEF_UNIFORM, LINK_CONST)
ALL_2D(COEF_STEP, LINK_CONST)

}  // namespace fused
}  // namespace dirac
