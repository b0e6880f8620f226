// What the fused time-step kernels of both dimensions share: the functional's
// terms, the batched launches' bookkeeping, resident worker counts.
#pragma once

#include "kernels.cuh"
#include "quad.cuh"

namespace dirac {
namespace fused {

__device__ __forceinline__ int wrapi(int i, int n) {
  i %= n;
  return i < 0 ? i + n : i;
}

// |value|^2 as the functional's terms are formed
__device__ __forceinline__ float n2(float2 v) { return fmaf(v.x, v.x, v.y * v.y); }
// the functional's terms of one component cell: the sum of |value|^2, and the
// cross terms conj(G) S' added to lc in the order of the two values
__device__ __forceinline__ float n2(const Quad& q) { return n2(qlane(q, 0)) + n2(qlane(q, 1)); }
__device__ __forceinline__ float cross(const Quad& G, const Quad& S, float lc) {
  lc = fmaf(G.re.x, S.re.x, fmaf(G.im.x, S.im.x, lc));
  return fmaf(G.re.y, S.re.y, fmaf(G.im.y, S.im.y, lc));
}

// FP64 block reduction of the two conserved-functional accumulators into
// out[blockIdx.x][2] (all threads of the block call it)
__device__ __forceinline__ void block_store_e(double e_n, double e_c, double* out) {
  __shared__ double red[32][2];
  double n = e_n, c = e_c;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    n += __shfl_down_sync(0xffffffffu, n, o);
    c += __shfl_down_sync(0xffffffffu, c, o);
  }
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  __syncthreads();
  if (lane == 0) {
    red[w][0] = n;
    red[w][1] = c;
  }
  __syncthreads();
  if (w == 0) {
    n = lane < nw ? red[lane][0] : 0.0;
    c = lane < nw ? red[lane][1] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      n += __shfl_down_sync(0xffffffffu, n, o);
      c += __shfl_down_sync(0xffffffffu, c, o);
    }
    if (lane == 0) {
      out[2LL * blockIdx.x] = n;
      out[2LL * blockIdx.x + 1] = c;
    }
  }
}

// simulation of global item g: the last s with first[s] <= g
__device__ __forceinline__ int find_sim(const long long* first, int nsims, long long g) {
  int lo = 0, hi = nsims - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (__ldg(first + mid) <= g) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// copy one simulation's arguments into shared memory (nthreads cooperating)
template <class P>
__device__ __forceinline__ void copy_args(FusedArgs<P>* dst, const FusedArgs<P>* src, int tid,
                                          int nthreads) {
  static_assert(sizeof(FusedArgs<P>) % 4 == 0, "word copy");
  const int* s = reinterpret_cast<const int*>(src);
  int* d = reinterpret_cast<int*>(dst);
  for (int i = tid; i < (int)(sizeof(FusedArgs<P>) / 4); i += nthreads) d[i] = __ldg(s + i);
}

inline int sm_count() {
  static const int count = [] {
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n > 0 ? n : 1;
  }();
  return count;
}

template <class K>
int resident_blocks(K kernel, int threads, size_t smem = 0) {
  int per_sm = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem);
  return (per_sm < 1 ? 1 : per_sm) * sm_count();
}

// What the chunk rule (step_fused.cu) needs to know of a kernel on a grid: work
// items per chunk of levels, levels, resident workers, the shortest chunk worth
// starting and the cost of an item's restart in levels.
struct ChunkShape {
  long long tiles;
  int levels, workers, min_chunk;
  double restart;
};
ChunkShape shape3d(const int N[3]);
ChunkShape shape2d(const int N[3], int steps);  // steps per pass
// chunk length (levels per item) by that rule
int plan_chunk(const ChunkShape& g);

}  // namespace fused
}  // namespace dirac
