// Planning and dispatch of the fused time-step kernels (fused3d.cuh, fused2d.cu).
#include "fused_common.cuh"

namespace dirac {

namespace fused {

// the launchers, instantiated per field path in fused3d_*.cu and fused2d.cu
template <int COEF, int LINK>
int launch3d(FusedArgs<F32> a, cudaStream_t s);
template <int COEF, int LINK>
void launch3d_batch(BatchArgs<F32> b, long long total, cudaStream_t s);
template <int COEF, int LINK>
int launch2d(FusedArgs<F32> a, cudaStream_t s);
template <int COEF, int LINK>
int launch2d_tb2(FusedArgs<F32> a, cudaStream_t s);
template <int COEF, int LINK>
void launch2d_batch(BatchArgs<F32> b, long long total, cudaStream_t s);
template <int COEF, int LINK>
void launch2d_tb2_batch(BatchArgs<F32> b, long long total, cudaStream_t s);
// Chunk length (levels per item) for `tiles` items per level chunk, `levels`
// levels and `workers` persistent workers: maximise the busy fraction of the
// rounds times the useful fraction chunk/(chunk+restart) of each item, where
// `restart` is the cost of an item's extra first level in levels.
// The `max` best chunk lengths by that model, best first, into out; returns
// how many (at least one).
int rank_chunks(long long tiles, int levels, long long workers, int min_chunk, double restart, int* out,
                int max) {
  int n = 0, prev = -1;
  double eff_of[64];
  if (max > 64) max = 64;
  for (int c = 1; c <= levels; ++c) {
    const int len = (levels + c - 1) / c;  // non-increasing in c
    if (len < min_chunk && c > 1) break;
    if (len == prev) continue;
    prev = len;
    const int chunks = (levels + len - 1) / len;
    const long long items = tiles * chunks;
    const long long rounds = (items + workers - 1) / workers;
    // work of a round ~ len + restart levels; total time ~ rounds * (len + restart)
    const double eff = (double)tiles * levels / ((double)rounds * workers * (len + restart));
    // insert by efficiency (stable: on ties, fewer chunks first)
    int pos = n;
    while (pos > 0 && eff > eff_of[pos - 1] * 1.0001) --pos;
    if (pos >= max) continue;
    const int last = n < max ? n : max - 1;
    for (int i = last; i > pos; --i) {
      out[i] = out[i - 1];
      eff_of[i] = eff_of[i - 1];
    }
    out[pos] = len;
    eff_of[pos] = eff;
    if (n < max) ++n;
  }
  if (n == 0) out[n++] = levels;
  return n;
}

int plan_chunk(const ChunkShape& g) {
  int best = g.levels;
  rank_chunks(g.tiles, g.levels, g.workers, g.min_chunk, g.restart, &best, 1);
  return best;
}

}  // namespace fused

using namespace fused;

namespace {

template <int DIMS, int COEF, int LINK>
int launch_dims(const FusedArgs<F32>& a, cudaStream_t s) {
  if constexpr (DIMS == 3) {
    // (3+1)D plane waves are dispatched before reaching here (LINK_PLANE_ZX)
    if constexpr (LINK == LINK_PLANE) return launch3d<kAnyMode, kAnyMode>(a, s);
    else return launch3d<COEF, LINK>(a, s);
  } else {
    return launch2d<COEF, LINK>(a, s);
  }
}

template <int DIMS>
int dispatch(const FusedArgs<F32>& a, cudaStream_t s) {
  const int c = a.hu.coef_mode, l = a.hu.link_mode;
  if (c == COEF_GENERAL || l == LINK_GENERAL) return launch_dims<DIMS, kAnyMode, kAnyMode>(a, s);
  // the fused (3+1)D kernel stages plane-wave link factors per z level: a wave
  // along z polarised along x runs as LINK_PLANE_ZX, other plane waves take
  // the general path there
  if (DIMS == 3 && l == LINK_PLANE) {
    if (a.hu.ltab_axis != 2 || a.hu.lpol != 0) return launch3d<kAnyMode, kAnyMode>(a, s);
    if (c == COEF_UNIFORM) return launch3d<COEF_UNIFORM, LINK_PLANE_ZX>(a, s);
    if (c == COEF_STEP) return launch3d<COEF_STEP, LINK_PLANE_ZX>(a, s);
    if (c == COEF_TABLE) return launch3d<COEF_TABLE, LINK_PLANE_ZX>(a, s);
    if (c == COEF_SOFTCORE) return launch3d<COEF_SOFTCORE, LINK_PLANE_ZX>(a, s);
    if (c == COEF_SOFTCORR) return launch3d<COEF_SOFTCORR, LINK_PLANE_ZX>(a, s);
    return launch3d<kAnyMode, kAnyMode>(a, s);
  }
  if (c == COEF_SOFTCORE) {
    if (l == LINK_NONE) return launch_dims<DIMS, COEF_SOFTCORE, LINK_NONE>(a, s);
    if (l == LINK_PLANE) return launch_dims<DIMS, COEF_SOFTCORE, LINK_PLANE>(a, s);
    return launch_dims<DIMS, kAnyMode, kAnyMode>(a, s);
  }
  if (c == COEF_SOFTCORR) {
    if (l == LINK_NONE) return launch_dims<DIMS, COEF_SOFTCORR, LINK_NONE>(a, s);
    if (l == LINK_PLANE) return launch_dims<DIMS, COEF_SOFTCORR, LINK_PLANE>(a, s);
    return launch_dims<DIMS, kAnyMode, kAnyMode>(a, s);
  }
  if (l == LINK_TABLE) {
    if (c == COEF_UNIFORM) return launch_dims<DIMS, COEF_UNIFORM, LINK_TABLE>(a, s);
    if (c == COEF_STEP) return launch_dims<DIMS, COEF_STEP, LINK_TABLE>(a, s);
    return launch_dims<DIMS, COEF_TABLE, LINK_TABLE>(a, s);
  }
  if (c == COEF_TABLE && l == LINK_NONE) return launch_dims<DIMS, COEF_TABLE, LINK_NONE>(a, s);
  if (c == COEF_TABLE && l == LINK_PLANE) return launch_dims<DIMS, COEF_TABLE, LINK_PLANE>(a, s);
  if (c == COEF_TABLE) return launch_dims<DIMS, kAnyMode, kAnyMode>(a, s);
  if (c == COEF_UNIFORM && l == LINK_PLANE) return launch_dims<DIMS, COEF_UNIFORM, LINK_PLANE>(a, s);
  if (c == COEF_STEP && l == LINK_PLANE) return launch_dims<DIMS, COEF_STEP, LINK_PLANE>(a, s);
  if (c == COEF_UNIFORM && l == LINK_NONE) return launch_dims<DIMS, COEF_UNIFORM, LINK_NONE>(a, s);
  if (c == COEF_STEP && l == LINK_NONE) return launch_dims<DIMS, COEF_STEP, LINK_NONE>(a, s);
  if (c == COEF_UNIFORM && l == LINK_CONST) return launch_dims<DIMS, COEF_UNIFORM, LINK_CONST>(a, s);
  return launch_dims<DIMS, COEF_STEP, LINK_CONST>(a, s);
}

template <int DIMS, int COEF, int LINK>
void batch_dims(const BatchArgs<F32>& b, long long total, cudaStream_t s) {
  if (DIMS == 3) launch3d_batch<COEF, LINK>(b, total, s);
  else launch2d_batch<COEF, LINK>(b, total, s);
}

}  // namespace

int launch_fused2d_tb2(const FusedArgs<F32>& a, cudaStream_t s) {
  const int c = a.hu.coef_mode, l = a.hu.link_mode;
  if (c == COEF_UNIFORM && l == LINK_NONE) return launch2d_tb2<COEF_UNIFORM, LINK_NONE>(a, s);
  if (c == COEF_STEP && l == LINK_NONE) return launch2d_tb2<COEF_STEP, LINK_NONE>(a, s);
  if (c == COEF_UNIFORM && l == LINK_CONST) return launch2d_tb2<COEF_UNIFORM, LINK_CONST>(a, s);
  if (c == COEF_STEP && l == LINK_CONST) return launch2d_tb2<COEF_STEP, LINK_CONST>(a, s);
  if (c == COEF_TABLE && l == LINK_NONE) return launch2d_tb2<COEF_TABLE, LINK_NONE>(a, s);
  if (c == COEF_SOFTCORE && l == LINK_NONE) return launch2d_tb2<COEF_SOFTCORE, LINK_NONE>(a, s);
  if (c == COEF_SOFTCORR && l == LINK_NONE) return launch2d_tb2<COEF_SOFTCORR, LINK_NONE>(a, s);
  return 0;
}

static ChunkShape shape_of(int dims, const int N[3], int two_step) {
  return dims == 3 ? shape3d(N) : (two_step ? shape2d_tb2(N) : shape2d(N));
}
static long long items_of(const ChunkShape& g, int chunk) { return g.tiles * ((g.levels + chunk - 1) / chunk); }

int fused_chunk_tb2(const int N[3]) { return plan_chunk(shape2d_tb2(N)); }

long long fused_items_tb2(const int N[3], int chunk) { return items_of(shape2d_tb2(N), chunk); }

void launch_fused2d_tb2_batch(const BatchArgs<F32>& b, long long total, int coef, int link, cudaStream_t s) {
  if (coef == COEF_UNIFORM && link == LINK_NONE) return launch2d_tb2_batch<COEF_UNIFORM, LINK_NONE>(b, total, s);
  if (coef == COEF_STEP && link == LINK_NONE) return launch2d_tb2_batch<COEF_STEP, LINK_NONE>(b, total, s);
  if (coef == COEF_UNIFORM && link == LINK_CONST) return launch2d_tb2_batch<COEF_UNIFORM, LINK_CONST>(b, total, s);
  return launch2d_tb2_batch<COEF_STEP, LINK_CONST>(b, total, s);
}

int fused_chunk(int dims, const int N[3]) { return plan_chunk(shape_of(dims, N, 0)); }

int fused_candidates(int dims, const int N[3], int two_step, int* out, int max) {
  const ChunkShape g = shape_of(dims, N, two_step);
  return rank_chunks(g.tiles, g.levels, g.workers, g.min_chunk, g.restart, out, max);
}

long long fused_items(int dims, const int N[3], int chunk) { return items_of(shape_of(dims, N, 0), chunk); }

template <>
void launch_fused_batch<F32, 3>(const BatchArgs<F32>& b, long long total, int coef, int link,
                                cudaStream_t s) {
  if (coef == COEF_UNIFORM && link == LINK_NONE) return batch_dims<3, COEF_UNIFORM, LINK_NONE>(b, total, s);
  if (coef == COEF_STEP && link == LINK_NONE) return batch_dims<3, COEF_STEP, LINK_NONE>(b, total, s);
  if (coef == COEF_UNIFORM && link == LINK_CONST) return batch_dims<3, COEF_UNIFORM, LINK_CONST>(b, total, s);
  return batch_dims<3, COEF_STEP, LINK_CONST>(b, total, s);
}
template <>
void launch_fused_batch<F32, 2>(const BatchArgs<F32>& b, long long total, int coef, int link,
                                cudaStream_t s) {
  if (coef == COEF_UNIFORM && link == LINK_NONE) return batch_dims<2, COEF_UNIFORM, LINK_NONE>(b, total, s);
  if (coef == COEF_STEP && link == LINK_NONE) return batch_dims<2, COEF_STEP, LINK_NONE>(b, total, s);
  if (coef == COEF_UNIFORM && link == LINK_CONST) return batch_dims<2, COEF_UNIFORM, LINK_CONST>(b, total, s);
  return batch_dims<2, COEF_STEP, LINK_CONST>(b, total, s);
}

template <>
int launch_fused<F32, 3>(const FusedArgs<F32>& a, cudaStream_t s) {
  return dispatch<3>(a, s);
}
template <>
int launch_fused<F32, 2>(const FusedArgs<F32>& a, cudaStream_t s) {
  return dispatch<2>(a, s);
}

}  // namespace dirac
