// Planning and dispatch of the fused time-step kernels (fused3d.cuh, fused2d.cuh).
#include <algorithm>
#include <vector>

#include "fused_common.cuh"

namespace dirac {

namespace fused {

// the launchers, instantiated per field path in fused3d_*.cu and fused2d_*.cu
template <int COEF, int LINK>
int launch3d(FusedArgs<F32> a, cudaStream_t s);
template <int COEF, int LINK, bool kIso>
void launch3d_batch(BatchArgs<F32> b, long long total, cudaStream_t s);
template <int COEF, int LINK, int kT>
int launch2d(FusedArgs<F32> a, cudaStream_t s);
template <int COEF, int LINK, int kT, bool kIso>
void launch2d_batch(BatchArgs<F32> b, long long total, cudaStream_t s);
// Chunk length (levels per item) for `tiles` items per level chunk, `levels`
// levels and `workers` persistent workers: maximise the busy fraction of the
// rounds times the useful fraction chunk/(chunk+restart) of each item, where
// `restart` is the cost of an item's extra first level in levels.
// The `max` best chunk lengths by that model, best first, into out; returns
// how many (at least one).
int rank_chunks(long long tiles, int levels, long long workers, int min_chunk, double restart, int* out,
                int max) {
  int n = 0, len = 0;
  double eff_of[64];
  if (max > 64) max = 64;
  // every length that an even split into c chunks has, longest first, each once
  // (trying every c took 40 us of host time per launch at 20000 levels, more than the kernel)
  for (int c = 1; c <= levels; c = len > 1 ? (levels + len - 2) / (len - 1) : levels + 1) {
    len = (levels + c - 1) / c;
    if (len < min_chunk && c > 1) break;
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

// kT time steps per pass ((3+1)D: one)
template <int DIMS, int kT, int COEF, int LINK>
int launch_dims(const FusedArgs<F32>& a, cudaStream_t s) {
  if constexpr (DIMS == 3) {
    // (3+1)D plane waves are dispatched before reaching here (LINK_PLANE_ZX)
    if constexpr (LINK == LINK_PLANE) return launch3d<kAnyMode, kAnyMode>(a, s);
    else return launch3d<COEF, LINK>(a, s);
  } else if constexpr (COEF == kAnyMode && kT > 1) {
    return 0;  // the per-site paths take one step per pass
  } else {
    if constexpr (COEF == COEF_STEP)
      if (a.hu.step_axis == 0) return launch2d<COEF_STEP_X, LINK, kT>(a, s);
    return launch2d<COEF, LINK, kT>(a, s);
  }
}

template <int DIMS, int kT>
int dispatch(const FusedArgs<F32>& a, cudaStream_t s) {
  const int c = a.hu.coef_mode, l = a.hu.link_mode;
#define RUN(COEF, LINK) return launch_dims<DIMS, kT, COEF, LINK>(a, s)
  if (c == COEF_GENERAL || l == LINK_GENERAL) RUN(kAnyMode, kAnyMode);
  // the fused (3+1)D kernel stages plane-wave link factors per z level: a wave
  // along z polarised along x runs as LINK_PLANE_ZX, other plane waves take
  // the general path there
  if constexpr (DIMS == 3) {
    if (l == LINK_PLANE) {
      if (a.hu.ltab_axis != 2 || a.hu.lpol != 0) RUN(kAnyMode, kAnyMode);
      if (c == COEF_UNIFORM) RUN(COEF_UNIFORM, LINK_PLANE_ZX);
      if (c == COEF_STEP) RUN(COEF_STEP, LINK_PLANE_ZX);
      if (c == COEF_TABLE) RUN(COEF_TABLE, LINK_PLANE_ZX);
      if (c == COEF_SOFTCORE) RUN(COEF_SOFTCORE, LINK_PLANE_ZX);
      if (c == COEF_SOFTCORR) RUN(COEF_SOFTCORR, LINK_PLANE_ZX);
      RUN(kAnyMode, kAnyMode);
    }
  }
  if (c == COEF_SOFTCORE) {
    if (l == LINK_NONE) RUN(COEF_SOFTCORE, LINK_NONE);
    if (l == LINK_PLANE) RUN(COEF_SOFTCORE, LINK_PLANE);
    // (the run-time path takes one value at a time and each loads the pair's link
    // record: 96^3 574 us per step, 224 so; 512^2 42 and 22.5)
    if (l == LINK_TABLE) RUN(COEF_SOFTCORE, LINK_TABLE);
    RUN(kAnyMode, kAnyMode);
  }
  if (c == COEF_SOFTCORR) {
    if (l == LINK_NONE) RUN(COEF_SOFTCORR, LINK_NONE);
    if (l == LINK_PLANE) RUN(COEF_SOFTCORR, LINK_PLANE);
    RUN(kAnyMode, kAnyMode);
  }
  if (l == LINK_TABLE) {
    if (c == COEF_UNIFORM) RUN(COEF_UNIFORM, LINK_TABLE);
    if (c == COEF_STEP) RUN(COEF_STEP, LINK_TABLE);
    RUN(COEF_TABLE, LINK_TABLE);
  }
  if (c == COEF_TABLE && l == LINK_NONE) RUN(COEF_TABLE, LINK_NONE);
  if (c == COEF_TABLE && l == LINK_PLANE) RUN(COEF_TABLE, LINK_PLANE);
  if (c == COEF_TABLE) RUN(kAnyMode, kAnyMode);
  if (c == COEF_UNIFORM && l == LINK_PLANE) RUN(COEF_UNIFORM, LINK_PLANE);
  if (c == COEF_STEP && l == LINK_PLANE) RUN(COEF_STEP, LINK_PLANE);
  if (c == COEF_UNIFORM && l == LINK_NONE) RUN(COEF_UNIFORM, LINK_NONE);
  if (c == COEF_STEP && l == LINK_NONE) RUN(COEF_STEP, LINK_NONE);
  if (c == COEF_UNIFORM && l == LINK_CONST) RUN(COEF_UNIFORM, LINK_CONST);
  RUN(COEF_STEP, LINK_CONST);
#undef RUN
}

template <int DIMS, int kT, int COEF, int LINK>
void batch_dims(const BatchArgs<F32>& b, long long total, bool iso, cudaStream_t s) {
  if constexpr (DIMS == 3) {
    if (iso) launch3d_batch<COEF, LINK, true>(b, total, s);
    else launch3d_batch<COEF, LINK, false>(b, total, s);
  } else {
    if (iso) launch2d_batch<COEF, LINK, kT, true>(b, total, s);
    else launch2d_batch<COEF, LINK, kT, false>(b, total, s);
  }
}
template <int DIMS, int kT>
void dispatch_batch(const BatchArgs<F32>& b, long long total, int coef, int link, bool iso, cudaStream_t s) {
  if (coef == COEF_UNIFORM && link == LINK_NONE) batch_dims<DIMS, kT, COEF_UNIFORM, LINK_NONE>(b, total, iso, s);
  else if (coef == COEF_STEP && link == LINK_NONE) batch_dims<DIMS, kT, COEF_STEP, LINK_NONE>(b, total, iso, s);
  else if (coef == COEF_UNIFORM && link == LINK_CONST) batch_dims<DIMS, kT, COEF_UNIFORM, LINK_CONST>(b, total, iso, s);
  else batch_dims<DIMS, kT, COEF_STEP, LINK_CONST>(b, total, iso, s);
}

ChunkShape shape_of(int dims, const int N[3], int steps) { return dims == 3 ? shape3d(N) : shape2d(N, steps); }

}  // namespace

int launch_fused2d_two(const FusedArgs<F32>& a, cudaStream_t s) { return dispatch<2, 2>(a, s); }

int fused_candidates(int dims, const int N[3], int steps, int* out, int max) {
  const ChunkShape g = shape_of(dims, N, steps);
  return rank_chunks(g.tiles, g.levels, g.workers, g.min_chunk, g.restart, out, max);
}

long long fused_items(int dims, const int N[3], int steps, int chunk) {
  const ChunkShape g = shape_of(dims, N, steps);
  return g.tiles * ((g.levels + chunk - 1) / chunk);
}

// Chunks of a batched launch.  Each simulation's own rule cuts it into enough
// items to fill the GPU alone, at the price of an extra first level per item
// (64^3: items of 3 levels); together they need far fewer.  So one target length
// for all: the one whose rounds (items in order, `workers` at a time, each round
// as long as its longest item and the restart) add up to the least.  Eight
// residents of 64^3 .. 160^3 and 192^2 .. 576^2: 248 us per step, now 239
void fused_batch_chunks(int dims, const int* const* N, int n, int steps, int* chunk) {
  std::vector<ChunkShape> g(n);
  int longest = 0;
  for (int i = 0; i < n; ++i) {
    g[i] = shape_of(dims, N[i], steps);
    longest = std::max(longest, g[i].levels);
  }
  if (n == 1) {
    if (chunk[0] <= 0) chunk[0] = plan_chunk(g[0]);
    return;
  }
  auto length = [&](int i, int target) {  // the target's nearest even split of the levels
    if (chunk[i] > 0) return chunk[i];
    const int parts = (g[i].levels + target - 1) / target;
    return (g[i].levels + parts - 1) / parts;
  };
  const long long workers = g[0].workers;
  const double restart = g[0].restart;
  int best = longest, prev = 0;
  double best_time = 0.0;
  for (int parts = 1; parts <= 256; ++parts) {
    const int target = (longest + parts - 1) / parts;
    if (target == prev) continue;
    if (target < g[0].min_chunk && parts > 1) break;
    prev = target;
    double time = 0.0;
    long long used = 0;  // workers taken in the open round
    int open = 0;        // its longest item
    for (int i = 0; i < n; ++i) {
      const int len = length(i, target);
      long long items = g[i].tiles * ((g[i].levels + len - 1) / len);
      const long long first = std::min(items, workers - used);
      open = std::max(open, len);
      used += first;
      items -= first;
      if (used < workers) continue;
      time += (open + restart) + (double)(items / workers) * (len + restart);
      used = items % workers;
      open = used ? len : 0;
    }
    if (open) time += open + restart;
    if (best_time == 0.0 || time < best_time * 0.9999) best_time = time, best = target;
  }
  for (int i = 0; i < n; ++i) chunk[i] = length(i, best);
}

void launch_fused_batch(const BatchArgs<F32>& b, int dims, int steps, long long total, int coef, int link, bool iso,
                        cudaStream_t s) {
  if (dims == 3) dispatch_batch<3, 1>(b, total, coef, link, iso, s);
  else if (steps == 2) dispatch_batch<2, 2>(b, total, coef, link, iso, s);
  else dispatch_batch<2, 1>(b, total, coef, link, iso, s);
}

template <>
int launch_fused<F32, 3>(const FusedArgs<F32>& a, cudaStream_t s) {
  return dispatch<3, 1>(a, s);
}
template <>
int launch_fused<F32, 2>(const FusedArgs<F32>& a, cudaStream_t s) {
  return dispatch<2, 1>(a, s);
}

}  // namespace dirac
