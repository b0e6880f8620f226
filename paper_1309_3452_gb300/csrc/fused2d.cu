// The fused (2+1)D kernels: one time step per pass, two steps per pass, and the
// batched forms of both (see fused3d.cuh for the state's layout and the
// scheduling, which they share).
//
// (2+1)D: each warp owns a strip of 32 cells in x (30 interior) and marches
// along y with the same pipeline (u0 ~ A, u1 ~ B, v1 ~ C, v0 ~ D with y as the
// marching axis); x neighbours come from warp shuffles, no block barrier.
#include "fused_common.cuh"

namespace dirac {
namespace fused {

namespace {

__device__ __forceinline__ float2 shfl_up1(float2 v) {
  return make_float2(__shfl_up_sync(0xffffffffu, v.x, 1), __shfl_up_sync(0xffffffffu, v.y, 1));
}
__device__ __forceinline__ float2 shfl_down1(float2 v) {
  return make_float2(__shfl_down_sync(0xffffffffu, v.x, 1), __shfl_down_sync(0xffffffffu, v.y, 1));
}

// work items of a (2+1)D one-step launch: strips x chunks of the `rows` updated rows
__host__ __device__ __forceinline__ long long items2d(const int (&N)[3], int rows, int chunk) {
  return (long long)((N[0] + kCore - 1) / kCore) * ((rows + chunk - 1) / chunk);
}

// One row of the (2+1)D pipeline at march position k.  In: U = the old u0 of
// row k+1 (lane 0) and u1 of row k (lane 1); V, Vn = the old v records of rows
// k and k+1; nU0, nU1 = the new u0 of row k and u1 of row k-1.  Out: nU = the
// new u0 of row k+1 (lane 0) and u1 of row k (lane 1), nV = the new v record of
// row k and its difference part S.  Sublattices: u0 (0,0), u1 (1,1), v0 (1,0),
// v1 (0,1).
template <class P, int COEF, int LINK>
__device__ __forceinline__ void row2d(const FusedArgs<P>& a, bool iso, int hx, int yk, int yn, long long ok,
                                      long long on, const Quad& U, const Quad& V, const Quad& Vn, float2 nU0,
                                      float2 nU1, Quad& nU, Quad& nV, Quad* S) {
  const float2 v0n = qlane(Vn, 0), v1n = qlane(Vn, 1), v0 = qlane(V, 0), v1 = qlane(V, 1);
  {  // u0(k+1) from v0(k+1) (x), v1(k+1), v1(k) (y); u1(k) from v1(k) (x), v0(k+1), v0(k) (y)
    Quad up[3], dn[3];
    up[0] = mkquad(v0n, shfl_down1(v1));
    dn[0] = mkquad(shfl_up1(v0n), v1);
    up[1] = mkquad(v1n, v0n);
    dn[1] = mkquad(v1, v0);
    const int H0[3] = {hx, 2 * yn, 0}, H1[3] = {hx + 1, 2 * yk + 1, 0};
    nU = quad_update<2, COEF, LINK, false>(a.hu, a.f, iso, a.ry, a.rz, 0, U, up, dn, H0, H1, on, ok, a.pstride,
                                           nullptr, nullptr, nullptr, a.N);
  }
  {  // v0(k) from u0(k) (x), u1(k), u1(k-1) (y); v1(k) from u1(k) (x), u0(k+1), u0(k) (y)
    const float2 u0n = qlane(nU, 0), u1k = qlane(nU, 1);
    Quad up[3], dn[3];
    up[0] = mkquad(shfl_down1(nU0), u1k);
    dn[0] = mkquad(nU0, shfl_up1(u1k));
    up[1] = mkquad(u1k, u0n);
    dn[1] = mkquad(nU1, nU0);
    const int H0[3] = {hx + 1, 2 * yk, 0}, H1[3] = {hx, 2 * yk + 1, 0};
    nV = quad_update<2, COEF, LINK, true>(a.hl, a.f, iso, a.ry, a.rz, 1, V, up, dn, H0, H1, ok, ok, a.pstride, S,
                                          nullptr, nullptr, a.N);
  }
}

// the functional's terms of one (2+1)D row: new u1 and v of the row
__device__ __forceinline__ void row_terms(float2 u1, const Quad& V, const Quad& S, double& e_n, double& e_c) {
  e_n += (n2(u1) + n2(qlane(V, 0))) + n2(qlane(V, 1));
  e_c += fmaf(V.re.y, S.re.y, fmaf(V.im.y, S.im.y, fmaf(V.re.x, S.re.x, V.im.x * S.im.x)));
}

// One work item (one 32-cell strip over one chunk of rows) of one simulation,
// processed by one warp.
template <class P, int COEF, int LINK>
__device__ __forceinline__ void fused2d_item(const FusedArgs<P>& a, long long item, int lane, double& e_n,
                                             double& e_c) {
  const int Nx = a.N[0], Ny = a.N[1];
  const int strips = (Nx + kCore - 1) / kCore;
  const bool iso = a.iso != 0;
  const long long chunk = item / strips;
  const int strip = (int)(item - chunk * strips);
  // the updated rows zlo .. zlo + nzu - 1 (all rows of a whole grid, a slab's
  // own rows); fields at the global row (zorg + k, wrapped: in [-1, 2 Nzg))
  const int y0 = a.zlo + (int)chunk * a.chunk;
  const int y1 = min(a.zlo + a.nzu, y0 + a.chunk);
  auto gy = [&](int k) {
    const int g = a.zorg + k;
    return g < 0 ? g + a.Nzg : (g >= a.Nzg ? g - a.Nzg : g);
  };
  const int gx = strip * kCore + lane - 1;
  const int x = wrapi(gx, Nx);
  const bool core = lane >= 1 && lane <= kCore && gx < Nx;
  const int hx = 2 * x;
  // the loads of row k: the u and v records of row k+1 (u1 of row k comes from the row before)
  auto load = [&](int k, Quad& u, Quad& v) {
    const int yn = k + 1 >= Ny ? k + 1 - Ny : (k + 1 < 0 ? k + 1 + Ny : k + 1);
    const long long on = (long long)yn * Nx + x;
    u = ldq(a.in[0] + on);
    v = ldq(a.in[1] + on);
  };
  Quad V, Vn, Un;
  float2 u1;  // old u1 of row k
  {
    const long long o = (long long)wrapi(y0 - 1, Ny) * Nx + x;
    V = ldq(a.in[1] + o);
    u1 = qlane(ldq(a.in[0] + o), 1);
  }
  float2 nU0 = qlane(V, 0), nU1 = nU0;  // placeholders: only feed values never stored
  load(y0 - 1, Un, Vn);
  for (int k = y0 - 1; k < y1; ++k) {
    const int yk = k < 0 ? k + Ny : k;
    const int yn = k + 1 >= Ny ? k + 1 - Ny : k + 1;
    const long long ok = (long long)yk * Nx + x, on = (long long)yn * Nx + x;
    Quad pU = Un, pV = Vn;  // next row, loaded while this one computes
    if (k + 1 < y1) load(k + 1, pU, pV);
    Quad nU, nV, S;
    row2d<P, COEF, LINK>(a, iso, hx, gy(k), gy(k + 1), ok, on, mkquad(qlane(Un, 0), u1), V, Vn, nU0, nU1, nU, nV, &S);
    if (core && k >= y0) {
      a.out[0][ok] = pack4(mkquad(nU0, qlane(nU, 1)));  // the row's new u0 (formed one row earlier) and u1
      a.out[1][ok] = pack4(nV);
      if (a.e_partials) {
        row_terms(qlane(nU, 1), nV, S, e_n, e_c);
        e_n += n2(nU0);
      }
    }
    nU0 = qlane(nU, 0);
    nU1 = qlane(nU, 1);
    u1 = qlane(Un, 1);
    V = Vn;
    Un = pU;
    Vn = pV;
  }
}

// Two time steps per pass ((2+1)D, fields without time dependence).  Step 1
// runs the row pipeline on the old state; step 2 runs it one row behind on
// step 1's results, which never leave registers.  A strip keeps 28 interior
// lanes (lanes 2..29): step 1 is valid on lanes 1..30, step 2 on 2..29.
// Step 1 starts two rows and step 2 one row before the chunk.
constexpr int kCoreTb = 28;

template <class P, int COEF, int LINK>
__device__ __forceinline__ void fused2d_tb2_item(const FusedArgs<P>& a, long long item, int lane,
                                                 double& e_n, double& e_c) {
  const int Nx = a.N[0], Ny = a.N[1];
  const int strips = (Nx + kCoreTb - 1) / kCoreTb;
  const bool iso = a.iso != 0;
  const long long chunk = item / strips;
  const int strip = (int)(item - chunk * strips);
  const int y0 = (int)chunk * a.chunk;
  const int y1 = min(Ny, y0 + a.chunk);
  const int gx = strip * kCoreTb + lane - 2;
  const int x = wrapi(gx, Nx);
  const bool core = lane >= 2 && lane <= kCoreTb + 1 && gx < Nx;
  const int hx = 2 * x;
  auto wrapy = [&](int k) { return k < 0 ? k + Ny : (k >= Ny ? k - Ny : k); };
  auto load = [&](int k, Quad& u, Quad& v) {
    const long long on = (long long)wrapy(k + 1) * Nx + x;
    u = ldq(a.in[0] + on);
    v = ldq(a.in[1] + on);
  };
  // step-1 pipeline state: old v and u1 of row k; new u0 of row k, u1 of row k-1
  Quad V, Vn, Un;
  float2 u1;
  {
    const long long o = (long long)wrapy(y0 - 2) * Nx + x;
    V = ldq(a.in[1] + o);
    u1 = qlane(ldq(a.in[0] + o), 1);
  }
  float2 nU0 = qlane(V, 0), nU1 = nU0;  // placeholders: only feed values never stored
  // step-2 pipeline state: step-1 v of row k-1; step-2 u0 of row k-1, u1 of row k-2
  Quad qV = V;
  float2 mU0 = nU0, mU1 = nU0;
  load(y0 - 2, Un, Vn);
  for (int k = y0 - 2; k <= y1; ++k) {
    const int yk = wrapy(k), yn = wrapy(k + 1);
    const long long ok = (long long)yk * Nx + x, on = (long long)yn * Nx + x;
    Quad pU = Un, pV = Vn;
    if (k + 1 <= y1) load(k + 1, pU, pV);
    // step 1 at row k
    Quad sU, sV;
    row2d<P, COEF, LINK>(a, iso, hx, yk, yn, ok, on, mkquad(qlane(Un, 0), u1), V, Vn, nU0, nU1, sU, sV, nullptr);
    if (k >= y0) {
      // step 2 at row k-1: its old u0 of row k and u1 of row k-1 and v of rows k-1, k are step 1's
      const int ym = wrapy(k - 1);
      const long long om = (long long)ym * Nx + x;
      Quad tU, tV, S;
      row2d<P, COEF, LINK>(a, iso, hx, ym, yk, om, ok, mkquad(nU0, nU1), qV, sV, mU0, mU1, tU, tV, &S);
      if (core && k - 1 >= y0) {
        a.out[0][om] = pack4(mkquad(mU0, qlane(tU, 1)));
        a.out[1][om] = pack4(tV);
        if (a.e_partials) {
          row_terms(qlane(tU, 1), tV, S, e_n, e_c);
          e_n += n2(mU0);
        }
      }
      mU0 = qlane(tU, 0);
      mU1 = qlane(tU, 1);
    }
    qV = sV;  // step-1 v of row k becomes step 2's old row
    nU0 = qlane(sU, 0);
    nU1 = qlane(sU, 1);
    u1 = qlane(Un, 1);
    V = Vn;
    Un = pU;
    Vn = pV;
  }
}

template <class P, int COEF, int LINK>
__global__ void __launch_bounds__(32 * kFused2dWarps) fused2d_kernel(const FusedArgs<P> a) {
  const int lane = threadIdx.x & 31;
  const long long worker = (long long)blockIdx.x * kFused2dWarps + (threadIdx.x >> 5);
  const long long items = items2d(a.N, a.nzu, a.chunk);
  double e_n = 0.0, e_c = 0.0;
  for (long long item = worker; item < items; item += a.workers)  // uniform per warp
    fused2d_item<P, COEF, LINK>(a, item, lane, e_n, e_c);
  if (a.e_partials) block_store_e(e_n, e_c, a.e_partials);
}

template <class P, int COEF, int LINK>
__global__ void __launch_bounds__(32 * kFused2dWarps) fused2d_tb2_kernel(const FusedArgs<P> a) {
  const int lane = threadIdx.x & 31;
  const long long worker = (long long)blockIdx.x * kFused2dWarps + (threadIdx.x >> 5);
  const long long items = (long long)((a.N[0] + kCoreTb - 1) / kCoreTb) * ((a.N[1] + a.chunk - 1) / a.chunk);
  double e_n = 0.0, e_c = 0.0;
  for (long long item = worker; item < items; item += a.workers)  // uniform per warp
    fused2d_tb2_item<P, COEF, LINK>(a, item, lane, e_n, e_c);
  if (a.e_partials) block_store_e(e_n, e_c, a.e_partials);
}

template <class P, int COEF, int LINK>
__global__ void __launch_bounds__(32 * kFused2dWarps) fused2d_batch_kernel(const BatchArgs<P> b) {
  __shared__ FusedArgs<P> sa[kFused2dWarps];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long long worker = (long long)blockIdx.x * kFused2dWarps + w;
  const long long total = b.first_item[b.nsims];
  int cur = -1;
  for (long long g = worker; g < total; g += b.workers) {
    const int s = find_sim(b.first_item, b.nsims, g);
    if (s != cur) {
      __syncwarp();
      copy_args(&sa[w], b.sims + s, lane, 32);
      __syncwarp();
      cur = s;
    }
    double e_n = 0.0, e_c = 0.0;  // (batched launches never accumulate the functional)
    fused2d_item<P, COEF, LINK>(sa[w], g - b.first_item[s], lane, e_n, e_c);
  }
}

// Two time steps per pass for several (2+1)D simulations (time-independent
// fields): as fused2d_batch_kernel with the two-step item of each simulation.
template <class P, int COEF, int LINK>
__global__ void __launch_bounds__(32 * kFused2dWarps) fused2d_tb2_batch_kernel(const BatchArgs<P> b) {
  __shared__ FusedArgs<P> sa[kFused2dWarps];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long long worker = (long long)blockIdx.x * kFused2dWarps + w;
  const long long total = b.first_item[b.nsims];
  int cur = -1;
  for (long long g = worker; g < total; g += b.workers) {
    const int s = find_sim(b.first_item, b.nsims, g);
    if (s != cur) {
      __syncwarp();
      copy_args(&sa[w], b.sims + s, lane, 32);
      __syncwarp();
      cur = s;
    }
    double e_n = 0.0, e_c = 0.0;  // (batched launches never accumulate the functional)
    fused2d_tb2_item<P, COEF, LINK>(sa[w], g - b.first_item[s], lane, e_n, e_c);
  }
}

// resident warps of a kernel, computed once
template <auto K>
int workers2d() {
  static int r = resident_blocks(K, 32 * kFused2dWarps) * kFused2dWarps;
  return r;
}

}  // namespace

template <int COEF, int LINK>
int launch2d(FusedArgs<F32> a, cudaStream_t s) {
  auto k = fused2d_kernel<F32, COEF, LINK>;
  const int warps = workers2d<fused2d_kernel<F32, COEF, LINK>>();
  if (a.chunk <= 0 || a.chunk > a.nzu) {
    const int Np[3] = {a.N[0], a.nzu, 1};
    a.chunk = plan_chunk(shape2d(Np));
  }
  const long long items = items2d(a.N, a.nzu, a.chunk);
  long long w = items < warps ? items : warps;
  // one E partial per block: never more blocks than the partials hold
  if (a.e_partials && w > (long long)kFusedEMaxBlocks * kFused2dWarps) w = (long long)kFusedEMaxBlocks * kFused2dWarps;
  a.workers = (int)w;
  const int blocks = (int)((w + kFused2dWarps - 1) / kFused2dWarps);
  k<<<(unsigned)blocks, 32 * kFused2dWarps, 0, s>>>(a);
  return blocks;
}

template <int COEF, int LINK>
void launch2d_batch(BatchArgs<F32> b, long long total, cudaStream_t s) {
  auto k = fused2d_batch_kernel<F32, COEF, LINK>;
  const int warps = workers2d<fused2d_batch_kernel<F32, COEF, LINK>>();
  const long long w = total < warps ? total : warps;
  b.workers = (int)w;
  k<<<(unsigned)((w + kFused2dWarps - 1) / kFused2dWarps), 32 * kFused2dWarps, 0, s>>>(b);
}

template <int COEF, int LINK>
void launch2d_tb2_batch(BatchArgs<F32> b, long long total, cudaStream_t s) {
  auto k = fused2d_tb2_batch_kernel<F32, COEF, LINK>;
  const int warps = workers2d<fused2d_tb2_batch_kernel<F32, COEF, LINK>>();
  const long long w = total < warps ? total : warps;
  b.workers = (int)w;
  k<<<(unsigned)((w + kFused2dWarps - 1) / kFused2dWarps), 32 * kFused2dWarps, 0, s>>>(b);
}

template <int COEF, int LINK>
int launch2d_tb2(FusedArgs<F32> a, cudaStream_t s) {
  auto k = fused2d_tb2_kernel<F32, COEF, LINK>;
  const int warps = workers2d<fused2d_tb2_kernel<F32, COEF, LINK>>();
  const long long strips = (a.N[0] + kCoreTb - 1) / kCoreTb;
  if (a.chunk <= 0 || a.chunk > a.N[1]) a.chunk = plan_chunk(shape2d_tb2(a.N));
  const long long items = strips * ((a.N[1] + a.chunk - 1) / a.chunk);
  long long w = items < warps ? items : warps;
  if (a.e_partials && w > (long long)kFusedEMaxBlocks * kFused2dWarps) w = (long long)kFusedEMaxBlocks * kFused2dWarps;
  a.workers = (int)w;
  const int blocks = (int)((w + kFused2dWarps - 1) / kFused2dWarps);
  k<<<(unsigned)blocks, 32 * kFused2dWarps, 0, s>>>(a);
  return blocks;
}

ChunkShape shape2d(const int N[3]) {
  return {(N[0] + kCore - 1) / kCore, N[1], workers2d<fused2d_kernel<F32, COEF_UNIFORM, LINK_NONE>>(), 16, 1.0};
}
ChunkShape shape2d_tb2(const int N[3]) {
  return {(N[0] + kCoreTb - 1) / kCoreTb, N[1], workers2d<fused2d_tb2_kernel<F32, COEF_UNIFORM, LINK_NONE>>(), 32, 1.0};
}

#define STEP_2D(COEF, LINK) template int launch2d<COEF, LINK>(FusedArgs<F32>, cudaStream_t);
STEP_2D(COEF_UNIFORM, LINK_NONE)
STEP_2D(COEF_UNIFORM, LINK_PLANE)
STEP_2D(COEF_STEP, LINK_NONE)
STEP_2D(COEF_STEP, LINK_PLANE)
STEP_2D(COEF_TABLE, LINK_NONE)
STEP_2D(COEF_TABLE, LINK_PLANE)
STEP_2D(COEF_SOFTCORE, LINK_NONE)
STEP_2D(COEF_SOFTCORE, LINK_PLANE)
STEP_2D(COEF_SOFTCORR, LINK_NONE)
STEP_2D(COEF_SOFTCORR, LINK_PLANE)
STEP_2D(COEF_UNIFORM, LINK_CONST)
STEP_2D(COEF_STEP, LINK_CONST)
STEP_2D(COEF_UNIFORM, LINK_TABLE)
STEP_2D(COEF_STEP, LINK_TABLE)
STEP_2D(COEF_TABLE, LINK_TABLE)
STEP_2D(kAnyMode, kAnyMode)
#define STEPS_2D(COEF, LINK) template int launch2d_tb2<COEF, LINK>(FusedArgs<F32>, cudaStream_t);
STEPS_2D(COEF_UNIFORM, LINK_NONE)
STEPS_2D(COEF_STEP, LINK_NONE)
STEPS_2D(COEF_UNIFORM, LINK_CONST)
STEPS_2D(COEF_STEP, LINK_CONST)
STEPS_2D(COEF_TABLE, LINK_NONE)
STEPS_2D(COEF_SOFTCORE, LINK_NONE)
STEPS_2D(COEF_SOFTCORR, LINK_NONE)
#define BATCH_2D(COEF, LINK)                                                     \
  template void launch2d_batch<COEF, LINK>(BatchArgs<F32>, long long, cudaStream_t); \
  template void launch2d_tb2_batch<COEF, LINK>(BatchArgs<F32>, long long, cudaStream_t);
BATCH_2D(COEF_UNIFORM, LINK_NONE)
BATCH_2D(COEF_UNIFORM, LINK_CONST)
BATCH_2D(COEF_STEP, LINK_NONE)
BATCH_2D(COEF_STEP, LINK_CONST)

}  // namespace fused
}  // namespace dirac
