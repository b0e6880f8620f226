// The fused (2+1)D kernels: kT time steps per pass (1 or 2), for one
// simulation or a batch of them (see fused3d.cuh for the state's layout and the
// scheduling, which they share).
//
// Each warp owns a strip of 32 cells in x (32 - 2 kT interior) and marches along
// y with the (3+1)D kernels' pipeline (u0 ~ A, u1 ~ B, v1 ~ C, v0 ~ D with y as
// the marching axis); x neighbours come from warp shuffles, no block barrier.
// Stage s of a pass runs step s + 1 two rows behind stage s - 1 on its results,
// which never leave registers: a pass reads and writes the state once for kT
// steps, and the stages of one march position are independent chains of
// arithmetic.  Every step loses one lane and one row per side, so the arithmetic
// grows by 32 / (32 - 2 kT) and the restart of an item by kT rows.
//
// Bound: instruction issue (147 thread instructions per cell and step, 66 % of
// the issue slots, FP32 pipe 50 %, ALU 41 %; HBM at 68 % of its peak).  us per
// step with one warp row of (re, im) lanes per value / with quads and stages waiting for one another /
// now: 4096^2 Klein step 138 / 131 / 95, 1000^2 moving plane wave 35.0 / 26.8 /
// 13.5 (one step per pass before), 300 x 260 constant A 16.8 / 13.7 / 3.1 (blocks of
// eight warps and chunks of 32 rows left most SMs idle).  Four steps per pass
// were measured too: 4096^2 103 (spills or 8 warps per SM), 300 x 260 2.95.
#pragma once

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

// blocks per SM that the registers are planned for.  Two steps per pass: 16 warps
// of up to 128 registers (5 blocks: 4096^2 280 us per step instead of 95, the
// stages' chains spill; 3: the plane wave at 1000^2 26.3 instead of 22.5); links
// with per-value factors keep 168.
constexpr int min_blocks(int steps, int coef, int link) {
  return steps == 2 ? (link == LINK_NONE || link == LINK_PLANE ? 4 : 3) : (link == LINK_TABLE ? 4 : 6);
}
// rows of a strip in flight or at hand (u and v records of 32 lanes each)
constexpr int kRing = 4;
constexpr int kWaveRows = 8;
// float4 of shared memory per warp: the rows, a Klein step's coefficients per
// lane, a plane wave's factors
template <int COEF, int LINK>
constexpr int warp_slots() {
  return kRing * 64 + (COEF == COEF_STEP || COEF == COEF_STEP_X || COEF == COEF_LANES ? 256 : 0) +
         (LINK == LINK_PLANE ? 256 : 0);
}
// interior lanes of a strip, and strips of a grid
template <int kT>
constexpr int core_lanes() { return 32 - 2 * kT; }
template <int kT>
__host__ __device__ __forceinline__ int strips2d(int Nx) { return (Nx + core_lanes<kT>() - 1) / core_lanes<kT>(); }

// Where a row's plane-wave link factors are (LINK_PLANE): of u0 (row + 1), u1, v0, v1
struct WaveAt {
  const float4 *u0, *u1, *v0, *v1;
};

// One row of the (2+1)D pipeline at march position k.  In: U = the old u0 of
// row k+1 (lane 0) and u1 of row k (lane 1); V, Vn = the old v records of rows
// k and k+1; nU0, nU1 = the new u0 of row k and u1 of row k-1.  Out: nU = the
// new u0 of row k+1 (lane 0) and u1 of row k (lane 1), nV = the new v record of
// row k and its difference part S.  Sublattices: u0 (0,0), u1 (1,1), v0 (1,0),
// v1 (0,1).
template <class P, int COEF, int LINK, bool kIso>
__device__ __forceinline__ void row2d(const FusedArgs<P>& a, bool iso, int hx, int yk, int yn, long long ok,
                                      long long on, long long ck, long long cn, const Quad& U, const Quad& V, const Quad& Vn, float2 nU0,
                                      float2 nU1, const float4* lanes, const WaveAt& w, Quad& nU, Quad& nV, Quad* S) {
  const float2 v0n = qlane(Vn, 0), v1n = qlane(Vn, 1), v0 = qlane(V, 0), v1 = qlane(V, 1);
  {  // u0(k+1) from v0(k+1) (x), v1(k+1), v1(k) (y); u1(k) from v1(k) (x), v0(k+1), v0(k) (y)
    Quad up[3], dn[3];
    up[0] = mkquad(v0n, shfl_down1(v1));
    dn[0] = mkquad(shfl_up1(v0n), v1);
    up[1] = mkquad(v1n, v0n);
    dn[1] = mkquad(v1, v0);
    const int H0[3] = {hx, 2 * yn, 0}, H1[3] = {hx + 1, 2 * yk + 1, 0};
    nU = quad_update<2, COEF, LINK, false, kIso>(a.hu, a.f, iso, a.ry, a.rz, 0, U, up, dn, H0, H1, on, ok, cn, ck, a.pstride,
                                           nullptr, nullptr, nullptr, a.N, lanes, w.u0, w.u1);
  }
  {  // v0(k) from u0(k) (x), u1(k), u1(k-1) (y); v1(k) from u1(k) (x), u0(k+1), u0(k) (y)
    const float2 u0n = qlane(nU, 0), u1k = qlane(nU, 1);
    Quad up[3], dn[3];
    up[0] = mkquad(shfl_down1(nU0), u1k);
    dn[0] = mkquad(nU0, shfl_up1(u1k));
    up[1] = mkquad(u1k, u0n);
    dn[1] = mkquad(nU1, nU0);
    const int H0[3] = {hx + 1, 2 * yk, 0}, H1[3] = {hx, 2 * yk + 1, 0};
    nV = quad_update<2, COEF, LINK, true, kIso>(a.hl, a.f, iso, a.ry, a.rz, 1, V, up, dn, H0, H1, ok, ok, ck, ck, a.pstride, S,
                                          nullptr, nullptr, a.N, lanes + 128, w.v0, w.v1);
  }
}

// One work item (one strip over one chunk of rows) of one simulation, processed
// by one warp: kT time steps of the chunk's rows.
// kStepSlots: a Klein step's coefficients lie between the rows and the wave's factors
template <class P, int COEF, int LINK, int kT, bool kIso, int kStepSlots>
__device__ __forceinline__ void march2d(const FusedArgs<P>& a, float4* ring, int strip, long long chunk, int lane,
                                        double& e_n, double& e_c) {
  const int Nx = a.N[0], Ny = a.N[1];
  const bool iso = a.iso != 0;
  // the updated rows zlo .. zlo + nzu - 1 (all rows of a whole grid, a slab's
  // own rows; kT = 2: whole grids of at least four rows); fields at the global
  // row (zorg + k, wrapped: in [-kT, 2 Nzg))
  const int y0 = a.zlo + (int)chunk * a.chunk;
  const int y1 = min(a.zlo + a.nzu, y0 + a.chunk);
  auto gy = [&](int k) {
    const int g = a.zorg + k;
    return g < 0 ? g + a.Nzg : (g >= a.Nzg ? g - a.Nzg : g);
  };
  auto stored = [&](int k) { return k < 0 ? k + Ny : (k >= Ny ? k - Ny : k); };
  const int gx = strip * core_lanes<kT>() + lane - kT;
  const int x = wrapi(gx, Nx);
  const bool core = lane >= kT && lane < 32 - kT && gx < Nx;
  const int hx = 2 * x;
  using Off = unsigned;  // (a level has fewer than 2^31 cells)
  auto off = [&](int k) { return (Off)stored(k) * (Off)Nx + (Off)x; };
  auto class_of = [&](int k) -> long long {  // (COEF_TABLE)
    if constexpr (COEF == COEF_TABLE) return __ldg(a.hu.b_map + x) + __ldg(a.hu.b_map + Nx + stored(k));
    else return 0;
  };
  const float4* lanes = ring + kRing * 64 + lane;  // (COEF_LANES)
  // LINK_PLANE: the factors from the steps' tables, [stage][half][parity of the
  // half-lattice coordinate].  A wave along y has the same ones for the whole
  // row: they travel with the rows (loaded where they are used, an L2 latency
  // per row and stage is exposed: 1000^2 22.5 us per step against 16.6), kWaveRows
  // rows since stage 1 is two rows behind.  A wave along x: a lane's own, kept
  // through the march
  float4* wave = ring + kRing * 64 + 256 * kStepSlots;
  const bool wave_y = a.hu.ltab_axis == 1;
  auto wave_entry = [&](int e, int H) {  // e = 4 stage + 2 half + parity
    const PlaneLink32* t = static_cast<const PlaneLink32*>((e & 2) ? a.hl.ltab : a.hu.ltab);
    return &t[(e >> 2) * a.lstep + H + (e & 1)].v;
  };
  auto wave_at = [&](int s, int r) {
    WaveAt w{};
    if constexpr (LINK == LINK_PLANE) {
      const int row = wave_y ? 1 : 0, step = wave_y ? 1 : 32;
      const float4* here = wave + (wave_y ? (r & (kWaveRows - 1)) * 8 : lane) + 4 * s * step;
      const float4* above = wave_y ? wave + ((r + 1) & (kWaveRows - 1)) * 8 + 4 * s : here;
      w = WaveAt{above, here + step, here + (row ? 2 : 3) * step, here + (row ? 3 : 2) * step};
    }
    return w;
  };
  // State of stage s, which processes row r = k - 2 s at march position k, on
  // what stage s - 1 left in earlier positions (so the stages of one position
  // do not wait for one another): the old v of rows r and r + 1, the old u0 of
  // row r + 1 and u1 of row r, the new u0 of row r and u1 of row r - 1.  (Values
  // before a stage's first row only feed values that are never stored.)
  Quad V[kT], Vn[kT], U[kT];
  float2 nU0[kT], nU1[kT];
  const int k0 = y0 - kT;
  // the last position in which stage s has a row to do is kl + s; stage 0 reads
  // rows up to kl + 1
  const int kl = y1 + kT - 2;
  // rows ahead travel through shared memory by copies that bypass the registers
  // (loads into registers end up waited for within a position: the compiler
  // sinks them towards their use)
  auto fetch = [&](int row) {
    if (row <= kl + 1) {
      const Off o = off(row);
      float4* slot = ring + (row & (kRing - 1)) * 64 + lane;
      cp_async16(slot, a.in[0] + o);
      cp_async16(slot + 32, a.in[1] + o);
      if (LINK == LINK_PLANE && wave_y && lane < 4 * kT)
        cp_async16(wave + (row & (kWaveRows - 1)) * 8 + lane, wave_entry(lane, 2 * gy(row)));
    }
    cp_async_commit();
  };
  if (LINK == LINK_PLANE) {
    if (wave_y) {
      if (lane < 4 * kT) wave[(k0 & (kWaveRows - 1)) * 8 + lane] = *wave_entry(lane, 2 * gy(k0));
    } else {
#pragma unroll
      for (int e = 0; e < 4 * kT; ++e) wave[e * 32 + lane] = *wave_entry(e, hx);  // (ordinary loads, as ldq)
    }
  }
#pragma unroll
  for (int j = 1; j < kRing; ++j) fetch(k0 + j);
  {
    const Off o = off(k0);
    Vn[0] = ldq(a.in[1] + o);
    const Quad u = ldq(a.in[0] + o);
    U[0] = u;
    nU0[0] = nU1[0] = qlane(u, 1);
#pragma unroll
    for (int s = 1; s < kT; ++s) {
      V[s] = Vn[s] = U[s] = u;
      nU0[s] = nU1[s] = qlane(u, 1);
    }
  }
  float2 u1 = nU1[0];  // the old u1 of row k
  Quad oU, oV, oS;     // the last stage's new row and its difference part
  auto stage = [&](auto sc, int k) {
    constexpr int s = decltype(sc)::value;
    constexpr int next = s + 1 < kT ? s + 1 : 0;
    const int r = k - 2 * s;
    Quad nU, nV;
    row2d<P, COEF, LINK, kIso>(a, iso, hx, gy(r), gy(r + 1), off(r), off(r + 1), class_of(r), class_of(r + 1), U[s], V[s], Vn[s], nU0[s], nU1[s],
                               lanes, wave_at(s, r), nU, nV, s == kT - 1 ? &oS : nullptr);
    if constexpr (s == kT - 1) {
      oU = mkquad(nU0[s], qlane(nU, 1));  // the row's new u0 (formed one row earlier) and u1
      oV = nV;
    } else {  // the next stage's rows of the next position
      U[next] = mkquad(nU0[s], nU1[s]);
      V[next] = Vn[next];
      Vn[next] = nV;
    }
    nU0[s] = qlane(nU, 0);
    nU1[s] = qlane(nU, 1);
  };
  using S0 = std::integral_constant<int, 0>;
  using S1 = std::integral_constant<int, kT - 1>;
#pragma unroll 1
  for (int k = k0; k < kl + kT; ++k) {
    cp_async_wait<kRing - 2>();  // row k + 1 has arrived
    if (LINK == LINK_PLANE) __syncwarp();  // (for every lane: the wave's factors are copied by a few)
    {
      const float4* slot = ring + ((k + 1) & (kRing - 1)) * 64 + lane;
      const Quad u = quad(slot[0]);
      V[0] = Vn[0];
      Vn[0] = quad(slot[32]);
      U[0] = mkquad(qlane(u, 0), u1);
      u1 = qlane(u, 1);
    }
    fetch(k + kRing);  // into the slot of row k, read in the position before
    if (kT == 1 || (k >= k0 + 3 && k <= kl)) {
      if constexpr (kT == 2) stage(S1{}, k);
      stage(S0{}, k);
    } else {  // the first and last positions: stage s starts at row y0 - kT + s and ends with the rows the next needs
      if (k >= k0 + 3) stage(S1{}, k);
      else stage(S0{}, k);
    }
    const int r = k - 2 * (kT - 1);
    if (core && r >= y0) {  // (after all stages: a branch between them would keep their chains apart)
      const Off o = off(r);
      a.out[0][o] = pack4(oU);
      a.out[1][o] = pack4(oV);
      if (a.e_partials) {
        e_n += (n2(qlane(oU, 1)) + n2(qlane(oV, 0))) + n2(qlane(oV, 1));
        e_n += n2(qlane(oU, 0));
        e_c += fmaf(oV.re.y, oS.re.y, fmaf(oV.im.y, oS.im.y, fmaf(oV.re.x, oS.re.x, oV.im.x * oS.im.x)));
      }
    }
  }
  cp_async_wait<0>();  // nothing of this item lands in the next one's slots
  // every lane has read its last factors before a few lanes write the next item's
  // (the rows in the ring are each lane's own)
  if (LINK == LINK_PLANE) __syncwarp();
}

template <class P, int COEF, int LINK, int kT, bool kIso>
__device__ __forceinline__ void fused2d_item(const FusedArgs<P>& a, float4* ring, long long item, int lane,
                                             double& e_n, double& e_c) {
  const int strips = strips2d<kT>(a.N[0]);
  const long long chunk = item / strips;
  const int strip = (int)(item - chunk * strips);
  if constexpr (COEF == COEF_STEP_X) {
    // all but the strips the step cuts have one coefficient, and in those every
    // lane has its own throughout (a choice between two results per value made
    // these few strips 2.3 times slower, and every launch wait for them)
    const int hx = 2 * wrapi(strip * core_lanes<kT>() + lane - kT, a.N[0]);
    if (__all_sync(0xffffffffu, hx + 1 < a.hu.step_X))
      return march2d<P, COEF_UNIFORM, LINK, kT, kIso, 1>(a, ring, strip, chunk, lane, e_n, e_c);
    if (__all_sync(0xffffffffu, hx >= a.hu.step_X))
      return march2d<P, COEF_BEYOND, LINK, kT, kIso, 1>(a, ring, strip, chunk, lane, e_n, e_c);
    // (u0, v1 at hx; u1, v0 at hx + 1; a lane reads its own records only)
    float4* t = ring + kRing * 64 + lane;
    const bool b0 = hx >= a.hu.step_X, b1 = hx + 1 >= a.hu.step_X;
    lane_coefs(a.hu, b0, b1, t);
    lane_coefs(a.hl, b1, b0, t + 128);
    return march2d<P, COEF_LANES, LINK, kT, kIso, 1>(a, ring, strip, chunk, lane, e_n, e_c);
  }
  if constexpr (COEF != COEF_STEP_X) march2d<P, COEF, LINK, kT, kIso, COEF == COEF_STEP>(a, ring, strip, chunk, lane, e_n, e_c);
}

template <class P, int COEF, int LINK, int kT, bool kIso>
__global__ void __launch_bounds__(32 * kFused2dWarps, min_blocks(kT, COEF, LINK)) fused2d_kernel(const FusedArgs<P> a) {
  depends();
  const int lane = threadIdx.x & 31;
  const long long worker = (long long)blockIdx.x * kFused2dWarps + (threadIdx.x >> 5);
  const long long items = (long long)strips2d<kT>(a.N[0]) * ((a.nzu + a.chunk - 1) / a.chunk);
  __shared__ __align__(16) float4 ring[kFused2dWarps][warp_slots<COEF, LINK>()];
  double e_n = 0.0, e_c = 0.0;
  for (long long item = worker; item < items; item += a.workers)  // uniform per warp
    fused2d_item<P, COEF, LINK, kT, kIso>(a, ring[threadIdx.x >> 5], item, lane, e_n, e_c);
  if (a.e_partials) block_store_e(e_n, e_c, a.e_partials);
}

// Several simulations (time-independent fields) in one persistent launch.
template <class P, int COEF, int LINK, int kT, bool kIso>
__global__ void __launch_bounds__(32 * kFused2dWarps, min_blocks(kT, COEF, LINK)) fused2d_batch_kernel(const BatchArgs<P> b) {
  depends();
  __shared__ FusedArgs<P> sa[kFused2dWarps];
  __shared__ __align__(16) float4 ring[kFused2dWarps][warp_slots<COEF, LINK>()];
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
    if (COEF == COEF_STEP && sa[w].hu.step_axis == 0)
      fused2d_item<P, COEF == COEF_STEP ? COEF_STEP_X : COEF, LINK, kT, kIso>(sa[w], ring[w], g - b.first_item[s],
                                                                               lane, e_n, e_c);
    else fused2d_item<P, COEF, LINK, kT, kIso>(sa[w], ring[w], g - b.first_item[s], lane, e_n, e_c);
  }
}

// resident warps of a kernel, computed once
template <auto K>
int workers2d() {
  static int r = resident_blocks(K, 32 * kFused2dWarps) * kFused2dWarps;
  return r;
}

}  // namespace

template <int COEF, int LINK, int kT, bool kIso>
int launch2d_iso(FusedArgs<F32> a, cudaStream_t s) {
  constexpr auto k = fused2d_kernel<F32, COEF, LINK, kT, kIso>;
  const int warps = workers2d<k>();
  if (a.chunk <= 0 || a.chunk > a.nzu) {
    const int Np[3] = {a.N[0], a.nzu, 1};
    ChunkShape shape = shape2d(Np, kT);
    shape.workers = warps;  // this kernel's own
    a.chunk = plan_chunk(shape);
  }
  const long long items = (long long)strips2d<kT>(a.N[0]) * ((a.nzu + a.chunk - 1) / a.chunk);
  long long w = items < warps ? items : warps;
  // one E partial per block: never more blocks than the partials hold
  if (a.e_partials && w > (long long)kFusedEMaxBlocks * kFused2dWarps) w = (long long)kFusedEMaxBlocks * kFused2dWarps;
  a.workers = (int)w;
  const int blocks = (int)((w + kFused2dWarps - 1) / kFused2dWarps);
  launch_dependent(k, dim3((unsigned)blocks), dim3(32 * kFused2dWarps), 0, s, a);
  return blocks;
}
template <int COEF, int LINK, int kT>
int launch2d(FusedArgs<F32> a, cudaStream_t s) {
  if constexpr (COEF != kAnyMode)  // (the run-time path tests iso itself)
    if (!a.iso) return launch2d_iso<COEF, LINK, kT, false>(a, s);
  return launch2d_iso<COEF, LINK, kT, true>(a, s);
}

template <int COEF, int LINK, int kT, bool kIso>
void launch2d_batch(BatchArgs<F32> b, long long total, cudaStream_t s) {
  constexpr auto k = fused2d_batch_kernel<F32, COEF, LINK, kT, kIso>;
  const int warps = workers2d<k>();
  const long long w = total < warps ? total : warps;
  b.workers = (int)w;
  launch_dependent(k, dim3((unsigned)((w + kFused2dWarps - 1) / kFused2dWarps)), dim3(32 * kFused2dWarps), 0, s, b);
}

}  // namespace fused
}  // namespace dirac
