// Reductions of the stored state: the naive norm, the cross terms of the
// conserved functional (Lemma of Sect. 2, Eq. EPM, in its "lower" form; see
// dirac.h) and the partial density used for the Klein-step transmission; and
// the tables and layout conversions that a simulation is set up with.
#include <cfloat>

#include "kernels.cuh"
#include "fused_common.cuh"

namespace dirac {

namespace {

__device__ __forceinline__ double2 widen(double2 v) { return v; }
__device__ __forceinline__ double2 widen(float2 v) { return make_double2(v.x, v.y); }

__device__ __forceinline__ double2 mul_expm(double2 v, double phi) {  // v * exp(-i phi)
  double s, c;
  sincos(phi, &s, &c);
  return make_double2(c * v.x + s * v.y, c * v.y - s * v.x);
}

template <int NS>
__device__ __forceinline__ void block_reduce_store(double (&v)[NS], double* out) {
  __shared__ double sh[32][NS];
  const int tid = threadIdx.y * blockDim.x + threadIdx.x;
  const int lane = tid & 31, warp = tid >> 5;
#pragma unroll
  for (int k = 0; k < NS; ++k)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_down_sync(0xffffffffu, v[k], o);
  if (lane == 0)
#pragma unroll
    for (int k = 0; k < NS; ++k) sh[warp][k] = v[k];
  __syncthreads();
  if (warp == 0) {
    const int nw = (blockDim.x * blockDim.y) >> 5;
#pragma unroll
    for (int k = 0; k < NS; ++k) {
      double x = lane < nw ? sh[lane][k] : 0.0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
      if (lane == 0) out[k] = x;
    }
  }
}

// Running sums of a thread: FP64 for FP64 states.  For FP32 states the FP64
// pipe (1.6 lanes per clock and SM) would be the limit, so a cell's terms are
// added to an unevaluated sum h + m + l of three floats: the rounding error of
// h goes to m, that of m to l (TwoSum, both exact), so only l rounds, by 2^-24 of
// itself, at most 2^-64 of the largest partial sum over the kFlush cells after which
// the three go to FP64.  FP64 additions one by one round by 2^-53 of the sum each.
// Terms that kFlush of them could add up to beyond the floats' range, infinities
// and NaN (which TwoSum would turn into NaN) go to FP64 by themselves.
constexpr int kFlush = 16;
constexpr float kSumMax = 0x1p120f;
struct Sum32 {
  float h, m, l;
  // s becomes s + v, the result is what the rounding left out
  static __device__ __forceinline__ float two_sum(float& s, float v) {
    const float t = __fadd_rn(s, v), b = __fsub_rn(t, s);
    const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(v, b));
    s = t;
    return e;
  }
  __device__ __forceinline__ void add(float v) { l = __fadd_rn(l, two_sum(m, two_sum(h, v))); }
  __device__ __forceinline__ void flush(double& acc) {
    acc += (double)h + ((double)m + (double)l);
    h = m = l = 0.0f;
  }
};
struct Sum64 {
  double h;
  __device__ __forceinline__ void add(double v) { h += v; }
  __device__ __forceinline__ void flush(double& acc) {
    acc += h;
    h = 0.0;
  }
};
template <class P> struct SumOf { using type = Sum64; };
template <> struct SumOf<F32> { using type = Sum32; };

// L up - conj(M) dn of FP32 values rounded once: each part is a sum of four
// products formed as by Dot2 (Ogita, Rump, Oishi, SIAM J. Sci. Comput. 26, 2005),
// the products of the factors' lo parts among the corrections, so that what is
// left out is about 2^-47 of the neighbours.  (A product rounded to FP32 before the
// difference is taken leaves out 2^-24 of them, however small the difference;
// FP64 arithmetic would put 20 operations per link on the narrow FP64 pipe.)
struct Dot32 {
  float s, e;
  __device__ __forceinline__ Dot32(float f_hi, float f_lo, float v) {
    s = __fmul_rn(f_hi, v);
    e = __fmaf_rn(f_lo, v, __fmaf_rn(f_hi, v, -s));
  }
  __device__ __forceinline__ void add(float f_hi, float f_lo, float v) {
    const float p = __fmul_rn(f_hi, v), pe = __fmaf_rn(f_hi, v, -p);
    e = __fadd_rn(e, __fmaf_rn(f_lo, v, __fadd_rn(pe, Sum32::two_sum(s, p))));
  }
  // (an infinite product leaves no corrections)
  __device__ __forceinline__ float value() const { return fabsf(e) <= FLT_MAX ? __fadd_rn(s, e) : s; }
};
__device__ __forceinline__ float2 rotated_diff(const F32::Link& L, float2 up, const F32::Link& M, float2 dn) {
  Dot32 re(L.hi.x, L.lo.x, up.x), im(L.hi.x, L.lo.x, up.y);
  re.add(-L.hi.y, -L.lo.y, up.y);
  re.add(-M.hi.x, -M.lo.x, dn.x);
  re.add(-M.hi.y, -M.lo.y, dn.y);
  im.add(L.hi.y, L.lo.y, up.x);
  im.add(-M.hi.x, -M.lo.x, dn.y);
  im.add(M.hi.y, M.lo.y, dn.x);
  return make_float2(re.value(), im.value());
}

// Both values of a component in one cell (two planes, or one quad).
template <class P>
struct Pair {
  typename P::cplx v[2];
};
template <class P, bool kQuads>
__device__ __forceinline__ Pair<P> load_pair(const ObsArgs<P>& a, int comp, long long cell) {
  if constexpr (kQuads) {
    const float4 q = __ldg(a.quads[comp] + cell);
    return Pair<P>{{make_float2(q.x, q.z), make_float2(q.y, q.w)}};
  } else {
    return Pair<P>{{a.pl[2 * comp][cell], a.pl[2 * comp + 1][cell]}};
  }
}

// A warp takes 32 cells along x of one row at a time, rows dealt to a grid
// that fills the GPU once.  Per cell the terms are formed in the state's
// precision (FP32 states: products of two stored floats) and accumulated per
// thread (SumOf), then in FP64 per warp (shuffles), per block and over the
// blocks, in a fixed order, so the result is deterministic for a given grid.
// Plane-wave link factors c - i s come from a table.  kLink: LINK_TABLE is the
// quads' table of factors; any other vector potential (LINK_GENERAL) evaluates
// its phases in FP64.
// Bound: loads (14 16-byte records per cell, about 5 from L2 or HBM).
// us at 128^3 free / 4096^2 / 512^3 laser: with a block per 32 x 8 cells and z
// range, a sincos per link, FP64 sums per cell and up to 65536 partials summed
// by one warp 203 / 1449 / 79120; with this grid, link tables and FP64 sums
// 55 / 215 / 9840; with the sums' errors in one float and rotations rounded before
// their difference (fewer bits than the FP64 sums and rotations) 39 / 150 / 3890;
// now, the kernel alone, 43 / 135 / 3950 (128^3 static links 167 and 210).
template <class P, int DIMS, bool kQuads, int kLink, bool kDens>
__global__ void __launch_bounds__(256) observables_kernel(const ObsArgs<P> a) {
  using C = typename P::cplx;
  using R = typename P::real;
  constexpr int nc = nplanes<DIMS>() / 2;  // components, the lower ones from nc / 2
  const int Nx = a.N[0], Ny = a.N[1], Nz = DIMS == 3 ? a.N[2] : 1;
  const long long nxy = (long long)Nx * Ny;
  const int lane = threadIdx.x & 31, wpb = blockDim.x >> 5;
  const int tiles_x = (Nx + 31) / 32;
  // rows summed: all of a whole grid, a slab's own levels zlo .. zlo + nzu - 1
  // along the marching axis; fields at the global level
  const int rows_y = DIMS == 3 ? Ny : a.nzu;
  const long long items = (long long)tiles_x * rows_y * (DIMS == 3 ? a.nzu : 1);
  double acc[kObsSums] = {0.0, 0.0, 0.0, 0.0, 0.0};
  typename SumOf<P>::type sum[kObsSums] = {};
  int pending = 0;
  auto global_level = [&](int k) {  // in [-1, 2 Nzg): one wrap at most
    const int g = a.zorg + k;
    return g < 0 ? g + a.Nzg : (g >= a.Nzg ? g - a.Nzg : g);
  };
  for (long long it = (long long)blockIdx.x * wpb + (threadIdx.x >> 5); it < items; it += (long long)gridDim.x * wpb) {
    const long long row = it / tiles_x;
    const int x = (int)(it - row * tiles_x) * 32 + lane;
    if (x >= Nx) continue;
    const int zz = DIMS == 3 ? (int)(row / Ny) : 0;
    const int y = DIMS == 3 ? (int)(row - (long long)zz * Ny) : a.zlo + (int)row;
    const int z = DIMS == 3 ? a.zlo + zz : 0;
    const int yg = DIMS == 3 ? y : global_level(y), zg = DIMS == 3 ? global_level(z) : 0;
    const long long cell = z * nxy + (long long)y * Nx + x;
    const long long dxm = x == 0 ? Nx - 1 : -1, dxp = x == Nx - 1 ? 1 - Nx : 1;
    const long long dym = y == 0 ? nxy - Nx : -Nx, dyp = y == Ny - 1 ? Nx - nxy : Nx;
    Pair<P> own[nc];
#pragma unroll
    for (int c = 0; c < nc; ++c) own[c] = load_pair<P, kQuads>(a, c, cell);
    R cn = 0, cd = 0, cb[3] = {0, 0, 0};
#pragma unroll
    for (int c = 0; c < nc; ++c) {
#pragma unroll
      for (int l = 0; l < 2; ++l) {
        const C G = own[c].v[l];
        const R n2 = G.x * G.x + G.y * G.y;
        cn += n2;
        if (kDens) {
          const int plane = 2 * c + l;
          const int hd = a.dens_axis == 0 ? 2 * x + plane_off<DIMS>(plane, 0)
                         : (a.dens_axis == 1 ? 2 * yg + plane_off<DIMS>(plane, 1) : 2 * zg + plane_off<DIMS>(plane, 2));
          if (hd >= a.dens_X) cd += n2;
        }
      }
    }
#pragma unroll
    for (int c = nc / 2; c < nc; ++c) {
      // the x-y partner component around the cell, the z partner above / below;
      // sublattice 0 of C has its x+ neighbour in its own cell, of D (v) its x-
      const int cxy = DIMS == 3 ? 3 - c : 0;
      const bool kX = DIMS == 2 || c == 3;
      const Pair<P> q = own[cxy];
      const C xm = load_pair<P, kQuads>(a, cxy, cell + dxm).v[kX ? 1 : 0];
      const C xp = load_pair<P, kQuads>(a, cxy, cell + dxp).v[kX ? 0 : 1];
      const C ym1 = load_pair<P, kQuads>(a, cxy, cell + dym).v[1];
      const C yp0 = load_pair<P, kQuads>(a, cxy, cell + dyp).v[0];
      Pair<P> zu{}, zd{};
      if (DIMS == 3) {
        if (c == 2) {
          zu = load_pair<P, kQuads>(a, 0, cell + (z == Nz - 1 ? nxy - nxy * Nz : nxy));
          zd = own[0];
        } else {
          zu = own[1];
          zd = load_pair<P, kQuads>(a, 1, cell + (z == 0 ? nxy * Nz - nxy : -nxy));
        }
      }
#pragma unroll
      for (int l = 0; l < 2; ++l) {
        const int plane = 2 * c + l;
        const C G = own[c].v[l];
        const int p = sign_class<DIMS>(plane);
        const long long H[3] = {2LL * x + plane_off<DIMS>(plane, 0), 2LL * yg + plane_off<DIMS>(plane, 1),
                                DIMS == 3 ? 2LL * zg + plane_off<DIMS>(plane, 2) : 0};
#pragma unroll
        for (int ax = 0; ax < DIMS; ++ax) {
          const bool own_up = (l == 0) != kX;  // the x+ neighbour is in the own cell
          C up = ax == 0 ? (own_up ? q.v[l] : xp) : (ax == 1 ? (l == 0 ? q.v[1] : yp0) : zu.v[l]);
          C dn = ax == 0 ? (own_up ? xm : q.v[l]) : (ax == 1 ? (l == 0 ? ym1 : q.v[0]) : zd.v[l]);
          R re, im;
          if (kLink == LINK_PLANE && ax == a.f.Apw_pol) {
            // (the wave is across its own links: one factor c - i s for both, at
            // the value's half-lattice coordinate along the wave vector)
            const int h = a.wave_axis == 0 ? (int)H[0] : (a.wave_axis == 1 ? (int)H[1] : (int)H[2]);
            if constexpr (sizeof(R) == 4) {
              const float4 f = __ldg(&(static_cast<const PlaneLink32*>(a.wave) + h)->v);
              const F32::Link L{make_float2(f.x, -f.z), make_float2(f.y, -f.w)};
              const C w = rotated_diff(L, up, L, dn);
              re = w.x;
              im = w.y;
            } else {
              const double2 f = __ldg(static_cast<const double2*>(a.wave) + h);  // (cos phi, -sin phi)
              re = f.x * (up.x - dn.x) - f.y * (up.y + dn.y);
              im = f.x * (up.y - dn.y) + f.y * (up.x + dn.x);
            }
          } else if (kLink == LINK_GENERAL) {
            const double2 u = mul_expm(widen(up), link_phase_site(a.f, DIMS, H, ax, +1, a.t_links, plane, cell));
            const double2 v = mul_expm(widen(dn), -link_phase_site(a.f, DIMS, H, ax, -1, a.t_links, plane, cell));
            re = (R)(u.x - v.x);
            im = (R)(u.y - v.y);
          } else {
            if (kLink == LINK_CONST) {
              up = link_mul(a.L[ax], up);
              dn = link_mulc(a.L[ax], dn);
            }
            if constexpr (kLink == LINK_UP) {
              const long long below = plane_off<DIMS>(plane, ax) ? cell
                                      : (ax == 0 ? cell + dxm : (ax == 1 ? cell + dym : cell + (z == 0 ? nxy * Nz - nxy : -nxy)));
              const typename P::Link* t = a.larr + ax * a.larr_n;
              up = link_mul(up_link<P>(t + (plane * a.pstride + cell)), up);
              dn = link_mulc(up_link<P>(t + (partner<DIMS>(plane, ax) * a.pstride + below)), dn);
            }
            re = up.x - dn.x;
            im = up.y - dn.y;
            if constexpr (kLink == LINK_TABLE && kQuads) {
              const float4* t = a.lq + 2 * ((long long)(2 * ax * nc + c) * a.pstride + cell);
              const float4 u = quad_lane(t, l), d = quad_lane(t + 2 * nc * a.pstride, l);
              const C w = rotated_diff(F32::Link{make_float2(u.x, u.y), make_float2(u.z, u.w)}, up,
                                       F32::Link{make_float2(d.x, d.y), make_float2(d.z, d.w)}, dn);
              re = w.x;
              im = w.y;
            }
          }
          const R sre = ax == 1 ? (p ? -im : im) : (ax == 2 && p ? -re : re);
          const R sim = ax == 1 ? (p ? re : -re) : (ax == 2 && p ? -im : im);
          cb[ax] += G.x * sre + G.y * sim;  // Re(conj(G) s d)
        }
      }
    }
    // (one test for all of a cell's terms; no density term exceeds cn)
    if (sizeof(R) == 8 || fabs(cn) + (fabs(cb[0]) + fabs(cb[1]) + fabs(cb[2])) <= (R)kSumMax) {
      sum[0].add(cn);
#pragma unroll
      for (int ax = 0; ax < DIMS; ++ax) sum[1 + ax].add(cb[ax]);
      if (kDens) sum[4].add(cd);
    } else {
      acc[0] += cn;
#pragma unroll
      for (int ax = 0; ax < DIMS; ++ax) acc[1 + ax] += cb[ax];
      if (kDens) acc[4] += cd;
    }
    if (++pending == kFlush) {
      pending = 0;
#pragma unroll
      for (int k = 0; k < kObsSums; ++k) sum[k].flush(acc[k]);
    }
  }
#pragma unroll
  for (int k = 0; k < kObsSums; ++k) sum[k].flush(acc[k]);
  block_reduce_store<kObsSums>(acc, a.partials + (long long)blockIdx.x * kObsSums);
}

// exp(-i phi) in the plane-wave table's element type: F64::Link, or for the
// FP32 kernels c - i s as hi + lo pairs of cos phi and sin phi
__device__ __forceinline__ void plane_link_from(double phi, F64::Link* out) {
  *out = link_from(phi, (F64*)nullptr);
}
__device__ __forceinline__ void plane_link_from(double phi, PlaneLink32* out) {
  double sn, cs;
  sincos(phi, &sn, &cs);
  const float ch = __double2float_rn(cs), sh = __double2float_rn(sn);
  const float cl = __double2float_rn(cs - (double)ch), sl = __double2float_rn(sn - (double)sh);
  out->v = make_float4(ch, cl, sh, sl);
  out->ch = make_float2(ch, ch);
  out->cl = make_float2(cl, cl);
  out->sh = make_float2(sh, -sh);
  out->sl = make_float2(sl, -sl);
  out->sp = make_float2(sh, sh);
  out->lp = make_float2(sl, sl);
}

// one value's {re hi, im hi, re lo, im lo} into a quad record
__device__ __forceinline__ void store_quad_lane(float4* rec, int lane, float4 v) {
  float* r = reinterpret_cast<float*>(rec) + lane;
  r[0] = v.x;
  r[2] = v.y;
  r[4] = v.z;
  r[6] = v.w;
}

struct LinkTimes {
  double up[kTableSteps], lo[kTableSteps];
};
template <class P>
__global__ void link_table_kernel(typename PlaneLinkOf<P>::type* tab, int n, const FieldDesc f, int dims,
                                  int axis, int pol, const LinkTimes t, int steps) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x, per_step = 2LL * n;
  if (i >= per_step * steps) return;
  const int step = (int)(i / per_step);
  const long long j = i - step * per_step;
  const int half = j >= n;
  long long HH[3] = {0, 0, 0};
  HH[axis] = half ? j - n : j;
  // the same phase function as the per-link FP64 path
  plane_link_from(link_phase(f, dims, HH, pol, +1, half ? t.lo[step] : t.up[step]), tab + i);
}

// b = 1/(1 + i theta), theta = dt (beta m + V)/2 with V complex, of every site
// of one plane (blockIdx.y), V from the same FP64 potential functions as the
// per-site general path, at time 0 (the table serves time-independent
// potentials only); stored as {re hi, im hi, re lo, im lo}
template <int DIMS>
__global__ void coef_table_kernel(float4* __restrict__ tab, const FieldDesc f, int N0, int N1, int N2,
                                  long long pstride, int quads, const int* __restrict__ rep) {
  const int plane = blockIdx.y;
  const long long ncell = (long long)N0 * N1 * N2;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < ncell;
       c += (long long)gridDim.x * blockDim.x) {
    long long x = c % N0, y = (c / N0) % N1, z = c / ((long long)N0 * N1);
    if (rep) x = rep[x], y = rep[N0 + y], z = rep[N0 + N1 + z];
    const long long X = 2 * x + plane_off<DIMS>(plane, 0), Y = 2 * y + plane_off<DIMS>(plane, 1),
                    Z = DIMS == 3 ? 2 * z + plane_off<DIMS>(plane, 2) : 0;
    const double V = potential_at(f, DIMS, X, Y, Z, c, pstride, plane, 0.0);
    const double beta = is_upper<DIMS>(plane) ? 1.0 : -1.0;
    const double ta = f.dt * (beta * f.m + V) * 0.5;  // theta = ta + i tb
    const double tb = f.dt * potential_imag_at(f, DIMS, X, Y, Z) * 0.5;
    // b = 1/((1 - tb) + i ta)
    const double k = 1.0 / ((1.0 - tb) * (1.0 - tb) + ta * ta);
    const double re = (1.0 - tb) * k, im = -ta * k;
    const float rh = __double2float_rn(re), ih = __double2float_rn(im);
    const float4 b = make_float4(rh, ih, __double2float_rn(re - (double)rh), __double2float_rn(im - (double)ih));
    if (quads) store_quad_lane(tab + 2 * ((plane >> 1) * pstride + c), plane & 1, b);
    else tab[plane * pstride + c] = b;
  }
}

// COEF_TABLE of the FP64 kernels: alpha and gamma of every site, by the same
// operations as the per-site path
template <int DIMS>
__global__ void coef64_table_kernel(F64::Coef* __restrict__ tab, const FieldDesc f, int N0, int N1, int N2,
                                    long long pstride) {
  const int plane = blockIdx.y;
  const long long ncell = (long long)N0 * N1 * N2;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < ncell;
       c += (long long)gridDim.x * blockDim.x) {
    const long long x = c % N0, y = (c / N0) % N1, z = c / ((long long)N0 * N1);
    const long long X = 2 * x + plane_off<DIMS>(plane, 0), Y = 2 * y + plane_off<DIMS>(plane, 1),
                    Z = DIMS == 3 ? 2 * z + plane_off<DIMS>(plane, 2) : 0;
    const double beta = is_upper<DIMS>(plane) ? 1.0 : -1.0;
    double2 al, ga;
    site_coef(f, DIMS, X, Y, Z, c, pstride, plane, beta, 0.0, al, ga);
    tab[plane * pstride + c] = F64::Coef{al, ga};
  }
}

// COEF_SOFTCORR: the correction records (softcore_corr_index's layout) of a
// real soft-core potential: per value, (exact b) - (the kernels' FP32
// estimate softcore_fast2), b = 1/(1 + i dt (beta m + V)/2) with V from the
// same FP64 potential function as the per-site path, rounded to an integer
// multiple of 2^-35 per component and stored as two 16-bit integers; a value
// out of the 16-bit range sets *overflow (the estimate was off by more than
// the table can hold; the library then evaluates the soft core otherwise)
template <int DIMS>
__global__ void softcore_corr_kernel(unsigned* __restrict__ out, const HalfFields<F32> hu,
                                     const HalfFields<F32> hl, const FieldDesc f, int N0, int N1, int N2,
                                     int* overflow) {
  constexpr int np = nplanes<DIMS>();
  const int N[3] = {N0, N1, N2};
  const long long ncell = (long long)N0 * N1 * N2;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < ncell * np;
       i += (long long)gridDim.x * blockDim.x) {
    const long long r = i / np;
    const int plane = (int)(i - r * np);
    const int x = (int)(r % N0), y = (int)((r / N0) % N1), zr = (int)(r / ((long long)N0 * N1));
    int yy = y, zz = zr;
    const bool shifted = DIMS == 3 ? plane < 2 : plane == 0;
    if (shifted) {
      if (DIMS == 3) zz = zr + 1 == N2 ? 0 : zr + 1;
      else yy = y + 1 == N1 ? 0 : y + 1;
    }
    const int H[3] = {2 * x + plane_off<DIMS>(plane, 0), 2 * yy + plane_off<DIMS>(plane, 1),
                      DIMS == 3 ? 2 * zz + plane_off<DIMS>(plane, 2) : 0};
    const bool upper = is_upper<DIMS>(plane);
    const HalfFields<F32>& h = upper ? hu : hl;
    float Rh, Rl;
    softcore_R<DIMS>(h, H, Rh, Rl);
    float2 re, im;
    softcore_fast2(f2(Rh), f2(Rl), f2(softcore_t0(h, H).x), h.sc_K_hi, re, im);
    const double V = potential_at(f, DIMS, H[0], H[1], H[2], 0, 0, plane, 0.0);
    const double th = f.dt * ((upper ? 1.0 : -1.0) * f.m + V) * 0.5;
    const double k = 1.0 / (1.0 + th * th);
    long long q[2] = {llrint((k - (double)re.x) * 34359738368.0), llrint((-th * k - (double)im.x) * 34359738368.0)};
    for (int c = 0; c < 2; ++c) {
      if (q[c] > 32767 || q[c] < -32767) {
        atomicOr(overflow, 1);
        q[c] = q[c] > 0 ? 32767 : -32767;
      }
    }
    out[i] = (unsigned)(q[0] & 0xffff) | ((unsigned)(q[1] & 0xffff) << 16);
  }
}

// q times the link integrals of every value in the state layout: the value's
// own link towards +dx_a/2 (slot 2a; alone, dirs = 1: slot a) and the link from
// its neighbour at -dx_a/2 to it (slot 2a+1), which that neighbour (partner
// plane, cell shifted with the periodic wrap) carries as its own up link
template <int DIMS>
__global__ void link_integral_table_kernel(double* __restrict__ out, const double* __restrict__ raw, int N0,
                                           int N1, int N2, long long pstride, double q, int dirs) {
  const int plane = blockIdx.y, axis = blockIdx.z;
  const long long ncell = (long long)N0 * N1 * N2;
  const long long n = (long long)nplanes<DIMS>() * pstride;
  const double* raw_a = raw + (long long)axis * nplanes<DIMS>() * ncell;
  const int pp = partner<DIMS>(plane, axis);
  const int shift = nb_shift<DIMS>(plane, axis, -1);
  const int Nn[3] = {N0, N1, N2};
  const long long stride[3] = {1, N0, (long long)N0 * N1};
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < ncell;
       c += (long long)gridDim.x * blockDim.x) {
    const long long j[3] = {c % N0, (c / N0) % N1, c / ((long long)N0 * N1)};
    long long jm = j[axis] + shift;
    if (jm < 0) jm += Nn[axis];
    const long long cm = c + (jm - j[axis]) * stride[axis];
    out[(long long)(dirs * axis) * n + plane * pstride + c] = q * raw_a[(long long)plane * ncell + c];
    if (dirs == 2) out[(2LL * axis + 1) * n + plane * pstride + c] = q * raw_a[(long long)pp * ncell + cm];
  }
}

// LINK_TABLE: the link factors exp(-i phi) of every value of a time-independent
// vector potential, phi from the same FP64 function as the per-site path
// (slot 2 axis: the value's up link; 2 axis + 1: the link from its lower
// neighbour); LINK_UP (dirs == 1): the up links alone, slot = axis
template <class P, int DIMS>
__global__ void link_factor_table_kernel(typename P::Link* __restrict__ out, const FieldDesc f, int N0, int N1, int N2,
                                         long long pstride, int quads, int dirs) {
  const int plane = blockIdx.y, slot = blockIdx.z, axis = slot / dirs, dir = slot % dirs ? -1 : 1;
  const long long ncell = (long long)N0 * N1 * N2;
  const long long n = (long long)nplanes<DIMS>() * pstride;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < ncell;
       c += (long long)gridDim.x * blockDim.x) {
    const long long x = c % N0, y = (c / N0) % N1, z = c / ((long long)N0 * N1);
    const long long H[3] = {2 * x + plane_off<DIMS>(plane, 0), 2 * y + plane_off<DIMS>(plane, 1),
                            DIMS == 3 ? 2 * z + plane_off<DIMS>(plane, 2) : 0};
    const double phi = link_phase_site(f, DIMS, H, axis, dir, 0.0, plane, c);
    const typename P::Link L = link_from(phi, (P*)nullptr);
    if constexpr (sizeof(typename P::real) == 4) {
      if (quads) {  // the quads of slot, component: 2 * ((slot * components + component) * pstride + cell)
        store_quad_lane(reinterpret_cast<float4*>(out) + slot * n + 2 * ((plane >> 1) * pstride + c), plane & 1,
                        make_float4(L.hi.x, L.hi.y, L.lo.x, L.lo.y));
        continue;
      }
    }
    out[slot * n + plane * pstride + c] = L;
  }
}

// out[k] = sum over the blocks of partials[block][k]: one warp per column,
// eight loads in flight per lane, a fixed order
template <int NS>
__global__ void finish_sums_kernel(const double* __restrict__ partials, int nblocks, double* out) {
  const int lane = threadIdx.x & 31, k = threadIdx.x >> 5;
  double x = 0.0;
  for (int b0 = lane; b0 < nblocks; b0 += 256) {
    double v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = b0 + 32 * u < nblocks ? partials[(long long)(b0 + 32 * u) * NS + k] : 0.0;
#pragma unroll
    for (int u = 0; u < 8; ++u) x += v[u];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
  if (lane == 0) out[k] = x;
}

__global__ void convert_in_kernel(const double2* __restrict__ src, float2* __restrict__ dst,
                                  long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    dst[i] = make_float2(__double2float_rn(src[i].x), __double2float_rn(src[i].y));
}
__global__ void convert_out_kernel(const float2* __restrict__ src, double2* __restrict__ dst,
                                   long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    dst[i] = make_double2(src[i].x, src[i].y);
}

// Bound: HBM (32 B in and 16 B out per cell and component, or back): both planes
// of a component in one pass, so that the quads are written whole.
// two canonical planes <-> one component's quads; lane < 0: both planes, else
// the one plane of that sublattice (src0 / dst0)
__global__ void convert_in_quads_kernel(const double2* __restrict__ src0, const double2* __restrict__ src1,
                                        float4* __restrict__ dst, int lane, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const double2 v = src0[i];
    const float re = __double2float_rn(v.x), im = __double2float_rn(v.y);
    if (lane < 0) {
      const double2 w = src1[i];
      dst[i] = make_float4(re, __double2float_rn(w.x), im, __double2float_rn(w.y));
    } else {
      float* r = reinterpret_cast<float*>(dst + i) + lane;
      r[0] = re;
      r[2] = im;
    }
  }
}
__global__ void convert_out_quads_kernel(const float4* __restrict__ src, double2* __restrict__ dst0,
                                         double2* __restrict__ dst1, int lane, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const float4 q = src[i];
    if (lane < 0) {
      dst0[i] = make_double2(q.x, q.z);
      dst1[i] = make_double2(q.y, q.w);
    } else {
      dst0[i] = lane ? make_double2(q.y, q.w) : make_double2(q.x, q.z);
    }
  }
}

// FP64 FMA throughput: eight independent dependency chains of fused
// multiply-adds per thread (the FP64 pipe stays busy, nothing is read from
// memory); the result is stored only if it matches an impossible value, so
// the compiler keeps every operation
__global__ void __launch_bounds__(256) fp64_fma_rate_kernel(double* out, int iters) {
  const double m = 0.9999999999, c = 1e-12;
  double a[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) a[j] = 1e-3 * (threadIdx.x + 1) + j;
  for (int i = 0; i < iters; ++i) {
#pragma unroll
    for (int j = 0; j < 8; ++j) a[j] = fma(a[j], m, c);
  }
  double s = 0.0;
#pragma unroll
  for (int j = 0; j < 8; ++j) s += a[j];
  if (s == -1.0) out[blockIdx.x * blockDim.x + threadIdx.x] = s;
}

}  // namespace

// measured FP64 FMA rate of the current device in FP64 TFLOP/s (2 flops per
// FMA), or a negative value if a CUDA call failed
double measure_fp64_fma_tflops() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return -1.0;
  double* sink = nullptr;
  const int blocks = 8 * sms, threads = 256, iters = 4096;
  if (cudaMalloc(&sink, sizeof(double) * blocks * threads) != cudaSuccess) return -1.0;
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  float best = 1e30f;
  for (int rep = 0; rep < 4; ++rep) {  // the first launch warms up
    cudaEventRecord(e0);
    fp64_fma_rate_kernel<<<blocks, threads>>>(sink, iters);
    cudaEventRecord(e1);
    cudaEventSynchronize(e1);
    float ms = 0.0f;
    cudaEventElapsedTime(&ms, e0, e1);
    if (rep > 0 && ms < best) best = ms;
  }
  const bool ok = cudaGetLastError() == cudaSuccess;
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  cudaFree(sink);
  if (!ok || best <= 0.0f) return -1.0;
  return 2.0 * 8.0 * iters * (double)blocks * threads / (best * 1e-3) / 1e12;
}

// blocks of eight warps, a row piece of 32 cells per warp at a time: at most
// four blocks on every SM (the launcher takes fewer where registers hold fewer)
int observables_blocks(const int N[3], int dims) {
  const long long items = (long long)((N[0] + 31) / 32) * N[1] * (dims == 3 ? N[2] : 1);
  const long long b = (items + 7) / 8;
  const int most = 4 * fused::sm_count();
  return (int)(b < most ? b : most);
}

template <class P, int DIMS, bool kQuads, int kLink, bool kDens>
static int launch_observables_path(const ObsArgs<P>& a, int blocks, cudaStream_t s) {
  constexpr auto k = observables_kernel<P, DIMS, kQuads, kLink, kDens>;
  static const int resident = fused::resident_blocks(k, 256);  // a second, partial wave would idle most SMs
  const int grid = blocks < resident ? blocks : resident;
  k<<<grid, 256, 0, s>>>(a);
  return grid;
}
template <class P, int DIMS, bool kQuads, bool kDens>
static int launch_observables_link(const ObsArgs<P>& a, int blocks, cudaStream_t s) {
  const int l = a.link_mode;
  if (l == LINK_NONE) return launch_observables_path<P, DIMS, kQuads, LINK_NONE, kDens>(a, blocks, s);
  if (l == LINK_CONST) return launch_observables_path<P, DIMS, kQuads, LINK_CONST, kDens>(a, blocks, s);
  if (l == LINK_PLANE && a.wave) return launch_observables_path<P, DIMS, kQuads, LINK_PLANE, kDens>(a, blocks, s);
  if constexpr (sizeof(typename P::real) == 8)
    if (l == LINK_UP) return launch_observables_path<P, DIMS, kQuads, LINK_UP, kDens>(a, blocks, s);
  if (kQuads && l == LINK_TABLE)
    return launch_observables_path<P, DIMS, kQuads, kQuads ? LINK_TABLE : LINK_GENERAL, kDens>(a, blocks, s);
  return launch_observables_path<P, DIMS, kQuads, LINK_GENERAL, kDens>(a, blocks, s);
}
template <class P, int DIMS>
int launch_observables(const ObsArgs<P>& a, int blocks, cudaStream_t s) {
  if constexpr (sizeof(typename P::real) == 4) {
    if (a.quads[0])
      return a.dens_axis >= 0 ? launch_observables_link<P, DIMS, true, true>(a, blocks, s)
                              : launch_observables_link<P, DIMS, true, false>(a, blocks, s);
  }
  return a.dens_axis >= 0 ? launch_observables_link<P, DIMS, false, true>(a, blocks, s)
                          : launch_observables_link<P, DIMS, false, false>(a, blocks, s);
}
template int launch_observables<F64, 2>(const ObsArgs<F64>&, int, cudaStream_t);
template int launch_observables<F64, 3>(const ObsArgs<F64>&, int, cudaStream_t);
template int launch_observables<F32, 2>(const ObsArgs<F32>&, int, cudaStream_t);
template int launch_observables<F32, 3>(const ObsArgs<F32>&, int, cudaStream_t);

template <class P>
void launch_link_table(void* tab, int n, const FieldDesc& f, int dims, int axis, int pol, const double* t_up,
                       const double* t_lo, int steps, cudaStream_t s) {
  LinkTimes t{};
  for (int j = 0; j < steps; ++j) {
    t.up[j] = t_up[j];
    t.lo[j] = t_lo[j];
  }
  link_table_kernel<P><<<(unsigned)((2LL * n * steps + 127) / 128), 128, 0, s>>>(
      static_cast<typename PlaneLinkOf<P>::type*>(tab), n, f, dims, axis, pol, t, steps);
}
template void launch_link_table<F64>(void*, int, const FieldDesc&, int, int, int, const double*, const double*, int,
                                     cudaStream_t);
template void launch_link_table<F32>(void*, int, const FieldDesc&, int, int, int, const double*, const double*, int,
                                     cudaStream_t);

void launch_coef_table(float4* tab, const FieldDesc& f, int dims, const int N[3], long long pstride, int quads,
                       const int* rep, cudaStream_t s) {
  const long long ncell = (long long)N[0] * N[1] * (dims == 3 ? N[2] : 1);
  long long bx = (ncell + 255) / 256;
  if (bx > 152 * 16) bx = 152 * 16;
  const dim3 grid((unsigned)bx, dims == 3 ? 8 : 4);
  if (dims == 3)
    coef_table_kernel<3><<<grid, 256, 0, s>>>(tab, f, N[0], N[1], N[2], pstride, quads, rep);
  else
    coef_table_kernel<2><<<grid, 256, 0, s>>>(tab, f, N[0], N[1], 1, pstride, quads, rep);
}

void launch_coef64_table(F64::Coef* tab, const FieldDesc& f, int dims, const int N[3], long long pstride,
                         cudaStream_t s) {
  const long long ncell = (long long)N[0] * N[1] * (dims == 3 ? N[2] : 1);
  long long bx = (ncell + 255) / 256;
  if (bx > 152 * 16) bx = 152 * 16;
  const dim3 grid((unsigned)bx, dims == 3 ? 8 : 4);
  if (dims == 3)
    coef64_table_kernel<3><<<grid, 256, 0, s>>>(tab, f, N[0], N[1], N[2], pstride);
  else
    coef64_table_kernel<2><<<grid, 256, 0, s>>>(tab, f, N[0], N[1], 1, pstride);
}

void launch_softcore_corr(unsigned* out, const HalfFields<F32>& hu, const HalfFields<F32>& hl, const FieldDesc& f,
                          int dims, const int N[3], int* overflow, cudaStream_t s) {
  const long long n = (long long)N[0] * N[1] * (dims == 3 ? N[2] : 1) * (dims == 3 ? 8 : 4);
  long long bx = (n + 255) / 256;
  if (bx > 152 * 32) bx = 152 * 32;
  if (dims == 3)
    softcore_corr_kernel<3><<<(unsigned)bx, 256, 0, s>>>(out, hu, hl, f, N[0], N[1], N[2], overflow);
  else
    softcore_corr_kernel<2><<<(unsigned)bx, 256, 0, s>>>(out, hu, hl, f, N[0], N[1], 1, overflow);
}

void launch_link_integral_table(double* out, const double* raw, int dims, const int N[3], long long pstride,
                                double q, int dirs, cudaStream_t s) {
  const long long ncell = (long long)N[0] * N[1] * (dims == 3 ? N[2] : 1);
  long long bx = (ncell + 255) / 256;
  if (bx > 152 * 16) bx = 152 * 16;
  const dim3 grid((unsigned)bx, dims == 3 ? 8 : 4, dims);
  if (dims == 3)
    link_integral_table_kernel<3><<<grid, 256, 0, s>>>(out, raw, N[0], N[1], N[2], pstride, q, dirs);
  else
    link_integral_table_kernel<2><<<grid, 256, 0, s>>>(out, raw, N[0], N[1], 1, pstride, q, dirs);
}

template <class P>
void launch_link_factor_table(typename P::Link* out, const FieldDesc& f, int dims, const int N[3], long long pstride,
                              int quads, int dirs, cudaStream_t s) {
  const long long ncell = (long long)N[0] * N[1] * (dims == 3 ? N[2] : 1);
  long long bx = (ncell + 255) / 256;
  if (bx > 152 * 16) bx = 152 * 16;
  const dim3 grid((unsigned)bx, dims == 3 ? 8 : 4, dirs * dims);
  if (dims == 3)
    link_factor_table_kernel<P, 3><<<grid, 256, 0, s>>>(out, f, N[0], N[1], N[2], pstride, quads, dirs);
  else
    link_factor_table_kernel<P, 2><<<grid, 256, 0, s>>>(out, f, N[0], N[1], 1, pstride, quads, dirs);
}
template void launch_link_factor_table<F32>(F32::Link*, const FieldDesc&, int, const int[3], long long, int, int,
                                            cudaStream_t);
template void launch_link_factor_table<F64>(F64::Link*, const FieldDesc&, int, const int[3], long long, int, int,
                                            cudaStream_t);

void launch_finish_sums2(const double* partials, int nblocks, double* out, cudaStream_t s) {
  finish_sums_kernel<2><<<1, 64, 0, s>>>(partials, nblocks, out);
}

void launch_finish_sums(const double* partials, int nblocks, double* out, cudaStream_t s) {
  finish_sums_kernel<kObsSums><<<1, 32 * kObsSums, 0, s>>>(partials, nblocks, out);
}

static unsigned grid_for(long long n) {
  long long b = (n + 255) / 256;
  return (unsigned)(b > 152LL * 32 ? 152LL * 32 : (b < 1 ? 1 : b));
}
void launch_convert_in(const double2* src, float2* dst, long long n, cudaStream_t s) {
  convert_in_kernel<<<grid_for(n), 256, 0, s>>>(src, dst, n);
}
void launch_convert_out(const float2* src, double2* dst, long long n, cudaStream_t s) {
  convert_out_kernel<<<grid_for(n), 256, 0, s>>>(src, dst, n);
}
void launch_convert_in_quads(const double2* src0, const double2* src1, float4* dst, int lane, long long n,
                             cudaStream_t s) {
  convert_in_quads_kernel<<<grid_for(n), 256, 0, s>>>(src0, src1, dst, lane, n);
}
void launch_convert_out_quads(const float4* src, double2* dst0, double2* dst1, int lane, long long n,
                              cudaStream_t s) {
  convert_out_quads_kernel<<<grid_for(n), 256, 0, s>>>(src, dst0, dst1, lane, n);
}

}  // namespace dirac
