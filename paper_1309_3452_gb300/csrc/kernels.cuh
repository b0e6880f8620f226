// Kernel argument blocks and launcher declarations of libdirac.
#pragma once

#include <type_traits>

#include "common.cuh"

namespace dirac {

// Launches that follow one another on a stream are made as programmatic
// dependents: the next kernel's blocks are placed while the last blocks of the
// one before still run, and wait in depends() until that one has finished and
// its writes are visible.  Every kernel launched this way calls depends() before
// it touches memory, and reads what an earlier launch wrote by ordinary loads
// (the wait orders those, not the read-only path), so the order of all work is
// that of plain launches; what is saved is the launch latency between short kernels.
// us per step, before and after: 96^3 FP64 254 / 249, 64^2 FP64 5.5 / 5.0,
// 203x149x91 84.5 / 82.8, 300 x 260 3.16 / 3.09; long kernels unchanged.
__device__ __forceinline__ void depends() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
template <class... A, class... B>
inline void launch_dependent(void (*kernel)(A...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, const B&... args) {
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = grid;
  c.blockDim = block;
  c.dynamicSmemBytes = smem;
  c.stream = s;
  c.attrs = &attr;
  c.numAttrs = 1;
  cudaLaunchKernelEx(&c, kernel, static_cast<A>(args)...);
}

// One half-step (all upper or all lower values) of the scheme, one kernel.
template <class P>
struct HalfStepArgs {
  typename P::cplx* pl[8];  // plane base pointers (updated in place)
  int N[3];
  long long pstride;
  int iso;                  // r_x = r_y (= r_z)
  typename P::Ratio ry, rz; // r_y/r_x, r_z/r_x
  HalfFields<P> h;
  FieldDesc f;
  int early;                // at most a block per SM (set by the launcher)
};

template <class P, int DIMS>
void launch_half_step(const HalfStepArgs<P>& a, bool upper, cudaStream_t s);

// One full time step (both half-steps) in one kernel, out of place.
template <class P>
struct FusedArgs {
  const float4* in[4];      // components (quad.cuh): A, B, C, D or u, v
  float4* out[4];
  int N[3];
  int chunk;                // levels (z in (3+1)D, y in (2+1)D) per work item
  int workers;              // persistent workers: blocks ((3+1)D) or warps ((2+1)D)
  long long pstride;
  int iso;
  typename P::Ratio ry, rz;
  HalfFields<P> hu, hl;     // upper / lower half-step fields
  int lstep;                // LINK_PLANE: table entries from one time step of a pass to the next
  FieldDesc f;
  // non-null: accumulate the conserved functional of the new state (per block
  // [sum |psi|^2, Re sum_lower conj(G) S'_G]; E = first + r_x second)
  double* e_partials;
  // levels along the marching axis ((3+1)D: z, (2+1)D: y): the kernel updates
  // the nzu levels zlo .. zlo + nzu - 1 of the N[axis] stored ones; a level k
  // lies at global level (zorg + k) mod Nzg, where every field is evaluated.
  // A whole grid: zlo = 0, nzu = Nzg = N[axis], zorg = 0 (periodic wrap of
  // the stored levels); a slab of a decomposed grid: its own levels between
  // one halo level on either side (zlo = 1, nzu = N[axis] - 2), zorg = its
  // first global level - 1.  (Passes of several steps and the batched kernels
  // take whole grids only.)
  int zlo, nzu, zorg, Nzg;
};
constexpr int kFusedEMaxBlocks = 4096;  // capacity of the per-block E partials
// (2+1)D fused kernel geometry
constexpr int kFused2dWarps = 4;   // independent x strips per block (few, so that small grids spread over the SMs)
constexpr int kMaxSteps2d = 2;     // most time steps per pass
constexpr int kTableSteps = 32;    // most time steps whose plane-wave link tables one launch forms

// returns the number of blocks launched
template <class P, int DIMS>
int launch_fused(const FusedArgs<P>& a, cudaStream_t s);

// Two time steps per pass of the (2+1)D fused kernel, for every field path but
// the per-site ones; plane waves take one link table per step (lstep).  Grids
// of at least four rows.  Returns the number of blocks
// launched, or 0, launching nothing, for the per-site field paths.
int launch_fused2d_two(const FusedArgs<F32>& a, cudaStream_t s);

// Several simulations (same dims and time-independent field modes) in one
// persistent launch of the fused kernels.
template <class P>
struct BatchArgs {
  const FusedArgs<P>* sims;      // device array, one entry per simulation (chunk set)
  const long long* first_item;   // device array [nsims + 1]: prefix sums of the items
  int nsims;
  int workers;                   // set by the launcher
};
// (`steps`: time steps per pass, 1; (2+1)D: 1 or 2)
// levels per work item for n grids in one batched launch (N[i] the extents):
// every chunk[i] that is 0 is set (launches of one grid take the rule for
// themselves where FusedArgs's chunk is 0)
void fused_batch_chunks(int dims, const int* const* N, int n, int steps, int* chunk);
// chunk lengths worth timing, best first by the planner's model; returns the count
int fused_candidates(int dims, const int N[3], int steps, int* out, int max);
long long fused_items(int dims, const int N[3], int steps, int chunk);
// one launch: uniform / Klein-step coefficients, no / constant links, all members isotropic or none
void launch_fused_batch(const BatchArgs<F32>& b, int dims, int steps, long long total_items, int coef_mode,
                        int link_mode, bool iso, cudaStream_t s);
// Observables of the stored state: per-block FP64 partial sums of
// [sum|psi|^2, Bx, By, Bz, sum_{beyond} |psi|^2] with
// B_a = Re sum_lower conj(G) s_a d_a(G)  (E = naive + r_x Bx + r_y By + r_z Bz).
template <class P>
struct ObsArgs {
  const typename P::cplx* pl[8];
  const float4* quads[4];   // F32 states held as quads (quad.cuh), else null
  int N[3];
  long long pstride;
  int link_mode;
  typename P::Link L[3];
  FieldDesc f;
  double t_links;           // time of the upper sheet (t - dt/2)
  // LINK_PLANE: the link factors at t_links by half-lattice coordinate along the
  // wave vector, PlaneLinkOf<P> (null: phases evaluated per link); LINK_TABLE
  // of quads
  const void* wave;
  int wave_axis;
  const float4* lq;
  const typename P::Link* larr;  // LINK_UP: the up links, [axis * larr_n + plane * pstride + cell]
  long long larr_n;
  int dens_axis, dens_X;    // partial density: half-lattice index >= dens_X along axis
  double* partials;         // [gridDim.x][5]
  int zlo, nzu, zorg, Nzg;  // levels summed along the marching axis and their global position, as in FusedArgs
};
constexpr int kObsSums = 5;

// the most blocks (= partial sums) the observables kernel uses for a grid;
// the launcher returns how many ran
int observables_blocks(const int N[3], int dims);
template <class P, int DIMS>
int launch_observables(const ObsArgs<P>& a, int blocks, cudaStream_t s);
// fixed-order sum of partials[nblocks][5] into out[5]
void launch_finish_sums(const double* partials, int nblocks, double* out, cudaStream_t s);
// fixed-order sum of partials[nblocks][2] into out[2]
void launch_finish_sums2(const double* partials, int nblocks, double* out, cudaStream_t s);

// table of plane-wave link factors exp(-i phi) for both half-steps of one time
// step: tab[half * n + H], H = half-lattice coordinate along `axis`, n = 2 N_axis;
// elements of PlaneLinkOf<P>::type
// (steps tables of consecutive time steps one after another, t_up and t_lo given per step)
template <class P>
void launch_link_table(void* tab, int n, const FieldDesc& f, int dims, int axis, int pol, const double* t_up,
                       const double* t_lo, int steps, cudaStream_t s);

// coefficient table of a time-independent potential (COEF_TABLE): every
// plane of the state layout (pstride), b = 1/(1 + i dt (beta m + V)/2) as
// {re hi, im hi, re lo, im lo}, or (quads) as the quad records of quad.cuh.
// rep (device, or null): N are the classes per axis and rep, axis after axis,
// one cell coordinate of each
void launch_coef_table(float4* tab, const FieldDesc& f, int dims, const int N[3], long long pstride, int quads,
                       const int* rep, cudaStream_t s);

// the FP64 kernels' table: alpha and gamma of every value, tab[plane * pstride + cell]
void launch_coef64_table(F64::Coef* tab, const FieldDesc& f, int dims, const int N[3], long long pstride,
                         cudaStream_t s);

// COEF_SOFTCORR correction records of a soft-core potential (one 32-bit word
// per value, softcore_corr_index's layout); *overflow (device) is or-ed with 1
// if a correction does not fit
void launch_softcore_corr(unsigned* out, const HalfFields<F32>& hu, const HalfFields<F32>& hl, const FieldDesc& f,
                          int dims, const int N[3], int* overflow, cudaStream_t s);

// link integrals of an arbitrary vector potential (Sect. 4): raw = the
// caller's integrals [axis][plane][cell] (canonical layout, cells dense), out
// = q times them per value in the state layout, slot 2a = the value's up link
// and 2a+1 = its down link (dirs = 1: slot a, the up link alone):
// out[slot * P * pstride + plane * pstride + cell]
void launch_link_integral_table(double* out, const double* raw, int dims, const int N[3], long long pstride,
                                double q, int dirs, cudaStream_t s);

// exp(-i phi) of every value's links of a time-independent vector potential:
// out[slot * P * pstride + plane * pstride + cell], or (quads, F32) the quad
// records of quad.cuh, slot by slot.  dirs = 2 (LINK_TABLE): slot 2a the up
// link along axis a, 2a+1 the down link; dirs = 1 (LINK_UP): slot a the up link
template <class P>
void launch_link_factor_table(typename P::Link* out, const FieldDesc& f, int dims, const int N[3], long long pstride,
                              int quads, int dirs, cudaStream_t s);

// measured FP64 FMA rate of the current device (TFLOP/s), < 0 on a CUDA failure
double measure_fp64_fma_tflops();

// canonical complex128 plane <-> device plane of the simulation precision
void launch_convert_in(const double2* src, float2* dst, long long n, cudaStream_t s);
void launch_convert_out(const float2* src, double2* dst, long long n, cudaStream_t s);
// the same for states held as quads: two planes <-> one component (lane < 0),
// or one plane <-> that sublattice of it (lane 0 or 1: src0 / dst0)
void launch_convert_in_quads(const double2* src0, const double2* src1, float4* dst, int lane, long long n,
                             cudaStream_t s);
void launch_convert_out_quads(const float4* src, double2* dst0, double2* dst1, int lane, long long n,
                              cudaStream_t s);

}  // namespace dirac
