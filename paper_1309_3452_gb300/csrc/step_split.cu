// One kernel per half-step: every thread owns one cell and updates the values
// of one parity class (upper: A0,A1,B0,B1 / u0,u1; lower: C0,C1,D0,D1 /
// v0,v1) in place.  In-place is race-free: a half-step reads only values of
// the other parity (Eqs. ss1-ss4: A,B from C,D at t; C,D from the new A,B).
// This is the plain reference path (and the FP64 validation path); the fused
// kernels compute the same values with the same per-value arithmetic.
//
// Bound, FP64: the FP64 pipe (0.5e12 instructions per second on the whole GPU;
// 144 per free (3+1)D cell and step are 246 us at 96^3, measured 249), so what
// counts is that nothing but the update runs on it: potentials and link factors
// come from tables.  us per step, before and now: 64^3 soft core in a plane wave
// 1388 / 131 (per-site square roots, divisions and sines before), 96^3 free
// 254 / 249, 64^2 free 5.5 / 5.0 (two launches).
#include "fused_common.cuh"

namespace dirac {

namespace {

// depends() for half-steps: the next half-step's blocks are placed early only by
// grids of at most a block per SM.  Placed while this one's run they go where
// there is room, not where there is work left: with a few blocks per SM some SMs
// then get more than their share (67 x 39 x 24 Klein step, FP64, 720 blocks: 58 us
// per step, 37 so; 96^3 249 and 64^2 5.0 either way).
__device__ __forceinline__ void depends_half_step(bool early) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (early) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <class P, int DIMS, bool UPPER, int COEF, int LINK>
__global__ void __launch_bounds__(128) half_step_kernel(const HalfStepArgs<P> a) {
  depends_half_step(a.early != 0);
  using C = typename P::cplx;
  const int x = blockIdx.x * 32 + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z;
  const int Nx = a.N[0], Ny = a.N[1], Nz = DIMS == 3 ? a.N[2] : 1;
  if (x >= Nx || y >= Ny) return;
  const long long nxy = (long long)Nx * Ny;
  const long long cell = z * nxy + (long long)y * Nx + x;
  const int j[3] = {x, y, z};
  const int Nn[3] = {Nx, Ny, Nz};
  const long long stride[3] = {1, Nx, nxy};
  constexpr int half = nplanes<DIMS>() / 2;
  constexpr int first = UPPER ? 0 : half;
#pragma unroll
  for (int k = 0; k < half; ++k) {
    const int plane = first + k;
    C* self = a.pl[plane];
    int H[3];
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) H[ax] = 2 * j[ax] + plane_off<DIMS>(plane, ax);
    C nb[6];
#pragma unroll
    for (int ax = 0; ax < DIMS; ++ax) {
      const C* src = a.pl[partner<DIMS>(plane, ax)];
#pragma unroll
      for (int dir = 0; dir < 2; ++dir) {
        int jj = j[ax] + nb_shift<DIMS>(plane, ax, dir == 0 ? +1 : -1);
        jj = jj >= Nn[ax] ? jj - Nn[ax] : (jj < 0 ? jj + Nn[ax] : jj);
        nb[2 * ax + dir] = src[cell + (long long)(jj - j[ax]) * stride[ax]];
      }
    }
    self[cell] = site_update<P, DIMS, COEF, LINK>(a.h, a.f, a.iso != 0, a.ry, a.rz, plane, self[cell],
                                               nb, H, cell, a.pstride, nullptr, a.N);
  }
}

template <class P, int DIMS, bool UPPER>
void launch_one(HalfStepArgs<P> a, cudaStream_t s) {
  // blocks of four rows, or of one where that leaves SMs without work (the FP64
  // pipe is narrow: 64^2 in 32 blocks kept 32 of 152 busy, 5.55 us per step; 4.97 in 128)
  const long long blocks4 = (long long)((a.N[0] + 31) / 32) * ((a.N[1] + 3) / 4) * (DIMS == 3 ? a.N[2] : 1);
  const int rows = blocks4 < 2 * fused::sm_count() ? 1 : 4;
  dim3 block(32, rows);
  dim3 grid((a.N[0] + 31) / 32, (a.N[1] + rows - 1) / rows, DIMS == 3 ? a.N[2] : 1);
  a.early = (long long)grid.x * grid.y * grid.z <= fused::sm_count();
  const int c = a.h.coef_mode, l = a.h.link_mode;
  constexpr bool f32 = sizeof(typename P::real) == 4;
#define HALF_STEP(COEF, LINK) launch_dependent(half_step_kernel<P, DIMS, UPPER, COEF, LINK>, grid, block, 0, s, a)
  if (c == COEF_UNIFORM && l == LINK_NONE) HALF_STEP(COEF_UNIFORM, LINK_NONE);
  else if (c == COEF_STEP && l == LINK_NONE) HALF_STEP(COEF_STEP, LINK_NONE);
  else if (c == COEF_TABLE && l == LINK_NONE) HALF_STEP(COEF_TABLE, LINK_NONE);
  else if (c == COEF_UNIFORM && l == LINK_PLANE) HALF_STEP(COEF_UNIFORM, LINK_PLANE);
  else if (c == COEF_STEP && l == LINK_PLANE) HALF_STEP(COEF_STEP, LINK_PLANE);
  else if (c == COEF_TABLE && l == LINK_PLANE) HALF_STEP(COEF_TABLE, LINK_PLANE);
  else if (f32 && c == COEF_SOFTCORE && l == LINK_NONE) HALF_STEP(f32 ? COEF_SOFTCORE : COEF_TABLE, LINK_NONE);
  else if (f32 && c == COEF_SOFTCORE && l == LINK_PLANE) HALF_STEP(f32 ? COEF_SOFTCORE : COEF_TABLE, LINK_PLANE);
  else if (f32 && c == COEF_SOFTCORR && l == LINK_NONE) HALF_STEP(f32 ? COEF_SOFTCORR : COEF_TABLE, LINK_NONE);
  else if (f32 && c == COEF_SOFTCORR && l == LINK_PLANE) HALF_STEP(f32 ? COEF_SOFTCORR : COEF_TABLE, LINK_PLANE);
  // FP64 (the FP32 reference kernels take these through the run-time path)
  else if (!f32 && c == COEF_UNIFORM && l == LINK_CONST) HALF_STEP(COEF_UNIFORM, f32 ? LINK_NONE : LINK_CONST);
  else if (!f32 && c == COEF_STEP && l == LINK_CONST) HALF_STEP(COEF_STEP, f32 ? LINK_NONE : LINK_CONST);
  else if (!f32 && c == COEF_TABLE && l == LINK_CONST) HALF_STEP(COEF_TABLE, f32 ? LINK_NONE : LINK_CONST);
  else if (!f32 && c == COEF_UNIFORM && l == LINK_UP) HALF_STEP(COEF_UNIFORM, f32 ? LINK_NONE : LINK_UP);
  else if (!f32 && c == COEF_STEP && l == LINK_UP) HALF_STEP(COEF_STEP, f32 ? LINK_NONE : LINK_UP);
  else if (!f32 && c == COEF_TABLE && l == LINK_UP) HALF_STEP(COEF_TABLE, f32 ? LINK_NONE : LINK_UP);
  else HALF_STEP(kAnyMode, kAnyMode);
#undef HALF_STEP
}

}  // namespace

template <class P, int DIMS>
void launch_half_step(const HalfStepArgs<P>& a, bool upper, cudaStream_t s) {
  if (upper)
    launch_one<P, DIMS, true>(a, s);
  else
    launch_one<P, DIMS, false>(a, s);
}

template void launch_half_step<F64, 2>(const HalfStepArgs<F64>&, bool, cudaStream_t);
template void launch_half_step<F64, 3>(const HalfStepArgs<F64>&, bool, cudaStream_t);
template void launch_half_step<F32, 2>(const HalfStepArgs<F32>&, bool, cudaStream_t);
template void launch_half_step<F32, 3>(const HalfStepArgs<F32>&, bool, cudaStream_t);

}  // namespace dirac
