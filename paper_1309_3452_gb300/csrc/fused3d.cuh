// One kernel per full time step (both half-steps of Eqs. ss1-ss4 / Eqs.
// scheme2Deq ff.), out of place: every value is read once from HBM and
// written once, neighbours come from registers, shuffles and shared memory.
// The state is held as sublattice quads (quad.cuh): one 16-byte access per
// component and cell, both values of a component updated together.
//
// (3+1)D: a block of 480 threads covers a 34 x 28 tile of cells in (x, y), or
// 512 threads a 34 x 30 one, and marches along z; every thread updates two
// cells stacked in y (rows ly, ly + 1), so the y neighbour inside the pair
// comes from registers.  Columns 0, 33 and the first and last row are a one-cell
// halo: they load and compute the upper half-step like every other cell, so the
// new upper values the interior needs from outside the tile exist in shared
// memory, but they store nothing.  Per z level k the block
//   1. holds the old A(k+1), C(k+1), D(k+1) and B(k) (B, C sit at z+1/2) in
//      registers, loaded while level k-1 was computed, publishes C(k+1) and
//      D(k+1) in shared memory and starts the loads of level k+1,
//   2. (the old C(k), D(k) and the new A(k), B(k-1) are in shared memory,
//      every tile double-buffered by level parity),
//   3. computes the new A(k+1) and B(k)      (upper half-step, t -> t+dt/2),
//   4. publishes them,
//   5. computes the new C(k) and D(k)        (lower half-step, t -> t+dt),
// A run of levels starts one level early to rebuild that state (the upper
// half-step of that level only).
//
// Scheduling: the grid holds the blocks that fit on the GPU at once (fewer
// for small grids); these persistent workers (blocks in (3+1)D, warps in
// (2+1)D) take work items round-robin.  An item is one tile over one chunk of
// levels, ordered chunk-major and tile-minor, so every round processes
// neighbouring tiles at the same levels at the same time and the overlapping
// halo loads hit L2.  The chunk length balances full rounds against the one
// restart level of each item.
//
// Bound: without fields the shared-memory queue and the two barriers of a level
// (2.6 and 1.6 of the stalled warps per issue at 128^3, the FP32 pipe 31 % busy;
// 54 us per step, its 128 bytes per cell take 40 at the copy rate); with a soft
// core and a plane wave the FP32 pipe (52 % busy over the kernel, stalled on it
// in the long chains) and the barriers.  Tiles of 34 x 28 and 34 x 30 cells are
// the largest that one block per SM can hold two cells per thread of: smaller
// ones spend more on halo cells (14 rows: 6114 us per 512^3 laser step against
// 3940).  us per step, with (re, im) lanes per value / now: 128^3 free 59.6 / 54.4, 203 x 149 x
// 91 Klein step anisotropic 102 / 82.8, 512^3 laser 4879 / 3940, 160^3 layers
// 227 / 141, 128^3 static links 670 / 395.
//
// Cells outside the grid (ragged last tiles) are wrapped periodically, so
// they compute correct duplicates and only the owning interior thread stores.
#pragma once

#include "fused_common.cuh"

namespace dirac {
namespace fused {

// (3+1)D tile geometry: kPairs row pairs, two cells per thread stacked in y.
// Two sizes are built: 14 pairs (34 x 28 cells, 480 threads) and 15 (34 x 30,
// 512 threads: 16 warps, four to each scheduler); tile_pairs says which runs.
template <int kPairs>
struct Tile3 {
  static constexpr int TW = 34, TH = 2 * kPairs;  // tile in cells
  static constexpr int CX = TW - 2, CY = TH - 2;  // interior
  static constexpr int threads = 32 * kPairs + 32;  // interior warps + one warp of halo columns and spares
  // shared-memory rows: a row below the tile, its TH rows, the spare threads'
  // pair of rows and a row above, so that every neighbour of every thread is at
  // a fixed offset from the thread's own slot and inside the array (what lies
  // outside the tile only feeds values that are never used)
  static constexpr int smem_rows = TH + 4;
  static constexpr int slots = smem_rows * TW + 2;  // slots per array (and the x+ neighbour of the last)
  // two level parities, each with the tiles of old C, old D, new B and new A
  static constexpr int tile = 4 * slots;
  static constexpr int tC = 0, tD = tile, tB = 2 * tile, tA = 3 * tile, parity = 4 * tile;
  static constexpr size_t smem = (size_t)2 * parity * sizeof(float);
  static_assert(2 * kPairs <= 32, "the halo columns fill at most one warp");
};

// A shared-memory tile holds re 0, re 1, im 0, im 1 of every slot as four float
// arrays.  A neighbour is one sublattice's value, two of the four words: from
// 16-byte records the compiler loads them as two words at a stride of four,
// with four-way bank conflicts (174 shared-memory wavefronts per 32 cells, the
// LSU data path 72 % busy and the limit); from word arrays every access is
// free of conflicts (78 wavefronts), and the lanes of a record land where the
// packed arithmetic wants them.
// a cell's record, and one sublattice's value, of the tile at t (slot applied)
template <int kSlots>
__device__ __forceinline__ Quad lds_quad(const float* t) {
  return Quad{make_float2(t[0], t[kSlots]), make_float2(t[2 * kSlots], t[3 * kSlots])};
}
template <int kSlots>
__device__ __forceinline__ float2 lds_value(const float* t, int l) {
  return make_float2(t[l * kSlots], t[(2 + l) * kSlots]);
}
template <int kSlots>
__device__ __forceinline__ void sts_quad(float* t, const Quad& q) {
  t[0] = q.re.x;
  t[kSlots] = q.re.y;
  t[2 * kSlots] = q.im.x;
  t[3 * kSlots] = q.im.y;
}

// The four records of one level load: A, C, D at level k+1 and B at level k.
struct LevelLoad {
  Quad A, B, C, D;
};

// Thread geometry inside the (3+1)D tile (two cells per thread, rows ly and
// ly + 1).  Warp w < kPairs holds the columns 1..32 (lane -> x) of the row pair
// (2w, 2w + 1); the first and the last row are halo rows, so warp 0's lower cell
// and the last pair's upper cell are halo cells.  The last warp holds the
// halo columns 0 and 33 of every row pair (2 kPairs threads) and the spare
// threads that are left (four with 14 pairs, two with 15; rows of their own in shared
// memory, never stored).  Halo cells take part in the upper half-step only,
// whose values the interior needs.
struct Thread3d {
  int slot;                // the lower cell's shared-memory slot, (ly + 1) * TW + lx (upper: slot + TW)
  int lx, ly;              // position of the lower cell in the tile
  bool halo;               // warp-uniform: halo columns and spares (upper half-step only)
  bool h0, h1;             // warp-uniform: the lower / upper cell is a halo cell
};

template <int kPairs>
__device__ __forceinline__ Thread3d thread3d() {
  constexpr int TW = Tile3<kPairs>::TW, TH = Tile3<kPairs>::TH;
  Thread3d th;
  const int t = threadIdx.x, w = t >> 5;
  if (w < kPairs) {
    th.lx = (t & 31) + 1;
    th.ly = 2 * w;
    th.halo = false;
  } else {
    const int h = t - 32 * kPairs;
    th.halo = true;
    if (h < kPairs) { th.lx = 0; th.ly = 2 * h; }
    else if (h < 2 * kPairs) { th.lx = TW - 1; th.ly = 2 * (h - kPairs); }
    else { th.lx = h - 2 * kPairs; th.ly = TH; }  // spare: rows of their own
  }
  th.h0 = th.halo || th.ly == 0;
  th.h1 = th.halo || th.ly + 1 == TH - 1;
  th.slot = (th.ly + 1) * TW + th.lx;
  return th;
}

// The x and y neighbours (up: +dx_a/2, dn: -dx_a/2) of both values of a
// component from its x-y partner component: own cell q, xt its tile at the
// cell's slot (for the cells at x -+ 1), ym1 the sublattice-1 value at y - 1,
// yp0 the sublattice-0 value at y + 1.  Sublattice 0 of A, C (kX = 0) has its
// x+ neighbour in its own cell, of B, D (kX = 1) its x- neighbour; along y
// sublattice 0 has y+ and sublattice 1 y- in its own cell on every component.
template <int kX, int kSlots>
__device__ __forceinline__ void xy_neighbours(const Quad& q, const float* xt, float2 ym1, float2 yp0, Quad (&up)[3],
                                              Quad (&dn)[3]) {
  if (kX == 0) {
    up[0] = mkquad(qlane(q, 0), lds_value<kSlots>(xt + 1, 1));
    dn[0] = mkquad(lds_value<kSlots>(xt - 1, 0), qlane(q, 1));
  } else {
    up[0] = mkquad(lds_value<kSlots>(xt + 1, 0), qlane(q, 1));
    dn[0] = mkquad(qlane(q, 0), lds_value<kSlots>(xt - 1, 1));
  }
  up[1] = mkquad(qlane(q, 1), yp0);
  dn[1] = mkquad(ym1, qlane(q, 0));
}

// tiles of a grid, and work items of a (3+1)D launch: tiles x chunks of the
// `levels` updated levels
template <int kPairs>
__host__ __device__ __forceinline__ long long tiles3d(const int (&N)[3]) {
  using T = Tile3<kPairs>;
  return (long long)((N[0] + T::CX - 1) / T::CX) * ((N[1] + T::CY - 1) / T::CY);
}
template <int kPairs>
__host__ __device__ __forceinline__ long long items3d(const int (&N)[3], int levels, int chunk) {
  return tiles3d<kPairs>(N) * ((levels + chunk - 1) / chunk);
}

// One work item (one tile over one chunk of z levels) of one simulation, two
// cells per thread stacked in y: cell 0 at row ly, cell 1 at row ly + 1.  The
// y neighbour of a cell inside the pair comes from the other cell's registers;
// the pair's outer y neighbours and all x neighbours come from shared memory.
// `a` may live in the constant bank (kernel parameter) or in shared memory.
template <class P, int COEF, int LINK, bool kE, int kPairs, bool kIso>
__device__ __forceinline__ void fused3d_item(const FusedArgs<P>& a, long long item, const Thread3d& th,
                                             unsigned char* smem_raw, double* e_acc) {
  using T = Tile3<kPairs>;
  constexpr int TW = T::TW, CX = T::CX, CY = T::CY, kSlots = T::slots, kThreads3d = T::threads;
  const int lx = th.lx, ly = th.ly;
  const int Nx = a.N[0], Ny = a.N[1], Nz = a.N[2];
  // global level of the stored level k (wrapped on the global grid), for the
  // fields; zorg + k lies in [-1, 2 Nzg) (zorg in [-1, Nzg), k <= N[2] <= Nzg + 1)
  auto gz = [&](int k) {
    const int g = a.zorg + k;
    return g < 0 ? g + a.Nzg : (g >= a.Nzg ? g - a.Nzg : g);
  };
  const int tiles_x = (Nx + CX - 1) / CX;
  const long long tiles = (long long)tiles_x * ((Ny + CY - 1) / CY);
  const bool iso = a.iso != 0;
  // record offsets inside a component: 32-bit (the host runs the fused kernels
  // only on grids of fewer than 2^31 cells), so an address is one wide
  // multiply-add
  using Off = unsigned;
  const Off nxy = (Off)Nx * (Off)Ny;
  const long long chunk = item / tiles, tile = item - chunk * tiles;
  const int z0 = a.zlo + (int)chunk * a.chunk;
  const int z1 = min(a.zlo + a.nzu, z0 + a.chunk);
  const int gx = (int)(tile % tiles_x) * CX + lx - 1;
  const int gy0 = (int)(tile / tiles_x) * CY + ly - 1, gy1 = gy0 + 1;
  const int x = wrapi(gx, Nx), y0 = wrapi(gy0, Ny), y1 = wrapi(gy1, Ny);
  const bool xin = lx >= 1 && lx <= CX && gx < Nx;
  const bool core0 = xin && !th.h0 && gy0 < Ny;
  const bool core1 = xin && !th.h1 && gy1 < Ny;
  const Off cxy0 = (Off)y0 * (Off)Nx + (Off)x, cxy1 = (Off)y1 * (Off)Nx + (Off)x;
  const int hx = 2 * x, hy0 = 2 * y0, hy1 = 2 * y1;
  // COEF_SOFTCORE: the x-y part of R = |x - c|^2 + a^2 of each cell of the
  // pair, as (hi, lo) pairs of two values: lanes (A0/C0, A1/C1) at (hx, hy),
  // (hx+1, hy+1) and (B0/D0, B1/D1) at (hx+1, hy), (hx, hy+1), kept in
  // shared memory (one record per thread and cell) so that they take no
  // registers through the z-march
  constexpr bool kSoft = COEF == COEF_SOFTCORE || COEF == COEF_SOFTCORR;
  __shared__ __align__(16) float4 sRxy[2][2][kSoft ? kThreads3d : 1];
  if constexpr (kSoft) {
    const float2 x0 = __ldg(a.hu.sc_sq[0] + hx), x1 = __ldg(a.hu.sc_sq[0] + hx + 1);
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int hy = c ? hy1 : hy0;
      const float2 ya = __ldg(a.hu.sc_sq[1] + hy), yb = __ldg(a.hu.sc_sq[1] + hy + 1);
      const float2 d00 = padd(x0, ya), d11 = padd(x1, yb), a10 = padd(x1, ya), a01 = padd(x0, yb);
      sRxy[c][0][threadIdx.x] = make_float4(d00.x, d11.x, d00.y, d11.y);
      sRxy[c][1][threadIdx.x] = make_float4(a10.x, a01.x, a10.y, a01.y);
    }
  }
  // COEF_TABLE: the x-y part of the two cells' classes
  constexpr bool kTab = COEF == COEF_TABLE;
  const unsigned* class_z = kTab ? a.hu.b_map + Nx + Ny : nullptr;
  Off cls0 = 0, cls1 = 0;
  if constexpr (kTab) {
    const Off cx = __ldg(a.hu.b_map + x);
    cls0 = cx + __ldg(a.hu.b_map + Nx + y0);
    cls1 = cx + __ldg(a.hu.b_map + Nx + y1);
  }
  // Per-level field constants, the same for the whole block, staged in
  // shared memory by threads 0..6 with copies that bypass the registers,
  // double-buffered by level parity (level k's copies are issued after the
  // first barrier of level k-1, when no thread reads that parity any more,
  // and waited for before the first barrier of level k):
  //   sLk[p][0..3]: plane-wave link factors along z (LINK_PLANE_ZX)
  //                 of A (upper half, Z = 2zn), B (upper, 2zk+1), C (lower,
  //                 2zk+1), D (lower, 2zk)
  //   sZq[p][0..2]: soft-core z terms sc_sq[2][Z] of Z = 2zn, 2zk+1, 2zk
  using PL = PlaneLink32;
  __shared__ __align__(16) PL sLk[2][4];
  __shared__ __align__(16) float2 sZq[2][3];
  // (the (3+1)D launchers run a plane wave along z polarised along x as
  // LINK_PLANE_ZX and send other plane waves to the general path)
  constexpr bool lk_z = LINK == LINK_PLANE_ZX;
  auto stage_level = [&](int k) {
    const int tid = threadIdx.x;
    if (tid >= 7) return;
    const int p = k & 1;
    const int zk = gz(k), zn = gz(k + 1);  // global levels: the tables are indexed by global Z
    if constexpr (lk_z) {
      if (tid < 4) {
        const int Z = tid == 0 ? 2 * zn : (tid == 3 ? 2 * zk : 2 * zk + 1);
        const PL* tab = static_cast<const PL*>(tid < 2 ? a.hu.ltab : a.hl.ltab);
        static_assert(sizeof(PL) % 16 == 0, "16-byte copies");
        for (int q = 0; q < (int)(sizeof(PL) / 16); ++q)
          cp_async16(reinterpret_cast<char*>(&sLk[p][tid]) + 16 * q,
                     reinterpret_cast<const char*>(tab + Z) + 16 * q);
      }
    }
    if constexpr (kSoft) {
      if (tid >= 4) {
        const int Z = tid == 4 ? 2 * zn : (tid == 5 ? 2 * zk + 1 : 2 * zk);
        cp_async8(&sZq[p][tid - 4], a.hu.sc_sq[2] + Z);
      }
    }
    cp_async_commit();
  };
  // the soft-core coefficients of the pair of values of a component of cell c:
  // xy 0 for A, C and 1 for B, D; z term z and positions H0, H1 (softcore_R's
  // sums, same order).  COEF_SOFTCORR: rec, slot of the correction words
  auto pair_b = [&](const HalfFields<P>& h, int c, int xy, float2 z, const int (&H0)[3], const int (&H1)[3],
                    Off rec, int slot) {
    SoftB2 b;
    if constexpr (kSoft) {
      const float4 r = sRxy[c][xy][threadIdx.x];
      const float2 Rh = padd(make_float2(r.x, r.y), f2(z.x)), Rl = padd(make_float2(r.z, r.w), f2(z.y));
      float2 th = f2(h.sc_t0[0].x), tl = f2(h.sc_t0[0].y);
      if (h.sc_step) {
        const float2 t0 = softcore_t0(h, H0), t1 = softcore_t0(h, H1);
        th = make_float2(t0.x, t1.x);
        tl = make_float2(t0.y, t1.y);
      }
      if constexpr (COEF == COEF_SOFTCORE) {
        b = softcore_b2(Rh, Rl, th, tl, h.sc_K_hi, h.sc_K_lo);
      } else {
        // the pair's two words of the level's correction record (read where used)
        const uint2 w = __ldg(reinterpret_cast<const uint2*>(a.hu.sc_corr + 8 * (long long)rec + slot));
        softcore_fast2(Rh, Rl, th, h.sc_K_hi, b.re_hi, b.im_hi);
        const float2 c0 = corr_decode(w.x), c1 = corr_decode(w.y);
        b.re_lo = make_float2(c0.x, c1.x);
        b.im_lo = make_float2(c0.y, c1.y);
      }
    }
    return b;
  };
  // both values of component comp (0 A, 1 B, 2 C, 3 D) of one cell: F the old
  // record, q, xt, ym1, yp0 the partner component around it (xy_neighbours), zu
  // and zd the z partner's records, Z the level's half-lattice z, site the cell,
  // rec its class (COEF_TABLE) or the cell of the level's correction record
  auto update = [&](auto comp_c, int cell, const Quad& F, const Quad& q, const float* xt, float2 ym1, float2 yp0,
                    const Quad& zu, const Quad& zd, int Z, float2 zq, Off site, Off rec, Quad* S, const PL* lk) {
    constexpr int comp = decltype(comp_c)::value;
    constexpr int xy = comp & 1;  // B, D: sublattice 0 at hx + 1
    const HalfFields<P>& h = comp < 2 ? a.hu : a.hl;
    const int hy = cell ? hy1 : hy0;
    const int H0[3] = {hx + xy, hy, Z}, H1[3] = {hx + 1 - xy, hy + 1, Z};
    Quad up[3], dn[3];
    xy_neighbours<xy, kSlots>(q, xt, ym1, yp0, up, dn);
    up[2] = zu;
    dn[2] = zd;
    SoftB2 b;
    if constexpr (kSoft) b = pair_b(h, cell, xy, zq, H0, H1, rec, 2 * comp);
    return quad_update<3, COEF, LINK, true, kIso>(h, a.f, iso, a.ry, a.rz, comp, F, up, dn, H0, H1, site, site, rec, rec, a.pstride, S,
                                            kSoft ? &b : nullptr, lk, a.N);
  };

  auto load = [&](int k, LevelLoad& l0, LevelLoad& l1) {
    const int zk = k < 0 ? k + Nz : k;
    const int zn = k + 1 >= Nz ? k + 1 - Nz : k + 1;
    const Off ok = (Off)zk * nxy, on = (Off)zn * nxy;
    l0.A = ldq(a.in[0] + (on + cxy0));
    l1.A = ldq(a.in[0] + (on + cxy1));
    l0.B = ldq(a.in[1] + (ok + cxy0));
    l1.B = ldq(a.in[1] + (ok + cxy1));
    l0.C = ldq(a.in[2] + (on + cxy0));
    l1.C = ldq(a.in[2] + (on + cxy1));
    l0.D = ldq(a.in[3] + (on + cxy0));
    l1.D = ldq(a.in[3] + (on + cxy1));
  };

  // the lower cell's slot in the parity of level k (tk) and of levels k - 1 and
  // k + 1 (tn), exchanged from level to level; the upper cell's is TW further
  float* tk = reinterpret_cast<float*>(smem_raw) + th.slot + ((z0 - 1) & 1) * T::parity;
  float* tn = reinterpret_cast<float*>(smem_raw) + th.slot + (z0 & 1) * T::parity;
  constexpr int YM = -TW, YP = 2 * TW;  // the pair's outer y neighbours
  {  // old C, D of level z0-1 (the z- neighbours of the first level)
    const Off zo = (Off)wrapi(z0 - 1, Nz) * nxy;
    sts_quad<kSlots>(tk + T::tC, ldq(a.in[2] + (zo + cxy0)));
    sts_quad<kSlots>(tk + T::tD, ldq(a.in[3] + (zo + cxy0)));
    sts_quad<kSlots>(tk + T::tC + TW, ldq(a.in[2] + (zo + cxy1)));
    sts_quad<kSlots>(tk + T::tD + TW, ldq(a.in[3] + (zo + cxy1)));
  }
  LevelLoad c0, c1;  // the level loads of the two cells
  load(z0 - 1, c0, c1);
  constexpr bool kStage = lk_z || kSoft;
  if (kStage) stage_level(z0 - 1);
  using IA = std::integral_constant<int, 0>;
  using IB = std::integral_constant<int, 1>;
  using IC = std::integral_constant<int, 2>;
  using ID = std::integral_constant<int, 3>;

  Off class_n = 0;  // COEF_TABLE: the z part of the classes of level k + 1
  if constexpr (kTab) class_n = __ldg(class_z + (z0 ? z0 - 1 : Nz - 1));
#pragma unroll 1
  for (int k = z0 - 1; k < z1; ++k) {
    const int zk = k < 0 ? k + Nz : k;
    const int zn = k + 1 >= Nz ? k + 1 - Nz : k + 1;
    const Off ok0 = (Off)zk * nxy + cxy0, on0 = (Off)zn * nxy + cxy0;
    const Off ok1 = (Off)zk * nxy + cxy1, on1 = (Off)zn * nxy + cxy1;
    Off rk0 = ok0, rn0 = ok0, rk1 = ok1, rn1 = ok1;
    if constexpr (kTab) {
      rk0 = class_n + cls0, rk1 = class_n + cls1;
      class_n = __ldg(class_z + zn);
      rn0 = class_n + cls0, rn1 = class_n + cls1;
    }
    const int pk = k & 1;
    const int Zk = 2 * gz(k), Zn = 2 * gz(k + 1);  // half-lattice z of levels k, k+1 (global)
    sts_quad<kSlots>(tn + T::tC, c0.C);  // old C(k+1), D(k+1): z+ / x,y neighbours now,
    sts_quad<kSlots>(tn + T::tD, c0.D);  // own old values at the next level
    sts_quad<kSlots>(tn + T::tC + TW, c1.C);
    sts_quad<kSlots>(tn + T::tD + TW, c1.D);
    // prefetch the next level while this one computes
    LevelLoad n0 = c0, n1 = c1;
    if (k + 1 < z1) load(k + 1, n0, n1);
    if (kStage && threadIdx.x < 7) cp_async_wait_all();  // this level's staged constants
    __syncthreads();
    if (kStage && k + 1 < z1) stage_level(k + 1);
    const float2 zq0 = kSoft ? sZq[pk][0] : make_float2(0.0f, 0.0f), zq1 = kSoft ? sZq[pk][1] : zq0;

    // upper half-step: A(k+1) from C(k+1), C(k), D(k+1); B(k) from D(k+1), D(k), C(k)
    const Quad oC0 = lds_quad<kSlots>(tk + T::tC), oC1 = lds_quad<kSlots>(tk + T::tC + TW);  // old C(k) of the two cells
    const Quad nA0 = update(IA{}, 0, c0.A, c0.D, tn + T::tD, lds_value<kSlots>(tn + T::tD + YM, 1), qlane(c1.D, 0), c0.C, oC0, Zn,
                            zq0, on0, rn0, nullptr, &sLk[pk][0]);
    const Quad nA1 = update(IA{}, 1, c1.A, c1.D, tn + T::tD + TW, qlane(c0.D, 1), lds_value<kSlots>(tn + T::tD + YP, 0), c1.C, oC1,
                            Zn, zq0, on1, rn1, nullptr, &sLk[pk][0]);
    const Quad nB0 = update(IB{}, 0, c0.B, oC0, tk + T::tC, lds_value<kSlots>(tk + T::tC + YM, 1), qlane(oC1, 0), c0.D,
                            lds_quad<kSlots>(tk + T::tD), Zk + 1, zq1, ok0, rk0, nullptr, &sLk[pk][1]);
    const Quad nB1 = update(IB{}, 1, c1.B, oC1, tk + T::tC + TW, qlane(oC0, 1), lds_value<kSlots>(tk + T::tC + YP, 0), c1.D,
                            lds_quad<kSlots>(tk + T::tD + TW), Zk + 1, zq1, ok1, rk1, nullptr, &sLk[pk][1]);
    sts_quad<kSlots>(tk + T::tB, nB0);
    sts_quad<kSlots>(tn + T::tA, nA0);
    sts_quad<kSlots>(tk + T::tB + TW, nB1);
    sts_quad<kSlots>(tn + T::tA + TW, nA1);
    __syncthreads();

    // lower half-step: C(k) from A(k+1), A(k), B(k); D(k) from B(k), B(k-1), A(k)
    // (interior cells only: nothing needs the halo's lower values; the
    // first level of a run only rebuilds A(z0) and B(z0-1))
    if (!th.halo) {
      if (k >= z0) {
        const float2 zq2 = kSoft ? sZq[pk][2] : zq0;
        const Quad oA0 = lds_quad<kSlots>(tk + T::tA), oA1 = lds_quad<kSlots>(tk + T::tA + TW);  // new A(k) of the two cells
        Quad S;
        Quad* Sp = kE ? &S : nullptr;
        if (!th.h0) {  // cell 0 (warp-uniform; one block of code per cell: computing
                       // the halo cells too, to interleave the two cells, was slower)
          float lc = 0.0f;
          const Quad nC = update(IC{}, 0, oC0, nB0, tk + T::tB, lds_value<kSlots>(tk + T::tB + YM, 1), qlane(nB1, 0), nA0, oA0,
                                 Zk + 1, zq1, ok0, rk0, Sp, &sLk[pk][2]);
          if (kE) lc = cross(nC, S, lc);
          const Quad nD = update(ID{}, 0, lds_quad<kSlots>(tk + T::tD), oA0, tk + T::tA, lds_value<kSlots>(tk + T::tA + YM, 1),
                                 qlane(oA1, 0), nB0, lds_quad<kSlots>(tn + T::tB), Zk, zq2, ok0, rk0, Sp, &sLk[pk][3]);
          if (core0) {
            if (kE) {  // this level's few terms in FP32, the running sums in FP64 (shared memory)
              e_acc[1] += cross(nD, S, lc);
              e_acc[0] += (n2(nB0) + n2(nC)) + n2(nD);
            }
            a.out[1][ok0] = pack4(nB0);
            a.out[2][ok0] = pack4(nC);
            a.out[3][ok0] = pack4(nD);
          }
        }
        if (!th.h1) {  // cell 1 (warp-uniform)
          float lc = 0.0f;
          const Quad nC = update(IC{}, 1, oC1, nB1, tk + T::tB + TW, qlane(nB0, 1), lds_value<kSlots>(tk + T::tB + YP, 0), nA1,
                                 oA1, Zk + 1, zq1, ok1, rk1, Sp, &sLk[pk][2]);
          if (kE) lc = cross(nC, S, lc);
          const Quad nD = update(ID{}, 1, lds_quad<kSlots>(tk + T::tD + TW), oA1, tk + T::tA + TW, qlane(oA0, 1),
                                 lds_value<kSlots>(tk + T::tA + YP, 0), nB1, lds_quad<kSlots>(tn + T::tB + TW), Zk, zq2, ok1, rk1, Sp,
                                 &sLk[pk][3]);
          if (core1) {
            if (kE) {
              e_acc[1] += cross(nD, S, lc);
              e_acc[0] += (n2(nB1) + n2(nC)) + n2(nD);
            }
            a.out[1][ok1] = pack4(nB1);
            a.out[2][ok1] = pack4(nC);
            a.out[3][ok1] = pack4(nD);
          }
        }
      }
      if (k + 1 < z1) {
        if (core0) {
          if (kE) e_acc[0] += n2(nA0);
          a.out[0][on0] = pack4(nA0);
        }
        if (core1) {
          if (kE) e_acc[0] += n2(nA1);
          a.out[0][on1] = pack4(nA1);
        }
      }
    }
    c0 = n0;
    c1 = n1;
    float* t = tk;
    tk = tn;
    tn = t;
  }
  __syncthreads();  // the next item rewrites the shared tiles
}

// kE: the launch also accumulates the conserved functional of the new state (a
// kernel of its own, so that the others carry neither its terms nor its tests)
template <class P, int COEF, int LINK, bool kE, int kPairs, bool kIso>
__global__ void __launch_bounds__(Tile3<kPairs>::threads, 1) fused3d_kernel(const FusedArgs<P> a) {
  depends();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int kThreads3d = Tile3<kPairs>::threads;
  const Thread3d th = thread3d<kPairs>();
  const long long items = items3d<kPairs>(a.N, a.nzu, a.chunk);
  // running sums of the functional, one FP64 pair per thread, kept in shared
  // memory so that they take no registers in the z-march
  __shared__ double e_acc[kE ? kThreads3d : 1][2];
  double* acc = e_acc[kE ? threadIdx.x : 0];
  if (kE) acc[0] = acc[1] = 0.0;
  for (long long item = blockIdx.x; item < items; item += a.workers)
    fused3d_item<P, COEF, LINK, kE, kPairs, kIso>(a, item, th, smem_raw, acc);
  if (kE) block_store_e(acc[0], acc[1], a.e_partials);
}

// tiles of the batched launches (one size, so that a simulation's items do not
// depend on its companions)
constexpr int kBatchPairs = 14;

// Several simulations in one persistent launch: global items are the
// simulations' items back to back; each block copies the arguments of the
// simulation its current item belongs to into shared memory.
template <class P, int COEF, int LINK, bool kIso>
__global__ void __launch_bounds__(Tile3<kBatchPairs>::threads, 1) fused3d_batch_kernel(const BatchArgs<P> b) {
  depends();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ FusedArgs<P> sa;
  const Thread3d th = thread3d<kBatchPairs>();
  const long long total = b.first_item[b.nsims];
  int cur = -1;
  for (long long g = blockIdx.x; g < total; g += b.workers) {
    const int s = find_sim(b.first_item, b.nsims, g);
    if (s != cur) {
      __syncthreads();  // everyone is done with the previous arguments
      copy_args(&sa, b.sims + s, (int)threadIdx.x, Tile3<kBatchPairs>::threads);
      __syncthreads();
      cur = s;
    }
    // (batched launches never accumulate the functional: e_partials is null)
    fused3d_item<P, COEF, LINK, false, kBatchPairs, kIso>(sa, g - b.first_item[s], th, smem_raw, nullptr);
  }
}

// resident blocks of a kernel, computed once (the template argument is the
// kernel itself), with its dynamic shared-memory limit raised
template <auto K, int kPairs>
int workers3d() {
  static int r = [] {
    cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Tile3<kPairs>::smem);
    return resident_blocks(K, Tile3<kPairs>::threads, Tile3<kPairs>::smem);
  }();
  return r;
}

// Row pairs of a grid's tiles: the fewer rows computed (tiles along y times
// their rows, halo and ragged last tile included); 15 pairs at equal rows are 5 %
// faster with a soft core (its arithmetic fills the four schedulers evenly; 512^3 laser
// 3940 us per step against 4084 with 14 pairs, 570 rows against 560) and even
// otherwise (160^3 layers with a coefficient record per cell 189 us per step with
// 15 pairs, 180 rows, against 206 with 14, 196 rows; 128^3 free 57.7 against 54.2, 150 rows against 140).
template <int COEF>
bool taller_tile(const int N[3]) {
  const long long r14 = (N[1] + Tile3<14>::CY - 1) / Tile3<14>::CY * Tile3<14>::TH;
  const long long r15 = (N[1] + Tile3<15>::CY - 1) / Tile3<15>::CY * Tile3<15>::TH;
  return COEF == COEF_SOFTCORE ? 95 * r15 < 100 * r14 : r15 < r14;
}
// the field paths built with both tiles (the others, the launches that
// accumulate the functional and anisotropic grids run with 14 pairs)
template <int COEF, int LINK>
constexpr bool both_tiles() {
  return COEF != kAnyMode && COEF != COEF_SOFTCORR && LINK != LINK_TABLE;
}

template <int COEF, int LINK, bool kE, int kPairs, bool kIso>
int launch3d_tile(FusedArgs<F32> a, cudaStream_t s) {
  constexpr auto k = fused3d_kernel<F32, COEF, LINK, kE, kPairs, kIso>;
  const int resident = workers3d<k, kPairs>();
  if (a.chunk <= 0 || a.chunk > a.nzu) a.chunk = plan_chunk(ChunkShape{tiles3d<kPairs>(a.N), a.nzu, resident, 4, 0.5});
  const long long items = items3d<kPairs>(a.N, a.nzu, a.chunk);
  a.workers = (int)(items < resident ? items : resident);
  // one E partial per block: never more blocks than the partials hold
  if (kE && a.workers > kFusedEMaxBlocks) a.workers = kFusedEMaxBlocks;
  launch_dependent(k, dim3((unsigned)a.workers), dim3(Tile3<kPairs>::threads), Tile3<kPairs>::smem, s, a);
  return a.workers;
}

template <int COEF, int LINK>
int launch3d(FusedArgs<F32> a, cudaStream_t s) {
  if constexpr (COEF != kAnyMode) {  // (the run-time path tests iso itself)
    if (!a.iso)
      return a.e_partials ? launch3d_tile<COEF, LINK, true, 14, false>(a, s)
                          : launch3d_tile<COEF, LINK, false, 14, false>(a, s);
  }
  if (a.e_partials) return launch3d_tile<COEF, LINK, true, 14, true>(a, s);
  if constexpr (both_tiles<COEF, LINK>())
    if (taller_tile<COEF>(a.N)) return launch3d_tile<COEF, LINK, false, 15, true>(a, s);
  return launch3d_tile<COEF, LINK, false, 14, true>(a, s);
}

template <int COEF, int LINK, bool kIso>
void launch3d_batch(BatchArgs<F32> b, long long total, cudaStream_t s) {
  constexpr auto k = fused3d_batch_kernel<F32, COEF, LINK, kIso>;
  const int resident = workers3d<k, kBatchPairs>();
  b.workers = (int)(total < resident ? total : resident);
  launch_dependent(k, dim3((unsigned)b.workers), dim3(Tile3<kBatchPairs>::threads), Tile3<kBatchPairs>::smem, s, b);
}

}  // namespace fused
}  // namespace dirac
