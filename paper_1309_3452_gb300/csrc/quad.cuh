// The FP32 state of the fused kernels and its packed update.
//
// Layout: one array of float4 per component (A, B, C, D in (3+1)D; u, v in
// (2+1)D), [z][y][x]; a cell's record holds the component's two sublattice
// values as {re 0, re 1, im 0, im 1} (plane 2c in slot 0, plane 2c + 1 in slot
// 1; component c starts at c * pstride records).  Both values of a component
// obey the same equation with the same sign class, so every packed .f32x2
// operation of the update works on the two sublattices at once: products with
// i are a change of register names, per-value coefficients sit in the lanes
// they are used in, and a cell moves through memory and shared memory as one
// 16-byte access per component.  (Lanes (re, im) of one value, the layout
// before, need a swap per product with an imaginary part and every coefficient
// broadcast to both lanes: 345 thread instructions per free (3+1)D cell and
// step and 651 with the laser's fields.)
//
// Every operation is the one site_update performs on the same value, in the
// same order and rounding, so the two agree bit for bit.
#pragma once

#include "common.cuh"

namespace dirac {

struct Quad {
  float2 re, im;  // lane x: sublattice 0, lane y: sublattice 1
};
__device__ __forceinline__ Quad quad(float4 v) { return Quad{make_float2(v.x, v.y), make_float2(v.z, v.w)}; }
__device__ __forceinline__ float4 pack4(const Quad& q) { return make_float4(q.re.x, q.re.y, q.im.x, q.im.y); }
// A record of the evolving state: an ordinary load.  The read-only path (__ldg) may
// be used for what no kernel writes while this one is resident, and a step is
// resident (waiting in depends()) while the step before writes the state and the
// launch before that a wave's link table.
__device__ __forceinline__ Quad ldq(const float4* p) { return quad(*p); }
__device__ __forceinline__ float2 qlane(const Quad& q, int l) {
  return l ? make_float2(q.re.y, q.im.y) : make_float2(q.re.x, q.im.x);
}
__device__ __forceinline__ Quad mkquad(float2 v0, float2 v1) {
  return Quad{make_float2(v0.x, v1.x), make_float2(v0.y, v1.y)};
}

// up - dn lane by lane: the lanes of an x or y difference come from different
// records, where packed operands would first have to be moved together
__device__ __forceinline__ Quad qsub_lanes(const Quad& a, const Quad& b) {
  return Quad{make_float2(rsub(a.re.x, b.re.x), rsub(a.re.y, b.re.y)),
              make_float2(rsub(a.im.x, b.im.x), rsub(a.im.y, b.im.y))};
}
__device__ __forceinline__ Quad qadd_lanes(const Quad& a, const Quad& b) {
  return Quad{make_float2(radd(a.re.x, b.re.x), radd(a.re.y, b.re.y)),
              make_float2(radd(a.im.x, b.im.x), radd(a.im.y, b.im.y))};
}
__device__ __forceinline__ Quad qsub(const Quad& a, const Quad& b) {
  return Quad{psub(a.re, b.re), psub(a.im, b.im)};
}

// link_mul / link_mulc of both values, the link's parts per lane
struct QuadLink {
  float2 c_hi, c_lo, s_hi, s_lo;  // the link is c + i s (s = -sin phi)
};
__device__ __forceinline__ QuadLink quad_link(const F32::Link& L) {
  return QuadLink{f2(L.hi.x), f2(L.lo.x), f2(L.hi.y), f2(L.lo.y)};
}
__device__ __forceinline__ Quad link_mul(const QuadLink& L, const Quad& v) {
  float2 re = pfma(L.c_lo, v.re, pneg(pmul(L.s_lo, v.im)));
  float2 im = pfma(L.c_lo, v.im, pmul(L.s_lo, v.re));
  re = pfma(L.c_hi, v.re, pfma(pneg(L.s_hi), v.im, re));
  im = pfma(L.c_hi, v.im, pfma(L.s_hi, v.re, im));
  return Quad{re, im};
}
__device__ __forceinline__ Quad link_mulc(const QuadLink& L, const Quad& v) {
  float2 re = pfma(L.c_lo, v.re, pmul(L.s_lo, v.im));
  float2 im = pfma(L.c_lo, v.im, pneg(pmul(L.s_lo, v.re)));
  re = pfma(L.c_hi, v.re, pfma(L.s_hi, v.im, re));
  im = pfma(L.c_hi, v.im, pfma(pneg(L.s_hi), v.re, im));
  return Quad{re, im};
}
// plane_link_diff of both values: c (up - dn) - i s (up + dn)
__device__ __forceinline__ Quad plane_link_diff(float2 ch, float2 cl, float2 sp, float2 lp, const Quad& up,
                                                const Quad& dn) {
  const Quad D = qsub_lanes(up, dn), Q = qadd_lanes(up, dn);
  float2 re = pmul(cl, D.re), im = pmul(cl, D.im);
  re = pfma(lp, Q.im, re);
  im = pfma(pneg(lp), Q.re, im);
  re = pfma(sp, Q.im, re);
  im = pfma(pneg(sp), Q.re, im);
  return Quad{pfma(ch, D.re, re), pfma(ch, D.im, im)};
}

// combine<F32, DIMS> of both values
template <int DIMS, bool kIso>
__device__ __forceinline__ Quad combine_quad(const Quad& dx, const Quad& dy, const Quad& dz, int p,
                                             const F32::Ratio& ry, const F32::Ratio& rz) {
  if (!kIso) {
    const float2 tre = p ? pneg(dy.im) : dy.im, tim = p ? dy.re : pneg(dy.re);
    Quad s{padd(dx.re, ratio_mul(ry, tre)), padd(dx.im, ratio_mul(ry, tim))};
    if (DIMS == 3) {
      s.re = padd(s.re, ratio_mul(rz, p ? pneg(dz.re) : dz.re));
      s.im = padd(s.im, ratio_mul(rz, p ? pneg(dz.im) : dz.im));
    }
    return s;
  }
  Quad s = p ? Quad{psub(dx.re, dy.im), padd(dx.im, dy.re)} : Quad{padd(dx.re, dy.im), psub(dx.im, dy.re)};
  if (DIMS == 3) s = p ? Quad{psub(s.re, dz.re), psub(s.im, dz.im)} : Quad{padd(s.re, dz.re), padd(s.im, dz.im)};
  return s;
}

// apply of both values (one coefficient for both)
__device__ __forceinline__ Quad apply_quad(const F32::Coef& c, const Quad& F, const Quad& S) {
  float2 re = pmul(f2(c.g_lo.y), S.im), im = pmul(f2(-c.g_lo.y), S.re);
  re = pfma(f2(-c.g_lo.x), S.re, re);
  im = pfma(f2(-c.g_lo.x), S.im, im);
  re = pfma(f2(-c.a_lo.y), F.im, re);
  im = pfma(f2(c.a_lo.y), F.re, im);
  re = pfma(f2(c.a_lo.x), F.re, re);
  im = pfma(f2(c.a_lo.x), F.im, im);
  re = pfma(f2(c.g_hi.y), S.im, re);
  im = pfma(f2(-c.g_hi.y), S.re, im);
  re = pfma(f2(-c.g_hi.x), S.re, re);
  im = pfma(f2(-c.g_hi.x), S.im, im);
  re = pfma(f2(-c.a_hi.y), F.im, re);
  im = pfma(f2(c.a_hi.y), F.re, im);
  return Quad{pfma(f2(c.a_hi.x), F.re, re), pfma(f2(c.a_hi.x), F.im, im)};
}
// apply of both values with coefficients of their own, from lane_coefs' records
__device__ __forceinline__ Quad apply_lanes(const float4* t, const Quad& F, const Quad& S) {
  const Quad ah = quad(t[0]), gh = quad(t[32]), al = quad(t[64]), gl = quad(t[96]);
  float2 re = pmul(gl.im, S.im), im = pmul(pneg(gl.im), S.re);
  re = pfma(pneg(gl.re), S.re, re);
  im = pfma(pneg(gl.re), S.im, im);
  re = pfma(pneg(al.im), F.im, re);
  im = pfma(al.im, F.re, im);
  re = pfma(al.re, F.re, re);
  im = pfma(al.re, F.im, im);
  re = pfma(gh.im, S.im, re);
  im = pfma(pneg(gh.im), S.re, im);
  re = pfma(pneg(gh.re), S.re, re);
  im = pfma(pneg(gh.re), S.im, im);
  re = pfma(pneg(ah.im), F.im, re);
  im = pfma(ah.im, F.re, im);
  return Quad{pfma(ah.re, F.re, re), pfma(ah.re, F.im, im)};
}
// a lane's four records (alpha hi, gamma hi, alpha lo, gamma lo; 32 lanes
// interleaved) of a half-step, value l beyond the step where beyond[l]
__device__ __forceinline__ void lane_coefs(const HalfFields<F32>& h, bool beyond0, bool beyond1, float4* t) {
  auto rec = [&](float2 F32::Coef::*m) {
    const float2 i = h.c_in.*m, o = h.c_out.*m;
    return make_float4(beyond0 ? o.x : i.x, beyond1 ? o.x : i.x, beyond0 ? o.y : i.y, beyond1 ? o.y : i.y);
  };
  t[0] = rec(&F32::Coef::a_hi);
  t[32] = rec(&F32::Coef::g_hi);
  t[64] = rec(&F32::Coef::a_lo);
  t[96] = rec(&F32::Coef::g_lo);
}
// w = 2F - r_x S' of both values, small product first
__device__ __forceinline__ Quad two_f_minus_s(float rxh, float rxl, const Quad& F, const Quad& S) {
  return Quad{pfma(f2(-rxh), S.re, pfma(f2(-rxl), S.re, padd(F.re, F.re))),
              pfma(f2(-rxh), S.im, pfma(f2(-rxl), S.im, padd(F.im, F.im)))};
}
// apply_b of both values
__device__ __forceinline__ Quad apply_b_quad(const SoftB2& b, float rxh, float rxl, const Quad& F, const Quad& S) {
  const Quad w = two_f_minus_s(rxh, rxl, F, S);
  float2 re = pmul(b.re_lo, w.re), im = pmul(b.re_lo, w.im);
  re = pfma(b.im_lo, pneg(w.im), re);
  im = pfma(b.im_lo, w.re, im);
  re = pfma(b.im_hi, pneg(w.im), re);
  im = pfma(b.im_hi, w.re, im);
  re = pfma(b.re_hi, w.re, re);
  im = pfma(b.re_hi, w.im, im);
  return Quad{psub(re, F.re), psub(im, F.im)};
}
// apply_table of both values, the quad records of the two values (one record
// when both belong to the same cell)
__device__ __forceinline__ Quad apply_table_quad(float4 bh, float4 bl, float rxh, float rxl, const Quad& F,
                                                 const Quad& S) {
  const Quad w = two_f_minus_s(rxh, rxl, F, S);
  const Quad h = quad(bh), l = quad(bl);
  float2 re = pfma(l.re, w.re, pneg(pmul(l.im, w.im)));
  float2 im = pfma(l.re, w.im, pmul(l.im, w.re));
  re = pfma(h.re, w.re, pfma(pneg(h.im), w.im, re));
  im = pfma(h.re, w.im, pfma(h.im, w.re, im));
  return Quad{psub(re, F.re), psub(im, F.im)};
}

// both lanes' record: lane 0 from r0, lane 1 from r1 (the (2+1)D kernels
// update u0 and u1 of neighbouring rows together)
__device__ __forceinline__ float4 lanes_of(float4 r0, float4 r1) { return make_float4(r0.x, r1.y, r0.z, r1.w); }

// The update of both values of component comp (planes 2 comp and 2 comp + 1).
// up, dn: the neighbours at +-dx_a/2 of each lane's value; H0, H1, site0, site1
// and class0, class1: each lane's half-lattice point, cell and class (COEF_TABLE).  bpre: the coefficients of
// the pair where the caller forms them (COEF_SOFTCORE, COEF_SOFTCORR); lk: the
// staged link factor of LINK_PLANE_ZX; lanes: COEF_LANES; w0, w1: the lanes'
// factors (c_hi, c_lo, s_hi, s_lo) of LINK_PLANE.
// kOneCell: site0 == site1, class0 == class1.  kIso: r_x = r_y = r_z (a template parameter: a
// test here, uniform as it is, would end the compiler's basic block at every
// component and keep it from overlapping the chains of the others).
template <int DIMS, int COEF, int LINK, bool kOneCell, bool kIso>
__device__ __forceinline__ Quad quad_update(const HalfFields<F32>& h, const FieldDesc& f, bool iso,
                                            const F32::Ratio& ry, const F32::Ratio& rz, int comp, const Quad& F,
                                            const Quad (&up)[3], const Quad (&dn)[3], const int (&H0)[3],
                                            const int (&H1)[3], long long site0, long long site1, long long class0, long long class1, long long pstride,
                                            Quad* S_out, const SoftB2* bpre, const PlaneLink32* lk,
                                            const int (&N)[3], const float4* lanes = nullptr,
                                            const float4* w0 = nullptr, const float4* w1 = nullptr) {
  if constexpr (COEF == kAnyMode || LINK == kAnyMode) {
    // the per-site FP64 paths and rare combinations: one value at a time
    float2 r[2], S[2];
#pragma unroll
    for (int l = 0; l < 2; ++l) {
      float2 nb[6];
#pragma unroll
      for (int ax = 0; ax < 3; ++ax) {
        nb[2 * ax] = qlane(up[ax < DIMS ? ax : 0], l);
        nb[2 * ax + 1] = qlane(dn[ax < DIMS ? ax : 0], l);
      }
      r[l] = site_update<F32, DIMS, kAnyMode, kAnyMode>(h, f, iso, ry, rz, 2 * comp + l, qlane(F, l), nb,
                                                        l ? H1 : H0, l ? site1 : site0, pstride, &S[l], N);
    }
    if (S_out) *S_out = mkquad(S[0], S[1]);
    return mkquad(r[0], r[1]);
  } else {
    Quad d[3];
#pragma unroll
    for (int ax = 0; ax < DIMS; ++ax) {
      if constexpr (LINK == LINK_CONST) {
        const QuadLink L = quad_link(h.L[ax]);
        d[ax] = qsub(link_mul(L, up[ax]), link_mulc(L, dn[ax]));
      } else if constexpr (LINK == LINK_TABLE) {
        constexpr int nc = nplanes<DIMS>() / 2;
        QuadLink L[2];
#pragma unroll
        for (int dir = 0; dir < 2; ++dir) {
          const float4* t = h.lq + 2 * (long long)((2 * ax + dir) * nc + comp) * h.q_ps;
          float4 hi = __ldg(t + 2 * site0), lo = __ldg(t + 2 * site0 + 1);
          if (!kOneCell) {
            hi = lanes_of(hi, __ldg(t + 2 * site1));
            lo = lanes_of(lo, __ldg(t + 2 * site1 + 1));
          }
          L[dir] = QuadLink{quad(hi).re, quad(lo).re, quad(hi).im, quad(lo).im};
        }
        d[ax] = qsub(link_mul(L[0], up[ax]), link_mulc(L[1], dn[ax]));
      } else {
        d[ax] = ax == 2 ? qsub(up[ax], dn[ax]) : qsub_lanes(up[ax], dn[ax]);
      }
    }
    if constexpr (LINK == LINK_PLANE_ZX)  // the factor of the values' z level, staged by the caller
      d[0] = plane_link_diff(lk->ch, lk->cl, lk->sp, lk->lp, up[0], dn[0]);
    if constexpr (LINK == LINK_PLANE) {
      const float4 v0 = *w0, v1 = *w1;  // each lane's factor
      const float2 ch = make_float2(v0.x, v1.x), cl = make_float2(v0.y, v1.y);
      const float2 sp = make_float2(v0.z, v1.z), lp = make_float2(v0.w, v1.w);
      if (h.lpol == 0) d[0] = plane_link_diff(ch, cl, sp, lp, up[0], dn[0]);
      else if (h.lpol == 1) d[1] = plane_link_diff(ch, cl, sp, lp, up[1], dn[1]);
      else if (DIMS == 3) d[2] = plane_link_diff(ch, cl, sp, lp, up[2], dn[2]);
    }
    if (DIMS == 2) d[2] = d[0];
    const Quad S = combine_quad<DIMS, kIso>(d[0], d[1], d[2], sign_class<DIMS>(2 * comp), ry, rz);
    if (S_out) *S_out = S;
    if constexpr (COEF == COEF_UNIFORM) {
      return apply_quad(h.c_in, F, S);
    } else if constexpr (COEF == COEF_BEYOND) {
      return apply_quad(h.c_out, F, S);
    } else if constexpr (COEF == COEF_LANES) {
      return apply_lanes(lanes, F, S);
    } else if constexpr (COEF == COEF_STEP) {
      // both values on one side of the step almost everywhere: one apply, two
      // (and a choice per lane) only in the cells the step cuts
      const int a0 = h.step_axis == 0 ? H0[0] : (h.step_axis == 1 ? H0[1] : H0[2]);
      const int a1 = h.step_axis == 0 ? H1[0] : (h.step_axis == 1 ? H1[1] : H1[2]);
      const bool b0 = a0 >= h.step_X, b1 = a1 >= h.step_X;
      Quad r;
      if (!(b0 && b1)) r = apply_quad(h.c_in, F, S);
      if (b0 || b1) {
        const Quad q = apply_quad(h.c_out, F, S);
        if (b0) r.re.x = q.re.x, r.im.x = q.im.x;
        if (b1) r.re.y = q.re.y, r.im.y = q.im.y;
      }
      return r;
    } else if constexpr (COEF == COEF_TABLE) {
      const float4* t = h.bq + 2 * (long long)comp * h.b_ps;
      float4 bh = __ldg(t + 2 * class0), bl = __ldg(t + 2 * class0 + 1);
      if (!kOneCell) {
        bh = lanes_of(bh, __ldg(t + 2 * class1));
        bl = lanes_of(bl, __ldg(t + 2 * class1 + 1));
      }
      return apply_table_quad(bh, bl, h.rx_hi, h.rx_lo, F, S);
    } else if constexpr (COEF == COEF_SOFTCORE || COEF == COEF_SOFTCORR) {
      if (bpre) return apply_b_quad(*bpre, h.rx_hi, h.rx_lo, F, S);
      float Rh0, Rl0, Rh1, Rl1;
      softcore_R<DIMS>(h, H0, Rh0, Rl0);
      softcore_R<DIMS>(h, H1, Rh1, Rl1);
      const float2 Rh = make_float2(Rh0, Rh1), Rl = make_float2(Rl0, Rl1);
      const float2 t0 = softcore_t0(h, H0), t1 = softcore_t0(h, H1);
      SoftB2 b;
      if constexpr (COEF == COEF_SOFTCORE) {
        b = softcore_b2(Rh, Rl, make_float2(t0.x, t1.x), make_float2(t0.y, t1.y), h.sc_K_hi, h.sc_K_lo);
      } else {
        softcore_fast2(Rh, Rl, make_float2(t0.x, t1.x), h.sc_K_hi, b.re_hi, b.im_hi);
        const float2 c0 = corr_decode(__ldg(h.sc_corr + softcore_corr_index<DIMS>(2 * comp, H0, N)));
        const float2 c1 = corr_decode(__ldg(h.sc_corr + softcore_corr_index<DIMS>(2 * comp + 1, H1, N)));
        b.re_lo = make_float2(c0.x, c1.x);
        b.im_lo = make_float2(c0.y, c1.y);
      }
      return apply_b_quad(b, h.rx_hi, h.rx_lo, F, S);
    } else {
      static_assert(COEF == COEF_UNIFORM, "a coefficient path without a packed form");
      return F;
    }
  }
}

}  // namespace dirac
