// Double-float arithmetic and the RSST step in it.
//
// A double-float is the unevaluated sum hi + lo of two float32 values with
// |lo| <= ulp(hi)/2: a 48-bit significand (relative rounding ~2^-48) in the
// float32 exponent range, computed entirely on the float32 pipe.  The
// operations are the classical error-free transformations with a fused
// multiply-add (Dekker 1971; Knuth, TAOCP vol. 2, Sec. 4.2.2; Shewchuk 1997):
//   two_sum(a, b):  s = a + b exactly as s + e,
//   two_prod(a, b): a * b exactly as p + e with e = fma(a, b, -p),
// followed by renormalisation.  Reciprocal and square root take the float32
// hardware value and one Newton step carried in double-float.
//
// The step functions mirror the float64 ones (rsst_math_fp64.cuh) term for
// term, with the same readings of Sec. 4.2 (MC limiter, LLF with
// c_tot = |V| + a/xi, ties to the left state) and the same corrections
// (Sec. 3.2, App. A) and force (App. B).
#pragma once

#include "rsst_common.cuh"
#include "rsst_internal.h"

namespace rsst {

struct df {
  float hi, lo;
};

__device__ __forceinline__ df df_make(float h, float l = 0.0f) { return {h, l}; }

__device__ __forceinline__ df fast_two_sum(float a, float b) {  // |a| >= |b|
  const float s = a + b;
  return {s, b - (s - a)};
}
__device__ __forceinline__ df two_sum(float a, float b) {
  const float s = a + b;
  const float bb = s - a;
  return {s, (a - (s - bb)) + (b - bb)};
}

__device__ __forceinline__ df operator+(df x, df y) {
  const df s = two_sum(x.hi, y.hi);
  return fast_two_sum(s.hi, s.lo + (x.lo + y.lo));
}
__device__ __forceinline__ df operator-(df x) { return {-x.hi, -x.lo}; }
__device__ __forceinline__ df operator-(df x, df y) { return x + (-y); }
__device__ __forceinline__ df operator*(df x, df y) {
  const float p = __fmul_rn(x.hi, y.hi);  // rounded by itself: never contracted into the sums that follow
  float e = fmaf(x.hi, y.hi, -p);
  e = fmaf(x.hi, y.lo, e);
  e = fmaf(x.lo, y.hi, e);
  return fast_two_sum(p, e);
}
// a b + c: the product's leading part and its exact error go into the sum
// unnormalised, 15 float operations instead of the 18 of * and +, one rounding
// less.
__device__ __forceinline__ df df_fma(df a, df b, df c) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = fmaf(a.hi, b.hi, -p);
  e = fmaf(a.hi, b.lo, e);
  e = fmaf(a.lo, b.hi, e);
  const df s = two_sum(p, c.hi);
  return fast_two_sum(s.hi, s.lo + (e + c.lo));
}
// exact scaling by a power of two
__device__ __forceinline__ df scale(df x, float p2) { return {x.hi * p2, x.lo * p2}; }

// 1/y: float32 reciprocal r0, then r0 + r0 (1 - y r0) with 1 - y r0 formed
// from the exact product y.hi * r0 = p + pe.
__device__ __forceinline__ df rcp(df y) {
  const float r0 = 1.0f / y.hi;
  const float p = __fmul_rn(y.hi, r0);
  const float pe = fmaf(y.hi, r0, -p);
  const float e = ((1.0f - p) - pe) - y.lo * r0;
  return fast_two_sum(r0, __fmul_rn(r0, e));
}

// sqrt(x), 0 for x <= 0: s0 = sqrt(x.hi), then s0 + (x - s0^2)/(2 s0).
__device__ __forceinline__ df dsqrt(df x) {
  if (!(x.hi > 0.0f)) return {0.0f, 0.0f};
  const float s0 = sqrtf(x.hi);
  const float p = __fmul_rn(s0, s0);
  const float pe = fmaf(s0, s0, -p);
  const float d = ((x.hi - p) - pe) + x.lo;
  return fast_two_sum(s0, __fmul_rn(d, 0.5f / s0));
}

__device__ __forceinline__ bool df_lt(df a, df b) { return a.hi < b.hi || (a.hi == b.hi && a.lo < b.lo); }
__device__ __forceinline__ bool df_le(df a, df b) { return a.hi < b.hi || (a.hi == b.hi && a.lo <= b.lo); }
__device__ __forceinline__ bool df_pos(df a) { return a.hi > 0.0f || (a.hi == 0.0f && a.lo > 0.0f); }

__device__ __forceinline__ df df_from(double d) {
  const float h = __double2float_rn(d);
  return {h, __double2float_rn(d - (double)h)};
}
__device__ __forceinline__ double df_to(df x) { return (double)x.hi + (double)x.lo; }

// The same two conversions with one float64 operation each (see d2f_rn).
__device__ __forceinline__ df df_from_bits(double d) {
  const float h = d2f_rn(d);
  return {h, d2f_rn(d - f2d(h))};
}
__device__ __forceinline__ double df_to_bits(df x) { return f2d(x.hi) + f2d(x.lo); }

// Constants of the step in double-float (split once on the host).
struct PhysDF {
  df gamma, gm1, nhgm1, inv_gm1, gam_gm1;  // nhgm1 = -(gamma - 1)/2, gam_gm1 = gamma/(gamma - 1)
  df gx;                                   // gamma/xi^2 (constant xi) over xs^2: in [1, 4)
  float xs;                                // a power of two, 0 below the floats
  df nf, nf_gm1, inv_cmax4;                // -f, -f (gamma - 1)
  df grav[3], nhalf_inv_dx[3], sum_inv_dx;  // nhalf_inv_dx = -1/(2 dx): the faces hold twice the flux
  int variant, use_cmax, has_grav;
};

// Half the MC limited slope (Sec. 4.2): 0 unless a, b are nonzero with one
// sign; else a if |a| <= |b| and 4|a| <= |a+b|, b if 4|b| <= |a+b|, else
// (a+b)/4.  Taken on the values times a's sign, where same-sign operands are
// positive and order as (hi, lo).
__device__ __forceinline__ df flip(df a, unsigned s) {
  return {__uint_as_float(__float_as_uint(a.hi) ^ s), __uint_as_float(__float_as_uint(a.lo) ^ s)};
}
__device__ __forceinline__ df half_mc_df(df a, df b) {
  const unsigned sa = __float_as_uint(a.hi) & 0x80000000u;
  const df aa = flip(a, sa), bb = flip(b, sa);
  const df q = scale(aa + bb, 0.25f);
  df m = df_le(aa, bb) ? aa : bb;
  m = df_le(m, q) ? m : q;
  m = flip(m, sa);
  return aa.hi > 0.0f && bb.hi > 0.0f ? m : df{0.0f, 0.0f};
}

// 1/sqrt(w) factor of the C_max law, w = 1 + a^4/C_max^4: (a/xi)^2 = a^2 w^(-1/2).
__device__ __forceinline__ df cmax_factor_df(df a2, const PhysDF& p) {
  return rcp(dsqrt(df_fma(a2 * a2, p.inv_cmax4, df_make(1.0f))));
}
// a/xi from P/rho: constant xi (gamma/xi^2 itself leaves a float's range from xi
// = 1e19 on, long before a/xi does), or the C_max law.
template <bool CMAX>
__device__ __forceinline__ df sound_df(df p_rho, const PhysDF& p) {
  if constexpr (CMAX) {
    const df a2 = p.gamma * p_rho;
    return dsqrt(a2 * cmax_factor_df(a2, p));
  }
  return scale(dsqrt(p.gx * p_rho), p.xs);
}

// The Euler flux along D and c_tot of one state; k = rho |V|^2 = m.V feeds
// the pressure directly.
template <int NV, int D, bool CMAX>
__device__ __forceinline__ void euler_flux_df(const df (&q)[NV], const PhysDF& p, df (&F)[NV], df& c) {
  constexpr int ND = NV - 2;
  const df ir = rcp(q[0]);
  df v[ND];
#pragma unroll
  for (int e = 0; e < ND; ++e) v[e] = q[1 + e] * ir;
  df k = q[1] * v[0];
#pragma unroll
  for (int e = 1; e < ND; ++e) k = df_fma(q[1 + e], v[e], k);
  const df P = df_fma(p.nhgm1, k, p.gm1 * q[NV - 1]);
  c = dsqrt(k * ir) + sound_df<CMAX>(P * ir, p);
  F[0] = q[1 + D];
#pragma unroll
  for (int e = 0; e < ND; ++e) F[1 + e] = (e == D) ? df_fma(q[1 + e], v[D], P) : q[1 + e] * v[D];
  F[NV - 1] = (q[NV - 1] + P) * v[D];
}

// Twice the LLF flux, F(qL) + F(qR) - alpha (qR - qL); the 1/2 folds into 1/dx.
template <int NV, int D, bool CMAX>
__device__ __forceinline__ void llf_flux_x2_df(const df (&qL)[NV], const df (&qR)[NV], const PhysDF& p, df (&G)[NV]) {
  df FL[NV], FR[NV], cL, cR;
  euler_flux_df<NV, D, CMAX>(qL, p, FL, cL);
  euler_flux_df<NV, D, CMAX>(qR, p, FR, cR);
  const df alpha = df_le(cR, cL) ? cL : cR;
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    // one three-term sum: the product's and the sums' exact errors are added
    // up once, 34 float operations instead of 37 (the difference is normalised:
    // states that agree in their leading floats differ by the low ones alone)
    const df t0 = two_sum(qL[k].hi, -qR[k].hi);
    const df d = fast_two_sum(t0.hi, t0.lo + (qL[k].lo - qR[k].lo));
    const float pr = __fmul_rn(alpha.hi, d.hi);
    float e = fmaf(alpha.hi, d.hi, -pr);
    e = fmaf(alpha.hi, d.lo, e);
    e = fmaf(alpha.lo, d.hi, e);
    const df s = two_sum(FL[k].hi, FR[k].hi);
    const df t = two_sum(s.hi, pr);
    G[k] = fast_two_sum(t.hi, t.lo + ((s.lo + e) + (FL[k].lo + FR[k].lo)));
  }
}

// Reduced tendency and force (Sec. 3.2 Eqs. pvs_dt / pvs_dt_dpr, App. A, App. B).
template <int NV, bool CMAX>
__device__ __forceinline__ void rsst_rhs_df(const df (&q)[NV], df (&dU)[NV], const PhysDF& p) {
  constexpr int ND = NV - 2;
  const df rho = q[0];
  const int var = p.variant;
  if (var != RSST_EULER) {
    const df ir = rcp(rho);
    df v[ND];
#pragma unroll
    for (int e = 0; e < ND; ++e) v[e] = q[1 + e] * ir;
    df k = q[1] * v[0];
#pragma unroll
    for (int e = 1; e < ND; ++e) k = df_fma(q[1 + e], v[e], k);
    const df P = df_fma(p.nhgm1, k, p.gm1 * q[NV - 1]);
    const df kin = scale(k, 0.5f);
    df nf = p.nf, nf_gm1 = p.nf_gm1;  // -f, -f (gamma - 1)
    if constexpr (CMAX) {
      nf = cmax_factor_df(p.gamma * (P * ir), p) - df_make(1.0f);
      nf_gm1 = nf * p.gm1;
    }
    const bool mom = var == RSST_PVS || var == RSST_DVS;  // the correction moves momentum
    const df H = df_fma(p.gam_gm1, P, mom ? kin : -kin);  // e + P +- rho V^2/2
    if (var == RSST_PVS || var == RSST_PMS || var == RSST_PD) {
      df s = (kin * ir) * dU[0];  // the small terms first: one rounding at dE's size
#pragma unroll
      for (int e = 0; e < ND; ++e) s = df_fma(-v[e], dU[1 + e], s);
      const df nfs = nf_gm1 * (s + dU[NV - 1]);  // -f dP
      if (var == RSST_PD) {
        dU[NV - 1] = df_fma(nfs, p.inv_gm1, dU[NV - 1]);
      } else {
        const df ng = nfs * rcp(p.gamma * P);  // -f dP / (rho a^2)
        const df nw = ng * rho;
        dU[0] = dU[0] + nw;
        if (mom) {
#pragma unroll
          for (int e = 0; e < ND; ++e) dU[1 + e] = df_fma(nw, v[e], dU[1 + e]);
        }
        dU[NV - 1] = df_fma(ng, H, dU[NV - 1]);
      }
    } else {  // DVS, DMS: s = drho
      const df nw = nf * dU[0];
      dU[0] = dU[0] + nw;
      if (mom) {
#pragma unroll
        for (int e = 0; e < ND; ++e) dU[1 + e] = df_fma(nw, v[e], dU[1 + e]);
      }
      dU[NV - 1] = df_fma(nw * ir, H, dU[NV - 1]);
    }
  }
  if (p.has_grav) {
    df mg = q[1] * p.grav[0];
#pragma unroll
    for (int e = 0; e < ND; ++e) {
      dU[1 + e] = df_fma(rho, p.grav[e], dU[1 + e]);
      if (e > 0) mg = df_fma(q[1 + e], p.grav[e], mg);
    }
    dU[NV - 1] = dU[NV - 1] + mg;
  }
}

// CFL rate sum_d c_tot/dx_d of a cell and its physical check.
template <int NV>
__device__ __forceinline__ df cfl_rate_df(const df (&q)[NV], const PhysDF& p, bool& ok) {
  constexpr int ND = NV - 2;
  const df rho = q[0];
  const df ir = rcp(rho);
  bool fin = isfinite(q[0].hi) && isfinite(q[NV - 1].hi);
  df k = q[1] * (q[1] * ir);
#pragma unroll
  for (int e = 0; e < ND; ++e) {
    if (e > 0) k = df_fma(q[1 + e], q[1 + e] * ir, k);
    fin = fin && isfinite(q[1 + e].hi);
  }
  const df P = df_fma(p.nhgm1, k, p.gm1 * q[NV - 1]);
  ok = fin && df_pos(rho) && df_pos(P);
  const df a = p.use_cmax ? sound_df<true>(P * ir, p) : sound_df<false>(P * ir, p);
  return (dsqrt(k * ir) + a) * p.sum_inv_dx;
}

}  // namespace rsst
