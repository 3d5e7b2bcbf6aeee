// Float64 device arithmetic of the RSST step (arXiv:1812.04135).
//
// Each function states the passage of the paper it computes.  Variables:
// q = conservative state (rho, m_1..m_ND, E), ND = NV - 2 dimensions.
#pragma once

#include "rsst_internal.h"

namespace rsst {

// Equation of state (Sec. 3.2: the reduced equations hold for a general
// EOS; the pressure tendency needs (de/dP)_rho and (de/drho)_P, Eqs.
// pvs_cons_dpr / pvs_cons_therm).  The float64 step reads its
// thermodynamics only through these members.  Two gases, chosen at compile
// time (CV) so that the ideal-gas kernels carry no covolume arithmetic: the
// ideal gas (covolume b = 0, the only EOS the paper specifies),
// e = P/(gamma-1), and the covolume (Noble-Abel) gas,
// P = (gamma-1) e / (1 - b rho), a^2 = gamma P / (rho (1 - b rho)),
// (de/dP)_rho = (1 - b rho)/(gamma-1), (de/drho)_P = -b P/(gamma-1).  The
// launchers take CV = (b != 0) for a run.
__device__ __forceinline__ double rcp_nr(double x);

template <bool CV>
struct Eos {
  // 1 - b rho
  __device__ static __forceinline__ double omb(const Phys& p, double rho) { return fma(-p.covol, rho, 1.0); }
  // P from the total energy E and rho |V|^2
  __device__ static __forceinline__ double pressure(const Phys& p, double rho, double E, double rhov2) {
    const double Pi = p.gm1 * E - p.hgm1 * rhov2;
    if constexpr (CV) return Pi * rcp_nr(omb(p, rho));
    return Pi;
  }
  __device__ static __forceinline__ double sound2(const Phys& p, double rho, double P, double inv_rho) {
    if constexpr (CV) return p.gamma * P * inv_rho * rcp_nr(omb(p, rho));
    return p.gamma * P * inv_rho;
  }
  // (a/xi)^2 for a constant xi, with gamma/xi^2 folded into one constant
  __device__ static __forceinline__ double sound2_over_xi2(const Phys& p, double rho, double P, double inv_rho) {
    if constexpr (CV) return p.gamma_xi2 * (P * inv_rho) * rcp_nr(omb(p, rho));
    return p.gamma_xi2 * (P * inv_rho);
  }
  __device__ static __forceinline__ double internal_energy(const Phys& p, double rho, double P) {
    if constexpr (CV) return P * p.inv_gm1 * omb(p, rho);
    return P * p.inv_gm1;
  }
  __device__ static __forceinline__ double de_dP(const Phys& p, double rho, double P) {
    if constexpr (CV) return p.inv_gm1 * omb(p, rho);
    return p.inv_gm1;
  }
  __device__ static __forceinline__ double inv_de_dP(const Phys& p, double rho, double P) {
    if constexpr (CV) return p.gm1 * rcp_nr(omb(p, rho));
    return p.gm1;
  }
  // f [(de/dP)_rho]^-1
  __device__ static __forceinline__ double f_over_de_dP(const Phys& p, double f, double rho, double P) {
    if constexpr (CV) return f * inv_de_dP(p, rho, P);
    return p.use_cmax ? f * p.gm1 : p.f_gm1;
  }
  // e + P
  __device__ static __forceinline__ double enthalpy(const Phys& p, double rho, double P) {
    if constexpr (CV) return internal_energy(p, rho, P) + P;
    return p.gam_gm1 * P;
  }
  // 1/(rho a^2)
  __device__ static __forceinline__ double inv_rho_a2(const Phys& p, double rho, double P) {
    if constexpr (CV) return omb(p, rho) * rcp_nr(p.gamma * P);
    return rcp_nr(p.gamma * P);
  }
  // (0.5 |V|^2 - (de/drho)_P) of the pressure tendency, from 0.5 |V|^2
  __device__ static __forceinline__ double half_v2_minus_de_drho(const Phys& p, double hv2, double P) {
    if constexpr (CV) return fma(p.covol * p.inv_gm1, P, hv2);
    return hv2;
  }
  // a state the EOS admits: 1 - b rho > 0 (always true for the ideal gas)
  __device__ static __forceinline__ bool admissible(const Phys& p, double rho) {
    if constexpr (CV) return omb(p, rho) > 0.0;
    return true;
  }
};

// A positive double's leading 24 significant bits as a float h in [1, 2),
// the other 29 as a float l, and its biased exponent (<= 0 for zero,
// subnormal and negative values, 2047 for NaN and infinity).
__device__ __forceinline__ void split_pair(double x, float& h, float& l, int& be) {
  const int hi = __double2hiint(x);
  const unsigned lo = (unsigned)__double2loint(x);
  be = hi >> 20;
  h = __uint_as_float(0x3f800000u | (__funnelshift_l(lo, (unsigned)hi, 3) & 0x7fffffu));
  l = __uint2float_rn(lo & 0x1fffffffu) * __int_as_float((127 - 52) << 23);
}

// 1/x to full float64 accuracy with two float64-pipe instructions.  For a
// positive x = (h + l) 2^k the seed comes from the float32 and integer pipes:
// r = 1/h (hardware, 2^-23), its residual e = 1 - (h + l) r by two FMAs, and
// y0 = r + r e assembled as a double (relative error about 2^-45); one Newton
// step y0 + y0 (1 - x y0) squares that.  The float64 hardware seed is good
// to 2^-20 only and takes a third-order step: three float64 instructions, of
// about 22 that a face state costs.  Within an ulp of the correctly rounded
// quotient (checked against CUDA's division by rsst_math_selftest).  Values
// that are not positive normal numbers with room in the exponent (non-physical
// states) take the hardware seed: y <- y + y (e + e^2), e = 1 - x y.
__device__ __forceinline__ double rcp_nr(double x) {
  float h, l;
  int be;
  split_pair(x, h, l, be);
  if ((unsigned)(be - 64) < 1920u) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(h));
    const float e = fmaf(-l, r, fmaf(-h, r, 1.0f));
    // r in [1/2, 1]: units of 2^-53 (for r = 1 the correction is negative)
    const int li = __float2int_rn((r * e) * __int_as_float((127 + 53) << 23));
    const long long y0b = ((long long)__float_as_int(r) << 29) + ((long long)(896 + 1023 - be) << 52) + (long long)li;
    const double y0 = __longlong_as_double(y0b);
    return fma(y0, fma(-x, y0, 1.0), y0);
  }
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}

// sqrt(x) for the wave-speed estimate c_tot with three float64-pipe
// operations.  Seed: the float32 hardware reciprocal square root of
// m 2^odd, where x = m 2^e (m in [1, 2) holding x's leading 23 mantissa
// bits) and odd = e mod 2, so the argument lies in [1, 4); the result is
// rescaled by 2^(-(e - odd)/2) in the exponent field, all on the integer
// pipe.  One Newton step in Markstein's form, s = s0 + (y0/2)(x - s0^2) with
// s0 = x y0 and the residual x - s0^2 formed exactly by an FMA, squares the
// seed's relative error (about 2^-21) to below 2^-40.  Zero and subnormal x
// give 0, negative x NaN.  c_tot only sets the LLF dissipation speed and the
// CFL step, where this error is far below the 1e-10 the float64 path is
// held to; every other square root is the compiler's.
__device__ __forceinline__ double sqrt_ctot(double x) {
  const long long ix = __double_as_longlong(x);
  const int be = (int)(ix >> 52);  // biased exponent for x >= 0
  const int e = be - 1023;
  const int odd = e & 1;
  const float f = __int_as_float(((127 + odd) << 23) | (int)((ix >> 29) & 0x7fffff));
  const int ir = __float_as_int(rsqrtf(f));  // in (1/2, 1]
  const int k = (e - odd) >> 1;              // 1/sqrt(x) = rsqrt(f) 2^(-k)
  const long long yb = ((long long)(((ir >> 23) & 0xff) - 127 + 1023 - k) << 52) | ((long long)(ir & 0x7fffff) << 29);
  const double y0 = __longlong_as_double(yb);
  const double h0 = __longlong_as_double(yb - (1ll << 52));  // y0 / 2
  const double s0 = x * y0;
  const double s = fma(h0, fma(-s0, s0, x), s0);
  return be > 0 ? s : (ix >= 0 ? 0.0 : __longlong_as_double(0x7ff8000000000000ll));
}

// sqrt(x) as an unevaluated pair of floats s + c (relative error below
// 2^-42), for the LLF speed, on the integer and float32 pipes only: x =
// 2^(2k) y with y in [1, 4) read from the bit pattern, y = h + l with h its
// leading 24 significant bits and l the other 29 (rounded to a float);
// s = h rsqrt(h) and one Newton step c = (y - s^2) / (2 s) with s^2 split
// exactly by an FMA (h - s^2 is exact: Sterbenz), then both scaled by 2^k.
// Zero and subnormal x give 0, negative x and NaN give NaN, like sqrt_ctot;
// 2^k is kept to the float range (x in [2^-252, 2^256), far outside any
// physical speed^2).
//
// root_parts: s0 (in [1, 2]), c0 and k for a positive normal x (true), false
// for any other.
__device__ __forceinline__ bool root_parts(double x, float& s0, float& c0, int& k) {
  const long long ix = __double_as_longlong(x);
  const int be = (int)(ix >> 52);  // biased exponent for x >= 0, negative for x < 0
  const int e = be - 1023;
  const int odd = e & 1;
  const float h = __int_as_float(((127 + odd) << 23) | (int)((ix >> 29) & 0x7fffff));
  const float l = __uint2float_rn((unsigned)(ix & 0x1fffffff)) * __int_as_float((75 + odd) << 23);  // * 2^(odd-52)
  const float r = rsqrtf(h);
  s0 = h * r;
  const float p = s0 * s0;
  const float d = ((h - p) - fmaf(s0, s0, -p)) + l;
  c0 = d * (0.5f * r);
  k = (e - odd) >> 1;
  return be > 0 && be < 2047;
}
__device__ __forceinline__ void sqrt_pair(double x, float& s, float& c) {
  float s0, c0;
  int k;
  const bool fin = root_parts(x, s0, c0, k);
  const float sc = k < -126 ? 0.0f : (k > 127 ? __int_as_float(0x7f800000) : __int_as_float((127 + k) << 23));
  const long long ix = __double_as_longlong(x);
  const float special = (ix >= 0 && (ix >> 52) == 0) ? 0.0f : __int_as_float(0x7fc00000);
  s = fin ? s0 * sc : special;
  c = fin ? c0 * sc : special;
}

// A float as a double, on the integer pipe (subnormal floats read as 0).
__device__ __forceinline__ double f2d_bits(float f) {
  const unsigned b = __float_as_uint(f);
  const unsigned E = (b >> 23) & 0xffu;
  const unsigned long long sign = (unsigned long long)(b >> 31) << 63;
  const unsigned long long ex = E == 0u ? 0ull : (E == 255u ? 0x7ffull : (unsigned long long)(E + 896u)) << 52;
  const unsigned long long mant = E == 0u ? 0ull : (unsigned long long)(b & 0x7fffffu) << 29;
  return __longlong_as_double((long long)(sign | ex | mant));
}

// c_tot = |V| + a/xi from |V|^2 and (a/xi)^2 as a normalised float pair
// (h + l, |l| <= ulp(h)/2): both square roots by sqrt_pair, summed exactly
// in the leading parts (two-sum), relative error below 2^-41.
__device__ __forceinline__ void ctot_pair(double v2, double a2x, float& h, float& l) {
  float sv, cv, sa, ca;
  sqrt_pair(v2, sv, cv);
  sqrt_pair(a2x, sa, ca);
  const float t = sv + sa;
  const float bv = t - sv;
  const float lo = ((sv - (t - bv)) + (sa - bv)) + (cv + ca);
  h = t + lo;
  l = lo - (h - t);
}

// A normalised non-negative float pair (h + l, |l| <= ulp(h)/2) as a double,
// on the integer pipe: h's 24 bits shifted up plus l in units of the result's
// last place (2^-52 of h's exponent; half of that below a power of two), rounded
// as a float64 sum of the two would be.  Outside h in [2^-74, 2^126] (and for
// NaN) the two halves are added.
__device__ __forceinline__ double pair_to_double(float h, float l) {
  const unsigned hb = __float_as_uint(h);
  const int eh = (int)(hb >> 23);
  const unsigned mant = hb & 0x7fffffu;
  if (eh >= 53 && eh <= 253) {
    const int unit = mant == 0u && l < 0.0f ? 307 : 306;
    const int li = __float2int_rn(l * __int_as_float((unit - eh) << 23));
    return __longlong_as_double(((long long)(eh + 896) << 52) + ((long long)mant << 29) + (long long)li);
  }
  return f2d_bits(h) + f2d_bits(l);
}

// sqrt((h + l) 2^e) of a float pair with h in [1, 8) as a float pair: one
// Newton step from the hardware rsqrt, the square split exactly by an FMA.  The
// pair is normalised first, so that the correction stays as small as the seed's
// error, and the correction's own second-order term is kept.
__device__ __forceinline__ void sqrt_of_pair(float h, float l, int e, float& s, float& c) {
  const int odd = e & 1;
  const float f = odd ? 2.0f : 1.0f, h0 = h;
  h = (h + l) * f;
  l = fmaf(h0, f, -h) + l * f;
  const float r = rsqrtf(h);
  const float s0 = h * r;
  const float p = s0 * s0;
  const float d = ((h - p) - fmaf(s0, s0, -p)) + l;
  const int k = (e - odd) >> 1;
  const float sc = k < -126 ? 0.0f : (k > 127 ? __int_as_float(0x7f800000) : __int_as_float((127 + k) << 23));
  // the correction's own relative error: r is not quite 1/s0, and s0 + c0 not s0
  const float hr = 0.5f * r, c0 = d * hr;
  const float g = fmaf(-c0, hr, fmaf(-s0, r, 1.0f));
  s = s0 * sc;
  c = fmaf(c0, g, c0) * sc;
}

// Sum of two non-negative float pairs, normalised.
__device__ __forceinline__ void pair_sum(float sv, float cv, float sa, float ca, float& h, float& l) {
  const float t = sv + sa;
  const float bv = t - sv;
  const float lo = ((sv - (t - bv)) + (sa - bv)) + (cv + ca);
  h = t + lo;
  l = lo - (h - t);
}

// c_tot = |V| + a/xi as a float pair from k = rho |V|^2, P and 1/rho:
// |V|^2 = k/rho and (a/xi)^2 = (gamma/xi^2) P/rho are formed as products of
// float pairs (relative error below 2^-45) on the float32 and integer pipes,
// exponents apart, so any magnitude a double holds works.  Saves the three
// float64 products that formed the two squares, of the 22 float64 operations
// of a face state (the float64 pipe issues a 64th of the float32 pipe's rate).
// Error over 6.7e7 states, largest and rms: 2^-44.6, 2^-48.0; with the float64
// products and sqrt_pair 2^-44.0, 2^-47.8.
__device__ __forceinline__ void ctot_pair_of(double k, double P, double ir, const Phys& p, float& h, float& l) {
  float kh, kl, ph, pl, rh, rl;
  int ek, ep, er;
  split_pair(k, kh, kl, ek);
  split_pair(P, ph, pl, ep);
  split_pair(ir, rh, rl, er);
  const float v = kh * rh;
  const float ve = fmaf(kl, rh, fmaf(kh, rl, fmaf(kh, rh, -v)));
  const float t = ph * rh;
  const float te = fmaf(pl, rh, fmaf(ph, rl, fmaf(ph, rh, -t)));
  const float a = t * p.gxh;
  const float ae = fmaf(te, p.gxh, fmaf(t, p.gxl, fmaf(t, p.gxh, -a)));
  float sv, cv, sa, ca;
  sqrt_of_pair(v, ve, ek + er - 2046, sv, cv);
  sqrt_of_pair(a, ae, ep + er - 2046 + p.gxe, sa, ca);
  // zero (or subnormal) k or P: that speed is 0; negative or NaN anywhere: NaN
  const bool rok = (unsigned)(er - 1) < 2046u;
  const float nan = __int_as_float(0x7fc00000);
  if (!(rok && (unsigned)(ek - 1) < 2046u)) {
    sv = rok && ek == 0 ? 0.0f : nan;
    cv = 0.0f;
  }
  if (!(rok && (unsigned)(ep - 1) < 2046u)) {
    sa = rok && ep == 0 ? 0.0f : nan;
    ca = 0.0f;
  }
  pair_sum(sv, cv, sa, ca, h, l);
}

// 1/sqrt(w): the hardware approximation (20 bits) and one third-order step,
// y (1 + e/2 + 3 e^2/8) with e = 1 - w y^2, which cubes its error: about one
// ulp in five float64 operations instead of an IEEE square root and division.
// 0 for an infinite w.
__device__ __forceinline__ double rsqrt_nr(double w) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(w));
  const double e = fma(-(w * y), y, 1.0);
  return __double2hiint(w) == 0x7ff00000 ? 0.0 : fma(y * e, fma(0.375, e, 0.5), y);
}

// A float pair s + c with |c| within some ulps of s as a double, on the float32
// and integer pipes.
__device__ __forceinline__ double sum_to_double(float s, float c) {
  const float h = s + c;
  return pair_to_double(h, c - (h - s));
}

// x times 2^k, on the integer pipe (x and the result positive normal).
__device__ __forceinline__ double scale2(double x, int k) {
  return __hiloint2double(__double2hiint(x) + (k << 20), __double2loint(x));
}

// c_tot under the C_max law from |V|^2 and (a/xi)^2, with three float64
// instructions: the roots as float pairs (2^-42), one float64 Newton step on the
// sound term, which carries c_tot in slow flow (a float pair's accuracy showed
// there against a 64-bit evaluation).  The LLF speed is a float pair in the end,
// so its roots may have a float's range: beyond it, and for NaN, they come as
// sqrt_pair gives them.  dt (WIDE) takes any magnitude of a double: there the
// roots' exponents are added as integers.  (WIDE in the faces too cost 3.7 % of
// the 250^2 case.)
template <bool REFINE>
__device__ __forceinline__ double root_any(double x) {
  const long long ix = __double_as_longlong(x);
  if (ix == 0) return 0.0;
  const bool tiny = ix > 0 && ix < (1ll << 52);  // subnormal
  if (tiny) x *= 0x1p108;
  float s, c;
  int k;
  if (!root_parts(x, s, c, k)) return ix == 0x7ff0000000000000ll ? x : __longlong_as_double(0x7ff8000000000000ll);
  double y = scale2(sum_to_double(s, c), k);
  if constexpr (REFINE) y = fma(fma(-y, y, x), scale2(f2d_bits(__fdividef(0.5f, s)), -k), y);
  return tiny ? scale2(y, -54) : y;
}
template <bool WIDE>
__device__ __forceinline__ double ctot_cmax(double v2, double a2x) {
  if constexpr (WIDE) return root_any<false>(v2) + root_any<true>(a2x);
  float s, c;
  sqrt_pair(a2x, s, c);
  const double y = sum_to_double(s, c);
  const double a = s > 0.0f && s < __int_as_float(0x7f800000) ? fma(fma(-y, y, a2x), f2d_bits(__fdividef(0.5f, s)), y) : y;
  sqrt_pair(v2, s, c);
  return sum_to_double(s, c) + a;
}

// A non-negative double as a float pair (2^-48), on the float32 and integer
// pipes; subnormal floats come as 0, NaN and negative values as NaN.
__device__ __forceinline__ void to_pair(double x, float& h, float& l) {
  int be;
  split_pair(x, h, l, be);
  const int k = be - 1023;
  const float sc = k < -126 ? 0.0f : (k > 127 ? __int_as_float(0x7f800000) : __int_as_float((127 + k) << 23));
  const bool fin = (unsigned)(be - 1) < 2046u;
  h = fin ? h * sc : (be == 0 ? 0.0f : __int_as_float(0x7fc00000));
  l = fin ? l * sc : 0.0f;
}

// sqrt(x) (2^-42) and its reciprocal (2^-41) as doubles on the float32 and
// integer pipes, for the adjoint's derivatives of c_tot at any magnitude of
// the speeds.  Both corrections are added to their leading parts before they
// become a double (a correction may exceed an ulp).  0 and 0 for zero and
// subnormal x, NaN and 0 for any other that is not a positive normal number.
__device__ __forceinline__ void sqrt_rcp(double x, double& s, double& r) {
  float h, c, y;
  int k;
  const bool fin = root_parts(x, h, c, k);
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(h));
  const double sd = scale2(sum_to_double(h, c), k);
  const double rd = scale2(sum_to_double(y, y * fmaf(-c, y, fmaf(-h, y, 1.0f))), -k);
  s = fin ? sd : (((unsigned long long)__double_as_longlong(x) >> 52) == 0 ? 0.0 : __longlong_as_double(0x7ff8000000000000ll));
  r = fin ? rd : 0.0;
}

// Effective sound speed a/xi from a^2 and the factor f = 1 - 1/xi^2: constant
// xi, or the C_max law xi = [1 + (a/C_max)^4]^(1/4) (Eq. cx, Sec. 4.3), for
// which a/xi = sqrt(a^2 / sqrt(w)) and f = 1 - 1/sqrt(w), w = 1 + a^4/C_max^4.
__device__ __forceinline__ double sound_over_xi(double a2, const Phys& p) {
  if (p.use_cmax) return sqrt(a2 / sqrt(fma(a2 * a2, p.inv_cmax4, 1.0)));
  return sqrt_ctot(a2) * p.inv_xi;
}
__device__ __forceinline__ double f_of(double a2, const Phys& p) {
  if (p.use_cmax) return 1.0 - rsqrt_nr(fma(a2 * a2, p.inv_cmax4, 1.0));
  return p.f;
}

// The approximate RSST characteristic speed c_tot = |V| + a/xi (Sec. 4.2) of
// a state with k = rho |V|^2 as a normalised float pair.
template <bool CV>
__device__ __forceinline__ void ctot_of(const Phys& p, double rho, double k, double P, double ir, float& h, float& l) {
  if (p.use_cmax) {
    const double a2 = Eos<CV>::sound2(p, rho, P, ir);
    to_pair(ctot_cmax<false>(k * ir, a2 * rsqrt_nr(fma(a2 * a2, p.inv_cmax4, 1.0))), h, l);
  } else if constexpr (CV) {
    ctot_pair(k * ir, Eos<CV>::sound2_over_xi2(p, rho, P, ir), h, l);
  } else {
    ctot_pair_of(k, P, ir, p, h, l);
  }
}

// The Euler flux along dimension D, F (Eq. pvs_dt0), and c_tot of one state
// as the float pair ch + cl.  k = rho |V|^2 = m.V feeds the pressure directly.
template <int NV, int D, bool CV = false>
__device__ __forceinline__ void euler_flux(const double (&q)[NV], const Phys& p,
                                           double (&F)[NV], float& ch, float& cl) {
  constexpr int ND = NV - 2;
  const double rho = q[0];
  const double ir = rcp_nr(rho);
  double v[ND];
  double k = 0.0;
#pragma unroll
  for (int e = 0; e < ND; ++e) {
    v[e] = q[1 + e] * ir;
    k = e == 0 ? q[1] * v[0] : fma(q[1 + e], v[e], k);
  }
  const double P = Eos<CV>::pressure(p, rho, q[NV - 1], k);
  ctot_of<CV>(p, rho, k, P, ir, ch, cl);
  F[0] = q[1 + D];
#pragma unroll
  for (int e = 0; e < ND; ++e) F[1 + e] = (e == D) ? fma(q[1 + e], v[D], P) : q[1 + e] * v[D];
  F[NV - 1] = (q[NV - 1] + P) * v[D];
}

// Twice the local Lax-Friedrichs flux, 2 F = F(qL) + F(qR) - alpha (qR - qL)
// with alpha = max(c_tot(qL), c_tot(qR)), ties to the left state (Sec. 4.2,
// step 4).  The factor 1/2 is exact and left to the caller (it folds into
// the divergence's 1/dx), which saves the halvings inside the fluxes.
template <int NV, int D, bool CV = false>
__device__ __forceinline__ void llf_flux_x2(const double (&qL)[NV], const double (&qR)[NV],
                                            const Phys& p, double (&G)[NV]) {
  double FL[NV], FR[NV];
  float hL, lL, hR, lR;
  euler_flux<NV, D, CV>(qL, p, FL, hL, lL);
  euler_flux<NV, D, CV>(qR, p, FR, hR, lR);
  const bool left = hL > hR || (hL == hR && lL >= lR);  // normalised pairs order like their values
  const double alpha = pair_to_double(left ? hL : hR, left ? lL : lR);
#pragma unroll
  for (int k = 0; k < NV; ++k) G[k] = fma(-alpha, qR[k] - qL[k], FL[k] + FR[k]);
}

// Monotonized-central limited slope (named in Sec. 4.2): 0 if ab <= 0, else
// the smallest in magnitude of 2a, 2b, (a+b)/2, ties in that order.
// Only a + b uses the float64 pipe.  A double's bit pattern shifted left by
// one (sign dropped) orders like its magnitude as an unsigned integer, so the
// magnitude comparisons run on the integer pipe (the shift, unlike a mask of
// the sign bit, is not turned back into float64 absolute values by the
// compiler), and scaling a normal double by 2, 4 or 1/2 is an exact change
// of its exponent field (2|a| <= |a+b|/2 is |a| * 4 <= |a+b|).  Same
// decisions and values as the direct form for normal operands.  A sum whose
// half is no normal number (a profile's far tail) gives 0, and beside a larger
// one a subnormal operand's double may be up to 2^-1022 off.  (The direct form
// in a branch for such sums cost 1.4 % of a 64^2 run.)
__device__ __forceinline__ double mc_slope(double a, double b) {
  const long long one = 1ll << 52;                // +1 in the exponent field
  const unsigned long long four = 1ull << 54;     // +2 in the shifted exponent field: x4
  const long long ia = __double_as_longlong(a), ib = __double_as_longlong(b);
  const unsigned long long ua = (unsigned long long)ia << 1, ub = (unsigned long long)ib << 1;
  const long long is = __double_as_longlong(a + b);
  const unsigned long long us = (unsigned long long)is << 1;
  const bool same = ((ia ^ ib) >= 0) && ua != 0 && ub != 0 && us >= 2ull << 53;
  const long long pick = (ua <= ub && ua + four <= us) ? ia + one : ((ub + four <= us) ? ib + one : is - one);
  return same ? __longlong_as_double(pick) : 0.0;
}

// Half the MC slope (Sec. 4.2) and the branch taken: 0 -> 0, 1 -> a, 2 -> b,
// 3 -> (a+b)/4; decisions and values on the integer pipe as in mc_slope (0 where
// a quarter of the sum is no normal number).
__device__ __forceinline__ double half_mc(double a, double b, int& br) {
  const long long two = 2ll << 52;             // x4 in the exponent field
  const unsigned long long four = 1ull << 54;  // x4 in the shifted exponent field
  const long long ia = __double_as_longlong(a), ib = __double_as_longlong(b);
  const unsigned long long ua = (unsigned long long)ia << 1, ub = (unsigned long long)ib << 1;
  const long long is = __double_as_longlong(a + b);
  const unsigned long long us = (unsigned long long)is << 1;
  const bool same = ((ia ^ ib) >= 0) && ua != 0 && ub != 0;
  const bool pa = ua <= ub && ua + four <= us, pb = ub + four <= us;
  br = !same ? 0 : (pa ? 1 : (pb ? 2 : 3));
  return same && us >= 3ull << 53 ? __longlong_as_double(pa ? ia : (pb ? ib : is - two)) : 0.0;
}
// Reduced tendency: dU <- dU - (1 - 1/xi^2) s r, then the external force.
//   PVS: s = dP,   r = (1/a^2, V/a^2, (e+P+rho V^2/2)/(rho a^2))   Sec. 3.2, Eqs. pvs_dt, pvs_cons_rhs
//   DVS: s = drho, r = (1, V, (e+P+rho V^2/2)/rho)                  App. A.1
//   PMS: s = dP,   r = (1/a^2, 0, (e+P-rho V^2/2)/(rho a^2))        App. A.2
//   DMS: s = drho, r = (1, 0, (e+P-rho V^2/2)/rho)                  App. A.3
//   PD : s = dP,   r = (0, 0, 1/(gamma-1))                          App. A.4
// with dP = (gamma-1)(V^2/2 drho - V.dm + dE) (Eq. pvs_dt_dpr, ideal gas),
// evaluated at the cell centre of the stage state; force terms
// (0, rho F, m.F) of App. B are added after (dP excludes them).
//
// In two parts: what depends on the state alone, and what needs the Euler
// tendency (the 1D line kernel forms the first while the fluxes are computed).
// s is scaled by a; b turns it into the E row's factor: 1/(rho a^2) (PVS, PMS),
// 1/rho (DVS, DMS) or (de/dP)_rho (PD).
template <int NV>
struct RhsPrep {
  double v[NV - 2], hv2, H, a, b;  // hv2: |V|^2/2 - (de/drho)_P; H = e + P +- rho V^2/2
};
template <int NV, bool CV = false>
__device__ __forceinline__ void rhs_prep(const double (&q)[NV], const Phys& p, RhsPrep<NV>& r) {
  constexpr int ND = NV - 2;
  const double rho = q[0];
  const double ir = rcp_nr(rho);
  double k = 0.0;  // rho |V|^2
#pragma unroll
  for (int e = 0; e < ND; ++e) {
    r.v[e] = q[1 + e] * ir;
    k = e == 0 ? q[1] * r.v[0] : fma(q[1 + e], r.v[e], k);
  }
  const double P = Eos<CV>::pressure(p, rho, q[NV - 1], k);
  const double kin = 0.5 * k;
  const int var = p.variant;
  const double f = p.use_cmax ? f_of(Eos<CV>::sound2(p, rho, P, ir), p) : p.f;
  r.H = fma(var == RSST_PVS || var == RSST_DVS ? 0.5 : -0.5, k, Eos<CV>::enthalpy(p, rho, P));
  if (var == RSST_PVS || var == RSST_PMS || var == RSST_PD) {
    r.hv2 = Eos<CV>::half_v2_minus_de_drho(p, kin * ir, P);
    r.a = Eos<CV>::f_over_de_dP(p, f, rho, P);
    r.b = var == RSST_PD ? Eos<CV>::de_dP(p, rho, P) : Eos<CV>::inv_rho_a2(p, rho, P);
  } else {
    r.hv2 = 0.0;
    r.a = f;
    r.b = ir;
  }
}
template <int NV>
__device__ __forceinline__ void rhs_apply(const double (&q)[NV], double (&dU)[NV], const Phys& p,
                                          const RhsPrep<NV>& r) {
  constexpr int ND = NV - 2;
  const int var = p.variant;
  if (var != RSST_EULER) {
    double w, wE;  // f s r0 and f s rE / H
    if (var == RSST_PVS || var == RSST_PMS || var == RSST_PD) {
      double s = r.hv2 * dU[0];  // the small terms first: one rounding at dE's size
#pragma unroll
      for (int e = 0; e < ND; ++e) s = fma(-r.v[e], dU[1 + e], s);
      const double fs = r.a * (s + dU[NV - 1]);
      wE = fs * r.b;
      if (var == RSST_PD) {
        dU[NV - 1] = fma(-fs, r.b, dU[NV - 1]);
        w = 0.0;
      } else {
        w = wE * q[0];
      }
    } else {  // DVS, DMS
      w = r.a * dU[0];
      wE = w * r.b;
    }
    if (var != RSST_PD) {
      dU[0] -= w;
      if (var == RSST_PVS || var == RSST_DVS) {
#pragma unroll
        for (int e = 0; e < ND; ++e) dU[1 + e] = fma(-w, r.v[e], dU[1 + e]);
      }
      dU[NV - 1] = fma(-wE, r.H, dU[NV - 1]);
    }
  }
  if (p.has_grav) {
    double mg = 0.0;
#pragma unroll
    for (int e = 0; e < ND; ++e) {
      dU[1 + e] += q[0] * p.grav[e];
      mg += q[1 + e] * p.grav[e];
    }
    dU[NV - 1] += mg;
  }
}
template <int NV, bool CV = false>
__device__ __forceinline__ void rsst_rhs(const double (&q)[NV], double (&dU)[NV], const Phys& p) {
  RhsPrep<NV> r = {};
  if (p.variant != RSST_EULER) rhs_prep<NV, CV>(q, p, r);
  rhs_apply<NV>(q, dU, p, r);
}

// Half of a double (as 0.5 * x rounds it), on the integer pipe.  The sign is
// taken off the high word (a 64-bit mask would become a float64 absolute value).
__device__ __forceinline__ double half_of(double x) {
  const int hi = __double2hiint(x), lo = __double2loint(x);
  const unsigned s = (unsigned)hi & 0x80000000u, e = ((unsigned)hi >> 20) & 0x7ffu;
  if (e >= 2u) return __hiloint2double(e == 2047u ? hi : hi - (1 << 20), lo);
  // at and below the smallest normal exponent the pattern counts units of 2^-1074
  const unsigned long long mag = ((unsigned long long)((unsigned)hi ^ s) << 32) | (unsigned)lo;
  const unsigned long long h = (mag + ((mag >> 1) & 1ull)) >> 1;
  return __hiloint2double((int)((unsigned)(h >> 32) | s), (int)(unsigned)h);
}

// From the bit pattern (a float64 compare occupies the float64 pipe).
__device__ __forceinline__ bool finite_bits(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }
__device__ __forceinline__ bool positive_finite(double x) {
  return __double_as_longlong(x) > 0 && __double2hiint(x) < 0x7ff00000;
}

// CFL rate sum_d c_tot/dx_d of a cell and its physical-state check.  c_tot is
// the float pair of the LLF speed (C_max law: in float64); the
// checks read bit patterns.
template <int NV, bool CV = false>
__device__ __forceinline__ double cfl_rate(const double (&q)[NV], const Phys& p, bool& ok) {
  constexpr int ND = NV - 2;
  const double rho = q[0];
  const double ir = rcp_nr(rho);
  double k = 0.0;
  bool fin = finite_bits(q[NV - 1]);
#pragma unroll
  for (int e = 0; e < ND; ++e) {
    k = e == 0 ? q[1] * (q[1] * ir) : fma(q[1 + e], q[1 + e] * ir, k);
    fin = fin && finite_bits(q[1 + e]);
  }
  const double P = Eos<CV>::pressure(p, rho, q[NV - 1], k);
  ok = fin && positive_finite(rho) && positive_finite(P) && Eos<CV>::admissible(p, rho);
  if (p.use_cmax) {
    const double a2 = Eos<CV>::sound2(p, rho, P, ir);
    return ctot_cmax<true>(k * ir, a2 * rsqrt_nr(fma(a2 * a2, p.inv_cmax4, 1.0))) * p.sum_inv_dx;
  }
  float ch, cl;
  ctot_of<CV>(p, rho, k, P, ir, ch, cl);
  return pair_to_double(ch, cl) * p.sum_inv_dx;
}

}  // namespace rsst
