// Float32 perturbation arithmetic of rsst_fp32_lean.cuh on pairs: one
// instruction (add/mul/fma.f32x2) does the same operation for two cells or
// two faces.  The float32 stage kernels are bound by instruction issue, not by
// the float32 units (an f32x2 instruction takes one issue slot for two lanes'
// worth of work), so a lane that owns two neighbouring cells spends about half
// the issue slots on arithmetic, and loads, table reads, address and loop
// instructions are shared by the two.  Reciprocals, square roots, minima and
// selections have no pair form and go component by component.
#pragma once

#include "rsst_fp32_lean.cuh"
#include "rsst_internal.h"
#include "rsst_math_fp32.cuh"

namespace rsst {

struct f2 {
  unsigned long long v;
};

__device__ __forceinline__ f2 mk2(float a, float b) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ f2 dup2(float a) { return mk2(a, a); }
__device__ __forceinline__ float lo2(f2 x) { return __uint_as_float((unsigned)x.v); }
__device__ __forceinline__ float hi2(f2 x) { return __uint_as_float((unsigned)(x.v >> 32)); }
__device__ __forceinline__ f2 operator+(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 operator*(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
__device__ __forceinline__ f2 operator-(f2 a, f2 b) { return fma2(b, dup2(-1.0f), a); }
__device__ __forceinline__ f2 rcp2(f2 x) { return mk2(rcp_f(lo2(x)), rcp_f(hi2(x))); }
__device__ __forceinline__ f2 sqrt2(f2 x) { return mk2(sqrt_f(lo2(x)), sqrt_f(hi2(x))); }
__device__ __forceinline__ f2 max2(f2 a, f2 b) { return mk2(fmaxf(lo2(a), lo2(b)), fmaxf(hi2(a), hi2(b))); }

// A table value (held twice in shared memory) as a pair; two in one load.
struct f2x2 {
  f2 a, b;
};
__device__ __forceinline__ f2x2 tab2(const float* row, int i) {  // i even
  const ulonglong2 q = *reinterpret_cast<const ulonglong2*>(row + 2 * i);
  f2x2 r;
  r.a.v = q.x;
  r.b.v = q.y;
  return r;
}

// The run's constants, twice each.
struct PhysF2 {
  f2 gm1, nhgm1, gx, cmax4;
};
__device__ __forceinline__ PhysF2 make_pf2(const PhysF& p) {
  PhysF2 q;
  q.gm1 = dup2(p.gm1);
  q.nhgm1 = dup2(-p.hgm1);
  q.gx = dup2(p.gx);
  q.cmax4 = dup2(p.inv_cmax4);
  return q;
}

// Half MC slopes from the two cells' backward and forward differences.
__device__ __forceinline__ float half_mc_of(float a, float b, float q) {  // q = (a + b)/4
  const unsigned sa = __float_as_uint(a) & 0x80000000u;
  const float bs = __uint_as_float(__float_as_uint(b) ^ sa);
  float m;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(m) : "f"(fabsf(a)), "f"(bs), "f"(fabsf(q)));
  m = fmaxf(m, 0.0f);
  return __uint_as_float(__float_as_uint(m) | sa);
}
__device__ __forceinline__ f2 half_mc2(f2 a, f2 b) {
  const f2 q = (a + b) * dup2(0.25f);
  return mk2(half_mc_of(lo2(a), lo2(b), lo2(q)), half_mc_of(hi2(a), hi2(b), hi2(q)));
}

// half_bg_slope_f for two cells of one vertical index; t: the component's
// entries d0L, d0R and the four halved background terms.
__device__ __forceinline__ float bg_pick(float A, float B, float C, float da, float db, float dq, float t2, float t3,
                                         float t4, float t5) {
  const float aa = fabsf(A), bb = fabsf(B), cc = fabsf(C);
  const bool same = A * B > 0.0f;
  const bool p1 = aa <= bb && aa <= cc;
  const bool p2 = !p1 && bb <= cc;
  const float lin = p1 ? da : (p2 ? db : dq);
  const float del = p1 ? t3 : (p2 ? t4 : t5);
  return same ? lin + del : t2;
}
__device__ __forceinline__ f2 half_bg_slope2(const float* row, int t, f2 da, f2 db) {
  const f2x2 d0 = tab2(row, t), t23 = tab2(row, t + 2), t45 = tab2(row, t + 4);
  const f2 A = d0.a + da, B = d0.b + db;
  const f2 C = (A + B) * dup2(0.25f), dq = (da + db) * dup2(0.25f);
  return mk2(bg_pick(lo2(A), lo2(B), lo2(C), lo2(da), lo2(db), lo2(dq), lo2(t23.a), lo2(t23.b), lo2(t45.a), lo2(t45.b)),
             bg_pick(hi2(A), hi2(B), hi2(C), hi2(da), hi2(db), hi2(dq), lo2(t23.a), lo2(t23.b), lo2(t45.a), lo2(t45.b)));
}

// Half slopes across the vertical axis from the differences below and above
// the cells; row = the cells' (doubled) table row.
template <int NV, bool BG>
__device__ __forceinline__ void vslope2(const f2 (&da)[NV], const f2 (&db)[NV], const float* row, f2 (&h)[NV]) {
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    if (BG && (v == 0 || v == NV - 1))
      h[v] = half_bg_slope2(row, v == 0 ? TR_SRHO : TR_SE, da[v], db[v]);
    else
      h[v] = half_mc2(da[v], db[v]);
  }
}

// sound_x and flux_lean on pairs (see rsst_fp32_lean.cuh).
template <bool CMAX>
__device__ __forceinline__ f2 sound_x2(f2 a2x, const PhysF2& pf) {
  if constexpr (CMAX) return sqrt2(a2x * rcp2(sqrt2(fma2(a2x * a2x, pf.cmax4, dup2(1.0f)))));
  return sqrt2(a2x);
}
template <int NV, int D, bool BG, bool WANT_DC, bool CMAX>
__device__ __forceinline__ void flux_lean2(const f2 (&q)[NV], f2 rho0, f2 P0, f2 gxP0, f2 H0, f2 a0x, f2 gxr0, f2 c0,
                                           const PhysF2& pf, f2 (&F)[NV], f2& c, f2& dc) {
  constexpr int ND = NV - 2;
  const f2 rho = BG ? rho0 + q[0] : q[0];
  const f2 ir = rcp2(rho);
  f2 v[ND];
#pragma unroll
  for (int e = 0; e < ND; ++e) v[e] = q[1 + e] * ir;
  f2 k = q[1] * v[0];  // rho |V|^2 = m.V
#pragma unroll
  for (int e = 1; e < ND; ++e) k = fma2(q[1 + e], v[e], k);
  const f2 P1 = fma2(pf.nhgm1, k, pf.gm1 * q[NV - 1]);
  const f2 a2x = (BG ? fma2(pf.gx, P1, gxP0) : pf.gx * P1) * ir;
  const f2 vm = sqrt2(k * ir);
  const f2 ax = sound_x2<CMAX>(a2x, pf);
  c = vm + ax;
  if constexpr (WANT_DC) {
    if constexpr (CMAX) {
      dc = vm + (ax - c0);
    } else {
      const f2 da2x = fma2(P1, rho0, P0 * (q[0] * dup2(-1.0f))) * (ir * gxr0);  // one product rounded by itself
      dc = fma2(da2x, rcp2(ax + a0x), vm);
    }
  }
  F[0] = q[1 + D];
#pragma unroll
  for (int e = 0; e < ND; ++e) F[1 + e] = e == D ? fma2(q[1 + e], v[D], P1) : q[1 + e] * v[D];
  F[NV - 1] = (BG ? H0 + (q[NV - 1] + P1) : q[NV - 1] + P1) * v[D];
}

// Twice the LLF flux of two faces across which the background is constant
// (row: the faces' table row).
template <int NV, int D, bool BG, bool CMAX>
__device__ __forceinline__ void face_flat2(const f2 (&qL)[NV], const f2 (&qR)[NV], const float* row, const PhysF2& pf,
                                           f2 (&G)[NV]) {
  f2 FL[NV], FR[NV], cL, cR, dum;
  f2x2 b0 = {}, b1 = {};
  const f2 z = {};
  if constexpr (BG) {
    b0 = tab2(row, TR_RHO0);
    b1 = tab2(row, TR_GXP0);
  }
  flux_lean2<NV, D, BG, false, CMAX>(qL, b0.a, b0.b, b1.a, b1.b, z, z, z, pf, FL, cL, dum);
  flux_lean2<NV, D, BG, false, CMAX>(qR, b0.a, b0.b, b1.a, b1.b, z, z, z, pf, FR, cR, dum);
  const f2 alpha = max2(cL, cR);
#pragma unroll
  for (int v = 0; v < NV; ++v) G[v] = fma2(alpha, qL[v] - qR[v], FL[v] + FR[v]);
}

// Twice the LLF flux of two faces across the vertical axis D (row: the faces'
// table row), as face_vertical.
template <int NV, int D, bool CMAX>
__device__ __forceinline__ void face_vertical2(const f2 (&qL)[NV], const f2 (&qR)[NV], const float* row,
                                               const PhysF2& pf, f2 (&G)[NV]) {
  const f2x2 ga = tab2(row, TR_FG), j = tab2(row, TR_FJRHO);  // c0L - c0R and alpha0; jumps of rho and E
  const float g = lo2(ga.a), a0 = lo2(ga.b);
  const f2 c0L = dup2(g >= 0.0f ? a0 : a0 + g), c0R = dup2(g >= 0.0f ? a0 - g : a0);
  f2 FL[NV], FR[NV], cL, cR, dcL, dcR;
  const f2x2 a0x = tab2(row, TR_FA0X), gr = tab2(row, TR_FA0X + 2);
  {
    const f2x2 b0 = tab2(row, TR_FL), b1 = tab2(row, TR_FL + 2);
    flux_lean2<NV, D, true, true, CMAX>(qL, b0.a, b0.b, b1.a, b1.b, a0x.a, gr.a, c0L, pf, FL, cL, dcL);
  }
  {
    const f2x2 b0 = tab2(row, TR_FR), b1 = tab2(row, TR_FR + 2);
    flux_lean2<NV, D, true, true, CMAX>(qR, b0.a, b0.b, b1.a, b1.b, a0x.b, gr.b, c0R, pf, FR, cR, dcR);
  }
  // g >= 0: alpha - alpha0 = max(dcL, dcR - g), else max(dcL + g, dcR)
  const f2 dalpha = max2(dcL + dup2(fminf(g, 0.0f)), dcR - dup2(fmaxf(g, 0.0f)));
  const f2 alpha = ga.b + dalpha;
#pragma unroll
  for (int v = 0; v < NV; ++v) G[v] = fma2(alpha, qL[v] - qR[v], FL[v] + FR[v]);
  const f2 nd = dalpha * dup2(-1.0f);
  G[0] = fma2(nd, j.a, G[0]);
  G[NV - 1] = fma2(nd, j.b, G[NV - 1]);
}
template <int NV, int D, bool BG, bool CMAX>
__device__ __forceinline__ void face_vert2(const f2 (&qL)[NV], const f2 (&qR)[NV], const float* row, const PhysF2& pf,
                                           f2 (&G)[NV]) {
  if constexpr (BG) face_vertical2<NV, D, CMAX>(qL, qR, row, pf, G);
  else face_flat2<NV, D, false, CMAX>(qL, qR, row, pf, G);
}

// Reduced tendency, force and RK combine of two cells of one vertical index,
// as cell_lean (the form is read at run time if FORM < 0).
template <int NV, int FORM, bool CMAX, int ST>
__device__ __forceinline__ void cell_lean2(const f2 (&q)[NV], f2 (&L)[NV], const f2 (&Dl)[NV], f2 rho0, f2 P0,
                                           const PhysF& pf, const PhysF2& p2, int form_rt, bool has_grav, f2 dt,
                                           const f2 (&b)[NV], f2 (&u)[NV], f2& rate, bool (&ok)[2]) {
  constexpr int ND = NV - 2;
  const int form = FORM >= 0 ? FORM : form_rt;
  if (form != RSST_EULER) {
    const f2 rho = rho0 + q[0];
    const f2 ir = rcp2(rho);
    f2 v[ND];
#pragma unroll
    for (int e = 0; e < ND; ++e) v[e] = q[1 + e] * ir;
    f2 k = q[1] * v[0];
#pragma unroll
    for (int e = 1; e < ND; ++e) k = fma2(q[1 + e], v[e], k);
    const f2 kin = k * dup2(0.5f);
    const f2 P = fma2(p2.gm1, q[NV - 1] - kin, P0);
    f2 fcell = dup2(pf.f);
    if constexpr (CMAX) {
      const f2 a2 = P * ir * dup2(pf.gamma);
      const f2 w = fma2(a2 * a2, p2.cmax4, dup2(1.0f));
      fcell = dup2(1.0f) - mk2(1.0f / sqrtf(lo2(w)), 1.0f / sqrtf(hi2(w)));
    }
    const bool mom = form == RSST_PVS || form == RSST_DVS;
    const f2 H = fma2(dup2(pf.gam_gm1), P, mom ? kin : kin * dup2(-1.0f));  // e + P +- rho V^2/2
    if (form == RSST_PVS || form == RSST_PMS || form == RSST_PD) {
      // minus dP/(gamma - 1), dE last: one rounding at its size (a float32 run
      // amplifies this term's round-off by xi^2)
      f2 ns = (k * dup2(-0.5f)) * ir * Dl[0];
#pragma unroll
      for (int e = 0; e < ND; ++e) ns = fma2(v[e], Dl[1 + e], ns);
      const f2 nfs = (ns - Dl[NV - 1]) * (fcell * dup2(pf.gm1));  // -f dP
      if (form == RSST_PD) {
        L[NV - 1] = fma2(nfs, dup2(pf.inv_gm1), L[NV - 1]);
      } else {
        const f2 nfg = nfs * rcp2(P * dup2(pf.gamma));  // -f dP / (rho a^2)
        const f2 nw = nfg * rho;                        // -f dP / a^2
        L[0] = L[0] + nw;
        if (mom) {
#pragma unroll
          for (int e = 0; e < ND; ++e) L[1 + e] = fma2(nw, v[e], L[1 + e]);
        }
        L[NV - 1] = fma2(nfg, H, L[NV - 1]);
      }
    } else {  // DVS, DMS: s = drho
      const f2 nfs = Dl[0] * (fcell * dup2(-1.0f));
      L[0] = L[0] + nfs;
      if (mom) {
#pragma unroll
        for (int e = 0; e < ND; ++e) L[1 + e] = fma2(nfs, v[e], L[1 + e]);
      }
      L[NV - 1] = fma2(nfs * ir, H, L[NV - 1]);
    }
  }
  if (has_grav) {  // perturbation force: rho1 F and m.F (rho0 F is in the background residual)
    f2 mg = q[1] * dup2(pf.grav[0]);
#pragma unroll
    for (int e = 0; e < ND; ++e) {
      L[1 + e] = fma2(q[0], dup2(pf.grav[e]), L[1 + e]);
      if (e > 0) mg = fma2(q[1 + e], dup2(pf.grav[e]), mg);
    }
    L[NV - 1] = L[NV - 1] + mg;
  }
  rate = dup2(0.0f);
  ok[0] = ok[1] = true;
  if constexpr (ST == 1) {
#pragma unroll
    for (int k = 0; k < NV; ++k) u[k] = fma2(dt, L[k], q[k]);
  } else {
#pragma unroll
    for (int k = 0; k < NV; ++k) u[k] = (b[k] + fma2(dt, L[k], q[k])) * dup2(0.5f);
    const f2 rn = rho0 + u[0];
    const f2 irn = rcp2(rn);
    f2 k = u[1] * u[1];
#pragma unroll
    for (int e = 1; e < ND; ++e) k = fma2(u[1 + e], u[1 + e], k);
    k = k * irn;
    const f2 Pn = fma2(p2.gm1, fma2(dup2(-0.5f), k, u[NV - 1]), P0);
    // rho and P positive and finite (a NaN or infinite component reaches one of them)
    ok[0] = (__float_as_uint(lo2(rn)) - 1u < 0x7f7fffffu) && (__float_as_uint(lo2(Pn)) - 1u < 0x7f7fffffu);
    ok[1] = (__float_as_uint(hi2(rn)) - 1u < 0x7f7fffffu) && (__float_as_uint(hi2(Pn)) - 1u < 0x7f7fffffu);
    rate = (sqrt2(k * irn) + sound_x2<CMAX>(p2.gx * Pn * irn, p2)) * dup2(pf.sum_inv_dx);
  }
}

}  // namespace rsst
