// Discrete adjoint of the float64 SSP-RK2 step (the transpose of the
// Jacobian of the discrete map U^n -> U^{n+1}, dt held fixed), with
// checkpoint-and-recompute.  The paper has no adjoint; the conventions
// (fixed dt, forward branch of every non-smooth operation: MC branch, LLF
// max with ties to the left state, zero subgradient of |V| at V = 0) are
// this library's and match the oracle's reverse-mode derivative.
//
// One stage is out = a * base + b * (in + dt L(in)).  Its adjoint needs the
// vector-Jacobian product mu^T dL/d(in) (mu = b dt lambda_out) and
// mu^T dL/dxi:
//   adj_cell: per interior cell, with the Euler tendency dU that the forward
//     kernel wrote while the segment was recomputed, nu = mu^T dC/d(dU) and
//     the pointwise part mu^T d(C + force)/dq (C = reduced tendency, Sec. 3.2 /
//     App. A; force of App. B) plus the identity part b lambda_out (and, in
//     stage 1, lambda^{n+1}/2), and the xi partial;
//   adj_face: per face of any axis, phi = (nu_right - nu_left)/dx, then
//     phi^T dF/dU_k for the four stencil cells k of the face (MC slopes, face
//     states, LLF flux of Sec. 4.2) and the xi partial;
//   adj_gather: each interior cell sums the contributions of the faces whose
//     stencil holds it or a ghost cell it is the image of (wrap, or mirror
//     with the normal momentum negated).
// The derivatives are hand-derived reverse mode: each VJP recomputes its
// forward values (holding the branches the forward pass took) and then runs
// the chain rule backwards once.
//
// What bounds it: the float64 pipe, in the face kernel above all.  A 2D face
// takes 154 float64 instructions (295 when both sides carried the wave speed's
// derivatives, speeds and their reciprocals came from float64 square roots,
// limiter and flux halves were multiplications and each block summed its xi
// partials by a float64 tree).  A stage's VJP on 256^2 (ncu, us): cells 21,
// faces 50 (80 % of the float64 pipe; one launch for both axes, 94 in two),
// gather 15; ghost fold, xi sum and axpby (together 18) are gone into these.
#include <cstring>
#include <vector>

#include "rsst_common.cuh"
#include "rsst_internal.h"
#include "rsst_check.h"
#include "rsst_math_fp64.cuh"

namespace rsst {

// d(half slope)/da and /db of the taken branch, times the half slope's adjoint ds.
__device__ __forceinline__ void mc_reverse(int br, double ds, double& da, double& db) {
  const double q = half_of(half_of(ds));
  da = br == 1 ? ds : (br == 3 ? q : 0.0);
  db = br == 2 ? ds : (br == 3 ? q : 0.0);
}

// a/xi under the C_max law (Eq. cx).
__device__ __forceinline__ double sound_cmax(double a2, const Phys& p) {
  return sqrt(a2 * rcp_nr(sqrt(1.0 + (a2 * a2) * p.inv_cmax4)));
}

// The forward values of one face state that the reverse of its flux reuses.
template <int NV>
struct StateFwd {
  double ir, v[NV - 2], hv2, P;  // 1/rho, V, |V|^2/2, P
  double k;                      // rho |V|^2
};
template <int NV>
__device__ __forceinline__ void state_fwd(const double (&q)[NV], const Phys& p, StateFwd<NV>& w) {
  constexpr int ND = NV - 2;
  w.ir = rcp_nr(q[0]);
#pragma unroll
  for (int e = 0; e < ND; ++e) {
    w.v[e] = q[1 + e] * w.ir;
    w.k = e == 0 ? q[1] * w.v[0] : fma(q[1 + e], w.v[e], w.k);
  }
  w.P = p.gm1 * q[NV - 1] - p.hgm1 * w.k;
  w.hv2 = half_of(w.k) * w.ir;
}

// Reverse of the Euler flux along the first momentum (F = (m_0, m V_0 + P e_0,
// (E + P) V_0)) at q for the cotangent f: adds f^T dF/dq to dq, through
// V_0 = m_0/rho and P = (gamma-1)(E - |m|^2/(2 rho)).
template <int NV>
__device__ __forceinline__ void flux_vjp(const double (&q)[NV], const Phys& p, const StateFwd<NV>& w,
                                         const double (&f)[NV], double (&dq)[NV]) {
  constexpr int ND = NV - 2;
  const double v0 = w.v[0];
  const double g = p.gm1 * fma(f[NV - 1], v0, f[1]);  // (gamma-1) dP
  double dv = f[NV - 1] * (q[NV - 1] + w.P);
#pragma unroll
  for (int e = 0; e < ND; ++e) dv = fma(f[1 + e], q[1 + e], dv);
  const double t = dv * w.ir;
  dq[0] = fma(-t, v0, fma(g, w.hv2, dq[0]));
  dq[1] += f[0] + t;
#pragma unroll
  for (int e = 0; e < ND; ++e) dq[1 + e] = fma(-g, w.v[e], fma(f[1 + e], v0, dq[1 + e]));
  dq[NV - 1] = fma(f[NV - 1], v0, dq[NV - 1]) + g;
}

// Reverse of twice the face's LLF flux (Sec. 4.2, steps 2-4, through its
// MUSCL-MC states) for half the cotangent, f = phi/2; fields ordered with the
// face's normal momentum first.  G[k] = phi^T dF/d(stencil cell k), and the
// return value phi^T dF/d(1/xi).  The forward branches (MC branch, LLF side)
// are recomputed and held; the LLF speed's derivatives are taken on the side
// it came from only.
template <int NV>
__device__ __forceinline__ double face_vjp(const double (&s)[4][NV], const double (&f)[NV], const Phys& p,
                                           double (&G)[4][NV]) {
  constexpr int ND = NV - 2;
  double qL[NV], qR[NV];
  int bL[NV], bR[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const double d0 = s[1][v] - s[0][v], d1 = s[2][v] - s[1][v], d2 = s[3][v] - s[2][v];
    qL[v] = s[1][v] + half_mc(d0, d1, bL[v]);
    qR[v] = s[2][v] - half_mc(d1, d2, bR[v]);
  }
  StateFwd<NV> wL, wR;
  state_fwd<NV>(qL, p, wL);
  state_fwd<NV>(qR, p, wR);
  double dalpha = 0.0;
#pragma unroll
  for (int v = 0; v < NV; ++v) dalpha = fma(f[v], qL[v] - qR[v], dalpha);
  // LLF speed and, on its side: |V|, d(c)/d(m_e) = v_e iv / rho, and with
  // ca = a/xi the products cP = dc dca/dP and cr = -dc dca/drho
  bool left;
  double alpha, sv, iv, cP, cr, dinv_xi = 0.0;
  if (p.use_cmax) {
    const double a2L = p.gamma * wL.P * wL.ir, a2R = p.gamma * wR.P * wR.ir;
    const double vL = wL.k * wL.ir, vR = wR.k * wR.ir;
    const double sL = vL > 0.0 ? sqrt_ctot(vL) : 0.0, sR = vR > 0.0 ? sqrt_ctot(vR) : 0.0;
    const double cL = sL + sound_cmax(a2L, p), cR = sR + sound_cmax(a2R, p);
    left = cL >= cR;
    alpha = left ? cL : cR;
    sv = left ? sL : sR;
    iv = sv > 0.0 ? rcp_nr(sv) : 0.0;
    // ca = sqrt(u), u = a2 / t, t = sqrt(w), w = 1 + a2^2 / C^4
    const double a2 = left ? a2L : a2R, ir = left ? wL.ir : wR.ir;
    const double t = sqrt(1.0 + (a2 * a2) * p.inv_cmax4), it = rcp_nr(t), u = a2 * it;
    double da2 = 0.0;
    if (u > 0.0) {
      const double du = dalpha * 0.5 * rcp_nr(sqrt(u));
      da2 = du * it - du * u * it * it * a2 * p.inv_cmax4;
    }
    cP = da2 * p.gamma * ir;
    cr = da2 * a2 * ir;
  } else {
    float hL, lL, hR, lR;
    ctot_pair_of(wL.k, wL.P, wL.ir, p, hL, lL);
    ctot_pair_of(wR.k, wR.P, wR.ir, p, hR, lR);
    left = hL > hR || (hL == hR && lL >= lR);
    const double ir = left ? wL.ir : wR.ir, k = left ? wL.k : wR.k, P = left ? wL.P : wR.P;
    alpha = pair_to_double(left ? hL : hR, left ? lL : lR);
    sqrt_rcp(k * ir, sv, iv);  // |V|
    const double gir = p.gamma_xi2 * ir;
    double ca, ica;
    sqrt_rcp(gir * P, ca, ica);  // a/xi
    const double dh = half_of(dalpha);
    cP = dh * (gir * ica);
    cr = dh * (ca * ir);
    dinv_xi = dalpha * (ca * p.xi);
  }
  double dqL[NV], dqR[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    dqL[v] = alpha * f[v];
    dqR[v] = -dqL[v];
  }
  flux_vjp<NV>(qL, p, wL, f, dqL);
  flux_vjp<NV>(qR, p, wR, f, dqR);
  {
    // dc on its side: d|V|/dm_e = v_e/(rho |V|), d|V|/drho = -|V|/rho, and a/xi
    // through P and rho
    const double ir = left ? wL.ir : wR.ir, hv2 = left ? wL.hv2 : wR.hv2;
    const double t = dalpha * ir, g = p.gm1 * cP, c = fma(t, iv, -g);
    double x[NV];
    x[0] = fma(g, hv2, fma(-t, sv, -cr));
#pragma unroll
    for (int e = 0; e < ND; ++e) x[1 + e] = c * (left ? wL.v[e] : wR.v[e]);
    x[NV - 1] = g;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const double y = (left ? dqL[v] : dqR[v]) + x[v];
      dqL[v] = left ? y : dqL[v];
      dqR[v] = left ? dqR[v] : y;
    }
  }
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    double da, db, ea, eb;
    mc_reverse(bL[v], dqL[v], da, db);  // qL = u0 + h(u0 - um, u1 - u0)
    mc_reverse(bR[v], dqR[v], ea, eb);  // qR = u1 - h(u1 - u0, up - u1)
    G[0][v] = -da;
    G[1][v] = (dqL[v] + (da - db)) + ea;
    G[2][v] = (dqR[v] - (ea - eb)) + db;
    G[3][v] = -eb;
  }
  return dinv_xi;
}

// Reverse of the reduced tendency plus force at one cell,
//   L = dU - f s r + (0, rho F, m.F)   (Sec. 3.2, App. A, App. B),
// for the cotangent mu: nu = mu^T dL/d(dU), dq = mu^T dL/dq, and the return
// value mu^T dL/df (zero under the C_max law, where f comes from the state).
// With w = mu . r the correction contributes -f s w, so ds = -f w, dw = -f s.
template <int NV>
__device__ __forceinline__ double rhs_vjp(const double (&q)[NV], const double (&dU)[NV], const double (&mu)[NV],
                                          const Phys& p, double (&nu)[NV], double (&dq)[NV]) {
  constexpr int ND = NV - 2;
  const double rho = q[0];
  double dfc_total = 0.0;
  for (int v = 0; v < NV; ++v) {
    nu[v] = mu[v];
    dq[v] = 0.0;
  }
  const int var = p.variant;
  if (var != RSST_EULER) {
    const double ir = rcp_nr(rho);
    double v[ND], dv[ND];
    double v2 = 0.0, vdm = 0.0, mv = 0.0;
    for (int e = 0; e < ND; ++e) {
      v[e] = q[1 + e] * ir;
      v2 += v[e] * v[e];
      vdm += v[e] * dU[1 + e];
      mv += mu[1 + e] * v[e];
      dv[e] = 0.0;
    }
    const double E = q[NV - 1];
    const double P = p.gm1 * (E - 0.5 * (rho * v2));
    const double kin = 0.5 * (rho * v2);
    const bool pform = var == RSST_PVS || var == RSST_PMS || var == RSST_PD;
    const double sgn = (var == RSST_PVS || var == RSST_DVS) ? 1.0 : -1.0;
    const double H = P * p.inv_gm1 + P + sgn * kin;  // e + P +- rho|V|^2/2
    double s, r0, rv, rE, ia2 = 0.0, igP = 0.0;  // igP = 1/(gamma P)
    if (pform) {
      s = p.gm1 * (0.5 * (v2 * dU[0]) - vdm + dU[NV - 1]);
      if (var == RSST_PD) {
        r0 = 0.0; rv = 0.0; rE = p.inv_gm1;
      } else {
        igP = rcp_nr(p.gamma * P);
        ia2 = rho * igP;
        r0 = ia2;
        rv = var == RSST_PVS ? ia2 : 0.0;
        rE = H * ia2 * ir;
      }
    } else {
      s = dU[0];
      r0 = 1.0;
      rv = var == RSST_DVS ? 1.0 : 0.0;
      rE = H * ir;
    }
    double a2 = 0.0, wc = 0.0, fc = p.f;
    if (p.use_cmax) {
      a2 = p.gamma * P * ir;
      wc = 1.0 + (a2 * a2) * p.inv_cmax4;
      fc = 1.0 - rcp_nr(sqrt(wc));
    }
    const double w = mu[0] * r0 + rv * mv + mu[NV - 1] * rE;
    const double ds = -fc * w, dw = -fc * s, dfc = -s * w;
    double dv2 = 0.0, drho = 0.0, dP = 0.0, dH = 0.0;
    if (pform) {
      nu[0] += ds * p.gm1 * 0.5 * v2;
      for (int e = 0; e < ND; ++e) {
        nu[1 + e] -= ds * p.gm1 * v[e];
        dv[e] -= ds * p.gm1 * dU[1 + e];
      }
      nu[NV - 1] += ds * p.gm1;
      dv2 += ds * p.gm1 * 0.5 * dU[0];
    } else {
      nu[0] += ds;
    }
    for (int e = 0; e < ND; ++e) dv[e] += dw * rv * mu[1 + e];
    if (var == RSST_PVS || var == RSST_PMS) {
      double dia2 = dw * mu[0] + (var == RSST_PVS ? dw * mv : 0.0);
      const double drE = dw * mu[NV - 1];
      dH = drE * ia2 * ir;
      dia2 += drE * H * ir;
      drho -= drE * rE * ir;
      drho += dia2 * igP;
      dP -= dia2 * ia2 * (p.gamma * igP);  // ia2 / P
    } else if (var == RSST_DVS || var == RSST_DMS) {
      dH = dw * mu[NV - 1] * ir;
      drho -= dw * mu[NV - 1] * rE * ir;
    }
    dP += dH * (p.inv_gm1 + 1.0);
    const double dkin = sgn * dH;
    if (p.use_cmax) {
      const double da2 = dfc * p.inv_cmax4 * a2 * rcp_nr(wc * sqrt(wc));
      dP += da2 * p.gamma * ir;
      drho -= da2 * a2 * ir;
    } else {
      dfc_total = dfc;
    }
    drho += dkin * 0.5 * v2;
    dv2 += dkin * 0.5 * rho;
    dq[NV - 1] += dP * p.gm1;
    drho -= dP * p.gm1 * 0.5 * v2;
    dv2 -= dP * p.gm1 * 0.5 * rho;
    for (int e = 0; e < ND; ++e) {
      dv[e] += 2.0 * v[e] * dv2;
      dq[1 + e] += dv[e] * ir;
      drho -= dv[e] * v[e] * ir;
    }
    dq[0] += drho;
  }
  if (p.has_grav) {
    for (int e = 0; e < ND; ++e) {
      dq[0] += mu[1 + e] * p.grav[e];
      dq[1 + e] += mu[NV - 1] * p.grav[e];
    }
  }
  return dfc_total;
}

struct AdjArgs {
  const double* U;   // stage input, padded
  const double* dU;  // its Euler tendency, padded (written by the forward kernel on recompute)
  const double* lam_out;  // lambda of the stage output, padded (interior used)
  double mu_scale;        // mu = mu_scale * lambda_out = b dt lambda_out
  double id_scale;        // the stage's identity part adds id_scale * lambda_out = b lambda_out
  const double* add;      // stage 1: lambda^{n+1}, half of which is added (may be lam itself); or null
  double* nu;        // padded, interior written
  double* lam;       // padded output (interior)
  double* faceG;     // [4 stencil cells][NV][all faces]: coalesced for the faces and for the cells that gather
  double* xi_part;   // [cells + all faces]: xi partials, accumulated over the stages
  double xi_cell, xi_face;  // df/dxi and d(1/xi)/dxi
  Geom g;
  Phys p;
  int64_t nfaces;       // of all axes
  int64_t face_off[3];  // first face of each axis
};

__device__ __forceinline__ int64_t pidx_c(const Geom& g, const int (&c)[3]) { return pidx(g, c[0], c[1], c[2]); }

__device__ __forceinline__ void block_sum_to(double x, double* dst, double* sh) {
  sh[threadIdx.x] = x;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) *dst = sh[0];
}

template <int NV>
__global__ void __launch_bounds__(128) adj_cell_kernel(AdjArgs a) {
  const Geom& g = a.g;
  const Phys& p = a.p;
  const int64_t id = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (id >= g.ncells) return;
  const int c[3] = {(int)(id % g.n[0]), (int)((id / g.n[0]) % g.n[1]), (int)(id / ((int64_t)g.n[0] * g.n[1]))};
  const int64_t o = pidx_c(g, c);
  double q[NV], dU[NV], lo[NV], mu[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    q[v] = a.U[v * g.fstride + o];
    lo[v] = a.lam_out[v * g.fstride + o];
    mu[v] = a.mu_scale * lo[v];
    dU[v] = a.dU[v * g.fstride + o];
  }
  // nu = mu^T dL/d(dU), pointwise mu^T dL/dq, xi partial (f = 1 - 1/xi^2)
  double nu[NV], dq[NV];
  const double df = rhs_vjp<NV>(q, dU, mu, p, nu, dq);
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    a.nu[v * g.fstride + o] = nu[v];
    double l = fma(a.id_scale, lo[v], dq[v]);
    if (a.add) l = fma(0.5, a.add[v * g.fstride + o], l);
    a.lam[v * g.fstride + o] = l;
  }
  a.xi_part[id] = fma(df, a.xi_cell, a.xi_part[id]);
}

// Faces of axis blockIdx.y: index (f, other coords) with f in [0, n_D] (face
// f - 1/2).  The axis enters through strides and the order of the momenta
// only, so one launch takes all axes.
template <int NV>
__global__ void __launch_bounds__(128) adj_face_kernel(AdjArgs a) {
  constexpr int ND = NV - 2;
  const Geom& g = a.g;
  const Phys& p = a.p;
  const int D = blockIdx.y;
  int ext[3] = {g.n[0], g.n[1], g.n[2]};
  ext[D] += 1;
  const int64_t id = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (id >= (int64_t)ext[0] * ext[1] * ext[2]) return;
  const int c[3] = {(int)(id % ext[0]), (int)((id / ext[0]) % ext[1]), (int)(id / ((int64_t)ext[0] * ext[1]))};
  const int f = c[D];
  const int64_t o = pidx_c(g, c);  // the cell right of the face
  const int64_t st = D == 0 ? 1 : (D == 1 ? g.pitch : g.plane);
  int fld[NV];  // normal momentum first
  fld[0] = 0;
  fld[NV - 1] = NV - 1;
#pragma unroll
  for (int e = 0; e < ND; ++e) fld[1 + e] = 1 + (e == 0 ? D : (e <= D ? e - 1 : e));
  double s[4][NV], phi[NV], G[4][NV];
  const bool has_r = f < g.n[D], has_l = f > 0;
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const double* u = a.U + fld[v] * g.fstride + o;
#pragma unroll
    for (int k = 0; k < 4; ++k) s[k][v] = u[(k - 2) * st];  // cells f - 2 .. f + 1
    // phi/2 = (nu_right - nu_left) / (2 dx), nu = 0 outside the interior
    const double* nu = a.nu + fld[v] * g.fstride + o;
    phi[v] = ((has_r ? nu[0] : 0.0) - (has_l ? nu[-st] : 0.0)) * p.half_inv_dx[D];
  }
  const double dinv_xi = face_vjp<NV>(s, phi, p, G);
  const int64_t fid = a.face_off[D] + id;
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int v = 0; v < NV; ++v) a.faceG[(k * NV + fld[v]) * a.nfaces + fid] = G[k][v];
  double* xp = a.xi_part + g.ncells + fid;
  *xp = fma(dinv_xi, a.xi_face, *xp);
}

// Contributions to extended cell x along axis d of the line through cell c:
// those of the faces f - 1/2, f in [x-1, x+2].
template <int NV>
__device__ __forceinline__ void gather_axis(const AdjArgs& a, const int (&c)[3], int d, int x, double (&acc)[NV]) {
  const Geom& g = a.g;
  int ext[3] = {g.n[0], g.n[1], g.n[2]};
  ext[d] += 1;
#pragma unroll
  for (int k = 0; k < 4; ++k) {  // the cell's place in the face's stencil
    const int f = x + 2 - k;
    if (f < 0 || f > g.n[d]) continue;
    int cf[3] = {c[0], c[1], c[2]};
    cf[d] = f;
    const double* G = a.faceG + a.face_off[d] + ((int64_t)cf[2] * ext[1] + cf[1]) * ext[0] + cf[0];
#pragma unroll
    for (int v = 0; v < NV; ++v) acc[v] += G[(k * NV + v) * a.nfaces];
  }
}

// Each interior cell adds the face contributions to itself and to every ghost
// cell that was copied from it.
template <int NV>
__global__ void __launch_bounds__(128) adj_gather_kernel(AdjArgs a) {
  constexpr int ND = NV - 2;
  const Geom& g = a.g;
  const Phys& p = a.p;
  const int64_t id = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (id >= g.ncells) return;
  const int c[3] = {(int)(id % g.n[0]), (int)((id / g.n[0]) % g.n[1]), (int)(id / ((int64_t)g.n[0] * g.n[1]))};
  double acc[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) acc[v] = 0.0;
#pragma unroll
  for (int d = 0; d < ND; ++d) {
    gather_axis<NV>(a, c, d, c[d], acc);
    const int n = g.n[d], cd = c[d];
    if (cd >= RSST_G && cd < n - RSST_G) continue;
    for (int side = 0; side < 2; ++side) {
      if (side == 0 ? cd >= RSST_G : cd < n - RSST_G) continue;
      const bool per = p.bc[d] == RSST_BC_PERIODIC;
      const int gp = per ? (side == 0 ? cd + n : cd - n) : (side == 0 ? -1 - cd : 2 * n - 1 - cd);
      double x[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) x[v] = 0.0;
      gather_axis<NV>(a, c, d, gp, x);
#pragma unroll
      for (int v = 0; v < NV; ++v) acc[v] += (!per && v == 1 + d) ? -x[v] : x[v];
    }
  }
  const int64_t o = pidx_c(g, c);
#pragma unroll
  for (int v = 0; v < NV; ++v) a.lam[v * g.fstride + o] += acc[v];
}

// caller layout <-> padded interior
__global__ void to_padded_kernel(const double* src, double* dst, Geom g, int nv) {
  const int64_t id = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (id >= g.ncells) return;
  const int c[3] = {(int)(id % g.n[0]), (int)((id / g.n[0]) % g.n[1]), (int)(id / ((int64_t)g.n[0] * g.n[1]))};
  const int64_t o = pidx_c(g, c);
  for (int v = 0; v < nv; ++v) dst[v * g.fstride + o] = src[v * g.ncells + id];
}
__global__ void from_padded_kernel(const double* src, double* dst, Geom g, int nv) {
  const int64_t id = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (id >= g.ncells) return;
  const int c[3] = {(int)(id % g.n[0]), (int)((id / g.n[0]) % g.n[1]), (int)(id / ((int64_t)g.n[0] * g.n[1]))};
  const int64_t o = pidx_c(g, c);
  for (int v = 0; v < nv; ++v) dst[v * g.ncells + id] = src[v * g.fstride + o];
}

// Kinetic energy J = sum |m|^2/(2 rho) dV and dJ/dU = (-|V|^2/2, V, 0) dV.
template <int NV>
__global__ void __launch_bounds__(128) ke_kernel(const double* U, Geom g, double vol, double* part, double* grad) {
  constexpr int ND = NV - 2;
  __shared__ double sh[128];
  const int64_t id = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  double J = 0.0;
  if (id < g.ncells) {
    const int c[3] = {(int)(id % g.n[0]), (int)((id / g.n[0]) % g.n[1]), (int)(id / ((int64_t)g.n[0] * g.n[1]))};
    const int64_t o = pidx_c(g, c);
    const double rho = U[o];
    double m2 = 0.0, v2 = 0.0;
    for (int e = 0; e < ND; ++e) {
      const double m = U[(1 + e) * g.fstride + o];
      m2 += m * m;
      v2 += (m / rho) * (m / rho);
      if (grad) grad[(1 + e) * g.ncells + id] = m / rho * vol;
    }
    J = 0.5 * m2 / rho * vol;
    if (grad) {
      grad[id] = -0.5 * v2 * vol;
      grad[(NV - 1) * g.ncells + id] = 0.0;
    }
  }
  block_sum_to(J, part + blockIdx.x, sh);
}

// Fixed-order sum of a block's share of x[0 .. n - 1] into part[blockIdx.x].
__global__ void __launch_bounds__(256) sum_share_kernel(const double* x, int64_t n, double* part) {
  __shared__ double sh[256];
  const int64_t chunk = (n + gridDim.x - 1) / gridDim.x, lo = blockIdx.x * chunk, hi = min(n, lo + chunk);
  double acc = 0.0;
  for (int64_t i = lo + threadIdx.x; i < hi; i += 256) acc += x[i];
  block_sum_to(acc, part + blockIdx.x, sh);
}

__global__ void sum_parts_kernel(const double* part, int n, double* out, int accumulate) {
  __shared__ double sh[256];
  double acc = 0.0;
  for (int i = threadIdx.x; i < n; i += 256) acc += part[i];
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = accumulate ? *out + sh[0] : sh[0];
}

}  // namespace rsst

using namespace rsst;

// ---------------------------------------------------------------------------
// Host orchestration
// ---------------------------------------------------------------------------

struct AdjState {
  double dt = 0.0;
  int nsteps = 0, every = 0, nseg = 0;
  std::vector<double*> ckpt;   // padded states at steps 0, every, 2 every, ...
  double* stages = nullptr;    // recompute storage: 2 * every padded states
  double* dUs = nullptr;       // their Euler tendencies (same layout)
  double* save = nullptr;      // the live state while a segment is recomputed
  double* scal = nullptr;      // and its scalars
  double* lamA = nullptr;      // padded work arrays
  double* lamB = nullptr;
  double* nu = nullptr;
  double* faceG = nullptr;
  double* xi_part = nullptr;   // xi partials of every cell and face of a segment
  double* dxi = nullptr;       // [0] their sum, [1 ..] the sum's partials
  int64_t face_off[3] = {0, 0, 0}, faces = 0;
};

constexpr int XI_BLOCKS = 256;  // blocks of the xi partials' sum

static AdjState* adj_of(rsst_handle* h) { return reinterpret_cast<AdjState*>(h->adj); }

void rsst_adjoint_free(rsst_handle* h) {
  AdjState* s = adj_of(h);
  if (!s) return;
  for (double* c : s->ckpt) cudaFree(c);
  cudaFree(s->stages);
  cudaFree(s->dUs);
  cudaFree(s->save);
  cudaFree(s->lamA);
  cudaFree(s->lamB);
  cudaFree(s->nu);
  cudaFree(s->faceG);
  cudaFree(s->xi_part);
  cudaFree(s->dxi);
  cudaFree(s->scal);
  delete s;
  h->adj = nullptr;
}

static size_t state_bytes(const rsst_handle* h) { return (size_t)(h->g.ndim + 2) * h->g.fstride * sizeof(double); }

static int blocks_for(int64_t n) { return (int)((n + 127) / 128); }

static int launch_err(const char* what) {
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    rsst_set_error("%s: %s", what, cudaGetErrorString(e));
    return RSST_ECUDA;
  }
  return RSST_OK;
}

extern "C" int rsst_adjoint_record(rsst_handle* h, double dt, int nsteps, int every) {
  if (!h || !(dt > 0.0) || !std::isfinite(dt) || nsteps < 1 || every < 1) {
    rsst_set_error("rsst_adjoint_record: need a handle, finite dt > 0, nsteps >= 1, every >= 1");
    return RSST_EINVAL;
  }
  if (h->cfg.precision != RSST_FP64) {
    rsst_set_error("rsst_adjoint_record: the adjoint is float64 only");
    return RSST_EUNSUPPORTED;
  }
  if (h->cfg.covolume != 0.0) {
    rsst_set_error("rsst_adjoint_record: the adjoint is derived for the ideal gas only");
    return RSST_EUNSUPPORTED;
  }
  // A recording of the same shape reuses the last one's memory (allocating
  // and freeing it costs milliseconds and synchronises the device).
  const int nseg = (nsteps + every - 1) / every;
  AdjState* s = adj_of(h);
  if (!s || s->every != every || s->nseg != nseg) {
    rsst_adjoint_free(h);
    s = new AdjState();
    h->adj = s;
    s->every = every;
    s->nseg = nseg;
    const size_t sb = state_bytes(h);
    const Geom& g = h->g;
    for (int d = 0; d < g.ndim; ++d) {
      s->face_off[d] = s->faces;
      s->faces += g.ncells / g.n[d] * (g.n[d] + 1);
    }
    const int nv = g.ndim + 2;
    bool ok = cudaMalloc((void**)&s->stages, 2 * (size_t)every * sb) == cudaSuccess &&
              cudaMalloc((void**)&s->dUs, 2 * (size_t)every * sb) == cudaSuccess &&
              cudaMalloc((void**)&s->save, sb) == cudaSuccess &&
              cudaMalloc((void**)&s->scal, 16 * sizeof(double)) == cudaSuccess &&
              cudaMalloc((void**)&s->lamA, sb) == cudaSuccess && cudaMalloc((void**)&s->lamB, sb) == cudaSuccess &&
              cudaMalloc((void**)&s->nu, sb) == cudaSuccess &&
              cudaMalloc((void**)&s->faceG, (size_t)s->faces * 4 * nv * sizeof(double)) == cudaSuccess &&
              cudaMalloc((void**)&s->xi_part, (size_t)(g.ncells + s->faces) * sizeof(double)) == cudaSuccess &&
              cudaMalloc((void**)&s->dxi, (1 + XI_BLOCKS) * sizeof(double)) == cudaSuccess;
    for (int k = 0; ok && k < s->nseg; ++k) {
      double* c = nullptr;
      ok = cudaMalloc((void**)&c, sb) == cudaSuccess;
      s->ckpt.push_back(c);
    }
    if (!ok) {
      cudaGetLastError();
      rsst_adjoint_free(h);
      rsst_set_error("rsst_adjoint_record: device allocation failed");
      return RSST_ENOMEM;
    }
  }
  s->dt = dt;
  s->nsteps = nsteps;
  const size_t sb = state_bytes(h);
  for (int step = 0; step < nsteps; ++step) {
    if (step % every == 0) {
      if (cudaMemcpyAsync(s->ckpt[step / every], h->buf[0], sb, cudaMemcpyDeviceToDevice, h->stream) != cudaSuccess) {
        rsst_set_error("rsst_adjoint_record: checkpoint copy failed");
        return RSST_ECUDA;
      }
    }
    const int rc = rsst_handle_steps(h, dt, 1);
    if (rc != RSST_OK) return rc;
  }
  return RSST_OK;
}

extern "C" int rsst_adjoint_segments(rsst_handle* h, int32_t* nseg) {
  if (!h || !nseg || !adj_of(h)) { rsst_set_error("rsst_adjoint_segments: no recorded run"); return RSST_EINVAL; }
  *nseg = adj_of(h)->nseg;
  return RSST_OK;
}

// lam_out (padded, interior) -> its contribution through one stage.
// in: the stage input state; b: coefficient of (in + dt L(in)).
// Writes b lam_out + (b dt lam_out)^T dL/d(in), plus add/2 if given, into
// `res` (padded, interior; may be `add`) and adds the xi partials.
static int stage_vjp(rsst_handle* h, AdjState* s, const double* in, const double* dU, const double* lam_out, double b,
                     const double* add, double* res) {
  const Geom& g = h->g;
  const int nv = g.ndim + 2;
  cudaStream_t st = h->stream;
  const double xi = h->p.xi;
  AdjArgs a;
  memset(&a, 0, sizeof a);
  a.U = in;
  a.dU = dU;
  a.lam_out = lam_out;
  a.mu_scale = b * s->dt;
  a.id_scale = b;
  a.add = add;
  a.nu = s->nu;
  a.lam = res;
  a.faceG = s->faceG;
  a.xi_part = s->xi_part;
  a.xi_cell = 2.0 / (xi * xi * xi);
  a.xi_face = -1.0 / (xi * xi);
  a.g = g;
  a.p = h->p;
  a.nfaces = s->faces;
  int64_t nf = 0;
  for (int d = 0; d < 3; ++d) a.face_off[d] = s->face_off[d];
  for (int d = 0; d < g.ndim; ++d) {
    const int64_t m = g.ncells / g.n[d] * (g.n[d] + 1);
    nf = m > nf ? m : nf;
  }
  const int cb = blocks_for(g.ncells);
  const dim3 fb(blocks_for(nf), g.ndim);
#define RSST_VJP(NVv)                                \
  adj_cell_kernel<NVv><<<cb, 128, 0, st>>>(a);       \
  adj_face_kernel<NVv><<<fb, 128, 0, st>>>(a);       \
  adj_gather_kernel<NVv><<<cb, 128, 0, st>>>(a)
  switch (nv) {
    case 3: RSST_VJP(3); break;
    case 4: RSST_VJP(4); break;
    default: RSST_VJP(5); break;
  }
#undef RSST_VJP
  h->launches += 3;
  return launch_err("adjoint stage kernels");
}

extern "C" int rsst_adjoint_step(rsst_handle* h, int32_t seg, double* lam, double* dJ_dxi) {
  AdjState* s = h ? adj_of(h) : nullptr;
  if (!s || !lam || !dJ_dxi || seg < 0 || seg >= s->nseg) {
    rsst_set_error("rsst_adjoint_step: bad arguments or no recorded run");
    return RSST_EINVAL;
  }
  if (rsst_check_buffer(lam, 0, "rsst_adjoint_step (lam)") != RSST_OK) return RSST_EINVAL;
  const Geom& g = h->g;
  const int nv = g.ndim + 2;
  const size_t sb = state_bytes(h);
  cudaStream_t st = h->stream;
  const int s0 = seg * s->every;
  const int k = (s0 + s->every <= s->nsteps) ? s->every : s->nsteps - s0;
  const int64_t fe = g.fstride * (int64_t)nv;
  // recompute the segment: stages[2i] = U^{s0+i}, stages[2i+1] = U*; the
  // live state and scalars are saved and put back afterwards
  cudaError_t ce = cudaSuccess;
  auto chk = [&](cudaError_t e) { if (ce == cudaSuccess && e != cudaSuccess) ce = e; };
  int rc = RSST_OK;
  const int slot0 = h->slot;
  chk(cudaMemcpyAsync(s->scal, h->d_scal, 16 * sizeof(double), cudaMemcpyDeviceToDevice, st));
  chk(cudaMemcpyAsync(s->save, h->buf[0], sb, cudaMemcpyDeviceToDevice, st));
  chk(cudaMemcpyAsync(h->buf[0], s->ckpt[seg], sb, cudaMemcpyDeviceToDevice, st));
  for (int i = 0; i < k && rc == RSST_OK && ce == cudaSuccess; ++i) {
    chk(cudaMemcpyAsync(s->stages + (2 * i) * fe, h->buf[0], sb, cudaMemcpyDeviceToDevice, st));
    h->rec_dU[0] = s->dUs + (2 * i) * fe;      // the forward kernels also write each stage's Euler tendency
    h->rec_dU[1] = s->dUs + (2 * i + 1) * fe;
    rc = rsst_handle_steps(h, s->dt, 1);
    h->rec_dU[0] = h->rec_dU[1] = nullptr;
    // buf[1] still holds U* of this step
    chk(cudaMemcpyAsync(s->stages + (2 * i + 1) * fe, h->buf[1], sb, cudaMemcpyDeviceToDevice, st));
  }
  chk(cudaMemcpyAsync(h->buf[0], s->save, sb, cudaMemcpyDeviceToDevice, st));
  chk(cudaMemcpyAsync(h->d_scal, s->scal, 16 * sizeof(double), cudaMemcpyDeviceToDevice, st));
  if (rc == RSST_OK && ce != cudaSuccess) {
    rsst_set_error("rsst_adjoint_step: segment recompute: %s", cudaGetErrorString(ce));
    rc = RSST_ECUDA;
  }
  h->slot = slot0;
  if (rc == RSST_OK) {
    const int64_t parts = g.ncells + s->faces;
    if (cudaMemsetAsync(s->xi_part, 0, (size_t)parts * sizeof(double), st) != cudaSuccess) {
      rsst_set_error("rsst_adjoint_step: clearing the xi partials failed");
      return RSST_ECUDA;
    }
    to_padded_kernel<<<blocks_for(g.ncells), 128, 0, st>>>(lam, s->lamA, g, nv);
    for (int i = k - 1; i >= 0 && rc == RSST_OK; --i) {
      const double* Un = s->stages + (2 * i) * fe;
      const double* Us = s->stages + (2 * i + 1) * fe;
      // stage 2: U^{n+1} = 1/2 U^n + 1/2 (U* + dt L(U*)):  lamB = lambda_*
      rc = stage_vjp(h, s, Us, s->dUs + (2 * i + 1) * fe, s->lamA, 0.5, nullptr, s->lamB);
      if (rc) break;
      // stage 1: U* = U^n + dt L(U^n):  lambda^n = lambda_* dU*/dU^n + 1/2 lambda^{n+1}, in place
      rc = stage_vjp(h, s, Un, s->dUs + (2 * i) * fe, s->lamB, 1.0, s->lamA, s->lamA);
    }
    sum_share_kernel<<<XI_BLOCKS, 256, 0, st>>>(s->xi_part, parts, s->dxi + 1);
    sum_parts_kernel<<<1, 256, 0, st>>>(s->dxi + 1, XI_BLOCKS, s->dxi, 0);
    from_padded_kernel<<<blocks_for(g.ncells), 128, 0, st>>>(s->lamA, lam, g, nv);
    rc = rc ? rc : launch_err("adjoint transfer");
  }
  double dx = 0.0;
  if (rc == RSST_OK) {
    if (cudaMemcpyAsync(h->h_small, s->dxi, sizeof(double), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess) {
      rsst_set_error("rsst_adjoint_step: read-back failed");
      rc = RSST_ECUDA;
    } else {
      dx = h->h_small[0];
    }
  } else {
    cudaStreamSynchronize(st);
  }
  if (rc == RSST_OK) *dJ_dxi += dx;
  return rc;
}

extern "C" int rsst_kinetic_energy(rsst_handle* h, double* J, double* grad) {
  if (!h || !J) { rsst_set_error("rsst_kinetic_energy: NULL argument"); return RSST_EINVAL; }
  if (grad && rsst_check_buffer(grad, 0, "rsst_kinetic_energy (grad)") != RSST_OK) return RSST_EINVAL;
  if (h->cfg.precision != RSST_FP64) { rsst_set_error("rsst_kinetic_energy: float64 runs only"); return RSST_EUNSUPPORTED; }
  const Geom& g = h->g;
  const int nb = blocks_for(g.ncells);
  if (nb > 1024 * 64) { rsst_set_error("rsst_kinetic_energy: grid too large"); return RSST_EINVAL; }
  double* part = nullptr;
  if (cudaMalloc((void**)&part, (nb + 1) * sizeof(double)) != cudaSuccess) {
    cudaGetLastError();
    rsst_set_error("rsst_kinetic_energy: allocation failed");
    return RSST_ENOMEM;
  }
  double vol = 1.0;
  for (int d = 0; d < g.ndim; ++d) vol *= h->cfg.dx[d];
  switch (g.ndim + 2) {
    case 3: ke_kernel<3><<<nb, 128, 0, h->stream>>>((const double*)h->buf[0], g, vol, part, grad); break;
    case 4: ke_kernel<4><<<nb, 128, 0, h->stream>>>((const double*)h->buf[0], g, vol, part, grad); break;
    default: ke_kernel<5><<<nb, 128, 0, h->stream>>>((const double*)h->buf[0], g, vol, part, grad); break;
  }
  sum_parts_kernel<<<1, 256, 0, h->stream>>>(part, nb, part + nb, 0);
  int rc = launch_err("kinetic energy");
  if (rc == RSST_OK) {
    if (cudaMemcpyAsync(h->h_small, part + nb, sizeof(double), cudaMemcpyDeviceToHost, h->stream) != cudaSuccess ||
        cudaStreamSynchronize(h->stream) != cudaSuccess) {
      rsst_set_error("rsst_kinetic_energy: read-back failed");
      rc = RSST_ECUDA;
    } else {
      *J = h->h_small[0];
    }
  }
  cudaFree(part);
  h->launches += 2;
  return rc;
}

namespace rsst {

// dJ/drho at fixed V and P from dJ/dU (ideal gas, (de/drho)_P = 0):
// lam_rho + V . lam_m + |V|^2/2 lam_E, cell by cell; caller layout, planes of
// `cells` values.
template <int NV>
__global__ void rho_fixed_vp_kernel(const double* __restrict__ U, const double* __restrict__ lam,
                                    double* __restrict__ out, int64_t cells) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < cells; i += (int64_t)gridDim.x * blockDim.x) {
    const double rho = U[i];
    double acc = lam[i], v2 = 0.0;
#pragma unroll
    for (int d = 0; d < NV - 2; ++d) {
      const double v = U[(1 + d) * cells + i] / rho;
      acc = fma(v, lam[(1 + d) * cells + i], acc);
      v2 = fma(v, v, v2);
    }
    out[i] = fma(0.5 * v2, lam[(NV - 1) * cells + i], acc);
  }
}

}  // namespace rsst

extern "C" int rsst_adjoint_rho_fixed_vp(const double* U, const double* lam, double* out, int32_t ndim,
                                         const int32_t* n, void* stream) {
  if (!U || !lam || !out || !n || ndim < 1 || ndim > 3) {
    rsst_set_error("rsst_adjoint_rho_fixed_vp: NULL pointer or ndim outside 1..3");
    return RSST_EINVAL;
  }
  int64_t cells = 1;
  for (int d = 0; d < ndim; ++d) {
    if (n[d] < 1) { rsst_set_error("rsst_adjoint_rho_fixed_vp: n[%d] < 1", d); return RSST_EINVAL; }
    cells *= n[d];
  }
  if (cells > (int64_t)1 << 31) { rsst_set_error("rsst_adjoint_rho_fixed_vp: grid too large"); return RSST_EINVAL; }
  if (rsst_check_buffer(U, 0, "rsst_adjoint_rho_fixed_vp (U)") != RSST_OK ||
      rsst_check_buffer(lam, 0, "rsst_adjoint_rho_fixed_vp (lam)") != RSST_OK ||
      rsst_check_buffer(out, 0, "rsst_adjoint_rho_fixed_vp (out)") != RSST_OK)
    return RSST_EINVAL;
  const int64_t want = (cells + 255) / 256;
  const int grid = (int)(want < 152 * 8 ? want : 152 * 8);
  cudaStream_t st = (cudaStream_t)stream;
  switch (ndim) {
    case 1: rsst::rho_fixed_vp_kernel<3><<<grid, 256, 0, st>>>(U, lam, out, cells); break;
    case 2: rsst::rho_fixed_vp_kernel<4><<<grid, 256, 0, st>>>(U, lam, out, cells); break;
    default: rsst::rho_fixed_vp_kernel<5><<<grid, 256, 0, st>>>(U, lam, out, cells); break;
  }
  return launch_err("rsst_adjoint_rho_fixed_vp");
}
