// Float32-pipe part of rsst_math_eval (rsst_selftest.cu), compiled with the
// flags of the kernels that hold these helpers.
#include "rsst_fp32_pair.cuh"
#include "rsst_internal.h"
#include "rsst_math_df.cuh"

namespace rsst {

__global__ void eval_fp32_kernel(int fn, int64_t n, const double* __restrict__ in, double* __restrict__ out,
                                 const PhysF pf, const PhysDF pd) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  auto x = [&](int k) { return in[k * n + i]; };
  if (fn == RSST_EVAL_DF_FLUX) {
    // gas at rest left and right: the mass flux is the dissipation alone
    const df qL[3] = {df_from(x(0)), df_make(0.0f), df_from(x(2))}, qR[3] = {df_from(x(1)), df_make(0.0f), df_from(x(2))};
    df G[3];
    llf_flux_x2_df<3, 0, false>(qL, qR, pd, G);
    out[i] = df_to(G[0]);
  } else if (fn == RSST_EVAL_PAIR_TENDENCY) {
    // f (gamma - 1) = 1 and PD on L_E = 0 leave minus the pressure tendency
    const f2 z = dup2(0.0f), one = dup2(1.0f);
    const f2 q[4] = {dup2((float)x(0)), dup2((float)x(1)), dup2((float)x(2)), one};
    const f2 D[4] = {dup2((float)x(3)), dup2((float)x(4)), dup2((float)x(5)), dup2((float)x(6))};
    const f2 b[4] = {z, z, z, z};
    f2 L[4] = {z, z, z, z}, u[4], rate;
    bool ok[2];
    cell_lean2<4, RSST_PD, false, 1>(q, L, D, z, z, pf, make_pf2(pf), RSST_PD, false, z, b, u, rate, ok);
    out[i] = -(double)lo2(L[3]);
  } else {  // RSST_EVAL_PAIR_DC: c_tot - c0 of a state at rest about (rho0, P0)
    const float r0 = (float)x(2), P0 = (float)x(3), c0 = sqrtf(pf.gx * P0 / r0);
    const f2 q[4] = {dup2((float)x(0)), dup2(0.0f), dup2(0.0f), dup2((float)x(1))};
    f2 F[4], c, dc;
    flux_lean2<4, 1, true, true, false>(q, dup2(r0), dup2(P0), dup2(pf.gx * P0), dup2(0.0f), dup2(c0), dup2(pf.gx / r0),
                                        dup2(c0), make_pf2(pf), F, c, dc);
    out[i] = lo2(dc);
  }
}

}  // namespace rsst

void rsst_launch_eval_fp32(int fn, int64_t n, const double* in, double* out) {
  PhysF pf = {};
  pf.gamma = 2.0f;  // gamma - 1 = 1: the pressure of a state at rest is its energy
  pf.gm1 = pf.inv_gm1 = pf.f = 1.0f;
  pf.hgm1 = 0.5f;
  pf.gam_gm1 = 2.0f;
  pf.gx = 1.0f;
  rsst::PhysDF pd = {};
  pd.gm1 = pd.inv_gm1 = pd.gx = {1.0f, 0.0f};
  pd.xs = 1.0f;
  pd.nhgm1 = {-0.5f, 0.0f};
  rsst::eval_fp32_kernel<<<(unsigned)((n + 255) / 256), 256>>>(fn, n, in, out, pf, pd);
}
