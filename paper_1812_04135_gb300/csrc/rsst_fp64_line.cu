// Float64 steps of a short 1D line: many steps in one launch, the whole line on
// one thread-block cluster.
//
// What bounds a short line is not work but latency: with a launch per stage
// (rsst_fp64.cu) a 256-cell line took 7.3 us a stage, most of it one warp's
// chain of float64 instructions (a warp issues one per 64 SM clocks, however
// few lanes it has active and however independent they are) behind a launch, a
// reload of the state and a dt division.  Here up to 16 CTAs of a cluster each
// keep T cells in shared memory for all steps and exchange halo cells and CFL
// maxima through distributed shared memory, and each CTA spreads a stage over
// warps on different schedulers:
//   A. warps by side: the left (right) state of each face, its flux and c_tot;
//      further warps: what the reduced tendency needs of each cell's state
//      alone, and before stage 1 the state's CFL rate and physical check;
//   B. a lane per face and field: the LLF flux; one warp: dt, once the CFL
//      maxima of all CTAs are in;
//   C. a lane per cell: divergence, reduced tendency, RK combine, and the new
//      value to every CTA whose window holds it (neighbours' halos and the
//      ghosts it is the image of).
// The arithmetic is that of the stage kernel.  Measured a stage (us, a launch
// per stage -> here): 256 cells 7.25 -> 3.33, 1024 7.3 -> 4.0, 2048 7.3 -> 5.3;
// at 256 cells a stage's 6100 SM clocks are A 2600, B 750, C 1800, the cluster
// barrier 500.
#include <cooperative_groups.h>

#include "rsst_attr.h"
#include "rsst_common.cuh"
#include "rsst_internal.h"
#include "rsst_math_fp64.cuh"

namespace rsst {

namespace cg = cooperative_groups;

constexpr int LINE_CTAS = 16;       // cluster size (16 needs the non-portable opt-in)
constexpr int LINE_LEAST = 16;        // cells a CTA takes at least
constexpr int LINE_MOST = 128;      // and at most (4096 cells would take as long as a launch per stage)
constexpr int LINE_STEPS = 1024;    // steps a launch takes at most (bounds its run time to a few ms)

struct LineCfg {
  int T, ctas, wf, wc;  // cells a CTA; CTAs; warps per face side; warps of cells
  int threads() const { return 32 * (2 * wf + wc); }
  size_t smem() const {
    return sizeof(double) * ((size_t)6 * (T + 4) + (size_t)17 * (T + 1) + (size_t)5 * T + LINE_CTAS * 4 + 2);
  }
};
static LineCfg line_cfg(int n) {
  LineCfg c;
  c.T = (n + LINE_CTAS - 1) / LINE_CTAS;
  if (c.T < LINE_LEAST) c.T = LINE_LEAST;
  c.ctas = (n + c.T - 1) / c.T;
  c.wf = (c.T + 1 + 31) / 32;
  c.wc = (c.T + 31) / 32;
  return c;
}

template <bool CV>
__global__ void __launch_bounds__(448, 1) line_fp64_kernel(const StageArgs<double> a, int nsteps, int T, int wf,
                                                           int wc) {
  constexpr int NV = 3;
  extern __shared__ __align__(16) double sm[];
  cg::cluster_group cl = cg::this_cluster();
  const Geom& g = a.g;
  const Phys& p = a.p;
  const int n = g.n[0], rank = (int)cl.block_rank(), ctas = (int)cl.num_blocks();
  const int i0 = rank * T, cnt = min(T, n - i0);
  const int W = T + 4, F = T + 1;
  double* su = sm;              // [2][NV][W]: U^n and U* with two halo cells at each end
  double* sq = su + 2 * NV * W; // [2][NV][F]: face states, left and right
  double* sF = sq + 2 * NV * F; // [2][NV][F]: their fluxes
  double* sG = sF + 2 * NV * F; // [NV][F]: twice the LLF flux
  float2* sc = reinterpret_cast<float2*>(sG + NV * F);  // [2][F]: c_tot
  double* sp = sG + NV * F + 2 * F;                     // [5][T]: RhsPrep of each cell
  double* red = sp + 5 * T;                             // [ctas][4]: CFL maxima of all CTAs' cell warps
  double* sdt = red + LINE_CTAS * 4;                    // dt, simulated time
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool cellwarp = warp >= 2 * wf;
  const int cw = warp - 2 * wf;

  for (int id = tid; id < NV * (cnt + 4); id += blockDim.x) {
    const int v = id / (cnt + 4), x = id - v * (cnt + 4);
    su[v * W + x] = a.in[v * g.fstride + pidx(g, i0 + x - 2, 0, 0)];
  }
  if (tid == 0) {
    sdt[0] = a.dt_fixed > 0.0 ? a.dt_fixed : p.cfl / a.scal[a.slot];
    sdt[1] = a.scal[3] + sdt[0];
  }
  // CFL rate and physical check of the state in buffer 0 (cell warps): the
  // warp's maximum goes to every CTA
  bool bad = false;
  auto rates = [&]() {
    const int c = cw * 32 + lane;
    double r = 0.0;
    if (c < cnt) {
      double q[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) q[v] = su[v * W + c + 2];
      bool ok;
      const double x = cfl_rate<NV, CV>(q, p, ok);
      if (ok) r = x;
      bad = bad || !ok;
    }
    r = warp_max(r);
    if (lane < ctas) cl.map_shared_rank(red, lane)[rank * 4 + cw] = r;
  };
  auto rate_max = [&]() {  // by one whole warp, after a cluster barrier
    double r = 0.0;
    for (int i = lane; i < ctas * wc; i += 32) r = max_nonneg(r, red[i / wc * 4 + i % wc]);
    return warp_max(r);
  };
  // Where my cell's new value goes, fixed for the launch: the windows (other
  // than my own) that hold extended cell gx, at most two of them as neighbours
  // are at least LINE_LEAST cells wide
  auto window = [&](int gx, int skip, int which) -> double* {
    const int r0 = (gx + T) / T - 1;  // floor(gx / T) for gx >= -T
    int found = 0;
    for (int r = max(r0 - 1, 0); r <= min(r0 + 1, ctas - 1); ++r) {
      const int x = gx - r * T;
      if (r == skip || x < -2 || x > min(T, n - r * T) + 1) continue;
      if (found++ == which) return cl.map_shared_rank(su, r) + x + 2;
    }
    return nullptr;
  };
  const bool mine = tid < cnt;  // phase C: a lane per cell, in the first wc warps
  const int gi = i0 + tid;
  double* nb[2] = {nullptr, nullptr};                             // neighbours' halos
  double* gh[2][2] = {{nullptr, nullptr}, {nullptr, nullptr}};    // ghosts I am the image of, by end
  double gsign = 1.0, gd[2][2] = {{0.0, 0.0}, {0.0, 0.0}};        // their momentum sign and background difference
  if (mine) {
#pragma unroll
    for (int k = 0; k < 2; ++k) nb[k] = window(gi, rank, k);
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      if (side == 0 ? gi >= RSST_G : gi < n - RSST_G) continue;
      int gx;
      if (p.bc[0] == RSST_BC_PERIODIC) {
        gx = side == 0 ? gi + n : gi - n;
      } else {
        gx = side == 0 ? -1 - gi : 2 * n - 1 - gi;
        gsign = -1.0;
        if (a.bg != nullptr && p.vertical == 0) {
          gd[side][0] = a.bg[gx + RSST_G] - a.bg[gi + RSST_G];
          gd[side][1] = a.bg[a.bg_len + gx + RSST_G] - a.bg[a.bg_len + gi + RSST_G];
        }
      }
#pragma unroll
      for (int k = 0; k < 2; ++k) gh[side][k] = window(gx, -1, k);
    }
  }
  const bool edge = gh[0][0] != nullptr || gh[1][0] != nullptr;
  auto put = [&](int off, const double (&u)[NV]) {
    double* own = su + off + tid + 2;
#pragma unroll
    for (int v = 0; v < NV; ++v) own[v * W] = u[v];
#pragma unroll
    for (int k = 0; k < 2; ++k)
      if (nb[k]) {
#pragma unroll
        for (int v = 0; v < NV; ++v) nb[k][off + v * W] = u[v];
      }
    if (edge) {
#pragma unroll
      for (int side = 0; side < 2; ++side)
#pragma unroll
        for (int k = 0; k < 2; ++k)
          if (double* d = gh[side][k]) {
            d[off] = u[0] + gd[side][0];
            d[off + W] = gsign < 0.0 ? -u[1] : u[1];
            d[off + 2 * W] = u[2] + gd[side][1];
          }
    }
  };
  cl.sync();  // every CTA of the cluster runs; windows are loaded

  double q0[NV] = {0.0, 0.0, 0.0};  // my cell's U^n (phase C lanes)
  for (int s = 0; s < nsteps; ++s) {
#pragma unroll 1
    for (int st = 1; st <= 2; ++st) {
      const double* u = su + (st - 1) * NV * W;
      const bool newdt = st == 1 && s > 0;  // the first step's maximum came with the state
      // A
      if (!cellwarp) {
        const int side = warp >= wf ? 1 : 0, f = (warp - side * wf) * 32 + lane;
        if (f <= cnt) {
          const double* c = u + f + 1 + side;  // the cell left (right) of face f: local f - 1 + side
          const double h = side ? -0.5 : 0.5;
          double q[NV], Fq[NV];
#pragma unroll
          for (int v = 0; v < NV; ++v) {
            const double um = c[v * W - 1], u0 = c[v * W], up = c[v * W + 1];
            q[v] = fma(h, mc_slope(u0 - um, up - u0), u0);
          }
          float ch, cll;
          euler_flux<NV, 0, CV>(q, p, Fq, ch, cll);
#pragma unroll
          for (int v = 0; v < NV; ++v) {
            sq[(side * NV + v) * F + f] = q[v];
            sF[(side * NV + v) * F + f] = Fq[v];
          }
          sc[side * F + f] = make_float2(ch, cll);
        }
      } else {
        if (newdt) rates();
        const int c = cw * 32 + lane;
        if (c < cnt && p.variant != RSST_EULER) {
          double q[NV];
#pragma unroll
          for (int v = 0; v < NV; ++v) q[v] = u[v * W + c + 2];
          RhsPrep<NV> r;
          rhs_prep<NV, CV>(q, p, r);
          sp[c] = r.v[0];
          sp[T + c] = r.hv2;
          sp[2 * T + c] = r.H;
          sp[3 * T + c] = r.a;
          sp[4 * T + c] = r.b;
        }
      }
      __syncthreads();
      // the CFL maxima travel while B and the first half of C run; dt is formed
      // by a cell warp beside them and first needed by the RK combine
      if (newdt) cl.barrier_arrive();
      // B
      if (!cellwarp) {
        for (int id = tid; id < NV * (cnt + 1); id += 64 * wf) {
          const int v = id / (cnt + 1), f = id - v * (cnt + 1);
          const float2 cL = sc[f], cR = sc[F + f];
          const bool left = cL.x > cR.x || (cL.x == cR.x && cL.y >= cR.y);
          const double alpha = pair_to_double(left ? cL.x : cR.x, left ? cL.y : cR.y);
          sG[v * F + f] = fma(-alpha, sq[(NV + v) * F + f] - sq[v * F + f], sF[v * F + f] + sF[(NV + v) * F + f]);
        }
        asm volatile("bar.sync 1, %0;" ::"r"(64 * wf) : "memory");  // the face warps, which also take C
      } else if (newdt) {
        cl.barrier_wait();
        if (cw == 0) {
          const double m = rate_max();
          if (lane == 0) {
            const double dt = a.dt_fixed > 0.0 ? a.dt_fixed : p.cfl / m;
            sdt[0] = dt;
            sdt[1] += dt;
          }
        }
      }
      // C
      double q[NV], L[NV];
      if (mine) {
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          q[v] = u[v * W + tid + 2];
          L[v] = -(sG[v * F + tid + 1] - sG[v * F + tid]) * p.half_inv_dx[0];
        }
        RhsPrep<NV> r = {};
        if (p.variant != RSST_EULER) {
          r.v[0] = sp[tid];
          r.hv2 = sp[T + tid];
          r.H = sp[2 * T + tid];
          r.a = sp[3 * T + tid];
          r.b = sp[4 * T + tid];
        }
        rhs_apply<NV>(q, L, p, r);
      }
      __syncwarp();
      if (newdt) {
        if (!cellwarp) cl.barrier_wait();
        __syncthreads();
      }
      if (mine) {
        const double dt = sdt[0];
        double un[NV];
        if (st == 1) {
#pragma unroll
          for (int v = 0; v < NV; ++v) {
            q0[v] = q[v];
            un[v] = fma(dt, L[v], q[v]);
          }
          put(NV * W, un);
        } else {
#pragma unroll
          for (int v = 0; v < NV; ++v) un[v] = half_of(q0[v] + fma(dt, L[v], q[v]));
          put(0, un);
        }
      }
      __syncwarp();
      cl.sync();
    }
  }
  // the final state's CFL maximum, time and state
  if (cellwarp) rates();
  if (bad) atomicOr(a.flag, RSST_FLAG_NONPHYSICAL);
  cl.sync();
  if (rank == 0 && cellwarp && cw == 0) {
    const double m = rate_max();
    if (lane == 0) {
      a.scal[a.slot ^ (nsteps & 1)] = m;
      a.scal[2] = sdt[0];
      a.scal[3] = sdt[1];
    }
  }
  if (mine) {
    double u[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) u[v] = su[v * W + tid + 2];
    store_with_ghosts<NV>(a.out, g, p, a.bg, a.bg_len, gi, 0, 0, u);
  }
}

static int set_line_attrs(void (*kern)(const StageArgs<double>, int, int, int, int), std::atomic<unsigned long long>& done) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return RSST_ECUDA;
  const unsigned long long bit = dev < 64 ? 1ull << dev : 0ull;
  if (bit && (done.load(std::memory_order_acquire) & bit)) return RSST_OK;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
    cudaGetLastError();
    return RSST_ECUDA;
  }
  if (bit) done.fetch_or(bit, std::memory_order_acq_rel);
  return RSST_OK;
}

static void line_launch_config(const LineCfg& c, cudaStream_t s, cudaLaunchConfig_t* lc, cudaLaunchAttribute* at) {
  *lc = {};
  lc->gridDim = dim3(c.ctas);
  lc->blockDim = dim3(c.threads());
  lc->dynamicSmemBytes = c.smem();
  lc->stream = s;
  at->id = cudaLaunchAttributeClusterDimension;
  at->val.clusterDim.x = c.ctas;
  at->val.clusterDim.y = 1;
  at->val.clusterDim.z = 1;
  lc->attrs = at;
  lc->numAttrs = 1;
}

}  // namespace rsst

using namespace rsst;

// Whether a 1D float64 line runs on the cluster kernel: lines of up to 16 x 128
// cells, on a device that can hold such a cluster.
int rsst_line_fp64_ok(const Geom& g, const Phys& p) {
  if (g.ndim != 1 || g.n[0] > LINE_CTAS * LINE_MOST) return 0;
  static std::atomic<unsigned long long> attr[2];
  auto kern = p.covol != 0.0 ? line_fp64_kernel<true> : line_fp64_kernel<false>;
  if (set_line_attrs(kern, attr[p.covol != 0.0]) != RSST_OK) return 0;
  cudaLaunchConfig_t lc;
  cudaLaunchAttribute at[1];
  line_launch_config(line_cfg(g.n[0]), nullptr, &lc, at);
  int clusters = 0;
  if (cudaOccupancyMaxActiveClusters(&clusters, kern, &lc) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return clusters >= 1;
}

// nsteps steps of a line (a.in = a.out: U^n in place); returns the launches in *launches.
int rsst_launch_line_fp64(const StageArgs<double>& a0, int nsteps, int* launches, cudaStream_t s) {
  const LineCfg c = line_cfg(a0.g.n[0]);
  StageArgs<double> a = a0;
  *launches = 0;
  while (nsteps > 0) {
    const int k = nsteps < LINE_STEPS ? nsteps : LINE_STEPS;
    cudaLaunchConfig_t lc;
    cudaLaunchAttribute at[1];
    line_launch_config(c, s, &lc, at);
    const cudaError_t e = a.p.covol != 0.0 ? cudaLaunchKernelEx(&lc, line_fp64_kernel<true>, a, k, c.T, c.wf, c.wc)
                                           : cudaLaunchKernelEx(&lc, line_fp64_kernel<false>, a, k, c.T, c.wf, c.wc);
    if (e != cudaSuccess) {
      cudaGetLastError();
      rsst_set_error("float64 line kernel launch: %s", cudaGetErrorString(e));
      return RSST_ECUDA;
    }
    ++*launches;
    a.slot ^= k & 1;
    nsteps -= k;
  }
  return RSST_OK;
}
