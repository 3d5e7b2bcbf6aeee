// Double-float kernels (precision RSST_FP64_DF): the state is stored as
// float32 pairs (hi, lo) in the padded layout (8 bytes per value, like
// float64) and the fused stage kernel computes in double-float on the
// float32 pipe.  Tile structure as in the float64 kernel (rsst_fp64.cu): the
// halo tile by one TMA copy in 2D and 3D, 1D/2D tiles with every axis at once,
// 3D tiles axis by axis.
//
// What bounds it: instruction issue and the float32 pipe (a double-float
// operation is 7 to 15 float32 instructions).  Thread instructions a 2D cell
// in stage 1 (ncu, 512^2): 4100 -> 2785, by products fed unnormalised into
// sums (df_fma, the three-term sum of the LLF flux), twice-flux faces, slopes
// in pairs that share a difference, rho |V|^2 = m.V, the C_max law and the
// stage as template arguments, and the tile by TMA instead of loads and index
// arithmetic.  512^2: 40.9 -> 27.4 us a stage; 3D 90 x 70 x 50: 112 -> 74 us.
#include <climits>
#include <cmath>

#include "rsst_common.cuh"
#include "rsst_internal.h"
#include "rsst_attr.h"
#include "rsst_math_df.cuh"
#include "rsst_tma.cuh"
#include "rsst_transfer.cuh"

namespace rsst {

__device__ __forceinline__ df ld_df(const float2* p, int64_t i) {
  const float2 v = p[i];
  return {v.x, v.y};
}
__device__ __forceinline__ void st_df(float2* p, int64_t i, df v) { p[i] = make_float2(v.hi, v.lo); }

// Store a cell and the edge ghosts it is the image of (wrap, or mirror with
// the normal momentum negated and the background difference added).
template <int NV>
__device__ __forceinline__ void store_ghosts_df(float2* __restrict__ out, const Geom& g, const Phys& p,
                                                const double* __restrict__ bg, int bg_len, int i, int j, int k,
                                                const df (&u)[NV]) {
  constexpr int ND = NV - 2;
  const int64_t fs = g.fstride;
  const int64_t o = pidx(g, i, j, k);
#pragma unroll
  for (int v = 0; v < NV; ++v) st_df(out, v * fs + o, u[v]);
  const int c[3] = {i, j, k};
#pragma unroll
  for (int d = 0; d < ND; ++d) {
    const int n = g.n[d], cd = c[d];
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      const bool hit = side == 0 ? (cd < RSST_G) : (cd >= n - RSST_G);
      if (!hit) continue;
      df w[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) w[v] = u[v];
      int gp;
      if (p.bc[d] == RSST_BC_PERIODIC) {
        gp = side == 0 ? cd + n : cd - n;
      } else {
        gp = side == 0 ? -1 - cd : 2 * n - 1 - cd;
        w[1 + d] = -w[1 + d];
        if (bg != nullptr && d == p.vertical) {
          w[0] = w[0] + df_from(bg[gp + RSST_G] - bg[cd + RSST_G]);
          w[NV - 1] = w[NV - 1] + df_from(bg[bg_len + gp + RSST_G] - bg[bg_len + cd + RSST_G]);
        }
      }
      const int ii = d == 0 ? gp : i, jj = d == 1 ? gp : j, kk = d == 2 ? gp : k;
      const int64_t og = pidx(g, ii, jj, kk);
#pragma unroll
      for (int v = 0; v < NV; ++v) st_df(out, v * fs + og, w[v]);
    }
  }
}

__device__ __forceinline__ df warp_max_df(df x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const df y = {__shfl_xor_sync(0xffffffffu, x.hi, o), __shfl_xor_sync(0xffffffffu, x.lo, o)};
    if (df_lt(x, y)) x = y;
  }
  return x;
}

// Block maximum of non-negative double-floats, one float64 atomicMax.
template <int NT>
__device__ __forceinline__ void block_max_df(df x, double* dst, df* sred) {
  x = warp_max_df(x);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) sred[wid] = x;
  __syncthreads();
  if (wid == 0) {
    df y = lane < NT / 32 ? sred[lane] : df_make(0.0f);
    y = warp_max_df(y);
    if (lane == 0 && df_pos(y))
      atomicMax(reinterpret_cast<unsigned long long*>(dst), (unsigned long long)__double_as_longlong(df_to(y)));
  }
}

// Tile structure of the float64 kernel (rsst_fp64.cu): 1D/2D tiles hold the
// half slopes and faces of every axis at once, 3D tiles go axis by axis.
template <int NDIM, int BX, int BY, int BZ, int NT>
struct TileCfgDF {
  static constexpr int NV = NDIM + 2;
  static constexpr int HX = 2, HY = NDIM >= 2 ? 2 : 0, HZ = NDIM >= 3 ? 2 : 0;
  static constexpr int SX = BX + 2 * HX, SY = BY + 2 * HY, SZ = BZ + 2 * HZ;
  static constexpr int SCELLS = SX * SY * SZ;
  static constexpr int NCELL = BX * BY * BZ;
  static constexpr int CPT = (NCELL + NT - 1) / NT;
  static constexpr int F0 = (BX + 1) * BY * BZ, F1 = NDIM >= 2 ? BX * (BY + 1) * BZ : 0;
  static constexpr int F2 = NDIM >= 3 ? BX * BY * (BZ + 1) : 0;
  static constexpr int E0 = (BX + 2) * BY * BZ, E1 = NDIM >= 2 ? BX * (BY + 2) * BZ : 0;
  static constexpr int E2 = NDIM >= 3 ? BX * BY * (BZ + 2) : 0;
  static constexpr int max3(int a, int b, int c) { return a > b ? (a > c ? a : c) : (b > c ? b : c); }
  static constexpr bool ALL = NDIM <= 2;
  static constexpr int FMAX = ALL ? F0 + F1 : max3(F0, F1, F2);
  static constexpr int EMAX = ALL ? E0 + E1 : max3(E0, E1, E2);
  // halo tile, faces, half slopes, the block reduction and dt (64 values), two mbarriers (the tile copy; the
  // failure-detection test wait)
  static constexpr size_t SMEM = sizeof(df) * ((size_t)NV * (SCELLS + FMAX + EMAX) + 64) + 16;
  static constexpr uint32_t TILE_BYTES = (uint32_t)(sizeof(df) * NV * SCELLS);
  static_assert(BX % 2 == 0 && (NDIM < 2 || BY % 2 == 0) && (NDIM < 3 || BZ % 2 == 0), "slopes are taken in pairs");
};

// Half MC slopes along D of the pair of neighbouring slope cells e (tile
// coordinates -1 .. B along D, 0 .. B-1 across); the two share a difference.
template <class C, int BX, int BY, int BZ, int D>
__device__ __forceinline__ void slope_pair_df(const df* __restrict__ su, df* __restrict__ ss, int e) {
  constexpr int STRIDE = D == 0 ? 1 : (D == 1 ? C::SX : C::SX * C::SY);
  constexpr int XX = BX + 2 * (D == 0), YY = BY + 2 * (D == 1);
  constexpr int PX = D == 0 ? XX / 2 : XX, PY = D == 1 ? YY / 2 : YY;
  const int ex = e % PX * (D == 0 ? 2 : 1);
  const int t = e / PX;
  const int ey = t % PY * (D == 1 ? 2 : 1);
  const int ez = t / PY * (D == 2 ? 2 : 1);
  const int s0 = (ez - (D == 2) + C::HZ) * C::SX * C::SY + (ey - (D == 1) + C::HY) * C::SX + (ex - (D == 0) + C::HX);
  const int o = (ez * YY + ey) * XX + ex;
  constexpr int STRIDE_E = D == 0 ? 1 : (D == 1 ? XX : XX * YY);
#pragma unroll
  for (int v = 0; v < C::NV; ++v) {
    const df* sv = su + v * C::SCELLS + s0;
    const df um = sv[-STRIDE], u0 = sv[0], u1 = sv[STRIDE], up = sv[2 * STRIDE];
    const df d = u1 - u0;
    ss[v * C::EMAX + o] = half_mc_df(u0 - um, d);
    ss[v * C::EMAX + o + STRIDE_E] = half_mc_df(d, up - u1);
  }
}

// Twice the LLF flux of the face between tile cells sl | s0 (slopes el, er);
// fld lists the fields with the normal momentum second.
template <class C, bool CMAX, int D>
__device__ __forceinline__ void face_df(const df* __restrict__ su, const df* __restrict__ ss, df* __restrict__ sf,
                                        const PhysDF& p, int sl, int s0, int el, int er, int f,
                                        const int (&fld)[C::NV]) {
  constexpr int NV = C::NV;
  df qL[NV], qR[NV], F[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    qL[v] = su[fld[v] * C::SCELLS + sl] + ss[fld[v] * C::EMAX + el];
    qR[v] = su[fld[v] * C::SCELLS + s0] - ss[fld[v] * C::EMAX + er];
  }
  llf_flux_x2_df<NV, D, CMAX>(qL, qR, p, F);
#pragma unroll
  for (int v = 0; v < NV; ++v) sf[fld[v] * C::FMAX + f] = F[v];
}

// 2F above minus 2F below tile cell (cx, cy, cz) along D, per field.
template <class C, int BX, int BY, int BZ, int D>
__device__ __forceinline__ void face_diff_df(const df* __restrict__ sf, int cx, int cy, int cz, df (&d)[C::NV]) {
  constexpr int EX = BX + (D == 0), EY = BY + (D == 1);
  const int flo = (cz * EY + cy) * EX + cx;
  const int fhi = flo + (D == 0 ? 1 : (D == 1 ? EX : EX * EY));
#pragma unroll
  for (int v = 0; v < C::NV; ++v) d[v] = sf[v * C::FMAX + fhi] - sf[v * C::FMAX + flo];
}

// One axis of a 3D tile: slopes, faces, and each thread's cells' divergence.
template <int NDIM, int BX, int BY, int BZ, int NT, int D, bool CMAX>
__device__ __forceinline__ void axis_pass_df(const df* __restrict__ su, df* __restrict__ sf, df* __restrict__ ss,
                                             const PhysDF& p, const Geom& g, int i0, int j0, int k0,
                                             df (&dU)[TileCfgDF<NDIM, BX, BY, BZ, NT>::CPT][NDIM + 2]) {
  using C = TileCfgDF<NDIM, BX, BY, BZ, NT>;
  constexpr int NE = D == 0 ? C::E0 : (D == 1 ? C::E1 : C::E2), NF = D == 0 ? C::F0 : (D == 1 ? C::F1 : C::F2);
  constexpr int EX = BX + (D == 0), EY = BY + (D == 1);
  constexpr int STRIDE = D == 0 ? 1 : (D == 1 ? C::SX : C::SX * C::SY);
  constexpr int XX = BX + 2 * (D == 0), YY = BY + 2 * (D == 1);
  constexpr int STRIDE_E = D == 0 ? 1 : (D == 1 ? XX : XX * YY);
  constexpr int fld[5] = {0, 1, 2, 3, 4};
  for (int e = threadIdx.x; e < NE / 2; e += NT) slope_pair_df<C, BX, BY, BZ, D>(su, ss, e);
  __syncthreads();
  for (int f = threadIdx.x; f < NF; f += NT) {
    const int fx = f % EX, t = f / EX, fy = t % EY, fz = t / EY;
    if (i0 + fx > g.n[0] - (D == 0 ? 0 : 1) || j0 + fy > g.n[1] - (D == 1 ? 0 : 1) ||
        k0 + fz > g.n[2] - (D == 2 ? 0 : 1))
      continue;
    const int s0 = (fz + C::HZ) * C::SX * C::SY + (fy + C::HY) * C::SX + (fx + C::HX);
    const int er = ((fz + (D == 2)) * YY + (fy + (D == 1))) * XX + (fx + (D == 0));
    face_df<C, CMAX, D>(su, ss, sf, p, s0 - STRIDE, s0, er - STRIDE_E, er, f, fld);
  }
  __syncthreads();
#pragma unroll
  for (int c = 0; c < C::CPT; ++c) {
    const int cell = threadIdx.x + c * NT;
    if (cell >= C::NCELL) break;
    df d[C::NV];
    face_diff_df<C, BX, BY, BZ, D>(sf, cell % BX, cell / BX % BY, cell / BX / BY, d);
#pragma unroll
    for (int v = 0; v < C::NV; ++v)
      dU[c][v] = D == 0 ? d[v] * p.nhalf_inv_dx[D] : df_fma(d[v], p.nhalf_inv_dx[D], dU[c][v]);
  }
}

struct DFArgs {
  const float2* in;
  const float2* base;
  float2* out;
  Geom g;
  Phys p;
  PhysDF q;
  const double* bg;
  int bg_len;
  double* scal;
  unsigned int* flag;
  int slot, stage;
  double dt_fixed;
  int64_t stall_ns;  // as in StageArgs
};

template <int NDIM, int BX, int BY, int BZ, int NT, int MINB, bool CMAX, int ST>
__global__ void __launch_bounds__(NT, MINB)
    stage_df_kernel(const __grid_constant__ CUtensorMap tin, const DFArgs a) {
  using C = TileCfgDF<NDIM, BX, BY, BZ, NT>;
  constexpr int NV = C::NV;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  df* su = reinterpret_cast<df*>(smem_raw);
  df* sf = su + NV * C::SCELLS;
  df* ss = sf + NV * C::FMAX;  // half slopes
  df* sred = ss + NV * C::EMAX;
  double* sdt = reinterpret_cast<double*>(sred + 32);
  const Geom& g = a.g;
  const PhysDF& p = a.q;
  const int i0 = blockIdx.x * BX, j0 = blockIdx.y * BY, k0 = blockIdx.z * BZ;
  if (threadIdx.x == 0) {
    const double dt = a.dt_fixed > 0.0 ? a.dt_fixed : a.p.cfl / a.scal[a.slot];
    *sdt = dt;
    if (ST == 1 && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0) {
      a.scal[a.slot ^ 1] = 0.0;
      a.scal[2] = dt;
      a.scal[3] += dt;
    }
  }
  if constexpr (NDIM >= 2) {
    // the halo tile of all fields by one TMA copy (as in rsst_fp64.cu: a
    // double-float is an 8-byte element of the same layout)
    uint64_t* bar = reinterpret_cast<uint64_t*>(sred + 64);
    uint64_t* test_bar = bar + 1;
    const bool stall = a.stall_ns > 0;
    if (threadIdx.x == 32) {
      mbar_init(bar, 1);
      if (stall) mbar_init(test_bar, 1);
      fence_mbar_init();
      fence_proxy_async_smem();
      mbar_expect_tx(bar, C::TILE_BYTES);
      if constexpr (NDIM == 2) tma_load_3d(su, &tin, bar, i0 + g.xoff - C::HX, j0, 0);
      else tma_load_4d(su, &tin, bar, i0 + g.xoff - C::HX, j0, k0, 0);
      if (stall) mbar_expect_tx(test_bar, 16);  // bytes that no copy delivers, waited on while the tile's is in flight
    }
    __syncthreads();  // the barriers are initialised, dt is there
    const bool landed = mbar_wait_bounded(stall ? test_bar : bar, 0u, stall ? (uint64_t)a.stall_ns : RSST_WAIT_NS);
    // giving up (flag, one more bounded wait for the copy) is decided by the whole block
    if (__syncthreads_or(!landed)) {
      if (threadIdx.x == 0) {
        atomicOr(a.flag, RSST_FLAG_TIMEOUT);
        mbar_wait_bounded(bar, 0u);
      }
      return;
    }
  } else {
    for (int id = threadIdx.x; id < NV * C::SCELLS; id += NT) {
      const int v = id / C::SCELLS, lx = id - v * C::SCELLS;
      const int gi = i0 + lx - C::HX;
      su[id] = gi <= g.n[0] + 1 ? ld_df(a.in, v * g.fstride + pidx(g, gi, 0, 0)) : df{0.0f, 0.0f};
    }
    __syncthreads();
  }
  const df dt = df_from(*sdt);

  df dU[C::CPT][NV];
  if constexpr (C::ALL) {
    constexpr int PE = (C::E0 / 2 + 31) / 32 * 32;  // axis y starts at a whole warp
    for (int e = threadIdx.x; e < (NDIM == 1 ? C::E0 / 2 : PE + C::E1 / 2); e += NT) {
      if (e < PE) {
        if (e < C::E0 / 2) slope_pair_df<C, BX, BY, BZ, 0>(su, ss, e);
      } else if constexpr (NDIM == 2) {
        slope_pair_df<C, BX, BY, BZ, 1>(su, ss + C::E0, e - PE);
      }
    }
    __syncthreads();
    // the x and y faces as one list; the axis enters through strides and the
    // order of the momenta only (no divergence in a warp that holds both)
    for (int f = threadIdx.x; f < C::F0 + C::F1; f += NT) {
      const bool isy = NDIM == 2 && f >= C::F0;
      const int fid = isy ? f - C::F0 : f;
      const int fy = isy ? fid / BX : fid / (BX + 1);
      const int fx = fid - fy * (isy ? BX : BX + 1);
      if (i0 + fx > g.n[0] - (isy ? 1 : 0) || (NDIM == 2 && j0 + fy > g.n[1] - (isy ? 0 : 1))) continue;
      const int s0 = (fy + C::HY) * C::SX + (fx + C::HX);
      const int er = isy ? C::E0 + (fy + 1) * BX + fx : fy * (BX + 2) + fx + 1;
      if constexpr (NDIM == 1) {
        const int fld[3] = {0, 1, 2};
        face_df<C, CMAX, 0>(su, ss, sf, p, s0 - 1, s0, er - 1, er, f, fld);
      } else {
        const int fld[4] = {0, isy ? 2 : 1, isy ? 1 : 2, 3};
        face_df<C, CMAX, 0>(su, ss, sf, p, s0 - (isy ? C::SX : 1), s0, er - (isy ? BX : 1), er, f, fld);
      }
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < C::CPT; ++c) {
      const int cell = threadIdx.x + c * NT;
      if (cell >= C::NCELL) break;
      df d[NV];
      face_diff_df<C, BX, BY, BZ, 0>(sf, cell % BX, cell / BX, 0, d);
#pragma unroll
      for (int v = 0; v < NV; ++v) dU[c][v] = d[v] * p.nhalf_inv_dx[0];
      if constexpr (NDIM == 2) {
        face_diff_df<C, BX, BY, BZ, 1>(sf + C::F0, cell % BX, cell / BX, 0, d);
#pragma unroll
        for (int v = 0; v < NV; ++v) dU[c][v] = df_fma(d[v], p.nhalf_inv_dx[1], dU[c][v]);
      }
    }
  } else {
    axis_pass_df<NDIM, BX, BY, BZ, NT, 0, CMAX>(su, sf, ss, p, g, i0, j0, k0, dU);
    axis_pass_df<NDIM, BX, BY, BZ, NT, 1, CMAX>(su, sf, ss, p, g, i0, j0, k0, dU);
    axis_pass_df<NDIM, BX, BY, BZ, NT, 2, CMAX>(su, sf, ss, p, g, i0, j0, k0, dU);
  }

  df rmax = {0.0f, 0.0f};
  bool ok_all = true;
#pragma unroll
  for (int c = 0; c < C::CPT; ++c) {
    const int cell = threadIdx.x + c * NT;
    if (cell >= C::NCELL) break;
    const int cx = cell % BX;
    const int t = cell / BX;
    const int cy = t % BY;
    const int cz = t / BY;
    const int i = i0 + cx, j = j0 + cy, k = k0 + cz;
    if (i >= g.n[0] || (NDIM >= 2 && j >= g.n[1]) || (NDIM >= 3 && k >= g.n[2])) continue;
    const int s0 = (cz + C::HZ) * C::SX * C::SY + (cy + C::HY) * C::SX + (cx + C::HX);
    df q[NV], L[NV], u[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      q[v] = su[v * C::SCELLS + s0];
      L[v] = dU[c][v];
    }
    rsst_rhs_df<NV, CMAX>(q, L, p);
    if constexpr (ST == 1) {
#pragma unroll
      for (int v = 0; v < NV; ++v) u[v] = df_fma(dt, L[v], q[v]);
    } else {
      const int64_t o = pidx(g, i, j, k);
#pragma unroll
      for (int v = 0; v < NV; ++v) u[v] = scale(ld_df(a.base, v * g.fstride + o) + df_fma(dt, L[v], q[v]), 0.5f);
      bool ok;
      const df r = cfl_rate_df<NV>(u, p, ok);
      if (ok && df_lt(rmax, r)) rmax = r;
      ok_all = ok_all && ok;
    }
    store_ghosts_df<NV>(a.out, g, a.p, a.bg, a.bg_len, i, j, k, u);
  }
  if constexpr (ST == 2) {
    if (!ok_all) atomicOr(a.flag, RSST_FLAG_NONPHYSICAL);
    block_max_df<NT>(rmax, a.scal + (a.slot ^ 1), sred);
  }
}

// ---------------------------------------------------------------------------
// Packing, CFL maximum, sums (double-float storage)
// ---------------------------------------------------------------------------

// Storage of a double-float run (rsst_transfer.cuh), ghosts as in float64.
template <int NV_>
struct StoreDF {
  static constexpr int NV = NV_;
  float2* u;
  int64_t fs;
  const double* bg;
  int bg_len;
  PhysDF p;
  __device__ __forceinline__ void store(int64_t o, double (&w)[NV], int sv, int gv) const {
    if (gv != INT_MIN && bg != nullptr) {
      w[0] += bg[gv + RSST_G] - bg[sv + RSST_G];
      w[NV - 1] += bg[bg_len + gv + RSST_G] - bg[bg_len + sv + RSST_G];
    }
#pragma unroll
    for (int v = 0; v < NV; ++v) st_df(u, v * fs + o, df_from_bits(w[v]));
  }
  __device__ __forceinline__ double rate(const double (&w)[NV], int, bool& ok) const {
    df q[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) q[v] = df_from_bits(w[v]);
    return df_to_bits(cfl_rate_df<NV>(q, p, ok));
  }
  __device__ __forceinline__ double load(int64_t o, int v, int) const { return df_to_bits(ld_df(u, v * fs + o)); }
};

constexpr int SUM_BLOCKS_DF = 1024;
constexpr int SUM_THREADS_DF = 256;

__global__ void __launch_bounds__(SUM_THREADS_DF) sums_partial_df_kernel(const float2* __restrict__ U, Geom g,
                                                                         double* __restrict__ partial) {
  __shared__ double sh[SUM_THREADS_DF];
  const int nv = g.ndim + 2;
  const int64_t chunk = (g.ncells + SUM_BLOCKS_DF - 1) / SUM_BLOCKS_DF;
  const int64_t lo = blockIdx.x * chunk;
  const int64_t hi = min(g.ncells, lo + chunk);
  for (int v = 0; v < nv; ++v) {
    double acc = 0.0;
    for (int64_t id = lo + threadIdx.x; id < hi; id += SUM_THREADS_DF) {
      const int i = (int)(id % g.n[0]);
      const int j = (int)((id / g.n[0]) % g.n[1]);
      const int k = (int)(id / ((int64_t)g.n[0] * g.n[1]));
      acc += df_to(ld_df(U, v * g.fstride + pidx(g, i, j, k)));
    }
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int s = SUM_THREADS_DF / 2; s > 0; s >>= 1) {
      if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
      __syncthreads();
    }
    if (threadIdx.x == 0) partial[v * SUM_BLOCKS_DF + blockIdx.x] = sh[0];
    __syncthreads();
  }
}

__global__ void __launch_bounds__(SUM_THREADS_DF) sums_final_df_kernel(const double* __restrict__ partial, int nv,
                                                                       double scale_, double* __restrict__ out) {
  __shared__ double sh[SUM_THREADS_DF];
  for (int v = 0; v < nv; ++v) {
    double acc = 0.0;
    for (int b = threadIdx.x; b < SUM_BLOCKS_DF; b += SUM_THREADS_DF) acc += partial[v * SUM_BLOCKS_DF + b];
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int s = SUM_THREADS_DF / 2; s > 0; s >>= 1) {
      if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
      __syncthreads();
    }
    if (threadIdx.x == 0) out[v] = sh[0] * scale_;
    __syncthreads();
  }
}

static df split_host(double x) {
  const float h = (float)x;
  return {h, (float)(x - (double)h)};
}

static PhysDF make_physdf(const Phys& p) {
  PhysDF q;
  q.gamma = split_host(p.gamma);
  q.gm1 = split_host(p.gm1);
  q.nhgm1 = split_host(-p.hgm1);
  q.inv_gm1 = split_host(p.inv_gm1);
  q.gam_gm1 = split_host(p.gam_gm1);
  int e = 0;
  std::frexp(p.gamma_xi2, &e);
  const int m = (e - 1) >> 1;
  q.gx = p.gamma_xi2 > 0.0 ? split_host(std::ldexp(p.gamma_xi2, -2 * m)) : df{1.0f, 0.0f};
  q.xs = p.gamma_xi2 > 0.0 ? (float)std::ldexp(1.0, m) : 0.0f;
  q.nf = split_host(-p.f);
  q.nf_gm1 = split_host(-p.f_gm1);
  q.inv_cmax4 = split_host(p.inv_cmax4);
  for (int d = 0; d < 3; ++d) {
    q.grav[d] = split_host(p.grav[d]);
    q.nhalf_inv_dx[d] = split_host(-p.half_inv_dx[d]);
  }
  q.sum_inv_dx = split_host(p.sum_inv_dx);
  q.variant = p.variant;
  q.use_cmax = p.use_cmax;
  q.has_grav = p.has_grav;
  return q;
}

template <int NDIM, int BX, int BY, int BZ, int NT, int MINB, bool CMAX, int ST>
static int launch_df_kernel(const CUtensorMap* tin, const DFArgs& a, cudaStream_t s) {
  using C = TileCfgDF<NDIM, BX, BY, BZ, NT>;
  auto kern = stage_df_kernel<NDIM, BX, BY, BZ, NT, MINB, CMAX, ST>;
  const size_t smem = C::SMEM;
  static const CUtensorMap none = {};
  static std::atomic<unsigned long long> attr{0};
  if (set_smem_limit_once(kern, smem, attr) != cudaSuccess) {
    rsst_set_error("cudaFuncSetAttribute failed for the double-float stage kernel");
    return RSST_ECUDA;
  }
  dim3 grid((a.g.n[0] + BX - 1) / BX, NDIM >= 2 ? (a.g.n[1] + BY - 1) / BY : 1, NDIM >= 3 ? (a.g.n[2] + BZ - 1) / BZ : 1);
  kern<<<grid, NT, smem, s>>>(NDIM >= 2 ? *tin : none, a);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    rsst_set_error("double-float stage kernel launch: %s", cudaGetErrorString(e));
    return RSST_ECUDA;
  }
  return RSST_OK;
}

// The C_max law and the stage are compile-time (no branches on them in the flux).
template <int NDIM, int BX, int BY, int BZ, int NT, int MINB>
static int launch_df(const CUtensorMap* tin, const DFArgs& a, cudaStream_t s) {
  if (a.q.use_cmax)
    return a.stage == 1 ? launch_df_kernel<NDIM, BX, BY, BZ, NT, MINB, true, 1>(tin, a, s)
                        : launch_df_kernel<NDIM, BX, BY, BZ, NT, MINB, true, 2>(tin, a, s);
  return a.stage == 1 ? launch_df_kernel<NDIM, BX, BY, BZ, NT, MINB, false, 1>(tin, a, s)
                      : launch_df_kernel<NDIM, BX, BY, BZ, NT, MINB, false, 2>(tin, a, s);
}

}  // namespace rsst

using namespace rsst;

// 2D tiles: the one that finishes first by a linear model, as for float64
// (rsst_stage_fp64_tile): 16 x 16, or 8 x 8 where a grid is too small to fill
// the SMs.  Measured per stage (us, 16 x 16 / 8 x 8): 64^2 7.4 / 5.5, 128^2
// 7.5 / 6.2, 160^2 7.6 / 6.5, 192^2 7.9 / 7.2, 224^2 10.2 / 9.7, 256^2 10.1 /
// 13.4, 512^2 27.4 / 39.2, 2048^2 388 / 558; the model takes the faster of each.
static const int TILE2_DF[2] = {16, 8};

int rsst_stage_df_tile(const Geom& g, int sms) {
  static const double offset[2] = {4.3, 2.6}, slope[2] = {3.55, 1.29};
  if (g.ndim != 2) return 0;
  if ((g.n[1] + TILE2_DF[1] - 1) / TILE2_DF[1] > RSST_GRID_Y) return 0;  // beyond the launch grid's y limit
  double us[2];
  for (int t = 0; t < 2; ++t) {
    const int b = TILE2_DF[t];
    const int64_t tiles = (int64_t)((g.n[0] + b - 1) / b) * ((g.n[1] + b - 1) / b);
    us[t] = offset[t] + slope[t] * (double)((tiles + sms - 1) / sms);
  }
  return us[1] < us[0] ? 1 : 0;
}

void rsst_stage_df_box(const Geom& g, int tile, int* sx, int* sy, int* sz) {
  *sx = *sy = (g.ndim == 3 ? 8 : TILE2_DF[tile]) + 2 * RSST_G;
  *sz = g.ndim == 3 ? 4 + 2 * RSST_G : 1;
}

int rsst_launch_stage_df(const CUtensorMap* tin, const StageArgs<float2>& sa, cudaStream_t s) {
  DFArgs a;
  a.in = sa.in;
  a.base = sa.base;
  a.out = sa.out;
  a.g = sa.g;
  a.p = sa.p;
  a.q = make_physdf(sa.p);
  a.bg = sa.bg;
  a.bg_len = sa.bg_len;
  a.scal = sa.scal;
  a.flag = sa.flag;
  a.slot = sa.slot;
  a.stage = sa.stage;
  a.dt_fixed = sa.dt_fixed;
  a.stall_ns = sa.stall_ns;
  switch (a.g.ndim) {
    case 1:
      if (a.g.n[0] <= RSST_SMALL_1D) return launch_df<1, 16, 1, 1, 32, 1>(nullptr, a, s);
      return launch_df<1, 256, 1, 1, 256, 1>(nullptr, a, s);
    case 2:
      return sa.tile ? launch_df<2, 8, 8, 1, 160, 6>(tin, a, s) : launch_df<2, 16, 16, 1, 288, 4>(tin, a, s);
    case 3:
      return launch_df<3, 8, 8, 4, 320, 3>(tin, a, s);  // 10 warps: each face pass in one round
  }
  rsst_set_error("ndim must be 1, 2 or 3");
  return RSST_EINVAL;
}

static int err_df(const char* what) {
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    rsst_set_error("%s launch: %s", what, cudaGetErrorString(e));
    return RSST_ECUDA;
  }
  return RSST_OK;
}

int rsst_launch_pack_df(const double* src, float2* dst, const Geom& g, const Phys& p, const double* bg, int bg_len,
                        double* cfl, unsigned int* flag, cudaStream_t s) {
  const PhysDF q = make_physdf(p);
#define PACK(NV) launch_pack(src, g, p, StoreDF<NV>{dst, g.fstride, bg, bg_len, q}, cfl, flag, "pack (double-float)", s)
  return g.ndim == 1 ? PACK(3) : (g.ndim == 2 ? PACK(4) : PACK(5));
#undef PACK
}

int rsst_launch_unpack_df(const float2* src, double* dst, const Geom& g, cudaStream_t s) {
#define UNPACK(NV) \
  launch_unpack(dst, g, -1, StoreDF<NV>{const_cast<float2*>(src), g.fstride, nullptr, 0, PhysDF{}}, "unpack (double-float)", s)
  return g.ndim == 1 ? UNPACK(3) : (g.ndim == 2 ? UNPACK(4) : UNPACK(5));
#undef UNPACK
}

int rsst_launch_sums_df(const float2* U, const Geom& g, double* partial, double* out, double scale_, cudaStream_t s) {
  sums_partial_df_kernel<<<SUM_BLOCKS_DF, SUM_THREADS_DF, 0, s>>>(U, g, partial);
  const int rc = err_df("sums (double-float)");
  if (rc) return rc;
  sums_final_df_kernel<<<1, SUM_THREADS_DF, 0, s>>>(partial, g.ndim + 2, scale_, out);
  return err_df("sums final (double-float)");
}
