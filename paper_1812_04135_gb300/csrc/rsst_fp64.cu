// Float64 kernels of the RSST step: one fused kernel per SSP-RK2 stage
// (Sec. 4.2 steps 2-8 of arXiv:1812.04135), plus state packing, the
// standalone CFL maximum (step 1) and deterministic conservation sums.
//
// Fused stage kernel, one CTA per tile of BX x BY x BZ cells:
//   1. the tile plus two halo layers on every active axis (all fields) is
//      copied from the padded state into shared memory: in 2D and 3D by one
//      cp.async.bulk.tensor of the whole box (x origin on a 16-byte
//      boundary, rows and planes beyond the padded state zero-filled, a
//      bounded mbarrier wait), in 1D (tiles wider than a TMA box) with
//      coalesced loads;
//   2. the MC slope of every cell along each axis is computed once into
//      shared memory (1D/2D tiles: all axes at once; 3D tiles: axis by axis),
//      then every face of the tile gets twice its LLF flux,
//      F(qL) + F(qR) - alpha (qR - qL), from the face states of the two cells
//      beside it; a face shared by two tiles is computed the same way in both,
//      so both get bit-identical values (discrete conservation);
//   3. each cell takes -(2F_{+} - 2F_{-}) / (2 dx_D) of every axis;
//   4. epilogue per cell: RSST correction, force, RK combine, store, the
//      edge ghost cells the cell is the image of, and in stage 2 the CFL
//      maximum for the next step and the physical-state flag.
//
// What bounds it: the float64 pipe, which takes one warp instruction per 16
// SM clocks (a warp alone one per 64, however few lanes it has active) while
// every other pipe idles.  So the work is arranged for few float64
// instructions: 164.7 a 2D cell in stage 1 and 181.7 in stage 2 (ncu), 205.5
// and 227.5 with the wave speeds' squares, the reciprocal's third-order step,
// the block maximum, a per-thread dt division, unshared slope differences and
// the RK halving's sign on that pipe.  512^2: 123 -> 89 us a stage; 3D 256 x
// 128 x 128: 3090 -> 2457 us; 2048^2 runs the pipe 86 % busy.
#include <climits>
#include <cstdio>

#include "rsst_common.cuh"
#include "rsst_internal.h"
#include "rsst_attr.h"
#include "rsst_math_fp64.cuh"
#include "rsst_tma.cuh"
#include "rsst_transfer.cuh"

namespace rsst {

template <int NDIM, int BX, int BY, int BZ, int NT>
struct TileCfg {
  static constexpr int NV = NDIM + 2;
  static constexpr int HX = 2, HY = NDIM >= 2 ? 2 : 0, HZ = NDIM >= 3 ? 2 : 0;
  static constexpr int SX = BX + 2 * HX, SY = BY + 2 * HY, SZ = BZ + 2 * HZ;
  static constexpr int SCELLS = SX * SY * SZ;
  static constexpr int NCELL = BX * BY * BZ;
  static constexpr int CPT = (NCELL + NT - 1) / NT;
  // faces and slope cells (-1 .. B along the axis) per axis
  static constexpr int F0 = (BX + 1) * BY * BZ, F1 = NDIM >= 2 ? BX * (BY + 1) * BZ : 0;
  static constexpr int F2 = NDIM >= 3 ? BX * BY * (BZ + 1) : 0;
  static constexpr int E0 = (BX + 2) * BY * BZ, E1 = NDIM >= 2 ? BX * (BY + 2) * BZ : 0;
  static constexpr int E2 = NDIM >= 3 ? BX * BY * (BZ + 2) : 0;
  static constexpr int max3(int a, int b, int c) { return a > b ? (a > c ? a : c) : (b > c ? b : c); }
  // 1D/2D tiles hold the slopes and faces of every axis at once: three block
  // barriers a tile instead of six, and the axes' passes fill each other's
  // gaps.  3D tiles (three axes would leave room for one CTA an SM) go axis
  // by axis through one slope and one face array.
  static constexpr bool ALL = NDIM <= 2;
  static constexpr int FMAX = ALL ? F0 + F1 : max3(F0, F1, F2);
  static constexpr int EMAX = ALL ? E0 + E1 : max3(E0, E1, E2);
  static constexpr int up32(int x) { return (x + 31) / 32 * 32; }
  // halo tile, faces, slopes, the block reduction's 64 doubles, dt, and two
  // mbarriers (the tile copy; the failure-detection test wait)
  static constexpr size_t SMEM = sizeof(double) * ((size_t)NV * (SCELLS + FMAX + EMAX) + 64 + 1) + 16;
  static constexpr uint32_t TILE_BYTES = (uint32_t)(sizeof(double) * NV * SCELLS);
  static_assert(NDIM == 1 || (SX <= 256 && SY <= 256 && SZ <= 256), "TMA box dimensions are at most 256");
  static_assert(BX % 2 == 0 && (NDIM < 2 || BY % 2 == 0) && (NDIM < 3 || BZ % 2 == 0), "slopes are taken in pairs");
  static_assert((SX * sizeof(double)) % 16 == 0 && (HX * sizeof(double)) % 16 == 0,
                "the box's row bytes and the x origin (interior x0 - HX) stay on 16-byte boundaries");
};

// MC slopes along D of the pair of neighbouring slope cells e (tile
// coordinates -1 .. B along D, 0 .. B-1 across; pairs lie along D): the two
// share a difference, five float64 additions a field instead of six.
template <class C, int BX, int BY, int BZ, int D>
__device__ __forceinline__ void slope_pair(const double* __restrict__ su, double* __restrict__ ss, int e) {
  constexpr int STRIDE = D == 0 ? 1 : (D == 1 ? C::SX : C::SX * C::SY);
  constexpr int XX = BX + 2 * (D == 0), YY = BY + 2 * (D == 1);
  constexpr int PX = D == 0 ? XX / 2 : XX, PY = D == 1 ? YY / 2 : YY;  // pairs per axis
  const int ex = e % PX * (D == 0 ? 2 : 1);
  const int t = e / PX;
  const int ey = t % PY * (D == 1 ? 2 : 1);
  const int ez = t / PY * (D == 2 ? 2 : 1);
  const int s0 = (ez - (D == 2) + C::HZ) * C::SX * C::SY + (ey - (D == 1) + C::HY) * C::SX + (ex - (D == 0) + C::HX);
  const int o = (ez * YY + ey) * XX + ex;
  constexpr int STRIDE_E = D == 0 ? 1 : (D == 1 ? XX : XX * YY);
#pragma unroll
  for (int v = 0; v < C::NV; ++v) {
    const double* sv = su + v * C::SCELLS + s0;
    const double um = sv[-STRIDE], u0 = sv[0], u1 = sv[STRIDE], up = sv[2 * STRIDE];
    const double d = u1 - u0;
    ss[v * C::EMAX + o] = mc_slope(u0 - um, d);
    ss[v * C::EMAX + o + STRIDE_E] = mc_slope(d, up - u1);
  }
}

// Twice the LLF flux of face fid along D: index space
// (BX + [D==0]) x (BY + [D==1]) x (BZ + [D==2]), the face below that cell.
template <class C, int NDIM, int BX, int BY, int BZ, int D, bool CV>
__device__ __forceinline__ void face_flux(const double* __restrict__ su, const double* __restrict__ ss,
                                          double* __restrict__ sf, const Phys& p, const Geom& g, int i0, int j0,
                                          int k0, int fid) {
  constexpr int NV = C::NV;
  constexpr int EX = BX + (D == 0), EY = BY + (D == 1);
  constexpr int STRIDE = D == 0 ? 1 : (D == 1 ? C::SX : C::SX * C::SY);
  constexpr int XX = BX + 2 * (D == 0), YY = BY + 2 * (D == 1);
  const int fx = fid % EX;
  const int t = fid / EX;
  const int fy = t % EY;
  const int fz = t / EY;
  // face fD - 1/2 of tile cell (fx, fy, fz); valid if its cells exist
  const bool valid = (i0 + fx <= g.n[0] - (D == 0 ? 0 : 1)) && (NDIM < 2 || j0 + fy <= g.n[1] - (D == 1 ? 0 : 1)) &&
                     (NDIM < 3 || k0 + fz <= g.n[2] - (D == 2 ? 0 : 1));
  if (!valid) return;
  // shared-memory index of the cell right of the face; its slope index (the left one is STRIDE_E before)
  const int s0 = (fz + C::HZ) * C::SX * C::SY + (fy + C::HY) * C::SX + (fx + C::HX);
  constexpr int STRIDE_E = D == 0 ? 1 : (D == 1 ? XX : XX * YY);
  const int er = ((fz + (D == 2)) * YY + (fy + (D == 1))) * XX + (fx + (D == 0));
  double qL[NV], qR[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const double* sv = su + v * C::SCELLS + s0;
    qL[v] = fma(0.5, ss[v * C::EMAX + er - STRIDE_E], sv[-STRIDE]);
    qR[v] = fma(-0.5, ss[v * C::EMAX + er], sv[0]);
  }
  double F[NV];
  llf_flux_x2<NV, D, CV>(qL, qR, p, F);
#pragma unroll
  for (int v = 0; v < NV; ++v) sf[v * C::FMAX + fid] = F[v];
}

// The x and y faces of a 2D tile as one list (f < F0: x, then y): the axis
// only enters through strides and through which momentum is the normal one,
// so a warp that holds faces of both axes does not diverge (16 x 16 tiles: 17
// warps of faces; 18 with each axis padded to whole warps).
template <class C, int BX, int BY, bool CV>
__device__ __forceinline__ void face_flux_xy(const double* __restrict__ su, const double* __restrict__ ss,
                                             double* __restrict__ sf, const Phys& p, const Geom& g, int i0, int j0,
                                             int f) {
  const bool isy = f >= C::F0;
  const int fid = isy ? f - C::F0 : f;
  const int ex = isy ? BX : BX + 1;
  const int fy = isy ? fid / BX : fid / (BX + 1);
  const int fx = fid - fy * ex;
  if (i0 + fx > g.n[0] - (isy ? 1 : 0) || j0 + fy > g.n[1] - (isy ? 0 : 1)) return;
  const int s0 = (fy + C::HY) * C::SX + (fx + C::HX);
  const int sl = s0 - (isy ? C::SX : 1);
  const int er = isy ? C::E0 + (fy + 1) * BX + fx : fy * (BX + 2) + fx + 1;
  const int el = er - (isy ? BX : 1);
  const int n = isy ? 2 : 1, t = 3 - n;  // fields of the normal and the transverse momentum
  const int fld[4] = {0, n, t, 3};
  double qL[4], qR[4], F[4];
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    const double* sv = su + fld[v] * C::SCELLS;
    const double* se = ss + fld[v] * C::EMAX;
    qL[v] = fma(0.5, se[el], sv[sl]);
    qR[v] = fma(-0.5, se[er], sv[s0]);
  }
  llf_flux_x2<4, 0, CV>(qL, qR, p, F);
#pragma unroll
  for (int v = 0; v < 4; ++v) sf[fld[v] * C::FMAX + f] = F[v];
}

// 2F above minus 2F below tile cell (cx, cy, cz) along D, per field.
template <class C, int BX, int BY, int BZ, int D>
__device__ __forceinline__ void face_diff(const double* __restrict__ sf, int cx, int cy, int cz, double (&d)[C::NV]) {
  constexpr int EX = BX + (D == 0), EY = BY + (D == 1);
  const int flo = (cz * EY + cy) * EX + cx;
  const int fhi = flo + (D == 0 ? 1 : (D == 1 ? EX : EX * EY));
#pragma unroll
  for (int v = 0; v < C::NV; ++v) d[v] = sf[v * C::FMAX + fhi] - sf[v * C::FMAX + flo];
}

// One axis of a 3D tile: slopes, faces, and each thread's cells' divergence.
// The next axis may overwrite the slopes at once (every face was formed) and
// the faces after its own slope barrier (every divergence was taken).
template <int NDIM, int BX, int BY, int BZ, int NT, int D, bool CV>
__device__ __forceinline__ void axis_pass(const double* __restrict__ su, double* __restrict__ sf,
                                          double* __restrict__ ss, const Phys& p, const Geom& g, int i0, int j0,
                                          int k0, double (&dU)[TileCfg<NDIM, BX, BY, BZ, NT>::CPT][NDIM + 2]) {
  using C = TileCfg<NDIM, BX, BY, BZ, NT>;
  constexpr int NE = D == 0 ? C::E0 : (D == 1 ? C::E1 : C::E2), NF = D == 0 ? C::F0 : (D == 1 ? C::F1 : C::F2);
  for (int e = threadIdx.x; e < NE / 2; e += NT) slope_pair<C, BX, BY, BZ, D>(su, ss, e);
  __syncthreads();
  for (int f = threadIdx.x; f < NF; f += NT) face_flux<C, NDIM, BX, BY, BZ, D, CV>(su, ss, sf, p, g, i0, j0, k0, f);
  __syncthreads();
  const double idx = p.half_inv_dx[D];  // the faces hold 2 F
#pragma unroll
  for (int c = 0; c < C::CPT; ++c) {
    const int cell = threadIdx.x + c * NT;
    if (cell >= C::NCELL) break;
    double d[C::NV];
    face_diff<C, BX, BY, BZ, D>(sf, cell % BX, cell / BX % BY, cell / BX / BY, d);
#pragma unroll
    for (int v = 0; v < C::NV; ++v) dU[c][v] = D == 0 ? -d[v] * idx : fma(-d[v], idx, dU[c][v]);
  }
}

template <int NDIM, int BX, int BY, int BZ, int NT, int MINB, bool TMA, bool CV>
__global__ void __launch_bounds__(NT, MINB)
    stage_fp64_kernel(const __grid_constant__ CUtensorMap tin, const StageArgs<double> a) {
  using C = TileCfg<NDIM, BX, BY, BZ, NT>;
  constexpr int NV = C::NV;
  extern __shared__ __align__(128) double smem[];
  double* su = smem;
  double* sf = smem + NV * C::SCELLS;
  double* ss = sf + NV * C::FMAX;
  double* sred = ss + NV * C::EMAX;
  double* sdt = sred + 64;
  const Geom& g = a.g;
  const Phys& p = a.p;
  const int i0 = blockIdx.x * BX, j0 = blockIdx.y * BY, k0 = blockIdx.z * BZ;
  uint64_t* bar = reinterpret_cast<uint64_t*>(sdt + 1);
  uint64_t* test_bar = bar + 1;
  const bool stall = TMA && a.stall_ns > 0;
  if (TMA && threadIdx.x == 0) {
    mbar_init(bar, 1);
    if (stall) mbar_init(test_bar, 1);
    fence_mbar_init();
  }

  // 1. halo tile -> shared memory; dt once per CTA (a float64 division)
  if (threadIdx.x == (TMA ? NT - 1 : 0)) {
    const double dt = a.dt_fixed > 0.0 ? a.dt_fixed : p.cfl / a.scal[a.slot];
    *sdt = dt;
    if (a.stage == 1 && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0) {
      a.scal[a.slot ^ 1] = 0.0;
      a.scal[2] = dt;
      a.scal[3] += dt;
    }
  }
  if constexpr (TMA) {
    // The box of the padded state [nvar][pz][py][pitch] whose first cell is
    // interior (i0 - HX, j0 - HY, k0 - HZ): padded x i0 + xoff - HX, padded
    // y j0 (HY = gy), padded z k0 (HZ = gz).
    if (threadIdx.x == 0) {
      fence_proxy_async_smem();
      mbar_expect_tx(bar, C::TILE_BYTES);
      if constexpr (NDIM == 2) tma_load_3d(su, &tin, bar, i0 + g.xoff - C::HX, j0, 0);
      else tma_load_4d(su, &tin, bar, i0 + g.xoff - C::HX, j0, k0, 0);
      // failure-detection test: a barrier that expects 16 bytes no copy
      // delivers, waited on while the tile copy is still in flight
      if (stall) mbar_expect_tx(test_bar, 16);
    }
    __syncthreads();  // the barriers are initialised
    const bool landed = stall ? mbar_wait_bounded(test_bar, 0u, (uint64_t)a.stall_ns) : mbar_wait_bounded(bar, 0u);
    // Giving up is decided by the whole block: flag the run and, before
    // leaving, wait (bounded) for the tile copy, so that it cannot land in
    // shared memory the next CTA on this SM may own.
    if (__syncthreads_or(!landed)) {
      if (threadIdx.x == 0) {
        atomicOr(a.flag, RSST_FLAG_TIMEOUT);
        mbar_wait_bounded(bar, 0u);
      }
      return;
    }
  } else {
    for (int id = threadIdx.x; id < NV * C::SCELLS; id += NT) {
      const int v = id / C::SCELLS;
      const int r = id - v * C::SCELLS;
      const int lx = r % C::SX;
      const int t = r / C::SX;
      const int ly = t % C::SY;
      const int lz = t / C::SY;
      const int gi = i0 + lx - C::HX, gj = j0 + ly - C::HY, gk = k0 + lz - C::HZ;
      double val = 0.0;
      if (gi <= g.n[0] + 1 && (NDIM < 2 || gj <= g.n[1] + 1) && (NDIM < 3 || gk <= g.n[2] + 1))
        val = a.in[v * g.fstride + pidx(g, gi, gj, gk)];
      su[id] = val;
    }
    __syncthreads();
  }

  // 2-3. slopes, face fluxes and divergence
  double dU[C::CPT][NV];
  if constexpr (C::ALL) {
    constexpr int PE = C::up32(C::E0 / 2);  // axis y starts at a whole warp
    for (int e = threadIdx.x; e < (NDIM == 1 ? C::E0 / 2 : PE + C::E1 / 2); e += NT) {
      if (e < PE) {
        if (e < C::E0 / 2) slope_pair<C, BX, BY, BZ, 0>(su, ss, e);
      } else if constexpr (NDIM == 2) {
        slope_pair<C, BX, BY, BZ, 1>(su, ss + C::E0, e - PE);
      }
    }
    __syncthreads();
    if constexpr (NDIM == 1) {
      for (int f = threadIdx.x; f < C::F0; f += NT) face_flux<C, 1, BX, BY, BZ, 0, CV>(su, ss, sf, p, g, i0, j0, k0, f);
    } else {
      for (int f = threadIdx.x; f < C::F0 + C::F1; f += NT) face_flux_xy<C, BX, BY, CV>(su, ss, sf, p, g, i0, j0, f);
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < C::CPT; ++c) {
      const int cell = threadIdx.x + c * NT;
      if (cell >= C::NCELL) break;
      double d[NV];
      face_diff<C, BX, BY, BZ, 0>(sf, cell % BX, cell / BX, 0, d);
#pragma unroll
      for (int v = 0; v < NV; ++v) dU[c][v] = -d[v] * p.half_inv_dx[0];  // the faces hold 2 F
      if constexpr (NDIM == 2) {
        face_diff<C, BX, BY, BZ, 1>(sf + C::F0, cell % BX, cell / BX, 0, d);
#pragma unroll
        for (int v = 0; v < NV; ++v) dU[c][v] = fma(-d[v], p.half_inv_dx[1], dU[c][v]);
      }
    }
  } else {
    axis_pass<NDIM, BX, BY, BZ, NT, 0, CV>(su, sf, ss, p, g, i0, j0, k0, dU);
    axis_pass<NDIM, BX, BY, BZ, NT, 1, CV>(su, sf, ss, p, g, i0, j0, k0, dU);
    axis_pass<NDIM, BX, BY, BZ, NT, 2, CV>(su, sf, ss, p, g, i0, j0, k0, dU);
  }

  // 4. epilogue
  const double dt = *sdt;
  double rmax = 0.0;
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
    double q[NV], L[NV], u[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      q[v] = su[v * C::SCELLS + s0];
      L[v] = dU[c][v];
    }
    if (a.dU_out) {
      const int64_t o = pidx(g, i, j, k);
#pragma unroll
      for (int v = 0; v < NV; ++v) a.dU_out[v * g.fstride + o] = L[v];
    }
    rsst_rhs<NV, CV>(q, L, p);
    if (a.stage == 1) {
#pragma unroll
      for (int v = 0; v < NV; ++v) u[v] = fma(dt, L[v], q[v]);
    } else {
      const int64_t o = pidx(g, i, j, k);
#pragma unroll
      for (int v = 0; v < NV; ++v) u[v] = half_of(a.base[v * g.fstride + o] + fma(dt, L[v], q[v]));
      bool ok;
      const double r = cfl_rate<NV, CV>(u, p, ok);
      if (ok) rmax = max_nonneg(rmax, r);
      ok_all = ok_all && ok;
    }
    store_with_ghosts<NV>(a.out, g, p, a.bg, a.bg_len, i, j, k, u);
  }
  if (a.stage == 2) {
    if (!ok_all) atomicOr(a.flag, RSST_FLAG_NONPHYSICAL);
    block_max_to<NT>(rmax, a.scal + (a.slot ^ 1), sred);
  }
}

// ---------------------------------------------------------------------------
// Packing, CFL maximum, sums
// ---------------------------------------------------------------------------

// Storage of a float64 run (rsst_transfer.cuh): values as they are; a ghost
// mirrored across a wall of the vertical axis gets the background's difference.
template <int NV_, bool CV>
struct StoreF64 {
  static constexpr int NV = NV_;
  double* u;
  int64_t fs;
  const double* bg;
  int bg_len;
  Phys p;
  __device__ __forceinline__ void store(int64_t o, double (&w)[NV], int sv, int gv) const {
    if (gv != INT_MIN && bg != nullptr) {
      w[0] += bg[gv + RSST_G] - bg[sv + RSST_G];
      w[NV - 1] += bg[bg_len + gv + RSST_G] - bg[bg_len + sv + RSST_G];
    }
#pragma unroll
    for (int v = 0; v < NV; ++v) u[v * fs + o] = w[v];
  }
  __device__ __forceinline__ double rate(const double (&w)[NV], int, bool& ok) const {
    return cfl_rate<NV, CV>(w, p, ok);
  }
  __device__ __forceinline__ double load(int64_t o, int v, int) const { return u[v * fs + o]; }
};

// Deterministic sums: block b reduces a fixed contiguous chunk of cells with a
// fixed thread striding and shared-memory tree; a single block then reduces
// the per-block partials in index order.
constexpr int SUM_BLOCKS = 1024;
constexpr int SUM_THREADS = 256;

__global__ void __launch_bounds__(SUM_THREADS) sums_partial_fp64_kernel(const double* __restrict__ U, Geom g,
                                                                        double* __restrict__ partial) {
  __shared__ double sh[SUM_THREADS];
  const int nv = g.ndim + 2;
  const int64_t chunk = (g.ncells + SUM_BLOCKS - 1) / SUM_BLOCKS;
  const int64_t lo = blockIdx.x * chunk;
  const int64_t hi = min(g.ncells, lo + chunk);
  for (int v = 0; v < nv; ++v) {
    double acc = 0.0;
    for (int64_t id = lo + threadIdx.x; id < hi; id += SUM_THREADS) {
      const int i = (int)(id % g.n[0]);
      const int j = (int)((id / g.n[0]) % g.n[1]);
      const int k = (int)(id / ((int64_t)g.n[0] * g.n[1]));
      acc += U[v * g.fstride + pidx(g, i, j, k)];
    }
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int s = SUM_THREADS / 2; s > 0; s >>= 1) {
      if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
      __syncthreads();
    }
    if (threadIdx.x == 0) partial[v * SUM_BLOCKS + blockIdx.x] = sh[0];
    __syncthreads();
  }
}

__global__ void __launch_bounds__(SUM_THREADS) sums_final_kernel(const double* __restrict__ partial, int nv,
                                                                 double scale, double* __restrict__ out) {
  __shared__ double sh[SUM_THREADS];
  for (int v = 0; v < nv; ++v) {
    double acc = 0.0;
    for (int b = threadIdx.x; b < SUM_BLOCKS; b += SUM_THREADS) acc += partial[v * SUM_BLOCKS + b];
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int s = SUM_THREADS / 2; s > 0; s >>= 1) {
      if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
      __syncthreads();
    }
    if (threadIdx.x == 0) out[v] = sh[0] * scale;
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------

template <int NDIM, int BX, int BY, int BZ, int NT, int MINB, bool TMA, bool CV>
static int launch_stage_eos(const CUtensorMap* tin, const StageArgs<double>& a, cudaStream_t s) {
  using C = TileCfg<NDIM, BX, BY, BZ, NT>;
  auto kern = stage_fp64_kernel<NDIM, BX, BY, BZ, NT, MINB, TMA, CV>;
  static std::atomic<unsigned long long> attr{0};
  if (set_smem_limit_once(kern, C::SMEM, attr) != cudaSuccess) {
    rsst_set_error("cudaFuncSetAttribute failed for the float64 stage kernel");
    return RSST_ECUDA;
  }
  static const CUtensorMap none = {};
  dim3 grid((a.g.n[0] + BX - 1) / BX, NDIM >= 2 ? (a.g.n[1] + BY - 1) / BY : 1, NDIM >= 3 ? (a.g.n[2] + BZ - 1) / BZ : 1);
  kern<<<grid, NT, C::SMEM, s>>>(TMA ? *tin : none, a);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    rsst_set_error("float64 stage kernel launch: %s", cudaGetErrorString(e));
    return RSST_ECUDA;
  }
  return RSST_OK;
}

// The gas law is a compile-time choice (no covolume arithmetic in ideal-gas runs).
template <int NDIM, int BX, int BY, int BZ, int NT, int MINB, bool TMA>
static int launch_stage(const CUtensorMap* tin, const StageArgs<double>& a, cudaStream_t s) {
  if (a.p.covol != 0.0) return launch_stage_eos<NDIM, BX, BY, BZ, NT, MINB, TMA, true>(tin, a, s);
  return launch_stage_eos<NDIM, BX, BY, BZ, NT, MINB, TMA, false>(tin, a, s);
}

}  // namespace rsst

using namespace rsst;

// Tiles.  1D: short lines take 16-cell tiles (17 faces, one per thread of a
// warp) to spread the float64 work over SMs, longer ones 256 cells.  3D
// 8 x 8 x 4 with 10 warps (each face pass in one round).
// 2D: the tile that finishes first by a linear model, offset + slope x the
// most tiles any SM gets (the float64 pipe of an SM serves its tiles one
// after the other).  16 x 16 has the fewest halo faces a cell, smaller tiles
// spread a small grid over more SMs.  Measured per stage (us, GB300; 16 x 16
// / 16 x 8 / 8 x 8): 64^2 16.9 / 12.6 / 9.0, 128^2 16.9 / 12.9 / 11.0, 160^2
// 17.1 / 17.3 / 13.7, 192^2 17.2 / 17.4 / 17.7, 224^2 28.6 / 23.3 / 25.3, 256^2
// 28.6 / 29.7 / 33.2, 512^2 89.5 / 95.5 / 104, 2048^2 1338 / 1428 / 1610; with
// these constants the model takes the fastest of each.  (4 x 4 tiles gained
// 0.1 us on 64^2 and lost elsewhere.)  A shape whose rows of tiles exceed the
// launch grid's y limit is not taken (tall, narrow grids).
static const int TILE2[3][2] = {{16, 16}, {16, 8}, {8, 8}};

int rsst_stage_fp64_tile(const Geom& g, int sms) {
  static const double offset[3] = {4.5, 5.0, 3.3}, slope[3] = {12.35, 6.6, 3.72};
  if (g.ndim != 2) return 0;
  int best = 0;
  double tbest = 0.0;
  for (int t = 0; t < 3; ++t) {
    const int rows = (g.n[1] + TILE2[t][1] - 1) / TILE2[t][1];
    const int64_t tiles = (int64_t)((g.n[0] + TILE2[t][0] - 1) / TILE2[t][0]) * rows;
    if (t > 0 && rows > RSST_GRID_Y) continue;
    const double us = offset[t] + slope[t] * (double)((tiles + sms - 1) / sms);
    if (t == 0 || us < tbest) {
      best = t;
      tbest = us;
    }
  }
  return best;
}

void rsst_stage_fp64_box(const Geom& g, int tile, int* sx, int* sy, int* sz) {
  *sx = (g.ndim == 3 ? 8 : TILE2[tile][0]) + 2 * RSST_G;
  *sy = (g.ndim == 3 ? 8 : TILE2[tile][1]) + 2 * RSST_G;
  *sz = g.ndim == 3 ? 4 + 2 * RSST_G : 1;
}

int rsst_launch_stage_fp64(const CUtensorMap* tin, const StageArgs<double>& a, cudaStream_t s) {
  switch (a.g.ndim) {
    case 1:
      if (a.g.n[0] <= RSST_SMALL_1D) return launch_stage<1, 16, 1, 1, 32, 1, false>(nullptr, a, s);
      return launch_stage<1, 256, 1, 1, 256, 1, false>(nullptr, a, s);
    case 2:
      switch (a.tile) {
        case 0: return launch_stage<2, 16, 16, 1, 288, 4, true>(tin, a, s);
        case 1: return launch_stage<2, 16, 8, 1, 160, 6, true>(tin, a, s);
        default: return launch_stage<2, 8, 8, 1, 160, 6, true>(tin, a, s);
      }
    case 3:
      return launch_stage<3, 8, 8, 4, 320, 3, true>(tin, a, s);
  }
  rsst_set_error("ndim must be 1, 2 or 3");
  return RSST_EINVAL;
}

static int check_launch(const char* what) {
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    rsst_set_error("%s launch: %s", what, cudaGetErrorString(e));
    return RSST_ECUDA;
  }
  return RSST_OK;
}

namespace rsst {
__global__ void reset_kernel(double* scal, int slot, unsigned int* flag) {
  scal[slot] = 0.0;
  scal[3] = 0.0;  // simulated time
  *flag = 0u;
}
}  // namespace rsst

int rsst_launch_reset(double* scal, int slot, unsigned int* flag, cudaStream_t s) {
  reset_kernel<<<1, 1, 0, s>>>(scal, slot, flag);
  return check_launch("reset");
}

int rsst_launch_pack_fp64(const double* src, double* dst, const Geom& g, const Phys& p, const double* bg, int bg_len,
                          double* cfl, unsigned int* flag, cudaStream_t s) {
#define PACK(NV, CV) launch_pack(src, g, p, StoreF64<NV, CV>{dst, g.fstride, bg, bg_len, p}, cfl, flag, "pack", s)
  if (p.covol != 0.0) return g.ndim == 1 ? PACK(3, true) : (g.ndim == 2 ? PACK(4, true) : PACK(5, true));
  return g.ndim == 1 ? PACK(3, false) : (g.ndim == 2 ? PACK(4, false) : PACK(5, false));
#undef PACK
}

int rsst_launch_unpack_fp64(const double* src, double* dst, const Geom& g, cudaStream_t s) {
#define UNPACK(NV) launch_unpack(dst, g, -1, StoreF64<NV, false>{const_cast<double*>(src), g.fstride, nullptr, 0, Phys{}}, "unpack", s)
  return g.ndim == 1 ? UNPACK(3) : (g.ndim == 2 ? UNPACK(4) : UNPACK(5));
#undef UNPACK
}

int rsst_launch_sums_fp64(const double* U, const Geom& g, double* partial, double* out, double scale, cudaStream_t s) {
  sums_partial_fp64_kernel<<<SUM_BLOCKS, SUM_THREADS, 0, s>>>(U, g, partial);
  int rc = check_launch("sums");
  if (rc) return rc;
  sums_final_kernel<<<1, SUM_THREADS, 0, s>>>(partial, g.ndim + 2, scale, out);
  return check_launch("sums final");
}
