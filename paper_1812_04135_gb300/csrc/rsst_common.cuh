// Device helpers shared by the float64 and float32 kernels.
#pragma once

#include "rsst_internal.h"

namespace rsst {

// Padded-layout offset of interior cell (i, j, k) (ghosts at -2, -1, n, n+1).
__device__ __forceinline__ int64_t pidx(const Geom& g, int i, int j, int k) {
  return (int64_t)(k + g.gz) * g.plane + (int64_t)(j + g.gy) * g.pitch + (i + g.xoff);
}

// Maximum of non-negative doubles, whose bit patterns order like their
// values: on the integer pipe (a float64 compare or maximum occupies the
// float64 pipe as long as an FMA).
__device__ __forceinline__ double max_nonneg(double a, double b) {
  const long long x = __double_as_longlong(a), y = __double_as_longlong(b);
  return __longlong_as_double(x > y ? x : y);
}
__device__ __forceinline__ double warp_max(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
  const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? lo : 0u);
  return __hiloint2double((int)mh, (int)ml);
}

// Block-wide maximum of non-negative values, then one atomicMax on the bit
// pattern (monotone for non-negative doubles).  All threads must call it.
template <int NT>
__device__ __forceinline__ void block_max_to(double x, double* dst, double* sred) {
  x = warp_max(x);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) sred[wid] = x;
  __syncthreads();
  if (wid == 0) {
    double y = lane < NT / 32 ? sred[lane] : 0.0;
    y = warp_max(y);
    if (lane == 0 && __double_as_longlong(y) > 0)
      atomicMax(reinterpret_cast<unsigned long long*>(dst), (unsigned long long)__double_as_longlong(y));
  }
}

// Store a float64 cell and the edge ghost cells that mirror or wrap it (across a
// wall along the vertical axis with the background difference added).
template <int NV>
__device__ __forceinline__ void store_with_ghosts(double* __restrict__ out, const Geom& g,
                                                  const Phys& p, const double* __restrict__ bg,
                                                  int bg_len, int i, int j, int k,
                                                  const double (&u)[NV]) {
  constexpr int ND = NV - 2;
  const int64_t fs = g.fstride;
  const int64_t o = pidx(g, i, j, k);
#pragma unroll
  for (int v = 0; v < NV; ++v) out[v * fs + o] = u[v];
  const int c[3] = {i, j, k};
#pragma unroll
  for (int d = 0; d < ND; ++d) {
    const int n = g.n[d], cd = c[d];
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      const bool hit = side == 0 ? (cd < RSST_G) : (cd >= n - RSST_G);
      if (!hit) continue;
      int gp;
      double w[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) w[v] = u[v];
      if (p.bc[d] == RSST_BC_PERIODIC) {
        gp = side == 0 ? cd + n : cd - n;
      } else {
        gp = side == 0 ? -1 - cd : 2 * n - 1 - cd;
        w[1 + d] = -w[1 + d];
        if (bg != nullptr && d == p.vertical) {
          const double* rho0 = bg;
          const double* e0 = bg + bg_len;
          w[0] += rho0[gp + RSST_G] - rho0[cd + RSST_G];
          w[NV - 1] += e0[gp + RSST_G] - e0[cd + RSST_G];
        }
      }
      const int ii = d == 0 ? gp : i, jj = d == 1 ? gp : j, kk = d == 2 ? gp : k;
      const int64_t og = pidx(g, ii, jj, kk);
#pragma unroll
      for (int v = 0; v < NV; ++v) out[v * fs + og] = w[v];
    }
  }
}

// Store a perturbation-state cell and the edge ghost cells that wrap it or
// mirror it (normal momentum negated).  The perturbation about a background
// is mirrored without a background term: U1(ghost) = mirror(U1(image)).
template <typename T, int NV>
__device__ __forceinline__ void store_mirror_ghosts(T* __restrict__ out, const Geom& g, const Phys& p, int i, int j,
                                                    int k, const T (&u)[NV]) {
  constexpr int ND = NV - 2;
  const int64_t fs = g.fstride;
  const int64_t o = pidx(g, i, j, k);
#pragma unroll
  for (int v = 0; v < NV; ++v) out[v * fs + o] = u[v];
  const int c[3] = {i, j, k};
#pragma unroll
  for (int d = 0; d < ND; ++d) {
    const int n = g.n[d], cd = c[d];
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      const bool hit = side == 0 ? (cd < RSST_G) : (cd >= n - RSST_G);
      if (!hit) continue;
      const bool per = p.bc[d] == RSST_BC_PERIODIC;
      const int gp = per ? (side == 0 ? cd + n : cd - n) : (side == 0 ? -1 - cd : 2 * n - 1 - cd);
      const int ii = d == 0 ? gp : i, jj = d == 1 ? gp : j, kk = d == 2 ? gp : k;
      const int64_t og = pidx(g, ii, jj, kk);
#pragma unroll
      for (int v = 0; v < NV; ++v) out[v * fs + og] = (!per && v == 1 + d) ? -u[v] : u[v];
    }
  }
}

}  // namespace rsst
