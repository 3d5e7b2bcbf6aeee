// Device helpers shared by the float64 and float32 kernels.
#pragma once

#include "rsst_internal.h"

namespace rsst {

// Padded-layout offset of interior cell (i, j, k) (ghosts at -2, -1, n, n+1).
__device__ __forceinline__ int64_t pidx(const Geom& g, int i, int j, int k) {
  return (int64_t)(k + g.gz) * g.plane + (int64_t)(j + g.gy) * g.pitch + (i + g.xoff);
}

// Conversions between float64 and float32 on the integer pipe: the conversion
// instructions run at the float64 pipe's rate (a warp instruction per 16 SM
// clocks), which bounds a kernel that only moves data.  The same values and
// rounding (to nearest even, subnormals included; a NaN becomes the quiet one).
// Signs are taken off the high word: a 64-bit mask or xor of the sign is turned
// back into a float64 absolute value or negation.
static __device__ __noinline__ unsigned d2f_rare(unsigned long long m) {  // not a normal float (out of line: it rarely runs)
  const int e = (int)(m >> 52);
  if (e > 1150) return m > 0x7ff0000000000000ull ? 0x7fc00000u : 0x7f800000u;
  // units of 2^-149: the significand shifted by 29 + (897 - e)
  const int sh = min(926 - e, 63);
  const unsigned long long q = (m & 0xfffffffffffffull) | (e > 0 ? 1ull << 52 : 0ull);
  return (unsigned)((q + ((1ull << (sh - 1)) - 1ull) + ((q >> sh) & 1ull)) >> sh);
}
__device__ __forceinline__ float d2f_rn(double d) {
  const unsigned hi = (unsigned)__double2hiint(d), s = hi & 0x80000000u;
  const unsigned long long m = ((unsigned long long)(hi ^ s) << 32) | (unsigned)__double2loint(d);
  const int e = (int)(m >> 52);
  // normal floats; a carry past the largest gives infinity
  unsigned f = (unsigned)((m + 0x0fffffffull + ((m >> 29) & 1ull)) >> 29) - (896u << 23);
  if ((unsigned)(e - 897) >= 254u) f = m == 0ull ? 0u : d2f_rare(m);
  return __uint_as_float(s | f);
}
__device__ __forceinline__ double f2d(float x) {
  const unsigned b = __float_as_uint(x);
  unsigned m = b & 0x7fffffffu;
  int bias = 896;
  if (m < 0x00800000u) {  // subnormal: normalise
    const int n = __clz(m) - 8;
    m = m == 0u ? 0u : m << n;
    bias = m == 0u ? 0 : 896 - n;
  } else if (m >= 0x7f800000u) {
    bias = 1792;  // exponent 255 -> 2047
  }
  const unsigned long long v = ((unsigned long long)m << 29) + ((unsigned long long)bias << 52);
  return __hiloint2double((int)((unsigned)(v >> 32) | (b & 0x80000000u)), (int)(unsigned)v);
}
__device__ __forceinline__ double flip_sign(double x) {
  return __hiloint2double(__double2hiint(x) ^ (int)0x80000000u, __double2loint(x));
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
