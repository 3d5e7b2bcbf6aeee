// State transfer between the caller's layout [nvar][nz][ny][nx] (float64) and a
// run's padded storage, one kernel for every precision: a storage policy says
// how a cell is stored, read back and rated.
//
// What bounds it: at first the float64 pipe (conversions, and signs taken off or
// flipped by float64 operations: 10 warp instructions a float32 cell), a flat
// 64-bit index split per cell and a second pass for the CFL maximum; now the
// instructions of address arithmetic and conversions (60 % of issue), and in
// float64 runs the CFL rate on the float64 pipe.  Conversions run on the integer
// pipe, a thread takes one cell of a block shaped by the row, and the CFL maximum of the new
// state is taken from the values being packed.  Load (CFL included) / read-back,
// us: 4096^2 float32 535 / 313 -> 247 / 163, 3D 256 x 128 x 128 float32 194 / 116
// -> 93 / 72, float64 238 / 73 -> 144 / 67, 512^2 double-float 32 / 28 -> 16 / 25.
#pragma once

#include "rsst_common.cuh"
#include "rsst_internal.h"

namespace rsst {

struct XferGrid {
  dim3 grid, block;
};
// Blocks of 256 threads, one cell a thread: 32 x 8 (256-byte pieces of eight
// rows, so that a row of any length wastes less than one warp), for shorter
// rows the next power of two wide and the more rows (32 lanes to a row of two
// cells would idle), for fewer rows than eight wider (a line: 256 x 1).
static inline XferGrid xfer_grid(int cells_x, int64_t rows) {
  int bx = 32;
  while (bx > 2 && bx / 2 >= cells_x) bx /= 2;
  while (bx >= 32 && bx < 256 && 256 / bx > rows) bx *= 2;
  XferGrid x;
  x.block = dim3(bx, 256 / bx);
  const int64_t by = (rows + x.block.y - 1) / x.block.y;
  x.grid = dim3((cells_x + bx - 1) / bx, (unsigned)(by < RSST_GRID_Y ? by : RSST_GRID_Y));
  return x;
}

// Image of extended coordinate c of an axis (wrap, or mirror): the source
// coordinate, and whether it was mirrored.
__device__ __forceinline__ int image_of(int c, int n, int bc, bool& mirrored) {
  mirrored = false;
  if (c >= 0 && c < n) return c;
  if (bc == RSST_BC_PERIODIC) return (c + n) % n;
  mirrored = true;
  return c < 0 ? -1 - c : 2 * n - 1 - c;
}

// Policy S (NV fields):
//   store(offset, w, src_v, ghost_v): store the values w of a cell whose source
//     has vertical index src_v (-1: no vertical axis); ghost_v >= -RSST_G is the
//     extended vertical index if the cell mirrors across a wall of that axis,
//     else INT_MIN;
//   rate(w, src_v, ok): CFL rate of an interior cell, after store.
template <class S>
__global__ void __launch_bounds__(256) pack_kernel(const double* __restrict__ src, const Geom g, const Phys p,
                                                   const S st, double* cfl, unsigned int* flag) {
  constexpr int NV = S::NV, ND = NV - 2;
  __shared__ double sred[8];
  const int ex = g.n[0] + 2 * RSST_G, ey = ND >= 2 ? g.n[1] + 2 * RSST_G : 1, ez = ND >= 3 ? g.n[2] + 2 * RSST_G : 1;
  const int64_t rows = (int64_t)ey * ez;
  double rmax = 0.0;
  bool ok_all = true;
  const int tid = threadIdx.y * blockDim.x + threadIdx.x;
  // a maximum found by an earlier block (any age will do): read now, used at the end
  const long long seen = tid == 0 ? *reinterpret_cast<volatile long long*>(cfl) : 0;
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  if (x < ex) {
    int c[3] = {x - RSST_G, 0, 0}, s[3] = {0, 0, 0};
    bool m[3] = {false, false, false};
    s[0] = image_of(c[0], g.n[0], p.bc[0], m[0]);
    for (int64_t row = blockIdx.y * (int64_t)blockDim.y + threadIdx.y; row < rows; row += (int64_t)gridDim.y * blockDim.y) {
      if constexpr (ND >= 2) {
        const int k = ND >= 3 ? (int)(row / ey) : 0;
        c[1] = (int)(row - (int64_t)k * ey) - RSST_G;
        s[1] = image_of(c[1], g.n[1], p.bc[1], m[1]);
        if constexpr (ND >= 3) {
          c[2] = k - RSST_G;
          s[2] = image_of(c[2], g.n[2], p.bc[2], m[2]);
        }
      }
      const double* sp = src + ((int64_t)s[2] * g.n[1] + s[1]) * g.n[0] + s[0];
      double w[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) w[v] = sp[v * g.ncells];
#pragma unroll
      for (int e = 0; e < ND; ++e)
        if (m[e]) w[1 + e] = flip_sign(w[1 + e]);
      const bool v0 = p.vertical == 0, v1 = ND >= 2 && p.vertical == 1, v2 = ND >= 3 && p.vertical == 2;
      const int sv = v0 ? s[0] : (v1 ? s[1] : (v2 ? s[2] : -1));
      const bool vm = v0 ? m[0] : (v1 ? m[1] : (v2 ? m[2] : false));
      const int gv = vm ? (v0 ? c[0] : (v1 ? c[1] : c[2])) : INT_MIN;
      st.store(pidx(g, c[0], c[1], c[2]), w, sv, gv);
      if (s[0] == c[0] && s[1] == c[1] && s[2] == c[2]) {
        bool ok;
        const double r = st.rate(w, sv, ok);
        if (ok) rmax = max_nonneg(rmax, r);
        ok_all = ok_all && ok;
      }
    }
  }
  if (!ok_all) atomicOr(flag, RSST_FLAG_NONPHYSICAL);
  rmax = warp_max(rmax);
  if ((tid & 31) == 0) sred[tid >> 5] = rmax;
  __syncthreads();
  if (tid < 32) {
    const double r = warp_max(tid < 8 ? sred[tid] : 0.0);
    if (tid == 0 && __double_as_longlong(r) > seen)
      atomicMax(reinterpret_cast<unsigned long long*>(cfl), (unsigned long long)__double_as_longlong(r));
  }
}

// Policy S: load(offset, v, vertical index): field v of a stored interior cell.
template <class S>
__global__ void __launch_bounds__(256) unpack_kernel(double* __restrict__ dst, const Geom g, const int vertical,
                                                     const S st) {
  constexpr int NV = S::NV;
  const int64_t rows = (int64_t)g.n[1] * g.n[2];
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= g.n[0]) return;
  for (int64_t row = blockIdx.y * (int64_t)blockDim.y + threadIdx.y; row < rows; row += (int64_t)gridDim.y * blockDim.y) {
    const int k = (int)(row / g.n[1]), j = (int)(row - (int64_t)k * g.n[1]);
    const int64_t o = pidx(g, x, j, k);
    const int vi = vertical == 0 ? x : (vertical == 1 ? j : k);
    double w[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) w[v] = st.load(o, v, vi);
#pragma unroll
    for (int v = 0; v < NV; ++v) dst[v * g.ncells + row * g.n[0] + x] = w[v];
  }
}

template <class S>
static int launch_pack(const double* src, const Geom& g, const Phys& p, const S& st, double* cfl, unsigned int* flag,
                       const char* what, cudaStream_t s) {
  const XferGrid x = xfer_grid(g.n[0] + 2 * RSST_G, (int64_t)g.py * g.pz);
  pack_kernel<S><<<x.grid, x.block, 0, s>>>(src, g, p, st, cfl, flag);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    rsst_set_error("%s launch: %s", what, cudaGetErrorString(e));
    return RSST_ECUDA;
  }
  return RSST_OK;
}
template <class S>
static int launch_unpack(double* dst, const Geom& g, int vertical, const S& st, const char* what, cudaStream_t s) {
  const XferGrid x = xfer_grid(g.n[0], (int64_t)g.n[1] * g.n[2]);
  unpack_kernel<S><<<x.grid, x.block, 0, s>>>(dst, g, vertical, st);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    rsst_set_error("%s launch: %s", what, cudaGetErrorString(e));
    return RSST_ECUDA;
  }
  return RSST_OK;
}

}  // namespace rsst
