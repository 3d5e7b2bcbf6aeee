// 2D float32 perturbation tile routine (see rsst_fp32_2d.cu for the layout).
//
// The state is U = U0 + U1, U0 = (rho0, 0, 0, E0) a float64 background that
// varies along y only (or is absent), U1 the stored float32 perturbation.
// Every term that feeds an update is formed from perturbation-sized
// quantities (see rsst_math_fp32.cuh for the splitting).  A lane owns two
// neighbouring columns and works on them as pairs (rsst_fp32_pair.cuh):
//  - each cell's MC slope is computed once per axis, as a half slope h
//    (face states U +- h); along x a lane hands its right cell's right face
//    state to the next lane by a warp shuffle, along y the column march
//    carries it;
//  - faces hold twice the LLF flux, 2F = F(qL) + F(qR) - alpha (qR - qL),
//    and the exact 1/2 folds into 1/dx;
//  - the background enters through one table row per vertical index, each
//    value held twice so that a 16-byte load gives two pair operands.
#pragma once

#include "rsst_common.cuh"
#include "rsst_internal.h"
#include "rsst_fp32_lean.cuh"
#include "rsst_fp32_pair.cuh"
#include "rsst_math_fp32.cuh"
#include "rsst_tma.cuh"

namespace rsst {

// Tile geometry: BX_ x BY_ cells, each thread owning two columns of SEG_
// cells (BX_ * BY_ / (2 SEG_) threads).  Shared memory: the TMA box (halo
// tile, all fields), the x flux differences, the background rows, a barrier,
// dt, reduction.
template <int BX_, int BY_, int SEG_>
struct T2Cfg {
  static constexpr int NV = 4, BX = BX_, BY = BY_, SEG = SEG_;
  static constexpr int PX = BX / 2;    // pairs of columns per row
  static constexpr int NT = PX * (BY / SEG);
  static constexpr int SXP = BX + 8;   // TMA box width: 4 columns each side (3 used), 16-byte aligned origin
  static constexpr int SYP = BY + 4;   // halo rows
  static constexpr int XO = 4;         // smem column of tile x = 0
  static constexpr int U_FLOATS = NV * SYP * SXP;
  static constexpr int DX_FLOATS = NV * BY * BX;
  static constexpr int TR2 = 2 * TR_W;  // floats of a doubled table row
  static constexpr int TAB_FLOATS = TR2 * SYP;
  static constexpr size_t SCRATCH = (size_t)(U_FLOATS + DX_FLOATS + TAB_FLOATS) * 4;
  // A warp owns the cells its lanes march up: WX pairs of columns by WY rows
  // (64 x SEG cells; 32 x 2 SEG for BX = 32).  Its x pass takes the column
  // pairs -1 .. WX of those rows as one flat list, 32 at a time, chunks
  // starting every 30 (the first and the last lane only serve their
  // neighbours), so no warp waits for another between the passes.
  static constexpr int WX = PX < 32 ? PX : 32, WY = SEG * (32 / WX);
  static constexpr int PW = WX + 2;
  static constexpr int NPAIR = PW * WY;
  static constexpr int NCHUNK = (NPAIR - 2 + 29) / 30;
  static constexpr uint32_t BOX_BYTES = U_FLOATS * 4;
  static constexpr size_t smem_bytes() { return SCRATCH + 16 + 8 * 8 + 512 + 128; }
  static_assert(BY % SEG == 0, "column segments must tile BY");
  static_assert(PX % 32 == 0 || 32 % PX == 0, "a warp's columns");
  static_assert((U_FLOATS + DX_FLOATS) % 4 == 0, "the table rows start on a 16-byte boundary");
  static_assert(NT % 32 == 0, "whole warps");
  static_assert(SCRATCH % 8 == 0, "the barriers after the scratch area need 8-byte alignment");
  static_assert(SXP <= 256 && SYP <= 256, "TMA box dimensions are at most 256");
};

// Single-run tile: 128 x 8 with two 4-cell segments, so that four CTAs of four
// warps fit an SM (46.5 KB each).
using T2 = T2Cfg<128, 8, 4>;

template <class C>
__device__ __forceinline__ uint64_t* t2_barrier(unsigned char* smem) {
  return reinterpret_cast<uint64_t*>(smem + C::SCRATCH);
}
template <class C>
__device__ __forceinline__ double* t2_sred(unsigned char* smem) {
  return reinterpret_cast<double*>(smem + C::SCRATCH + 16);
}
// free shared memory after the reduction slots (used by the batched kernel)
template <class C>
__device__ __forceinline__ unsigned char* t2_extra(unsigned char* smem) {
  return smem + C::SCRATCH + 16 + 8 * 8;
}
// barrier of the failure-detection test wait (after the batched kernel's 512 bytes)
template <class C>
__device__ __forceinline__ uint64_t* t2_stall_barrier(unsigned char* smem) {
  return reinterpret_cast<uint64_t*>(smem + C::SCRATCH + 16 + 8 * 8 + 512);
}

// Everything one tile needs about its run.
struct TileRun {
  Geom g;
  Phys p;
  PhysF pf;
  const float* base;
  float* out;
  const float* tabr;  // row-major background table, or null (no background)
  int tab_len;
  unsigned int* flag;
  int stage;
  int64_t stall_ns;  // > 0 only in failure-detection tests (see tile2d_f)
};

// Process tile (tx, ty) of run r: returns false if a bounded wait gave up
// (flag set, nothing left in flight).  Accumulates the stage-2 CFL rate
// maximum and physical check.  The caller initialised the barrier; `phase` is
// its current parity.  *sdt (shared memory) may be written up to the routine's
// first barriers: the tile's copy does not wait for dt's float64 division.
// FORM (-1: read from the run), the C_max law and the stage are compile-time.
template <class T2, int VERT, int FORM, bool CM, int ST>
__device__ __forceinline__ bool tile2d_f(const CUtensorMap* tin, const TileRun& r, const float* sdt, int tx, int ty,
                                         unsigned char* smem, uint32_t& phase, float& rmax, bool& ok_all) {
  constexpr int NV = 4;
  constexpr bool BG = VERT >= 0;
  constexpr int PL = T2::SYP * T2::SXP;  // floats per field in the box
  float* sU = reinterpret_cast<float*>(smem);
  float* sDx = sU + T2::U_FLOATS;   // [NV][BY][BX]: twice the x flux above minus below each cell
  float* st = sDx + T2::DX_FLOATS;  // doubled table rows of padded y j0 .. j0 + SYP - 1
  uint64_t* bar = t2_barrier<T2>(smem);
  const Geom& g = r.g;
  const PhysF& pf = r.pf;
  const int i0 = tx * T2::BX, j0 = ty * T2::BY;
  const int tid = threadIdx.x;

  __syncthreads();  // previous tile's shared-memory reads are done
  if (tid == 0) {
    fence_proxy_async_smem();
    mbar_expect_tx(bar, T2::BOX_BYTES);
    tma_load_3d(sU, tin, bar, i0 + g.xoff - T2::XO, j0, 0);
  }
  if constexpr (BG) {
    // SYP consecutive table rows, every value twice
    const float2* src = reinterpret_cast<const float2*>(r.tabr);
    float4* dst = reinterpret_cast<float4*>(st);
    constexpr int N2 = TR_W * T2::SYP / 2;
    const int first = j0 * (TR_W / 2), last = r.tab_len * (TR_W / 2);
    for (int id = tid; id < N2; id += T2::NT) {
      const float2 q = first + id < last ? src[first + id] : make_float2(0.0f, 0.0f);
      dst[id] = make_float4(q.x, q.x, q.y, q.y);
    }
  }
  // the give-up decision is taken by the whole block (no thread may leave
  // while others wait at a barrier); a late copy gets one more bounded wait
  if (__syncthreads_or(!mbar_wait_bounded(bar, phase))) {
    if (tid == 0) atomicOr(r.flag, RSST_FLAG_TIMEOUT);
    mbar_wait_bounded(bar, phase);
    return false;
  }
  phase ^= 1u;
  if (r.stall_ns > 0) {
    // Failure-detection test: with the tile's copy landed (nothing in
    // flight), wait on a barrier that expects 16 bytes no copy delivers, so
    // the bounded wait runs out and the give-up path is taken.
    uint64_t* sb = t2_stall_barrier<T2>(smem);
    if (tid == 0) {
      mbar_init(sb, 1);
      fence_mbar_init();
      mbar_expect_tx(sb, 16);
    }
    __syncthreads();
    if (__syncthreads_or(!mbar_wait_bounded(sb, 0u, (uint64_t)r.stall_ns))) {
      if (tid == 0) atomicOr(r.flag, RSST_FLAG_TIMEOUT);
      return false;
    }
  }

  const float dt = *sdt;
  const int nx = g.n[0], ny = g.n[1];
  const int lane = tid & 31;
  const PhysF2 p2 = make_pf2(pf);
  // ---- x pass.  Lane l of chunk k holds the column pair A, A + 1 numbered
  // 30k + l of the flat list.  It takes both cells' half slopes (four loads
  // and three differences a field), and as one pair the face on A's left
  // (with the state B + h_B passed one lane up) and the face between its
  // cells; the face on its right comes from the next lane.  Lanes 1 .. 30
  // store the two cells' flux differences; faces across rows reach none.
  {
    const int wc = 2 * ((tid & ~31) % T2::PX), wr = (tid & ~31) / T2::PX * T2::SEG;  // my warp's first column and row
#pragma unroll 1
    for (int k = 0; k < T2::NCHUNK; ++k) {
      int P = 30 * k + lane;
      const bool inb = P < T2::NPAIR;
      P = inb ? P : T2::NPAIR - 1;  // keeps the loads inside the box
      const int row = wr + P / T2::PW;
      const int j = P % T2::PW;
      const int ca = wc + 2 * j - 2;  // tile column of A
      const int sr = row + 2;
      const float* ur = sU + sr * T2::SXP + T2::XO + ca;
      f2 qL[NV], qR[NV], G[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const float* uv = ur + v * PL;
        const float am = uv[-1], bp = uv[2];
        const float2 ab = *reinterpret_cast<const float2*>(uv);
        const float d1 = ab.x - am, d2 = ab.y - ab.x, d3 = bp - ab.y;
        const f2 u = mk2(ab.x, ab.y), h = half_mc2(mk2(d1, d2), mk2(d2, d3));
        const f2 up = u + h;
        qR[v] = u - h;
        qL[v] = mk2(__shfl_up_sync(0xffffffffu, hi2(up), 1), lo2(up));
      }
      face_flat2<NV, 0, BG, CM>(qL, qR, st + sr * T2::TR2, p2, G);
      const bool put = inb && lane >= 1 && lane <= 30 && j >= 1 && j <= T2::WX;
      float* dx = sDx + row * T2::BX + ca;
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const float f0 = lo2(G[v]), f1 = hi2(G[v]), fr = __shfl_down_sync(0xffffffffu, f0, 1);
        if (put) *reinterpret_cast<float2*>(dx + v * T2::BY * T2::BX) = make_float2(f1 - f0, fr - f1);
      }
    }
  }
  __syncwarp();

  // ---- column march with the fused epilogue: each thread owns tile columns
  // col, col + 1, rows jb .. jb + SEG - 1; a register window carries the cell
  // states, the y half slope and the lower face's flux.
  const int col = 2 * (tid % T2::PX);
  const int jb = (tid / T2::PX) * T2::SEG;
  const int x = i0 + col;
  if (x < nx && j0 + jb < ny) {
    const bool two = x + 1 < nx;  // an odd grid's last column stands alone
    const float* uc = sU + T2::XO + col;
    auto ld = [&](int srow, f2 (&u)[NV]) {
#pragma unroll
      for (int v = 0; v < NV; ++v)
        u[v].v = *reinterpret_cast<const unsigned long long*>(uc + v * PL + srow * T2::SXP);
    };
    f2 u0[NV], u1[NV], h0[NV], Fm[NV];
    {
      f2 umm[NV], um[NV], hm[NV], da[NV], db[NV], dc[NV];
      // cells jb-2 .. jb+1 live at smem rows jb .. jb+3
      ld(jb, umm);
      ld(jb + 1, um);
      ld(jb + 2, u0);
      ld(jb + 3, u1);
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        da[v] = um[v] - umm[v];
        db[v] = u0[v] - um[v];
        dc[v] = u1[v] - u0[v];
      }
      vslope2<NV, BG>(da, db, st + (jb + 1) * T2::TR2, hm);  // cell jb-1
      vslope2<NV, BG>(db, dc, st + (jb + 2) * T2::TR2, h0);  // cell jb
      f2 qL[NV], qR[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        qL[v] = um[v] + hm[v];
        qR[v] = u0[v] - h0[v];
      }
      face_vert2<NV, 1, BG, CM>(qL, qR, st + (jb + 2) * T2::TR2, p2, Fm);
    }
    const f2 nidx = dup2(-0.5f * pf.inv_dx[0]), nidy = dup2(-0.5f * pf.inv_dx[1]);  // the faces hold 2F
    const f2 dt2 = dup2(dt);
    const int64_t fs = g.fstride;
    const bool xghost = x < RSST_G || x + 1 >= nx - RSST_G;
    const int64_t o0 = pidx(g, x, j0 + jb, 0);
    // stage 2: U^n of the next row's cells is loaded one row ahead, so its
    // global-memory latency overlaps a row of arithmetic
    f2 bnext[NV] = {};
    if constexpr (ST == 2) {
#pragma unroll
      for (int v = 0; v < NV; ++v) bnext[v].v = *reinterpret_cast<const unsigned long long*>(r.base + v * fs + o0);
    }
#pragma unroll 1
    for (int jj = 0; jj < T2::SEG; ++jj) {
      const int j = jb + jj;  // tile row of the cells
      if (j0 + j >= ny) break;
      f2 bv[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) bv[v] = bnext[v];
      if (ST == 2 && jj + 1 < T2::SEG && j0 + j + 1 < ny) {
        const int64_t on = o0 + (int64_t)(jj + 1) * g.pitch;
#pragma unroll
        for (int v = 0; v < NV; ++v) bnext[v].v = *reinterpret_cast<const unsigned long long*>(r.base + v * fs + on);
      }
      const int sr = j + 2;  // their smem row
      f2 u2[NV], h1[NV], Fp[NV];
      ld(j + 4, u2);  // cells j+2
      {
        f2 da[NV], db[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          da[v] = u1[v] - u0[v];
          db[v] = u2[v] - u1[v];
        }
        vslope2<NV, BG>(da, db, st + (j + 3) * T2::TR2, h1);  // cells j+1
      }
      {
        f2 qL[NV], qR[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          qL[v] = u0[v] + h0[v];
          qR[v] = u1[v] - h1[v];
        }
        face_vert2<NV, 1, BG, CM>(qL, qR, st + (j + 3) * T2::TR2, p2, Fp);
      }
      f2 L[NV], Dl[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        f2 dx;
        dx.v = *reinterpret_cast<const unsigned long long*>(sDx + (v * T2::BY + j) * T2::BX + col);
        L[v] = fma2(Fp[v] - Fm[v], nidy, dx * nidx);
      }
      f2 rho0 = {}, P0 = {};
      if constexpr (BG) {
        const float* tr = st + sr * T2::TR2;
        const f2x2 cb = tab2(tr, TR_RHO0), r01 = tab2(tr, TR_R0), r23 = tab2(tr, TR_R0 + 2);
        const f2x2 x0 = tab2(tr, TR_R0 + 4), x1 = tab2(tr, TR_R0 + 6);  // R0[4] (unused in 2D), D0 rho; mv, E
        rho0 = cb.a;
        P0 = cb.b;
        Dl[0] = L[0] + x0.b;
        Dl[1] = L[1];
        Dl[2] = L[2] + x1.a;
        Dl[3] = L[3] + x1.b;
        L[0] = L[0] + r01.a;
        L[1] = L[1] + r01.b;
        L[2] = L[2] + r23.a;
        L[3] = L[3] + r23.b;
      } else {
#pragma unroll
        for (int v = 0; v < NV; ++v) Dl[v] = L[v];
      }
      const int y = j0 + j;
      const int64_t o = o0 + (int64_t)jj * g.pitch;
      f2 u[NV], rate;
      bool ok[2];
      cell_lean2<NV, FORM, CM, ST>(u0, L, Dl, rho0, P0, pf, p2, r.p.variant, r.p.has_grav != 0, dt2, bv, u, rate, ok);
      if constexpr (ST == 2) {
        rmax = ok[0] ? fmaxf(rmax, lo2(rate)) : rmax;
        rmax = two && ok[1] ? fmaxf(rmax, hi2(rate)) : rmax;
        ok_all = ok_all && ok[0] && (ok[1] || !two);
      }
      if (two) {
#pragma unroll
        for (int v = 0; v < NV; ++v) *reinterpret_cast<unsigned long long*>(r.out + v * fs + o) = u[v].v;
      } else {
#pragma unroll
        for (int v = 0; v < NV; ++v) r.out[v * fs + o] = lo2(u[v]);
      }
      if (xghost || y < RSST_G || y >= ny - RSST_G) {
        float ua[NV], ub[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          ua[v] = lo2(u[v]);
          ub[v] = hi2(u[v]);
        }
        store_mirror_ghosts<float, 4>(r.out, g, r.p, x, y, 0, ua);
        if (two) store_mirror_ghosts<float, 4>(r.out, g, r.p, x + 1, y, 0, ub);
      }
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        u0[v] = u1[v];
        u1[v] = u2[v];
        h0[v] = h1[v];
        Fm[v] = Fp[v];
      }
    }
  }
  return true;
}

}  // namespace rsst
