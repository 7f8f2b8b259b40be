// One fused kernel per third-order TVD Runge-Kutta stage of the 2D hybrid
// HWENO scheme (Zhao & Qiu, arXiv:2002.08816, Sec. 2.2).
//
// A CTA owns a TX x TY tile of cells.  It stages the tile and a 3-cell halo
// of the stage input in shared memory, then, on chip:
//   1. alpha_x, alpha_y from the slots the producer of the stage input left
//      (global Lax-Friedrichs fluxes); stage 1 turns them into
//      dt = CFL / (alpha_x/dx + alpha_y/dy), clipped to t_final;
//   2. Step 4 for the tile and 2 halo cells: KXRCF flags (FP32 kernels decide
//      in FP32 when the rounding-error bound allows, else with float pairs;
//      a replayed stage of the adjoint takes its recorded flags) and the
//      first moments of troubled cells modified dimension by dimension with
//      the 1D Step 1 formula (Euler: characteristic fields of the x- and of
//      the y-Jacobian at the cell average), written back into the tile once
//      every flag and limiter has read the raw ones;
//   3. Step 5.1/5.2 at the interface Gauss points of the tile's cells and of
//      the one-cell cross halo: linear p0 (the quartic on the 3x3 stencil),
//      or HWENO when the 3x3 stencil holds a troubled cell (Euler: x-faces in
//      the x characteristic fields, y-faces in the y fields);
//   4. own cells: Step 5.3 at the interior Gauss points, Lax-Friedrichs
//      fluxes at the 4 ng interface points, Eq. (ode2) and Eq. (RK);
//   5. the tile's wave-speed maxima (x and y) into the slots for the next
//      stage, the troubled count and the status bits.
// The reconstruction arithmetic is generated straight-line code (square cells):
// the linear p0 by parity classes (hweno2d_sym.cuh, which gives what that
// saves), the HWENO candidates and smoothness indicators of
// hweno2d_coef.cuh; the FP32 Euler kernel runs it, the fluxes
// and the HWENO helpers on pairs (two components, two points or two
// characteristic fields) in packed FP32 (fma.rn.f32x2).
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include "hweno1d_fields.cuh"
#include "hweno1d_recon.cuh"
#include "hweno2d_common.cuh"
#include "hweno_device.cuh"
#include "hweno.h"
#include "hweno_internal.h"

namespace hw {
namespace {

// Cells per CTA: 32 in x (a warp per row), TY rows of the stage kernel (8 or 4,
// stage2d_rows), TYW of the wave-speed kernels.
constexpr int TX = 32, TYW = 8;
constexpr int NTW = TX * TYW, NWW = NTW / 32;
// raw tile: a 3-cell halo, and in x one more column on the left so that the
// tile's first column bx0 - 4 is 16-byte aligned (TMA); own-tile cell (ci, cj)
// is raw (ci + OXR, cj + OYR)
constexpr int RX = TX + 8;
constexpr int OXR = 4, OYR = 3;
constexpr int LX = TX + 4;                // flags and modified moments, 2-cell halo
constexpr unsigned kTmaPolls = 1u << 20;  // mbarrier polls before a tile copy is given up

template <typename R, int C, int NG, bool COMP, int TY, bool SPLIT>
struct Smem2D {
  static constexpr int NT = TX * TY * (SPLIT ? 2 : 1), NW = NT / 32, RY = TY + 6, LY = TY + 4;
  static constexpr int kPadX = 1;  // raw index of flag-grid column lx: lx + 2
  // stage input (the TMA box); after Step 4 its first moments are the
  // modified ones
  alignas(128) R u[C][3][RY][RX];
  // HWENO_FP32C: the low parts of the stage input's averages (a second box)
  alignas(128) R ulo[COMP ? C : 1][COMP ? RY : 1][COMP ? RX : 1];
  union {
    R xf[C][2 * NG][TY][TX + 2];  // x-face values (left NG, right NG) of cells -1..TX
    R lim[C == 4 ? LX * LY : 1][C][2];  // Step 4, Euler: modified x-, y-moments by list slot (into u once all have read it)
  };
  R yf[C][2 * NG][TY + 2][TX];  // y-face values (bottom NG, top NG) of cells -1..TY
  R half[SPLIT ? 5 * C : 1][SPLIT ? TX * TY : 1];  // the second thread's sums (SPLIT)
  uint8_t fl[LY][LX];
  R red[2][NW];
  int cnt[NW];
  R amax[2][NW];
  unsigned long long bar;                        // mbarrier of the tile copy
  int ntb, nhw;                                  // lengths of the two work lists
  unsigned short tbl[LX * LY];                   // troubled cells (Euler limiter)
  unsigned short hwl[TX * TY + 2 * TX + 2 * TY]; // interface items with HWENO
};

// --------------------------------------------------------- KXRCF (2D)
// Reading: I = |dy jx + dx jy| / (h (dx + dy) max(|u0|, 1e-12)), h =
// sqrt(dx^2 + dy^2)/2, jx / jy the degree-1 trace jumps across the inflow x-
// and y-faces (left / bottom when the velocity component is >= 0).

__device__ __forceinline__ double jump64(double u0, double v0, double unb, double vnb, bool low) {
  return low ? __dsub_rn(__dsub_rn(u0, __dmul_rn(6.0, v0)), __dadd_rn(unb, __dmul_rn(6.0, vnb)))
             : __dsub_rn(__dadd_rn(u0, __dmul_rn(6.0, v0)), __dsub_rn(unb, __dmul_rn(6.0, vnb)));
}

// u0/v0/w0 the cell, (uxn, vxn) its inflow x-neighbour, (uyn, wyn) its inflow
// y-neighbour; lowx / lowy: the inflow faces are the left / bottom ones.
// FP32 data: decide in FP32 when the rounding-error bound allows, else with
// float pairs (no FP64 on the FP32 kernel's path): the two jumps as exact-to-
// ~2^-46 pairs (jump_pair), num = dy jx + dx jy from pair products (fma gives
// each product's rounding error; dx and dy carry their own low parts), and the
// threshold thr den_h max(|u0|, 1e-12) as a pair; the sign of |num| - r is then
// that of the exact values unless they agree to ~1e-13 of dy S_x + dx S_y,
// far inside the 1e-6 band around the threshold.
__device__ __forceinline__ bool kxrcf2_troubled(float u0, float v0, float w0, float uxn, float vxn,
                                                float uyn, float wyn, bool lowx, bool lowy,
                                                const Kx2& k) {
  const float jx = lowx ? (u0 - 6.0f * v0) - (uxn + 6.0f * vxn) : (u0 + 6.0f * v0) - (uxn - 6.0f * vxn);
  const float jy = lowy ? (u0 - 6.0f * w0) - (uyn + 6.0f * wyn) : (u0 + 6.0f * w0) - (uyn - 6.0f * wyn);
  const float sx = fabsf(u0) + 6.0f * fabsf(v0) + fabsf(uxn) + 6.0f * fabsf(vxn);
  const float sy = fabsf(u0) + 6.0f * fabsf(w0) + fabsf(uyn) + 6.0f * fabsf(wyn);
  const float num = fabsf(k.fdy * jx + k.fdx * jy);
  // |num - exact| <= 2^-24 (3 dy sx + 3 dx sy + 3 |num|) to first order
  const float e = 1.0e-6f * (k.fdy * sx + k.fdx * sy);
  const float nrm = fmaxf(fabsf(u0), 1e-12f);
  const float r = k.fthr_den * nrm;
  if (num - e > r * (1.0f + 4.8e-7f)) return true;
  if (num + e < r * (1.0f - 4.8e-7f)) return false;
  float jxh, jxl, jyh, jyl;
  jump_pair(u0, v0, uxn, vxn, lowx, jxh, jxl);
  jump_pair(u0, w0, uyn, wyn, lowy, jyh, jyl);
  const float p1h = __fmul_rn(k.fdy, jxh);
  const float p1l = __fadd_rn(fmaf(k.fdy, jxh, -p1h),
                              __fadd_rn(__fmul_rn(k.fdy, jxl), __fmul_rn(k.fdy_lo, jxh)));
  const float p2h = __fmul_rn(k.fdx, jyh);
  const float p2l = __fadd_rn(fmaf(k.fdx, jyh, -p2h),
                              __fadd_rn(__fmul_rn(k.fdx, jyl), __fmul_rn(k.fdx_lo, jyh)));
  float nh, nl, t;
  two_sum(p1h, p2h, nh, t);
  two_sum(nh, __fadd_rn(t, __fadd_rn(p1l, p2l)), nh, nl);
  if (nh < 0.0f) {
    nh = -nh;
    nl = -nl;
  }
  const float rh = __fmul_rn(nrm, k.fthr_den);
  const float rl = __fadd_rn(fmaf(nrm, k.fthr_den, -rh), __fmul_rn(nrm, k.fthr_den_lo));
  return __fadd_rn(__fsub_rn(nh, rh), __fsub_rn(nl, rl)) > 0.0f;
}

// FP64 data: the decision of the reading, |dy jx + dx jy| / (den_h nrm) >
// thr, in its divide-free product form (it differs from the quotient form only
// within a few ulp of the threshold).
__device__ __forceinline__ bool kxrcf2_troubled(double u0, double v0, double w0, double uxn,
                                                double vxn, double uyn, double wyn, bool lowx,
                                                bool lowy, const Kx2& k) {
  {
    // decided in FP32 on the truncated data where the error bound allows (no FP64
    // instruction): as the FP32 form above, with the truncations' 2^-23 added
    const float fu = trunc32(u0), fv = trunc32(v0), fw = trunc32(w0);
    const float gx = trunc32(uxn), gvx = trunc32(vxn), gy = trunc32(uyn), gwy = trunc32(wyn);
    const float sx6 = lowx ? -6.0f : 6.0f, sy6 = lowy ? -6.0f : 6.0f;
    const float jxf = fmaf(sx6, fv, fu) - fmaf(-sx6, gvx, gx);
    const float jyf = fmaf(sy6, fw, fu) - fmaf(-sy6, gwy, gy);
    const float sx = fabsf(fu) + 6.0f * fabsf(fv) + fabsf(gx) + 6.0f * fabsf(gvx);
    const float sy = fabsf(fu) + 6.0f * fabsf(fw) + fabsf(gy) + 6.0f * fabsf(gwy);
    const float numf = fabsf(k.fdy * jxf + k.fdx * jyf);
    const float e = 1.3e-6f * (k.fdy * sx + k.fdx * sy) + 1e-28f;
    const float r = k.fthr_den * fmaxf(fabsf(fu), 1e-12f);
    if (numf - e > r * (1.0f + 8.0e-7f)) return true;   // (NaN decides nothing)
    if (numf + e < r * (1.0f - 8.0e-7f)) return false;
  }
  const double jx = jump64(u0, v0, uxn, vxn, lowx);
  const double jy = jump64(u0, w0, uyn, wyn, lowy);
  const double num = __dadd_rn(__dmul_rn(k.dy, jx), __dmul_rn(k.dx, jy));
  const double nrm = fmax(fabs(u0), 1e-12);
  return fabs(num) > __dmul_rn(k.thr, __dmul_rn(k.den_h, nrm));
}

// Float-pair averages (HWENO_FP32C: u0 + l0, uxn + lxn, uyn + lyn), in three
// tiers: the FP32 fast test on hi (its margins exceed what the low parts can
// change, below 2^-24 of the averages); where it cannot decide, the float-pair
// form of the FP32 kernel with the low parts added in (jump_pair_lo; the norm
// |u0 + l0| as a pair), decided when the difference clears 1e-12 (dy S_x + dx
// S_y + r), far above its rounding bound; and only inside that margin the FP64
// form on hi + lo.  The decision is the oracle's on the same state except
// within a few FP64 ulp of the threshold.
__device__ __forceinline__ bool kxrcf2_troubled_pair(float u0, float l0, float v0, float w0,
                                                     float uxn, float lxn, float vxn, float uyn,
                                                     float lyn, float wyn, bool lowx, bool lowy,
                                                     const Kx2& k) {
  const float jx = lowx ? (u0 - 6.0f * v0) - (uxn + 6.0f * vxn) : (u0 + 6.0f * v0) - (uxn - 6.0f * vxn);
  const float jy = lowy ? (u0 - 6.0f * w0) - (uyn + 6.0f * wyn) : (u0 + 6.0f * w0) - (uyn - 6.0f * wyn);
  const float sx = fabsf(u0) + 6.0f * fabsf(v0) + fabsf(uxn) + 6.0f * fabsf(vxn);
  const float sy = fabsf(u0) + 6.0f * fabsf(w0) + fabsf(uyn) + 6.0f * fabsf(wyn);
  const float num = fabsf(k.fdy * jx + k.fdx * jy);
  const float e = 1.0e-6f * (k.fdy * sx + k.fdx * sy);
  const float r = k.fthr_den * fmaxf(fabsf(u0), 1e-12f);
  if (num - e > r * (1.0f + 4.8e-7f)) return true;
  if (num + e < r * (1.0f - 4.8e-7f)) return false;
  float jxh, jxl, jyh, jyl;
  jump_pair_lo(u0, l0, v0, uxn, lxn, vxn, lowx, jxh, jxl);
  jump_pair_lo(u0, l0, w0, uyn, lyn, wyn, lowy, jyh, jyl);
  const float p1h = __fmul_rn(k.fdy, jxh);
  const float p1l = __fadd_rn(fmaf(k.fdy, jxh, -p1h),
                              __fadd_rn(__fmul_rn(k.fdy, jxl), __fmul_rn(k.fdy_lo, jxh)));
  const float p2h = __fmul_rn(k.fdx, jyh);
  const float p2l = __fadd_rn(fmaf(k.fdx, jyh, -p2h),
                              __fadd_rn(__fmul_rn(k.fdx, jyl), __fmul_rn(k.fdx_lo, jyh)));
  float mh, ml, t;
  two_sum(p1h, p2h, mh, t);
  two_sum(mh, __fadd_rn(t, __fadd_rn(p1l, p2l)), mh, ml);
  if (mh < 0.0f) {
    mh = -mh;
    ml = -ml;
  }
  float nh = fabsf(u0), nl = u0 < 0.0f ? -l0 : l0;
  if (nh < 1e-12f) {
    nh = 1e-12f;
    nl = 0.0f;
  }
  const float rh = __fmul_rn(nh, k.fthr_den);
  const float rl = __fadd_rn(fmaf(nh, k.fthr_den, -rh),
                             __fadd_rn(__fmul_rn(nh, k.fthr_den_lo), __fmul_rn(nl, k.fthr_den)));
  const float d = __fadd_rn(__fsub_rn(mh, rh), __fsub_rn(ml, rl));
  if (fabsf(d) > 1e-12f * (k.fdy * sx + k.fdx * sy + r)) return d > 0.0f;
  return kxrcf2_troubled((double)u0 + (double)l0, (double)v0, (double)w0, (double)uxn + (double)lxn,
                         (double)vxn, (double)uyn + (double)lyn, (double)wyn, lowx, lowy, k);
}

// The 19 data of component c of the cell at own-tile coordinates (ci, cj):
// ubar of cells 1..9, vbar and wbar (modified: read after Step 4) of cells
// 2, 4, 5, 6, 8.
template <typename S, typename R>
__device__ __forceinline__ void gather19(const S& sm, int c, int ci, int cj, R* d) {
#pragma unroll
  for (int k = 0; k < 9; ++k) d[k] = sm.u[c][0][cj + OYR + k / 3 - 1][ci + OXR + k % 3 - 1];
  const int mx[5] = {0, -1, 0, 1, 0}, my[5] = {-1, 0, 0, 0, 1};
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    d[9 + k] = sm.u[c][1][cj + OYR + my[k]][ci + OXR + mx[k]];
    d[14 + k] = sm.u[c][2][cj + OYR + my[k]][ci + OXR + mx[k]];
  }
}

// The 19 data as gather19 gives them, or (COMP: the float-pair averages of
// HWENO_FP32C) with the 9 averages as increments over the cell's own hi, low
// parts included: the p0 and HWENO maps are consistent (their average
// coefficients sum to one, their smoothness indicators are differences), so
// they map these increments to the point values' increments over hi.
template <bool COMP, typename S, typename R>
__device__ __forceinline__ void gather_data(const S& sm, int c, int ci, int cj, R* d) {
  gather19(sm, c, ci, cj, d);
  if constexpr (COMP) {
    const R b = d[4];
#pragma unroll
    for (int k = 0; k < 9; ++k)
      d[k] = __fadd_rn(__fsub_rn(d[k], b), sm.ulo[c][cj + OYR + k / 3 - 1][ci + OXR + k % 3 - 1]);
  }
}

// Value v of point p (order of hweno2d_coef.cuh) of component c of the cell at
// own-tile coordinates (ci, cj) into the face arrays.
template <typename S, typename R>
__device__ __forceinline__ void store_point(S& sm, int c, int p, int ci, int cj, R v) {
  constexpr int NG2 = sizeof(sm.xf[0]) / sizeof(sm.xf[0][0]);  // 2 NG
  if (p < NG2)
    sm.xf[c][p][cj][ci + 1] = v;        // left and right faces
  else
    sm.yf[c][p - NG2][cj + 1][ci] = v;  // bottom and top faces
}

template <typename S>
__device__ __forceinline__ void store_points(S& sm, int c, int p, int ci, int cj, float2 v) {
  store_point(sm, c, p, ci, cj, v.x);
  store_point(sm, c + 1, p, ci, cj, v.y);
}
template <typename S, typename R>
__device__ __forceinline__ void store_points(S& sm, int c, int p, int ci, int cj, R v) {
  store_point(sm, c, p, ci, cj, v);
}

// What the linear maps take per step: two FP32 components, or one value.
template <typename R, bool PACKED>
struct PairOf { typedef R type; };
template <>
struct PairOf<float, true> { typedef float2 type; };

// The parity classes (hw2::p0_classes) of component c of the cell at own-tile
// coordinates (ci, cj), PACKED: of components c and c + 1.
template <bool COMP, bool PACKED, typename S, typename T>
__device__ __forceinline__ void classes_of(const S& sm, int c, int ci, int cj, T* s) {
  if constexpr (PACKED) {
    float da[19], db[19];
    gather_data<COMP>(sm, c, ci, cj, da);
    gather_data<COMP>(sm, c + 1, ci, cj, db);
    float2 d[19];
#pragma unroll
    for (int k = 0; k < 19; ++k) d[k] = make_float2(da[k], db[k]);
    hw2::p0_classes(d, s);
  } else {
    T d[19];
    gather_data<COMP>(sm, c, ci, cj, d);
    hw2::p0_classes(d, s);
  }
}

// Step 5.1 for the n listed Euler items, cells whose 3x3 stencil holds a troubled
// cell: the interface points by HWENO in the x (x-faces) and y (y-faces)
// characteristic fields of the cell average (Remark 4; mean_eigen: of the mean of
// the two cells at each face).  (item, field) on four consecutive lanes, the two
// directions on different warps.  An item as one thread is one chain of 2
// directions x 4 fields, a tile's few items one warp while the rest of the SM
// waits: in FP64, where a warp instruction takes a sub-partition 64 cycles however
// few lanes work, ~6000 such instructions against ~550 for a task; in FP32 the
// eigen-system and the point values of all fields also cost the kernel its
// registers (108 bytes of spills and 1 KB of stack, none now).  FP32, an item per
// thread -> this: 512 x 512 quadrants, 3 points, 12 steps 2.66 -> 1.38 ms; 1024 x
// 1024 quadrants, 2 points, 12 steps 5.77 -> 3.21; 4096 x 4096 smooth, 2 points, 4
// steps 14.7 -> 13.6; 2048 x 2048 smooth, 3 points 5.56 -> 5.07.
template <int NG, int NT, bool COMP, typename R, typename S, typename F>
__device__ __noinline__ void hweno_tasks_euler2d(S& sm, int n, F item_of, R g0, R g1, R g2,
                                                 R g3, R g4, R eps, R gas,
                                                 bool mean_eigen) {
  const R gam[5] = {g0, g1, g2, g3, g4};
  const int lane = threadIdx.x & 31, f = lane & 3, base = lane & ~3;
  const int dir = (threadIdx.x >> 5) & 1;
  for (int q0 = (threadIdx.x >> 6) * 8; q0 < n; q0 += NT / 64 * 8) {  // uniform over the warp
    const int q = q0 + (lane >> 2);
    int ci, cj, p_lo, p_hi;
    item_of(sm.hwl[q < n ? q : q0], ci, cj, p_lo, p_hi);
    for (int side = 0; side < (mean_eigen ? 2 : 1); ++side) {
      const int lo = dir * 2 * NG + side * NG, hi = lo + (mean_eigen ? NG : 2 * NG);
      const int plo = max(p_lo, lo), phi = q < n ? min(p_hi, hi) : plo;
      if (!__any_sync(0xffffffffu, plo < phi)) continue;
      R U[4];
      const int dx = mean_eigen && dir == 0 ? 2 * side - 1 : 0, dy = mean_eigen && dir == 1 ? 2 * side - 1 : 0;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        U[c] = sm.u[c][0][cj + OYR][ci + OXR];
        if (mean_eigen) U[c] = R(0.5) * (U[c] + sm.u[c][0][cj + OYR + dy][ci + OXR + dx]);
      }
      R Rm[4][4], Lm[4][4], l[4], r[4];
      Euler2D<R>::eigen(gas, U, dir, Rm, Lm);
#pragma unroll
      for (int c = 0; c < 4; ++c) {  // the row of field f; for component f, its row of Rm
        l[c] = f == 0 ? Lm[0][c] : f == 1 ? Lm[1][c] : f == 2 ? Lm[2][c] : Lm[3][c];
        r[c] = f == 0 ? Rm[0][c] : f == 1 ? Rm[1][c] : f == 2 ? Rm[2][c] : Rm[3][c];
      }
      R e[19], ch[2 * NG];
#pragma unroll
      for (int k = 0; k < 19; ++k) e[k] = R(0);
#pragma unroll 1
      for (int c = 0; c < 4; ++c) {
        R t[19];
        const R lc = c == 0 ? l[0] : c == 1 ? l[1] : c == 2 ? l[2] : l[3];
        gather_data<COMP>(sm, c, ci, cj, t);
#pragma unroll
        for (int k = 0; k < 19; ++k) e[k] = fma(lc, t[k], e[k]);
      }
      if (dir == 0) hweno2d_dir_faces<NG, 0>(e, gam, eps, ch);
      else hweno2d_dir_faces<NG, 1>(e, gam, eps, ch);
      // component f at the points: sum over the fields, which the item's lanes hold
#pragma unroll
      for (int p = 0; p < 2 * NG; ++p) {
        R v = R(0);
#pragma unroll
        for (int g = 0; g < 4; ++g) v = fma(r[g], __shfl_sync(0xffffffffu, ch[p], base + g), v);
        const int pt = dir * 2 * NG + p;
        if (pt >= plo && pt < phi) {
          if (dir == 0) store_point(sm, f, p, ci, cj, v);
          else store_point(sm, f, 2 * NG + p, ci, cj, v);
        }
      }
    }
  }
}

// Step 4 for the n listed troubled Euler cells, the same way: vbar from the
// x-neighbours in the x characteristic fields, wbar from the y-neighbours in the y
// fields, with the 1D Step 1 formula, to sm.lim by list slot.
template <int NT, int LX_, typename R, typename S>
__device__ __noinline__ void limit_tasks_euler2d(S& sm, int n, R g0, R g1, R g2, R eps,
                                                 R gas) {
  const R gam[3] = {g0, g1, g2};
  const int lane = threadIdx.x & 31, f = lane & 3, dir = (lane >> 2) & 1, base = lane & ~3;
  for (int q0 = (threadIdx.x >> 5) * 4; q0 < n; q0 += NT / 32 * 4) {
    const int q = q0 + (lane >> 3);
    const int k = sm.tbl[q < n ? q : q0];
    const int rx = k % LX_ + 1 + S::kPadX, ry = k / LX_ + 1;
    const int sx = dir == 0 ? 1 : 0, sy = 1 - sx, mom = 1 + dir;
    R U[4], Rm[4][4], Lm[4][4], l[4], r[4], w[5] = {R(0), R(0), R(0), R(0), R(0)};
#pragma unroll
    for (int c = 0; c < 4; ++c) U[c] = sm.u[c][0][ry][rx];
    Euler2D<R>::eigen(gas, U, dir, Rm, Lm);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      l[c] = f == 0 ? Lm[0][c] : f == 1 ? Lm[1][c] : f == 2 ? Lm[2][c] : Lm[3][c];
      r[c] = f == 0 ? Rm[0][c] : f == 1 ? Rm[1][c] : f == 2 ? Rm[2][c] : Rm[3][c];
      w[0] = fma(l[c], sm.u[c][0][ry - sy][rx - sx], w[0]);
      w[1] = fma(l[c], U[c], w[1]);
      w[2] = fma(l[c], sm.u[c][0][ry + sy][rx + sx], w[2]);
      w[3] = fma(l[c], sm.u[c][mom][ry - sy][rx - sx], w[3]);
      w[4] = fma(l[c], sm.u[c][mom][ry + sy][rx + sx], w[4]);
    }
    const R m = fld::limit_moment(w[0], w[1], w[2], w[3], w[4], gam, eps);
    R v = R(0);
#pragma unroll
    for (int g = 0; g < 4; ++g) v = fma(r[g], __shfl_sync(0xffffffffu, m, base + g), v);
    if (q < n) sm.lim[q][f][dir] = v;
  }
}

// CTAs per SM the kernel is built for.  FP32 at 128 registers holds two; where its
// shared memory leaves room for more (Euler with 2 Gauss points: three, Burgers:
// four), a build at 80 or 64 registers with those is the faster one on grids of
// several waves of tiles (DENSE; 4096 x 4096 Euler, 2 points, 4 steps 18.7 -> 14.6
// ms, 13.6 with the troubled work in tasks; 2048 x 2048 Burgers, 3 points 2.50 ->
// 1.63), and the slower one on a single wave, which is bound by a tile's own chain
// (240 x 240 Euler, 2 points, 30 steps 1.08 -> 1.15): stage2d_dense decides.
template <typename R, int C, int NG, bool DENSE, int TY, bool SPLIT>
constexpr int stage2d_ctas() {
  return SPLIT ? 1 : (sizeof(R) == 8 ? 1 : !DENSE ? 2 : C == 1 ? 4 : 3) * 8 / TY;
}
template <typename R, int C, int NG>
constexpr bool has_dense() { return sizeof(R) == 4 && (C == 1 || NG == 2); }

// SPLIT: two threads per cell, for FP32 grids of at most one tile per SM (152),
// whose stage takes as long as one tile's chain.  Step 4 and the interface items
// take one round instead of two, a cell's second thread takes the halo items, the
// interior points and the y-faces (its sums go to the first through shared memory).
// 120 x 120 Euler, 3 points, 30 steps 936 -> 863 us (about half of it from the tasks above).  Beyond one tile per SM two CTAs
// of one thread per cell overlap each other instead.
template <typename R, int C, int NG, bool COMP, bool DENSE, int TY, bool SPLIT>
__global__ void __launch_bounds__(TX * TY * (SPLIT ? 2 : 1), (stage2d_ctas<R, C, NG, DENSE, TY, SPLIT>()))
    stage2d_kernel(Stage2DArgs a, const __grid_constant__ CUtensorMap tile_map,
                   const __grid_constant__ CUtensorMap lo_map) {
  static_assert(!COMP || sizeof(R) == 4, "the float-pair averages are FP32");
  extern __shared__ __align__(128) unsigned char smem_raw[];
  using SM = Smem2D<R, C, NG, COMP, TY, SPLIT>;
  constexpr int NT = SM::NT, NW = SM::NW, RY = SM::RY, LY = SM::LY;
  SM& sm = *reinterpret_cast<SM*>(smem_raw);
  constexpr int NF = 4 * NG, NI = NG * NG;
  // FP32 Euler: the linear p0 maps take two components at once (packed FP32)
  constexpr bool kPacked = C == 4 && sizeof(R) == 4;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nx = a.nx, ny = a.ny;
  const int bx0 = blockIdx.x * TX, by0 = blockIdx.y * TY;
  const size_t plane = (size_t)nx * ny;
  const R* __restrict__ w = static_cast<const R*>(a.w);

  asm volatile("griddepcontrol.wait;" ::: "memory");
  // Tiles whose halo lies inside the grid are copied by one TMA box (all 3 C
  // planes, RX x RY cells from (bx0 - 4, by0 - 3)); the others (periodic or
  // wall ghosts) by the threads, through the boundary map.
  const bool tma = a.tma && bx0 >= OXR && bx0 - OXR + RX <= nx && by0 >= OYR &&
                   by0 - OYR + RY <= ny;
  if (tma && threadIdx.x == 0) {
    mbar_init(&sm.bar, 1);
    mbar_expect_tx(&sm.bar, (unsigned)(sizeof(sm.u) + (COMP ? sizeof(sm.ulo) : 0)));
    tma_load_3d(&sm.u[0][0][0][0], &tile_map, &sm.bar, bx0 - OXR, by0 - OYR, 0);
    if constexpr (COMP) tma_load_3d(&sm.ulo[0][0][0], &lo_map, &sm.bar, bx0 - OXR, by0 - OYR, 0);
  }

  R gam[5], eps, gas, inv_dx, inv_dy;
  if constexpr (sizeof(R) == 4) {
#pragma unroll
    for (int k = 0; k < 5; ++k) gam[k] = a.f32[k];
    eps = a.f32[5]; gas = a.f32[6]; inv_dx = a.f32[7]; inv_dy = a.f32[8];
  } else {
#pragma unroll
    for (int k = 0; k < 5; ++k) gam[k] = a.gam[k];
    eps = a.eps; gas = a.gas; inv_dx = a.inv_dx; inv_dy = a.inv_dy;
  }

  // ---- 1. alpha_x, alpha_y, the time bookkeeping, the tile and its halo
  const R* a_in = static_cast<const R*>(a.a_in);
  R ax = R(0), ay = R(0);
  for (int k = tid; k < a.nin; k += NT) {
    ax = fmax(ax, a_in[k]);
    ay = fmax(ay, a_in[a.nin + k]);
  }
  // dt of the step: formed in FP64 by dt2d_kernel before stage 1
  R dt_prev = R(0);
  if (a.stage > 0) dt_prev = sc_dt<R>(a.sc);
  const int ox = tid % TX, oy = (tid / TX) % TY;  // own cell of this thread
  // what of it this thread does (uniform over the warp): with one thread per
  // cell everything, else the first thread faces, x-fluxes and the combination
  const bool first = !SPLIT || tid < TX * TY, second = !SPLIT || tid >= TX * TY;
  const int gi = bx0 + ox, gj = by0 + oy;
  const bool own = first && gi < nx && gj < ny;
  // u^n of the own cell (stages 2 and 3): brought into L2 now and loaded in
  // phase 4, so that no registers hold it through phases 2 and 3
  if (a.stage >= 2 && own) {
    const R* u0 = static_cast<const R*>(a.u0);
#pragma unroll
    for (int c = 0; c < C; ++c) {
#pragma unroll
      for (int m = 0; m < 3; ++m)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(u0 + (3 * c + m) * plane + (size_t)gj * nx + gi));
      if constexpr (COMP)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(a.u0_lo + c * plane + (size_t)gj * nx + gi));
    }
  }
  if (!tma) {
    for (int k = tid; k < RX * RY; k += NT) {
      const int rx = k % RX, ry = k / RX;
      const int si = bc_map(bx0 - OXR + rx, nx, a.bc), sj = bc_map(by0 - OYR + ry, ny, a.bc);
      const size_t s = (size_t)sj * nx + si;
#pragma unroll
      for (int c = 0; c < C; ++c) {
#pragma unroll
        for (int m = 0; m < 3; ++m) sm.u[c][m][ry][rx] = w[(3 * c + m) * plane + s];
        if constexpr (COMP) sm.ulo[c][ry][rx] = a.w_lo[c * plane + s];
      }
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    ax = fmax(ax, __shfl_xor_sync(0xffffffffu, ax, o));
    ay = fmax(ay, __shfl_xor_sync(0xffffffffu, ay, o));
  }
  if (lane == 0) {
    sm.amax[0][warp] = ax;
    sm.amax[1][warp] = ay;
  }
  if (tid == 0) sm.ntb = sm.nhw = 0;
  __syncthreads();
  if (tma && !mbar_wait_bounded(&sm.bar, 0, kTmaPolls)) {
    // the copy did not land: flag the stage (the host reports
    // HWENO_ERR_TIMEOUT) and give the copy, which writes this CTA's shared
    // memory, a second bounded wait; no thread leaves the common path
    atomicOr(&a.sc->status, ST_TIMEOUT);
    mbar_wait_bounded(&sm.bar, 0, kTmaPolls);
  }
  asm volatile("griddepcontrol.launch_dependents;");
  R alx = sm.amax[0][0], aly = sm.amax[1][0];
#pragma unroll
  for (int k = 1; k < NW; ++k) {
    alx = fmax(alx, sm.amax[0][k]);
    aly = fmax(aly, sm.amax[1][k]);
  }
  if (a.alpha_in) {  // replay: the recorded values (what the reduction gave)
    alx = static_cast<const R*>(a.alpha_in)[0];
    aly = static_cast<const R*>(a.alpha_in)[1];
  }
  R dt = dt_prev;
  if (a.stage == 1) {
    if (a.dt_in) {  // replay of a recorded step
      dt = *static_cast<const R*>(a.dt_in);
      if (blockIdx.x == 0 && blockIdx.y == 0 && tid == 0) {
        a.sc->dt = (double)dt;
        a.sc->dt_f = (float)dt;
        a.sc->last = 0u;
      }
    }
    if (a.rec_dt && blockIdx.x == 0 && blockIdx.y == 0 && tid == 0)
      *static_cast<R*>(a.rec_dt) = dt;
  }
  if (a.rec_alpha && blockIdx.x == 0 && blockIdx.y == 0 && tid == 0) {
    static_cast<R*>(a.rec_alpha)[0] = alx;
    static_cast<R*>(a.rec_alpha)[1] = aly;
  }
  if (a.stage > 0 && !(dt > R(0))) return;  // uniform over the grid
  if (a.a_zero && blockIdx.x == 0 && blockIdx.y == 0 && tid < 2 * kAlphaSlots)
    static_cast<R*>(a.a_zero)[tid] = R(0);

  // ---- 2. Step 4 on the tile plus 2 halo cells; the modified first moments
  // of the troubled cells replace the raw ones in the tile only after every
  // flag and limiter has read the raw ones
  constexpr int kRounds = (LX * LY + NT - 1) / NT;  // cells of Step 4 per thread at most
  R hv[kRounds][2];  // Burgers: the modified moments of this thread's troubled cells
  int hk[kRounds];
#pragma unroll
  for (int j = 0; j < kRounds; ++j) hk[j] = -1;
  int it = 0;
  for (int k = tid; k < LX * LY; k += NT, ++it) {
    const int lx = k % LX, ly = k / LX;
    const int rx = lx + 1 + SM::kPadX, ry = ly + 1;  // raw index of the cell
    int flag;
    if (a.flags_in) {  // replay: the recorded decision (periodic: a ghost's is its image's)
      flag = a.flags_in[(size_t)bc_map(by0 - 2 + ly, ny, a.bc) * nx + bc_map(bx0 - 2 + lx, nx, a.bc)] != 0;
    } else if (a.mode == 1) {
      flag = 1;
    } else if (a.mode == 2) {
      flag = 0;
    } else {
      bool lowx, lowy;
      if constexpr (C == 1) {
        lowx = lowy = sm.u[0][0][ry][rx] >= R(0);
      } else {
        lowx = inflow_left(sm.u[0][0][ry][rx], sm.u[1][0][ry][rx]);
        lowy = inflow_left(sm.u[0][0][ry][rx], sm.u[2][0][ry][rx]);
      }
      const int nxx = lowx ? rx - 1 : rx + 1, nyy = lowy ? ry - 1 : ry + 1;
      const int ci = 0;
      if constexpr (COMP) {  // on hi + lo
        flag = kxrcf2_troubled_pair(sm.u[ci][0][ry][rx], sm.ulo[ci][ry][rx], sm.u[ci][1][ry][rx],
                                    sm.u[ci][2][ry][rx], sm.u[ci][0][ry][nxx], sm.ulo[ci][ry][nxx],
                                    sm.u[ci][1][ry][nxx], sm.u[ci][0][nyy][rx], sm.ulo[ci][nyy][rx],
                                    sm.u[ci][2][nyy][rx], lowx, lowy, a.kx);
        if constexpr (C == 4)
          flag = flag || kxrcf2_troubled_pair(sm.u[3][0][ry][rx], sm.ulo[3][ry][rx],
                                              sm.u[3][1][ry][rx], sm.u[3][2][ry][rx],
                                              sm.u[3][0][ry][nxx], sm.ulo[3][ry][nxx],
                                              sm.u[3][1][ry][nxx], sm.u[3][0][nyy][rx],
                                              sm.ulo[3][nyy][rx], sm.u[3][2][nyy][rx], lowx,
                                              lowy, a.kx);
      } else {
        flag = kxrcf2_troubled(sm.u[ci][0][ry][rx], sm.u[ci][1][ry][rx], sm.u[ci][2][ry][rx],
                               sm.u[ci][0][ry][nxx], sm.u[ci][1][ry][nxx], sm.u[ci][0][nyy][rx],
                               sm.u[ci][2][nyy][rx], lowx, lowy, a.kx);
        if constexpr (C == 4) {
          flag = flag || kxrcf2_troubled(sm.u[3][0][ry][rx], sm.u[3][1][ry][rx], sm.u[3][2][ry][rx],
                                         sm.u[3][0][ry][nxx], sm.u[3][1][ry][nxx],
                                         sm.u[3][0][nyy][rx], sm.u[3][2][nyy][rx], lowx, lowy, a.kx);
        }
      }
    }
    sm.fl[ly][lx] = (uint8_t)flag;
    if constexpr (C == 1) {
      if (flag) {
        hk[it] = k;
        hv[it][0] = limit_first_moment(sm.u[0][0][ry][rx - 1], sm.u[0][0][ry][rx],
                                       sm.u[0][0][ry][rx + 1], sm.u[0][1][ry][rx - 1],
                                       sm.u[0][1][ry][rx + 1], gam, eps);
        hv[it][1] = limit_first_moment(sm.u[0][0][ry - 1][rx], sm.u[0][0][ry][rx],
                                       sm.u[0][0][ry + 1][rx], sm.u[0][2][ry - 1][rx],
                                       sm.u[0][2][ry + 1][rx], gam, eps);
      }
    }
    // Euler: the troubled cells are listed and limited by consecutive threads
    // below, so a warp holding one or two of them does not run the
    // characteristic limiter for its other lanes' sake
    if constexpr (C == 4) list_append(&sm.ntb, sm.tbl, k, flag != 0, LX * LY);
  }
  // the tile's flag grid holds a troubled cell (uniform over the CTA): else
  // no interface item of the tile needs HWENO and none tests its stencil
  bool tile_troubled;
  if constexpr (C == 1) {
    bool mine = false;
#pragma unroll
    for (int j = 0; j < kRounds; ++j) mine |= hk[j] >= 0;
    tile_troubled = __syncthreads_or(mine);
    if (tile_troubled) {
#pragma unroll
      for (int j = 0; j < kRounds; ++j)
        if (hk[j] >= 0) {
          const int rx = hk[j] % LX + 1 + SM::kPadX, ry = hk[j] / LX + 1;
          sm.u[0][1][ry][rx] = hv[j][0];
          sm.u[0][2][ry][rx] = hv[j][1];
        }
      __syncthreads();
    }
  } else {
    __syncthreads();
    tile_troubled = sm.ntb > 0;
    if (tile_troubled) {
      limit_tasks_euler2d<NT, LX>(sm, sm.ntb, gam[0], gam[1], gam[2], eps, gas);
      __syncthreads();
      for (int q = tid; q < sm.ntb; q += NT) {
        const int k = sm.tbl[q];
        const int rx = k % LX + 1 + SM::kPadX, ry = k / LX + 1;
#pragma unroll
        for (int c = 0; c < C; ++c) {
          sm.u[c][1][ry][rx] = sm.lim[q][c][0];
          sm.u[c][2][ry][rx] = sm.lim[q][c][1];
        }
      }
      __syncthreads();
    }
  }

  // ---- 3. interface values of the own cells (all faces) and of the cross
  //         halo (left column: right face, right column: left face, bottom
  //         row: top face, top row: bottom face)
  //         by linear p0, and of the own cells the interior points (Step 5.3)
  //         with their volume integrals, from the same parity classes (the
  //         second gather and fold of phase 4 cost more than the 2 C sums held
  //         through the barrier); the items whose stencil holds a troubled
  //         cell are listed and reconstructed by HWENO on consecutive threads
  //         below (the same arithmetic, fewer warps diverging on it)
  auto item_of = [](int item, int& ci, int& cj, int& p_lo, int& p_hi) {
    if (item < TX * TY) {  // own cell: every interface point
      ci = item % TX; cj = item / TX; p_lo = 0; p_hi = NF;
    } else {               // cross halo: the one face shared with the tile
      const int h = item - TX * TY;  // the y-faces first: a warp has items of one kind
      if (h < TX) { ci = h; cj = -1; p_lo = 3 * NG; p_hi = 4 * NG; }
      else if (h < 2 * TX) { ci = h - TX; cj = TY; p_lo = 2 * NG; p_hi = 3 * NG; }
      else if (h < 2 * TX + TY) { ci = -1; cj = h - 2 * TX; p_lo = NG; p_hi = 2 * NG; }
      else { ci = TX; cj = h - 2 * TX - TY; p_lo = 0; p_hi = NG; }
    }
  };
  constexpr double r15 = 0.38729833462074168852;  // sqrt(15)/10
  constexpr double r3 = 0.28867513459481288225;   // sqrt(3)/6
  const R gw[3] = {NG == 3 ? R(5.0 / 18.0) : R(0.5), NG == 3 ? R(4.0 / 9.0) : R(0.5), R(5.0 / 18.0)};
  const R gx[3] = {NG == 3 ? R(-r15) : R(-r3), NG == 3 ? R(0) : R(r3), R(r15)};
  const int ci = ox, cj = oy;  // the own cell, as the item of this thread
  // COMP: every point value is an increment over the own cell's hi B, every
  // flux an increment over f(B) (the base cancels from Eq. (ode2) exactly)
  R B[C];
#pragma unroll
  for (int c = 0; c < C; ++c) B[c] = sm.u[c][0][cj + OYR][ci + OXR];
  auto flux = [&](const R* U, int dir, R* F) {
    if constexpr (COMP) flux_inc2<C>(gas, B, U, dir, F);
    else phys_flux2<R, C>(gas, U, dir, F);
  };
  R Fv[C], Gv[C];  // the volume integrals of Eq. (ode2)
#pragma unroll
  for (int c = 0; c < C; ++c) Fv[c] = Gv[c] = R(0);
  using T = typename PairOf<R, kPacked>::type;
  auto near_troubled = [&](int i, int j) {
    bool hw = false;
    if (tile_troubled) {
#pragma unroll
      for (int dj = -1; dj <= 1; ++dj)
#pragma unroll
        for (int di = -1; di <= 1; ++di) hw |= sm.fl[j + 2 + dj][i + 2 + di] != 0;
    }
    return hw;
  };
  // the values at the points [p_lo, p_hi) of component c (packed: c and c + 1)
  // of cell (i, j) from its parity classes
  auto faces = [&](const T* s, int c, int i, int j, int p_lo, int p_hi) {
    if (p_lo < 2 * NG) {
      T v[2 * NG];
      p0s_xfaces<NG>(s, v);
#pragma unroll
      for (int p = 0; p < 2 * NG; ++p)
        if (p >= p_lo && p < p_hi) store_points(sm, c, p, i, j, v[p]);
    }
    if (p_hi > 2 * NG) {
      T v[2 * NG];
      p0s_yfaces<NG>(s, v);
#pragma unroll
      for (int p = 0; p < 2 * NG; ++p)
        if (p + 2 * NG >= p_lo && p + 2 * NG < p_hi) store_points(sm, c, p + 2 * NG, i, j, v[p]);
    }
  };
  {
    const bool hw = first && near_troubled(ci, cj);
    R inter[C][NI];
#pragma unroll
    for (int c = 0; c < C; c += kPacked ? 2 : 1) {
      T s[19], v[NI];
      classes_of<COMP, kPacked>(sm, c, ci, cj, s);
      if (first && !hw) faces(s, c, ci, cj, 0, NF);
      if (!second) continue;
      p0s_interior<NG>(s, v);
#pragma unroll
      for (int l = 0; l < NI; ++l) {
        if constexpr (kPacked) {
          inter[c][l] = v[l].x;
          inter[c + 1][l] = v[l].y;
        } else {
          inter[c][l] = v[l];
        }
      }
    }
    // the volume integrals of Eq. (ode2) at interior point p (weight
    // gw[p % NG] gw[p / NG])
    auto interior_point = [&](int p) {
      R U[C], f[C], g[C];
#pragma unroll
      for (int c = 0; c < C; ++c) U[c] = inter[c][p];
      flux(U, 0, f);
      flux(U, 1, g);
#pragma unroll
      for (int c = 0; c < C; ++c) {
        Fv[c] += gw[p % NG] * gw[p / NG] * f[c];
        Gv[c] += gw[p % NG] * gw[p / NG] * g[c];
      }
    };
    if (!second) {
    } else if constexpr (kPacked) {  // points in pairs, an odd last one alone
      auto flux_x2 = [&](const float2* U, int dir, float2* F) {
        if constexpr (COMP) flux_inc2_x2(gas, B, U, dir, F);
        else euler_flux_x2(gas, U, dir, F);
      };
      float2 Fv2[C], Gv2[C];
#pragma unroll
      for (int c = 0; c < C; ++c) Fv2[c] = Gv2[c] = make_float2(0.0f, 0.0f);
#pragma unroll
      for (int p = 0; p + 1 < NI; p += 2) {
        float2 U2[C], f2[C], g2[C];
#pragma unroll
        for (int c = 0; c < C; ++c) U2[c] = make_float2(inter[c][p], inter[c][p + 1]);
        flux_x2(U2, 0, f2);
        flux_x2(U2, 1, g2);
        const float2 w2 = make_float2(gw[p % NG] * gw[p / NG], gw[(p + 1) % NG] * gw[(p + 1) / NG]);
#pragma unroll
        for (int c = 0; c < C; ++c) {
          Fv2[c] = __ffma2_rn(w2, f2[c], Fv2[c]);
          Gv2[c] = __ffma2_rn(w2, g2[c], Gv2[c]);
        }
      }
#pragma unroll
      for (int c = 0; c < C; ++c) {
        Fv[c] = Fv2[c].x + Fv2[c].y;
        Gv[c] = Gv2[c].x + Gv2[c].y;
      }
      if constexpr (NI % 2 == 1) interior_point(NI - 1);
    } else {
#pragma unroll
      for (int p = 0; p < NI; ++p) interior_point(p);
    }
    if (first) list_append(&sm.nhw, sm.hwl, tid, hw, TX * TY + 2 * TX + 2 * TY);
  }
  constexpr int kItems = TX * TY + 2 * TX + 2 * TY;
  for (int item = !SPLIT ? NT + tid : first ? kItems : tid; item < kItems; item += NT) {
    int hi, hj, p_lo, p_hi;  // own-tile coordinates of the halo cell, point range
    item_of(item, hi, hj, p_lo, p_hi);
    const bool hw = near_troubled(hi, hj);
    if (!hw) {
#pragma unroll
      for (int c = 0; c < C; c += kPacked ? 2 : 1) {
        T s[19];
        classes_of<COMP, kPacked>(sm, c, hi, hj, s);
        faces(s, c, hi, hj, p_lo, p_hi);
      }
    }
    list_append(&sm.nhw, sm.hwl, item, hw, TX * TY + 2 * TX + 2 * TY);
  }
  __syncthreads();
  if (sm.nhw > 0) {  // uniform over the CTA
    if constexpr (C == 4) {
      hweno_tasks_euler2d<NG, NT, COMP>(sm, sm.nhw, item_of, gam[0], gam[1], gam[2], gam[3], gam[4], eps,
                                        gas, (a.variant & HWENO_VARIANT_MEAN_EIGEN) != 0);
    } else {
      for (int q = tid; q < sm.nhw; q += NT) {
        int ci, cj, p_lo, p_hi;
        item_of(sm.hwl[q], ci, cj, p_lo, p_hi);
        R d[19], v[NF];
        gather_data<COMP>(sm, 0, ci, cj, d);
        hweno2d_faces<NG>(d, gam, eps, p_lo, p_hi, v);
#pragma unroll
        for (int p = 0; p < NF; ++p)
          if (p >= p_lo && p < p_hi) store_point(sm, 0, p, ci, cj, v[p]);
      }
    }
    __syncthreads();
  }

  // ---- 4. own cells: fluxes, Eq. (ode2), Eq. (RK)
  int myflag = 0;
  R spx = R(0), spy = R(0);
  unsigned bad = 0;
  {
    R u0c[C][3], u0l[C];
    if (a.stage >= 2 && own) {
      const R* u0 = static_cast<const R*>(a.u0);
#pragma unroll
      for (int c = 0; c < C; ++c) {
#pragma unroll
        for (int m = 0; m < 3; ++m) u0c[c][m] = u0[(3 * c + m) * plane + (size_t)gj * nx + gi];
        if constexpr (COMP) u0l[c] = a.u0_lo[c * plane + (size_t)gj * nx + gi];
      }
    }
    myflag = sm.fl[cj + 2][ci + 2];
    const R hax = R(0.5) * alx, hay = R(0.5) * aly;
    // COMP: a neighbour's face value, held over its own hi, over B instead
    auto rebase = [&](R* v, int dx, int dy) {
      if constexpr (COMP) {
#pragma unroll
        for (int c = 0; c < C; ++c)
          v[c] = __fadd_rn(v[c], __fsub_rn(sm.u[c][0][cj + OYR + dy][ci + OXR + dx], B[c]));
      }
    };
    R sfx[C], sfs[C], sfxe[C], sgy[C], sgs[C], sgyx[C];
#pragma unroll
    for (int c = 0; c < C; ++c) sfx[c] = sfs[c] = sfxe[c] = sgy[c] = sgs[c] = sgyx[c] = R(0);
    // the Lax-Friedrichs fluxes of the four faces at Gauss point k and their
    // weighted sums
    auto face_point = [&](int k) {
      R am[C], ap[C], fa[C], fb[C], FLk[C], FRk[C], GBk[C], GTk[C];
      if (first) {
        // x_{i-1/2}: u^- = right face of cell i-1, u^+ = own left face
#pragma unroll
        for (int c = 0; c < C; ++c) { am[c] = sm.xf[c][NG + k][cj][ci]; ap[c] = sm.xf[c][k][cj][ci + 1]; }
        rebase(am, -1, 0);
        flux(am, 0, fa); flux(ap, 0, fb);
#pragma unroll
        for (int c = 0; c < C; ++c) FLk[c] = R(0.5) * (fa[c] + fb[c]) - hax * (ap[c] - am[c]);
        // x_{i+1/2}: u^- = own right face, u^+ = left face of cell i+1
#pragma unroll
        for (int c = 0; c < C; ++c) { am[c] = sm.xf[c][NG + k][cj][ci + 1]; ap[c] = sm.xf[c][k][cj][ci + 2]; }
        rebase(ap, 1, 0);
        flux(am, 0, fa); flux(ap, 0, fb);
#pragma unroll
        for (int c = 0; c < C; ++c) FRk[c] = R(0.5) * (fa[c] + fb[c]) - hax * (ap[c] - am[c]);
#pragma unroll
        for (int c = 0; c < C; ++c) {
          sfx[c] += gw[k] * (FRk[c] - FLk[c]);
          sfs[c] += gw[k] * (FLk[c] + FRk[c]);
          sfxe[c] += gw[k] * gx[k] * (FRk[c] - FLk[c]);
        }
      }
      if (second) {
        // y_{j-1/2}: u^- = top face of cell j-1, u^+ = own bottom face
#pragma unroll
        for (int c = 0; c < C; ++c) { am[c] = sm.yf[c][NG + k][cj][ci]; ap[c] = sm.yf[c][k][cj + 1][ci]; }
        rebase(am, 0, -1);
        flux(am, 1, fa); flux(ap, 1, fb);
#pragma unroll
        for (int c = 0; c < C; ++c) GBk[c] = R(0.5) * (fa[c] + fb[c]) - hay * (ap[c] - am[c]);
        // y_{j+1/2}: u^- = own top face, u^+ = bottom face of cell j+1
#pragma unroll
        for (int c = 0; c < C; ++c) { am[c] = sm.yf[c][NG + k][cj + 1][ci]; ap[c] = sm.yf[c][k][cj + 2][ci]; }
        rebase(ap, 0, 1);
        flux(am, 1, fa); flux(ap, 1, fb);
#pragma unroll
        for (int c = 0; c < C; ++c) GTk[c] = R(0.5) * (fa[c] + fb[c]) - hay * (ap[c] - am[c]);
#pragma unroll
        for (int c = 0; c < C; ++c) {
          sgy[c] += gw[k] * (GTk[c] - GBk[c]);
          sgs[c] += gw[k] * (GBk[c] + GTk[c]);
          sgyx[c] += gw[k] * gx[k] * (GTk[c] - GBk[c]);
        }
      }
    };
    if constexpr (kPacked) {
      // FP32 Euler: points in pairs, (interior p, p + 1) and (Gauss k, k + 1)
      // of every face, each flux, Lax-Friedrichs flux and weighted sum in
      // packed FP32; the pairs' halves are added at the end and an odd last
      // point (3 Gauss points) runs alone.  COMP: the fluxes are increments
      // over f(B), a neighbour's face values moved onto B by one broadcast add
      auto flux_x2 = [&](const float2* U, int dir, float2* F) {
        if constexpr (COMP) flux_inc2_x2(gas, B, U, dir, F);
        else euler_flux_x2(gas, U, dir, F);
      };
      auto rebase_x2 = [&](float2* v, int dx, int dy) {
        if constexpr (COMP) {
#pragma unroll
          for (int c = 0; c < C; ++c)
            v[c] = __fadd2_rn(v[c], bcast2(__fsub_rn(sm.u[c][0][cj + OYR + dy][ci + OXR + dx], B[c])));
        }
      };
      float2 sfx2[C], sfs2[C], sfxe2[C], sgy2[C], sgs2[C], sgyx2[C];
#pragma unroll
      for (int c = 0; c < C; ++c)
        sfx2[c] = sfs2[c] = sfxe2[c] = sgy2[c] = sgs2[c] = sgyx2[c] = make_float2(0.0f, 0.0f);
#pragma unroll
      for (int k = 0; k + 1 < NG; k += 2) {
        const float2 gw2 = make_float2(gw[k], gw[k + 1]);
        const float2 gwx2 = make_float2(gw[k] * gx[k], gw[k + 1] * gx[k + 1]);
        float2 am[C], ap[C], fa[C], fb[C], FL[C], FR[C], GB[C], GT[C];
        if (first) {
#pragma unroll
          for (int c = 0; c < C; ++c) {
            am[c] = make_float2(sm.xf[c][NG + k][cj][ci], sm.xf[c][NG + k + 1][cj][ci]);
            ap[c] = make_float2(sm.xf[c][k][cj][ci + 1], sm.xf[c][k + 1][cj][ci + 1]);
          }
          rebase_x2(am, -1, 0);
          flux_x2(am, 0, fa); flux_x2(ap, 0, fb);
#pragma unroll
          for (int c = 0; c < C; ++c) FL[c] = lf_x2(fa[c], fb[c], am[c], ap[c], hax);
#pragma unroll
          for (int c = 0; c < C; ++c) {
            am[c] = make_float2(sm.xf[c][NG + k][cj][ci + 1], sm.xf[c][NG + k + 1][cj][ci + 1]);
            ap[c] = make_float2(sm.xf[c][k][cj][ci + 2], sm.xf[c][k + 1][cj][ci + 2]);
          }
          rebase_x2(ap, 1, 0);
          flux_x2(am, 0, fa); flux_x2(ap, 0, fb);
#pragma unroll
          for (int c = 0; c < C; ++c) FR[c] = lf_x2(fa[c], fb[c], am[c], ap[c], hax);
#pragma unroll
          for (int c = 0; c < C; ++c) {
            const float2 dx = sub2(FR[c], FL[c]);
            sfx2[c] = __ffma2_rn(gw2, dx, sfx2[c]);
            sfs2[c] = __ffma2_rn(gw2, __fadd2_rn(FL[c], FR[c]), sfs2[c]);
            sfxe2[c] = __ffma2_rn(gwx2, dx, sfxe2[c]);
          }
        }
        if (second) {
#pragma unroll
          for (int c = 0; c < C; ++c) {
            am[c] = make_float2(sm.yf[c][NG + k][cj][ci], sm.yf[c][NG + k + 1][cj][ci]);
            ap[c] = make_float2(sm.yf[c][k][cj + 1][ci], sm.yf[c][k + 1][cj + 1][ci]);
          }
          rebase_x2(am, 0, -1);
          flux_x2(am, 1, fa); flux_x2(ap, 1, fb);
#pragma unroll
          for (int c = 0; c < C; ++c) GB[c] = lf_x2(fa[c], fb[c], am[c], ap[c], hay);
#pragma unroll
          for (int c = 0; c < C; ++c) {
            am[c] = make_float2(sm.yf[c][NG + k][cj + 1][ci], sm.yf[c][NG + k + 1][cj + 1][ci]);
            ap[c] = make_float2(sm.yf[c][k][cj + 2][ci], sm.yf[c][k + 1][cj + 2][ci]);
          }
          rebase_x2(ap, 0, 1);
          flux_x2(am, 1, fa); flux_x2(ap, 1, fb);
#pragma unroll
          for (int c = 0; c < C; ++c) GT[c] = lf_x2(fa[c], fb[c], am[c], ap[c], hay);
#pragma unroll
          for (int c = 0; c < C; ++c) {
            const float2 dy = sub2(GT[c], GB[c]);
            sgy2[c] = __ffma2_rn(gw2, dy, sgy2[c]);
            sgs2[c] = __ffma2_rn(gw2, __fadd2_rn(GB[c], GT[c]), sgs2[c]);
            sgyx2[c] = __ffma2_rn(gwx2, dy, sgyx2[c]);
          }
        }
      }
#pragma unroll
      for (int c = 0; c < C; ++c) {
        sfx[c] = sfx2[c].x + sfx2[c].y;
        sfs[c] = sfs2[c].x + sfs2[c].y;
        sfxe[c] = sfxe2[c].x + sfxe2[c].y;
        sgy[c] = sgy2[c].x + sgy2[c].y;
        sgs[c] = sgs2[c].x + sgs2[c].y;
        sgyx[c] = sgyx2[c].x + sgyx2[c].y;
      }
      if constexpr (NG % 2 == 1) face_point(NG - 1);
    } else {
#pragma unroll
      for (int k = 0; k < NG; ++k) face_point(k);
    }
    if constexpr (SPLIT) {  // the second thread's sums to the first
      const int k = tid % (TX * TY);
      if (second) {
#pragma unroll
        for (int c = 0; c < C; ++c) {
          sm.half[c][k] = sgy[c];
          sm.half[C + c][k] = sgs[c];
          sm.half[2 * C + c][k] = sgyx[c];
          sm.half[3 * C + c][k] = Fv[c];
          sm.half[4 * C + c][k] = Gv[c];
        }
      }
      __syncthreads();
      if (first) {
#pragma unroll
        for (int c = 0; c < C; ++c) {
          sgy[c] = sm.half[c][k];
          sgs[c] = sm.half[C + c][k];
          sgyx[c] = sm.half[2 * C + c][k];
          Fv[c] = sm.half[3 * C + c][k];
          Gv[c] = sm.half[4 * C + c][k];
        }
      }
    }
    R Uo[C];
    if (first) {
#pragma unroll
      for (int c = 0; c < C; ++c) {
        const R L0 = -sfx[c] * inv_dx - sgy[c] * inv_dy;
        const R L1 = -R(0.5) * sfs[c] * inv_dx + Fv[c] * inv_dx - sgyx[c] * inv_dy;
        const R L2 = -sfxe[c] * inv_dx - R(0.5) * sgs[c] * inv_dy + Gv[c] * inv_dy;
        // the stage input the combination uses: first moments as modified by
        // Step 4 (stored, the default), or unmodified (variant)
        // (the tile holds the modified ones; the raw ones of an own cell are
        // read back from the stage input)
        const bool raw = (a.variant & HWENO_VARIANT_RAW_COMBINE) != 0;
        const size_t sw = (size_t)gj * nx + gi;
        const R W[3] = {sm.u[c][0][cj + OYR][ci + OXR],
                        raw ? (own ? w[(3 * c + 1) * plane + sw] : R(0)) : sm.u[c][1][cj + OYR][ci + OXR],
                        raw ? (own ? w[(3 * c + 2) * plane + sw] : R(0)) : sm.u[c][2][cj + OYR][ci + OXR]};
        const R Lm[3] = {L0, L1, L2};
        R o[3];
#pragma unroll
        for (int m = 0; m < 3; ++m) {
          if (a.stage == 0) {
            o[m] = Lm[m];
          } else {
            const R s = W[m] + dt * Lm[m];
            if (a.stage == 1) o[m] = s;
            else {
              const R cb = a.stage == 2 ? R(0.25) : R(2.0 / 3.0);
              o[m] = rk_combine(cb, u0c[c][m], s);
            }
          }
          if (!is_finite(o[m])) bad |= ST_NONFINITE;
        }
        R olo = R(0);
        if constexpr (COMP) {
          // the average as a float pair: a u^n + b w in pair arithmetic (1/3
          // and 2/3 as pairs), then the increment b dt L
          constexpr float t1h = 1.0f / 3.0f, t2h = 2.0f / 3.0f;
          constexpr float t1l = (float)(1.0 / 3.0 - (double)t1h), t2l = (float)(2.0 / 3.0 - (double)t2h);
          const R wl = sm.ulo[c][cj + OYR][ci + OXR];
          R bh = W[0], bl = wl;
          if (a.stage == 2)
            pair_axpby(0.75f, 0.0f, u0c[c][0], u0l[c], 0.25f, 0.0f, W[0], wl, bh, bl);
          else if (a.stage == 3)
            pair_axpby(t1h, t1l, u0c[c][0], u0l[c], t2h, t2l, W[0], wl, bh, bl);
          const R cb = a.stage == 2 ? R(0.25) : a.stage == 3 ? R(2.0 / 3.0) : R(1);
          pair_add(bh, bl, (cb * dt) * L0, o[0], olo);
          if (!isfinite(o[0])) bad |= ST_NONFINITE;
        }
        if (own) {
          R* out = static_cast<R*>(a.out);
          const size_t s = (size_t)gj * nx + gi;
#pragma unroll
          for (int m = 0; m < 3; ++m) out[(3 * c + m) * plane + s] = o[m];
          if constexpr (COMP) a.out_lo[c * plane + s] = olo;
          if (a.lim_out) {  // rhs mode: the modified moments; stage 1: what stages 2-3 combine
            R* lo = static_cast<R*>(a.lim_out);
            const R M[3] = {W[0], sm.u[c][1][cj + OYR][ci + OXR], sm.u[c][2][cj + OYR][ci + OXR]};
#pragma unroll
            for (int m = 0; m < 3; ++m) lo[(3 * c + m) * plane + s] = a.stage == 0 ? M[m] : W[m];
          }
        }
        Uo[c] = o[0];
      }
    }
    if (own) {
      if (a.flags_out) a.flags_out[(size_t)gj * nx + gi] = (uint8_t)myflag;
      if (a.stage > 0 && a.a_out) {  // (a replayed stage needs no maxima)
        wave_speeds2<R, C>(gas, Uo, spx, spy);
        if (!(spx == spx) || !(spy == spy)) {
          bad |= ST_NONPHYSICAL;
          spx = spy = R(0);
        }
      }
    } else {
      myflag = 0;
      bad = 0;
    }
  }

  // ---- 5. epilogue
  for (int o = 16; o > 0; o >>= 1) {
    spx = fmax(spx, __shfl_xor_sync(0xffffffffu, spx, o));
    spy = fmax(spy, __shfl_xor_sync(0xffffffffu, spy, o));
  }
  const int wcnt = __popc(__ballot_sync(0xffffffffu, myflag));
  if (lane == 0) {
    sm.red[0][warp] = spx;
    sm.red[1][warp] = spy;
    sm.cnt[warp] = wcnt;
  }
  if (bad) atomicOr(&a.sc->status, bad);
  __syncthreads();
  if (warp == 0) {
    R mx = lane < NW ? sm.red[0][lane] : R(0);
    R my = lane < NW ? sm.red[1][lane] : R(0);
    int cn = lane < NW ? sm.cnt[lane] : 0;
    for (int o = 16; o > 0; o >>= 1) {
      mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      my = fmax(my, __shfl_xor_sync(0xffffffffu, my, o));
      cn += __shfl_xor_sync(0xffffffffu, cn, o);
    }
    if (lane == 0) {
      const int slot = (blockIdx.y * gridDim.x + blockIdx.x) % kAlphaSlots;
      if (a.a_out) {
        atomic_max_nonneg(static_cast<R*>(a.a_out) + slot, mx);
        atomic_max_nonneg(static_cast<R*>(a.a_out) + kAlphaSlots + slot, my);
      }
      if (cn) atomicAdd(&a.sc->troubled, (unsigned long long)cn);
      if (a.stage == 3 && blockIdx.x == 0 && blockIdx.y == 0) {
        DevScalars* sc = a.sc;
        const double tf = sc->t_final;
        const double t = sc->last ? tf : sc->t + sc->dt;
        const double r = tf > 0.0 ? tf - t : (double)INFINITY;
        sc->t = t;
        sc->rem = r;
        sc->rem_f = (float)r;
        sc->steps += 1;
      }
    }
  }
}

// dt of a 2D step (Sec. 3, CFL; reading: dt = CFL / (alpha_x / dx + alpha_y /
// dy)), in FP64: one warp folds the wave-speed maxima of the step's input
// (kernel precision, so exact in FP64), forms dt and its clip to t_final,
// and leaves dt (FP64 and FP32 copies) and the last-step flag in the
// scalars, where the three stage kernels read it.
template <typename R>
__global__ void __launch_bounds__(32) dt2d_kernel(const R* a_in, int nin,
                                                  DevScalars* sc, double cfl, double inv_dx,
                                                  double inv_dy) {
  // (programmatic dependent launch on both sides: this warp is resident before
  // the previous stage ends, and stage 1's tiles before this one does)
  asm volatile("griddepcontrol.launch_dependents;");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const double rem = sc->rem;
  R mx = R(0), my = R(0);  // the maxima in the kernel precision (exact), FP64 after them
  for (int k = threadIdx.x; k < nin; k += 32) {
    mx = fmax(mx, a_in[k]);
    my = fmax(my, a_in[nin + k]);
  }
  for (int o = 16; o > 0; o >>= 1) {
    mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    my = fmax(my, __shfl_xor_sync(0xffffffffu, my, o));
  }
  if (threadIdx.x == 0) {
    const double ax = (double)mx, ay = (double)my;
    double dt = cfl / (ax * inv_dx + ay * inv_dy);
    unsigned last = 0u;
    if (rem <= 0.0) {
      dt = 0.0;
    } else if (dt >= rem) {
      dt = rem;
      last = 1u;
    }
    if (!(ax + ay > 0.0) || !isfinite(dt)) dt = 0.0;
    sc->dt = dt;
    sc->dt_f = (float)dt;
    sc->last = last;
  }
}

template <typename R, int C>
__global__ void __launch_bounds__(NTW) alpha2d_kernel(const R* __restrict__ w, R* a_out, int nx,
                                                    int ny, double gas, DevScalars* sc,
                                                    int slots) {
  __shared__ R red[2][NWW];
  const int gi = blockIdx.x * TX + threadIdx.x % TX, gj = blockIdx.y * TYW + threadIdx.x / TX;
  const size_t plane = (size_t)nx * ny;
  R sx = R(0), sy = R(0);
  if (gi < nx && gj < ny) {
    R U[C];
#pragma unroll
    for (int c = 0; c < C; ++c) U[c] = w[(3 * c) * plane + (size_t)gj * nx + gi];
    wave_speeds2<R, C>(R(gas), U, sx, sy);
    if (!(sx == sx) || !(sy == sy)) {
      atomicOr(&sc->status, (unsigned)ST_NONPHYSICAL);
      sx = sy = R(0);
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    sx = fmax(sx, __shfl_xor_sync(0xffffffffu, sx, o));
    sy = fmax(sy, __shfl_xor_sync(0xffffffffu, sy, o));
  }
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = sx;
    red[1][threadIdx.x >> 5] = sy;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 0; k < NWW; ++k) {
      sx = fmax(sx, red[0][k]);
      sy = fmax(sy, red[1][k]);
    }
    const int b = blockIdx.y * gridDim.x + blockIdx.x;
    if (slots) {
      atomic_max_nonneg(a_out + b % kAlphaSlots, sx);
      atomic_max_nonneg(a_out + kAlphaSlots + b % kAlphaSlots, sy);
    } else {
      const int nt = gridDim.x * gridDim.y;
      a_out[b] = sx;
      a_out[nt + b] = sy;
    }
  }
}

// More than two tiles per SM: the dense build.
bool stage2d_dense(int tiles) { return tiles > 304; }

template <typename R, int C, int NG, bool COMP, bool DENSE, int TY, bool SPLIT = false>
cudaError_t launch_stage2d_d(const Stage2DArgs& a0, cudaStream_t s) {
  Stage2DArgs a = a0;
  CUtensorMap map, lo_map;
  a.tma = encode_box_map(a.w, a.nx, a.ny, 3 * C, (int)sizeof(R), RX, TY + 6, &map) ? 1 : 0;
  memset(&lo_map, 0, sizeof(lo_map));
  if (COMP && a.tma)  // both boxes, or neither
    a.tma = encode_box_map(a.w_lo, a.nx, a.ny, C, (int)sizeof(R), RX, TY + 6, &lo_map) ? 1 : 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((a.nx + TX - 1) / TX), (unsigned)((a.ny + TY - 1) / TY));
  cfg.blockDim = dim3(Smem2D<R, C, NG, COMP, TY, SPLIT>::NT);
  cfg.dynamicSmemBytes = sizeof(Smem2D<R, C, NG, COMP, TY, SPLIT>);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, stage2d_kernel<R, C, NG, COMP, DENSE, TY, SPLIT>, a, map, lo_map);
}

// Rows of a tile: 8, or in FP64 4 (128 threads, two CTAs per SM) while the 8-row
// tiles are a single wave: the FP64 pipes of the SMs bound those grids, and
// half-tiles use twice as many (3 points, 4 steps, 8 / 4 rows: 40 x 40 vortex 1.67
// / 0.98 ms, 150 x 120 1.66 / 1.22, four quadrants 3.08 / 2.35).  Beyond, smooth
// data gain 10-20 % and data with shocks lose as much (a tile's listed items have
// half the warps; 250 x 190 vortex 3.22 / 2.58, quadrants 3.94 / 4.42), so 8 stays.
// FP32 is faster with 8 at every size (120 x 120 equal, 512 x 512 quadrants 11 %).
int stage2d_rows(const Stage2DArgs& a) {
  return a.fp64 && stage2d_tiles(a.nx, a.ny) <= 152 ? 4 : 8;
}

template <typename R, int C, int NG, bool COMP>
cudaError_t launch_stage2d_t(const Stage2DArgs& a, cudaStream_t s) {
  if constexpr (has_dense<R, C, NG>()) {
    if (stage2d_dense(stage2d_tiles(a.nx, a.ny))) return launch_stage2d_d<R, C, NG, COMP, true, 8>(a, s);
  }
  if constexpr (sizeof(R) == 8) {
    if (stage2d_rows(a) == 4) return launch_stage2d_d<R, C, NG, COMP, false, 4>(a, s);
  } else {
    if (stage2d_tiles(a.nx, a.ny) <= 152) return launch_stage2d_d<R, C, NG, COMP, false, 8, true>(a, s);
  }
  return launch_stage2d_d<R, C, NG, COMP, false, 8>(a, s);
}

template <typename R, int C, int NG, bool COMP, bool DENSE, int TY, bool SPLIT = false>
cudaError_t prepare_one() {
  cudaError_t e = cudaFuncSetAttribute(stage2d_kernel<R, C, NG, COMP, DENSE, TY, SPLIT>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)sizeof(Smem2D<R, C, NG, COMP, TY, SPLIT>));
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(stage2d_kernel<R, C, NG, COMP, DENSE, TY, SPLIT>,
                              cudaFuncAttributePreferredSharedMemoryCarveout, 100);
}
template <typename R, int C, int NG>
cudaError_t prepare_t() {
  cudaError_t e = prepare_one<R, C, NG, false, false, 8>();
  if constexpr (sizeof(R) == 8) {
    if (e == cudaSuccess) e = prepare_one<R, C, NG, false, false, 4>();
  } else {
    if (e == cudaSuccess) e = prepare_one<R, C, NG, true, false, 8>();
    if (e == cudaSuccess) e = prepare_one<R, C, NG, false, false, 8, true>();
    if (e == cudaSuccess) e = prepare_one<R, C, NG, true, false, 8, true>();
  }
  if constexpr (has_dense<R, C, NG>()) {
    if (e == cudaSuccess) e = prepare_one<R, C, NG, false, true, 8>();
    if (e == cudaSuccess) e = prepare_one<R, C, NG, true, true, 8>();
  }
  return e;
}

}  // namespace

int stage2d_tiles(int nx, int ny) { return ((nx + TX - 1) / TX) * ((ny + TYW - 1) / TYW); }

bool encode_box_map(const void* w, int nx, int ny, int planes, int esize, int box_x, int box_y,
                    CUtensorMap* map) {
  static PFN_cuTensorMapEncodeTiled_v12000 encode = [] {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault,
                                         &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      fn = nullptr;
    return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
  }();
  memset(map, 0, sizeof(*map));
  if (!encode || !w || ((size_t)nx * esize) % 16 != 0 || ((uintptr_t)w) % 16 != 0 || nx < box_x ||
      ny < box_y || ((size_t)box_x * esize) % 16 != 0 || box_x > 256 || box_y > 256 || planes > 256)
    return false;
  const cuuint64_t dims[3] = {(cuuint64_t)nx, (cuuint64_t)ny, (cuuint64_t)planes};
  const cuuint64_t strides[2] = {(cuuint64_t)nx * esize, (cuuint64_t)nx * ny * esize};
  const cuuint32_t box[3] = {(cuuint32_t)box_x, (cuuint32_t)box_y, (cuuint32_t)planes};
  const cuuint32_t estr[3] = {1, 1, 1};
  return encode(map, esize == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_FLOAT64,
                3, const_cast<void*>(w), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

void finish_stage2d_args(Stage2DArgs& a) {
  a.inv_dx = 1.0 / a.dx;
  a.inv_dy = 1.0 / a.dy;
  const double h = 0.5 * sqrt(a.dx * a.dx + a.dy * a.dy);
  a.kx.dx = a.dx;
  a.kx.dy = a.dy;
  a.kx.den_h = h * (a.dx + a.dy);
  a.kx.thr = a.thr;
  a.kx.fdx = (float)a.dx;
  a.kx.fdy = (float)a.dy;
  a.kx.fthr_den = (float)(a.thr * a.kx.den_h);
  a.kx.fdx_lo = (float)(a.dx - (double)a.kx.fdx);
  a.kx.fdy_lo = (float)(a.dy - (double)a.kx.fdy);
  a.kx.fthr_den_lo = (float)(a.thr * a.kx.den_h - (double)a.kx.fthr_den);
  for (int k = 0; k < 5; ++k) a.f32[k] = (float)a.gam[k];
  a.f32[5] = (float)a.eps;
  a.f32[6] = (float)a.gas;
  a.f32[7] = (float)a.inv_dx;
  a.f32[8] = (float)a.inv_dy;
  a.f32[9] = (float)a.cfl;
}

cudaError_t prepare_stage2d(int system, int fp64, int ng) {
  if (system == 0) {
    if (fp64) return ng == 2 ? prepare_t<double, 1, 2>() : prepare_t<double, 1, 3>();
    return ng == 2 ? prepare_t<float, 1, 2>() : prepare_t<float, 1, 3>();
  }
  if (fp64) return ng == 2 ? prepare_t<double, 4, 2>() : prepare_t<double, 4, 3>();
  return ng == 2 ? prepare_t<float, 4, 2>() : prepare_t<float, 4, 3>();
}

cudaError_t launch_stage2d(const Stage2DArgs& a, cudaStream_t s) {
  if (a.comp) {  // HWENO_FP32C (stages 1-3 of a step)
    if (a.system == 0)
      return a.ng == 2 ? launch_stage2d_t<float, 1, 2, true>(a, s) : launch_stage2d_t<float, 1, 3, true>(a, s);
    return a.ng == 2 ? launch_stage2d_t<float, 4, 2, true>(a, s) : launch_stage2d_t<float, 4, 3, true>(a, s);
  }
  if (a.system == 0) {
    if (a.fp64) return a.ng == 2 ? launch_stage2d_t<double, 1, 2, false>(a, s) : launch_stage2d_t<double, 1, 3, false>(a, s);
    return a.ng == 2 ? launch_stage2d_t<float, 1, 2, false>(a, s) : launch_stage2d_t<float, 1, 3, false>(a, s);
  }
  if (a.fp64) return a.ng == 2 ? launch_stage2d_t<double, 4, 2, false>(a, s) : launch_stage2d_t<double, 4, 3, false>(a, s);
  return a.ng == 2 ? launch_stage2d_t<float, 4, 2, false>(a, s) : launch_stage2d_t<float, 4, 3, false>(a, s);
}

template <typename R>
static cudaError_t launch_dt2d_t(const Stage2DArgs& a, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(1);
  cfg.blockDim = dim3(32);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, dt2d_kernel<R>, static_cast<const R*>(a.a_in), a.nin, a.sc, a.cfl,
                            a.inv_dx, a.inv_dy);
}

cudaError_t launch_dt2d(const Stage2DArgs& a, cudaStream_t s) {
  return a.fp64 ? launch_dt2d_t<double>(a, s) : launch_dt2d_t<float>(a, s);
}

cudaError_t launch_alpha2d(const void* w, void* a_out, int nx, int ny, int system, int fp64,
                           double gas, DevScalars* sc, int slots, cudaStream_t s) {
  dim3 grid((nx + TX - 1) / TX, (ny + TYW - 1) / TYW);
  if (system == 0) {
    if (fp64)
      alpha2d_kernel<double, 1><<<grid, NTW, 0, s>>>(static_cast<const double*>(w), static_cast<double*>(a_out), nx, ny, gas, sc, slots);
    else
      alpha2d_kernel<float, 1><<<grid, NTW, 0, s>>>(static_cast<const float*>(w), static_cast<float*>(a_out), nx, ny, gas, sc, slots);
  } else {
    if (fp64)
      alpha2d_kernel<double, 4><<<grid, NTW, 0, s>>>(static_cast<const double*>(w), static_cast<double*>(a_out), nx, ny, gas, sc, slots);
    else
      alpha2d_kernel<float, 4><<<grid, NTW, 0, s>>>(static_cast<const float*>(w), static_cast<float*>(a_out), nx, ny, gas, sc, slots);
  }
  return cudaGetLastError();
}

}  // namespace hw
