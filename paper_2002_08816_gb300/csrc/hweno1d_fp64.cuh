// One third-order TVD Runge-Kutta stage of the 1D hybrid HWENO scheme (Zhao &
// Qiu, arXiv:2002.08816, Sec. 2.1) on one tile in FP64, split into small tasks.
//
// What bounds it: the FP64 pipe.  On GB300 an SM retires one FP64 warp
// instruction every ~19 cycles, and a single warp one every ~64, whatever the
// number of active lanes and independent chains (measured: dependent and
// 4-way independent DFMA chains, 1 to 32 active lanes, 1 to 16 warps).  So the
// cost of a phase is the number of FP64 warp instructions on the busiest SM
// sub-partition, and everything here serves that number:
//   * the work of a cell is cut into tasks of one component, one point or one
//     characteristic field, which consecutive lanes of all warps take, so a
//     small tile uses all four sub-partitions and no warp carries a
//     whole cell's chain (per cell ~210 FP64 instructions, ~95 on the longest
//     path of a tile of up to 30 cells);
//   * the characteristic work of a troubled cell runs as three lanes (its
//     fields) of a warp that holds up to ten such cells, instead of one lane
//     of an otherwise idle warp doing all three;
//   * the KXRCF decision is taken in FP32 on the truncated data when the error
//     bound allows (no FP64 instruction, not even a conversion), in FP64
//     otherwise: the same flags;
//   * each Lax-Friedrichs flux is formed once for the two cells that share it,
//     p0's four values share their even and odd parts, and signs, finiteness
//     and maxima are read off the bit patterns.
// A CTA of NTH cell threads works on Tq <= TMAX cells and 3 halo cells a side;
// slot e of every array is cell base - 3 + e.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "hweno1d_fields.cuh"
#include "hweno1d_stage.cuh"

namespace hw {
namespace f64 {

using s1d::bar_sync;
using s1d::kBarCells;

template <int C, int TMAX>
struct Smem64 {
  static constexpr int NE = TMAX + 6;
  double u[2][C][2][NE];             // stage input and output (they alternate)
  double vl[C][NE];                  // modified first moments, slots 1 .. Tq+4
  double P[4][C][NE];                // u^+_{i-1/2}, u^-_{i+1/2} (slots 2 .. Tq+3), the interior values
  double F[4][C == 3 ? 2 : 1][NE];   // their fluxes (Euler: of momentum and energy)
  double q[C][NE];                   // Lax-Friedrichs flux at x_{e-1/2}
  double alpha, dt;
  uint8_t fl[NE];
  unsigned short tb[NE], hw[NE];     // troubled cells; cells next to one
  int ntb, nhw;
};

// kxrcf_troubled(double ...) with the FP32 test in front: the truncated terms
// carry 2^-23 S, the FP32 jump four roundings (together below 8e-7 S, S as
// in the FP32 form), the threshold three roundings and a truncation (7e-7).
__device__ __forceinline__ bool troubled(double um, double u0, double up, double vm, double v0,
                                         double vp, bool left, double h, double thr, float hthr) {
  const double un = left ? um : up, vn = left ? vm : vp;
  const float fu = trunc32(u0), fv = trunc32(v0), gu = trunc32(un), gv = trunc32(vn);
  const float s6 = left ? -6.0f : 6.0f;
  const float j = fabsf(fmaf(s6, fv, fu) - fmaf(-s6, gv, gu));
  const float e = 8.0e-7f * (fabsf(fu) + 6.0f * fabsf(fv) + fabsf(gu) + 6.0f * fabsf(gv)) + 1e-28f;
  const float r = hthr * fmaxf(fabsf(fu), 1e-12f);
  if (fu == fu && j - e > r * (1.0f + 7.0e-7f)) return true;
  if (fu == fu && j + e < r * (1.0f - 7.0e-7f)) return false;
  return kxrcf_troubled(um, u0, up, vm, v0, vp, left, h, thr, 0.0f, 0.0f);
}

// Physical flux: Euler (momentum and energy; that of density is m), Burgers.
template <int C>
__device__ __forceinline__ void flux(double gas, const double* U, double* F) {
  if constexpr (C == 1) {
    F[0] = 0.5 * U[0] * U[0];
  } else {
    const double mu = U[1] / U[0];
    const double p = (gas - 1.0) * fma(-0.5 * U[1], mu, U[2]);
    F[0] = fma(U[1], mu, p);
    F[1] = mu * (U[2] + p);
  }
}

// The parameters of a stage.
struct Par {
  double gam[3], eps, gas, h, thr, inv_dx;
  float hthr;
  int mode, variant;
};

// Step 1 and the lists: flags and modified first moments of slots 1 .. Tq+4 of
// the stage input u, and the cells whose faces need Step 2.1.  Ends with a
// barrier of the cell threads.  Returns the number of own troubled cells seen
// by this thread.
template <int C, int TMAX, int NTH>
__device__ __forceinline__ int step1(Smem64<C, TMAX>& sm, const double (*u)[2][TMAX + 6], int Tq, int tid,
                                     const Par& a) {
  int mine = 0;
  if (tid == 0) sm.ntb = sm.nhw = 0;
  bar_sync(kBarCells, NTH);
  for (int e = 1 + tid; e <= Tq + 4; e += NTH) {
    bool flag;
    if (a.mode != 0) {
      flag = a.mode == 1;
    } else {
      const bool left = C == 1 ? ge0(u[0][0][e]) : inflow_left(u[0][0][e], u[C == 3 ? 1 : 0][0][e]);
      flag = troubled(u[0][0][e - 1], u[0][0][e], u[0][0][e + 1], u[0][1][e - 1], u[0][1][e],
                      u[0][1][e + 1], left, a.h, a.thr, a.hthr);
      if constexpr (C == 3)
        flag = flag || troubled(u[2][0][e - 1], u[2][0][e], u[2][0][e + 1], u[2][1][e - 1],
                                u[2][1][e], u[2][1][e + 1], left, a.h, a.thr, a.hthr);
    }
    sm.fl[e] = flag;
    mine += flag && e >= 3 && e < Tq + 3;
    if (flag) sm.tb[atomicAdd(&sm.ntb, 1)] = (unsigned short)e;
    else {
#pragma unroll
      for (int c = 0; c < C; ++c) sm.vl[c][e] = u[c][1][e];
    }
  }
  bar_sync(kBarCells, NTH);
  const int ntb = sm.ntb;
  if (ntb > 0) {  // uniform over the CTA
    constexpr int PW = 32 / C;  // cells a warp takes at once
    const int lane = tid & 31, f = lane % C, base = lane - f;
    for (int k0 = (tid >> 5) * PW; k0 < ntb; k0 += (NTH / 32) * PW) {  // uniform over the warp
      const int k = k0 + lane / C;
      const bool on = lane < PW * C && k < ntb;
      const int e = sm.tb[on ? k : k0];
      double U[C], l[C], r[C], d[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll
      for (int c = 0; c < C; ++c) U[c] = u[c][0][e];
      fld::field<double, C>(a.gas, U, f, l, r);
#pragma unroll
      for (int c = 0; c < C; ++c) {
        d[0] = fma(l[c], u[c][0][e - 1], d[0]);
        d[1] = fma(l[c], U[c], d[1]);
        d[2] = fma(l[c], u[c][0][e + 1], d[2]);
        d[3] = fma(l[c], u[c][1][e - 1], d[3]);
        d[4] = fma(l[c], u[c][1][e + 1], d[4]);
      }
      const double v = fld::to_component<double, C>(r, fld::limit_moment(d[0], d[1], d[2], d[3], d[4], a.gam, a.eps), f,
                                       min(base, 32 - C));
      if (on) sm.vl[f][e] = v;
    }
    for (int e = 2 + tid; e <= Tq + 3; e += NTH)
      if (sm.fl[e - 1] | sm.fl[e] | sm.fl[e + 1]) sm.hw[atomicAdd(&sm.nhw, 1)] = (unsigned short)e;
    bar_sync(kBarCells, NTH);
  }
  return mine;
}

// Step 2 and the physical fluxes: P and F.  Ends with a barrier.
template <int C, int TMAX, int NTH>
__device__ __forceinline__ void step2(Smem64<C, TMAX>& sm, const double (*u)[2][TMAX + 6], int Tq, int tid,
                                      const Par& a) {
  const int n1 = Tq + 2;
  for (int t = tid; t < C * n1; t += NTH) {  // (component, cell)
    const int c = t / n1, e = 2 + t - c * n1;
    const double um = u[c][0][e - 1], u0 = u[c][0][e], up = u[c][0][e + 1];
    const double vm = sm.vl[c][e - 1], v0 = sm.vl[c][e], vp = sm.vl[c][e + 1];
    const double d1 = u0 - um, d2 = up - u0, sV = vm + vp, dV = vm - vp;
    const double D = d2 + d1, cU = d2 - d1;
    double l, r, gm, gp;
    fld::p0_faces(u0, D, cU, sV, dV, v0, l, r);
    fld::p0_interior(u0, D, cU, sV, dV, v0, gm, gp);
    sm.P[0][c][e] = l;
    sm.P[1][c][e] = r;
    sm.P[2][c][e] = gm;
    sm.P[3][c][e] = gp;
  }
  bar_sync(kBarCells, NTH);
  const int nhw = sm.nhw;
  if (nhw > 0) {  // uniform over the CTA: Step 2.1 where the stencil holds a troubled cell
    constexpr int PW = 32 / C;
    const int lane = tid & 31, f = lane % C, base = lane - f;
    const bool mean = C == 3 && (a.variant & HWENO_VARIANT_MEAN_EIGEN);
    for (int k0 = (tid >> 5) * PW; k0 < nhw; k0 += (NTH / 32) * PW) {
      const int k = k0 + lane / C;
      const bool on = lane < PW * C && k < nhw;
      const int e = sm.hw[on ? k : k0];
      for (int side = 0; side < (mean ? 2 : 1); ++side) {
        double B[C], l[C], r[C], d[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll
        for (int c = 0; c < C; ++c)
          B[c] = mean ? 0.5 * (u[c][0][e - 1 + side] + u[c][0][e + side]) : u[c][0][e];
        fld::field<double, C>(a.gas, B, f, l, r);
#pragma unroll
        for (int c = 0; c < C; ++c)
#pragma unroll
          for (int j = 0; j < 3; ++j) {
            d[j] = fma(l[c], u[c][0][e - 1 + j], d[j]);
            d[3 + j] = fma(l[c], sm.vl[c][e - 1 + j], d[3 + j]);
          }
        double cl, cr;
        fld::hweno(d[0], d[1], d[2], d[3], d[4], d[5], a.gam, a.eps, cl, cr);
        const int b = min(base, 32 - C);
        if (!mean || side == 0) {
          const double v = fld::to_component<double, C>(r, cl, f, b);
          if (on) sm.P[0][f][e] = v;
        }
        if (!mean || side == 1) {
          const double v = fld::to_component<double, C>(r, cr, f, b);
          if (on) sm.P[1][f][e] = v;
        }
      }
    }
    bar_sync(kBarCells, NTH);
  }
  for (int t = tid; t < 4 * n1; t += NTH) {  // (point, cell)
    const int p = t / n1, e = 2 + t - p * n1;
    double U[C], F[C == 3 ? 2 : 1];
#pragma unroll
    for (int c = 0; c < C; ++c) U[c] = sm.P[p][c][e];
    flux<C>(a.gas, U, F);
#pragma unroll
    for (int k = 0; k < (C == 3 ? 2 : 1); ++k) sm.F[p][k][e] = F[k];
  }
  bar_sync(kBarCells, NTH);
}

template <int C, int TMAX>
__device__ __forceinline__ double flux_at(const Smem64<C, TMAX>& sm, int p, int c, int e) {
  if constexpr (C == 1) return sm.F[p][0][e];
  else return c == 0 ? sm.P[p][1][e] : sm.F[p][c - 1][e];
}

// The Lax-Friedrichs flux at every interface of the tile.  Ends with a barrier.
template <int C, int TMAX, int NTH>
__device__ __forceinline__ void lax_friedrichs(Smem64<C, TMAX>& sm, int Tq, int tid, double alpha) {
  const double ha = 0.5 * alpha;
  for (int t = tid; t < C * (Tq + 1); t += NTH) {
    const int c = t / (Tq + 1), e = 3 + t - c * (Tq + 1);
    sm.q[c][e] = fma(-ha, sm.P[0][c][e] - sm.P[1][c][e - 1],
                     0.5 * (flux_at(sm, 1, c, e - 1) + flux_at(sm, 0, c, e)));
  }
  bar_sync(kBarCells, NTH);
}

// dx Lu and dx Lv of Eq. (odeH) for component c of slot e.
template <int C, int TMAX>
__device__ __forceinline__ void rhs_at(const Smem64<C, TMAX>& sm, int c, int e, double& Gu, double& Gv) {
  const double ql = sm.q[c][e], qr = sm.q[c][e + 1];
  const double F = fma(5.0 / 12.0, flux_at(sm, 2, c, e) + flux_at(sm, 3, c, e),
                       (1.0 / 12.0) * (flux_at(sm, 0, c, e) + flux_at(sm, 1, c, e)));
  Gu = ql - qr;
  Gv = fma(-0.5, ql + qr, F);
}

// Maximum wave speed at an average (NaN when not physical), one reciprocal.
template <int C>
__device__ __forceinline__ double speed_at(double gas, const double* U) {
  if constexpr (C == 1) {
    return fabs(U[0]);
  } else {
    if (!gt0(U[0])) return NAN;
    const double ir = __drcp_rn(U[0]);
    const double mu = U[1] * ir;
    const double p = (gas - 1.0) * fma(-0.5 * U[1], mu, U[2]);
    if (!gt0(p)) return NAN;
    return fabs(mu) + sqrt(gas * p * ir);
  }
}

// The warp's largest bit pattern of non-negative doubles.
__device__ __forceinline__ unsigned long long warp_max_bits(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const unsigned hi = (unsigned)(b >> 32);
  const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
  const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? (unsigned)b : 0u);
  return ((unsigned long long)mh << 32) | ml;
}

}  // namespace f64
}  // namespace hw
