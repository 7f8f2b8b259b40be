// One FP64 stage on one tile, from and to global memory: the tasks of
// hweno1d_fp64.cuh under the per-stage and the persistent launches (batches,
// the right-hand side, and grids too large for the resident run).
#pragma once
#include "hweno1d_fp64.cuh"

namespace hw {
namespace f64 {

using s1d::H;
using s1d::kBarAll;
using s1d::ldx;

// A tile of TMAX cells, by a CTA of NTH cell threads and the scalar warp (whose
// work is the FP32 stages': s1d::scalar_warp).
template <int C, bool BATCH, int TMAX, int NTH>
__device__ __forceinline__ void stage64_tile(Stage1DArgs a, const int tile, Smem64<C, TMAX>& sm) {
  const int tid = threadIdx.x, lane = tid & 31;
  const s1d::TileAt at = s1d::tile_at<double, C, BATCH>(a, tile, TMAX);
  const int n = at.n, base = at.base, Tq = min(TMAX, n - base);
  // the producer of the stage input may still be finishing (programmatic
  // dependent launch): wait for its completion and memory before any read
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (tid >= NTH) {
    s1d::scalar_warp<double, BATCH>(a, tile, at.inst, at.lead, lane, NTH, &sm.alpha, &sm.dt);
    return;
  }
  const Par par = {{a.gam[0], a.gam[1], a.gam[2]}, a.eps, a.gas, a.h, a.thr, a.inv_dx,
                   a.hthr, a.mode, a.variant};
  const double* __restrict__ w = static_cast<const double*>(a.w);
  double(*u)[2][TMAX + 6] = sm.u[0];
  double(*un)[2][TMAX + 6] = sm.u[1];
  for (int e = tid; e < Tq + 2 * H; e += NTH) {
    bool mir = false;
    const int g = a.bc == 2 ? bc_map_wall(base - H + e, n, &mir) : bc_map(base - H + e, n, a.bc);
#pragma unroll
    for (int c = 0; c < C; ++c)
#pragma unroll
      for (int m = 0; m < 2; ++m) {
        const double x = ldx(w + (2 * c + m) * n + g);
        u[c][m][e] = mir ? (double)mirror_sign(c, m) * x : x;
      }
  }
  bar_sync(kBarCells, NTH);
  // the next stage's CTAs may be scheduled now; they wait for this grid above
  asm volatile("griddepcontrol.launch_dependents;");
  int mine = step1<C, TMAX, NTH>(sm, u, Tq, tid, par);
  step2<C, TMAX, NTH>(sm, u, Tq, tid, par);
  bar_sync(kBarAll, NTH + 32);  // alpha and dt from the scalar warp
  const double alpha = sm.alpha, dt = sm.dt;
  if (a.stage > 0 && !(dt > 0.0)) return;  // t_final reached: the stage writes nothing
  lax_friedrichs<C, TMAX, NTH>(sm, Tq, tid, alpha);
  const double kd = dt * par.inv_dx;
  const double cb = a.stage == 2 ? 0.25 : 2.0 / 3.0;
  const double* u0 = static_cast<const double*>(a.u0);
  double* out = static_cast<double*>(a.out);
  double* lim = static_cast<double*>(a.lim_out);
  unsigned bad = 0u;
  for (int t = tid; t < C * Tq; t += NTH) {
    const int c = t / Tq, i = t - c * Tq, e = i + H;
    const size_t gu = (size_t)(2 * c) * n + base + i, gv = gu + n;
    double z0 = 0.0, z1 = 0.0;
    if (a.stage >= 2) {
      z0 = ldx(u0 + gu);
      z1 = ldx(u0 + gv);
    }
    double Gu, Gv;
    rhs_at<C, TMAX>(sm, c, e, Gu, Gv);
    const double wu = u[c][0][e], wvm = sm.vl[c][e];
    const double wv = (a.variant & HWENO_VARIANT_RAW_COMBINE) ? u[c][1][e] : wvm;
    double ou, ov;
    if (a.stage == 0) {
      ou = Gu * par.inv_dx;
      ov = Gv * par.inv_dx;
    } else {
      ou = fma(kd, Gu, wu);
      ov = fma(kd, Gv, wv);
      if (a.stage >= 2) {
        ou = rk_combine(cb, z0, ou);
        ov = rk_combine(cb, z1, ov);
      }
    }
    out[gu] = ou;
    out[gv] = ov;
    un[c][0][e] = ou;
    if (lim) {
      lim[gu] = wu;
      lim[gv] = a.stage == 0 ? wvm : wv;  // rhs mode: the modified moment
    }
    if (!is_finite(ou) || !is_finite(ov)) bad |= ST_NONFINITE;
    if (c == 0 && a.flags_out) a.flags_out[base + i] = sm.fl[e];
  }
  if (a.stage > 0) {
    bar_sync(kBarCells, NTH);
    double sp = 0.0;
    for (int i = tid; i < Tq; i += NTH) {
      double U[C];
#pragma unroll
      for (int c = 0; c < C; ++c) U[c] = un[c][0][i + H];
      const double v = speed_at<C>(par.gas, U);
      if (v == v) sp = fmax(sp, v);
      else bad |= ST_NONPHYSICAL;
    }
    // each warp folds its maximum into the tile's slot (one per instance in a batch)
    if ((tid & ~31) < Tq) {
      const unsigned long long m = warp_max_bits(sp);
      if (lane == 0 && a.a_out)
        atomicMax(static_cast<unsigned long long*>(a.a_out) + (BATCH ? at.inst : tile % kAlphaSlots), m);
    }
  }
  mine = __reduce_add_sync(0xffffffffu, (unsigned)mine);
  if (lane == 0 && mine) atomicAdd(&a.sc->troubled, (unsigned long long)mine);
  if (bad) atomicOr(&a.sc->status, bad);
}

}  // namespace f64
}  // namespace hw
