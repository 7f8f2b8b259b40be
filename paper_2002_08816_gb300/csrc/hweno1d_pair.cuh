// One FP32 stage of the 1D scheme (Zhao & Qiu, arXiv:2002.08816, Sec. 2.1) on
// one tile from and to global memory, two cells per thread in packed FP32.
//
// What bounds it: issue (a cell per thread took 625 instructions per
// cell-stage at 71-79 % issue activity on the 512-instance batch).  So a thread
// works on slot e of two half-tiles at once, cell base - 3 + e in the x halves
// of its pairs and cell base + W - 3 + e in the y halves (W = half the tile's
// cells): every shared-memory access is 64 bits for two cells, and the maps,
// fluxes, quadratures and combinations run as fma.rn.f32x2, one instruction
// for both.  Only the decisions (KXRCF, wave speeds, status) are taken half by
// half.  The halves' halos overlap, 6 slots of a half-tile's W + 6.  A thread
// keeps its slot's data from the flags to the combination in registers (the
// interior values and their fluxes never leave them).
//
// Euler: troubled cells and the cells next to them are listed, and their
// characteristic work runs as one field per lane, ten cells to a warp: with
// thread-own work a warp with one troubled cell ran all three fields' chains
// for its other 31 lanes' sake.  Burgers has one field: the thread that holds the
// cell does it (two barriers and a list less).
//
// Measured (GB300, us per stage, a cell per thread -> this): 512 instances of
// 256-16384 cells, 128 threads 62.7 -> 43.3; 1000000 cells 36.5 -> 22.4; 300000
// 10.5 -> 8.4.  What bounds it now: issue 56 % with the load latency of a tile on
// 20 cell warps per SM; 72 registers (5 CTAs per SM) is the best of 102 / 72 /
// 64 / 56 (53.4 / 43.3 / 46.1 / 47.7 on the batch).  One record per batch tile and
// asynchronous copies into shared memory took 51.5 to 43.8.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "hweno1d_fields.cuh"
#include "hweno1d_stage.cuh"

namespace hw {
namespace pr {

using s1d::bar_sync;
using s1d::H;
using s1d::kBarAll;
using s1d::kBarCells;
using s1d::ldx;

template <int C, int NTH>
struct SmemPair {
  static constexpr int WMAX = NTH - 2 * H, NE = NTH;  // cells of a half-tile, slots
  float2 u[C][2][NE];                 // stage input
  float2 z[C][2][NE];                 // limited u^n of the own cells (stages 2, 3)
  float2 vl[C][NE];                   // modified first moments, slots 1 .. W+4
  float2 P[2][C][NE];                 // u^+_{i-1/2}, u^-_{i+1/2}, slots 2 .. W+3
  float2 F[2][C == 3 ? 2 : 1][NE];    // their fluxes (Euler: of momentum and energy)
  uint8_t fl[NE];                     // troubled: bit 0 the x half, bit 1 the y half
  unsigned short tb[2 * NE], hw[2 * NE];  // 2 slot + half of troubled cells, of cells next to one
  int ntb, nhw;
  unsigned wmax;                      // the tile's maximum wave speed (bits)
  float alpha, dt;
};

// An asynchronous 4-byte copy from global (through L2 or L1: data of an earlier
// launch, or of this one written before a grid barrier) into shared memory.
__device__ __forceinline__ void copy4(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ float half_of(float2 v, int y) { return y ? v.y : v.x; }
__device__ __forceinline__ float at(const float2* p, int e, int y) {
  return reinterpret_cast<const float*>(p + e)[y];
}
__device__ __forceinline__ float2 k2(double c) { return bcast2((float)c); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

// Physical flux of two states: Euler (momentum and energy; that of density is
// m), Burgers.
template <int C>
__device__ __forceinline__ void flux2(float gas, const float2* U, float2* F) {
  if constexpr (C == 1) {
    F[0] = mul2(mul2(k2(0.5), U[0]), U[0]);
  } else {
    const float2 ir = make_float2(rcp_approx(U[0].x), rcp_approx(U[0].y));
    const float2 mu = mul2(U[1], ir);
    const float2 p = mul2(bcast2(gas - 1.0f), fma2(mul2(k2(-0.5), U[1]), mu, U[2]));
    F[0] = fma2(U[1], mu, p);
    F[1] = mul2(mu, add2(U[2], p));
  }
}

// p0 of fld::p0_faces and fld::p0_interior on pairs.
__device__ __forceinline__ void p0_pair(float2 um, float2 u0, float2 up, float2 vm, float2 v0, float2 vp,
                                        float2& l, float2& r, float2& gm, float2& gp) {
  constexpr double r5 = 2.2360679774997896964;
  const float2 d1 = sub2(u0, um), d2 = sub2(up, u0), sV = add2(vm, vp), dV = sub2(vm, vp);
  const float2 D = add2(d2, d1), c = sub2(d2, d1);
  const float2 ef = fma2(k2(5.0 / 24.0), c, mul2(k2(0.75), dV));
  const float2 of = fma2(k2(19.0 / 216.0), D, fma2(k2(-31.0 / 108.0), sV, mul2(k2(241.0 / 54.0), v0)));
  l = add2(u0, sub2(ef, of));
  r = add2(u0, add2(ef, of));
  const float2 ei = fma2(k2(-1.0 / 24.0), c, mul2(k2(-0.15), dV));
  const float2 oi = fma2(k2(-101.0 / 5400.0 * r5), D,
                    fma2(k2(841.0 / 13500.0 * r5), sV, mul2(k2(10289.0 / 6750.0 * r5), v0)));
  gm = add2(u0, sub2(ei, oi));
  gp = add2(u0, add2(ei, oi));
}

// kxrcf_troubled(float ...) for the inflow face's two cells: the fast test here
// without a branch on the side, with the bounds of hweno1d_recon.cuh (8 %
// wider), the float-pair form out of line.
__device__ __noinline__ bool kxrcf_close(float u0, float v0, float un, float vn, bool left, float hthr,
                                         float hthr_lo) {
  float jh, jl;
  jump_pair(u0, v0, un, vn, left, jh, jl);
  if (jh < 0.0f) {
    jh = -jh;
    jl = -jl;
  }
  const float nrm = fmaxf(fabsf(u0), 1e-12f);
  const float rh = __fmul_rn(nrm, hthr);
  const float rl = __fadd_rn(fmaf(nrm, hthr, -rh), __fmul_rn(nrm, hthr_lo));
  return __fadd_rn(__fsub_rn(jh, rh), __fsub_rn(jl, rl)) > 0.0f;
}
__device__ __forceinline__ bool kxrcf_half(float um, float u0, float up, float vm, float v0, float vp,
                                           bool left, float hthr, float hthr_lo) {
  const float un = left ? um : up, vn = left ? vm : vp, s6 = left ? -6.0f : 6.0f;
  const float j = fabsf(fmaf(s6, v0, u0) - fmaf(-s6, vn, un));
  const float s = fmaf(6.0f, fabsf(v0), fabsf(u0)) + fmaf(6.0f, fabsf(vn), fabsf(un));
  const float r = hthr * fmaxf(fabsf(u0), 1e-12f);
  const float d = j - r, m = fmaf(6.5e-7f, s, 6.0e-7f * r);
  if (d > m) return true;
  if (d < -m) return false;
  return kxrcf_close(u0, v0, un, vn, left, hthr, hthr_lo);
}

// KXRCF of one half of a pair.
template <int C>
__device__ __forceinline__ bool troubled_half(const float2* um, const float2* u0, const float2* up,
                                              const float2* vm, const float2* v0, const float2* vp, int y,
                                              float hthr, float hthr_lo) {
  const bool left = C == 1 ? half_of(u0[0], y) >= 0.0f
                           : inflow_left(half_of(u0[0], y), half_of(u0[C == 1 ? 0 : 1], y));
  bool f = kxrcf_half(half_of(um[0], y), half_of(u0[0], y), half_of(up[0], y), half_of(vm[0], y),
                      half_of(v0[0], y), half_of(vp[0], y), left, hthr, hthr_lo);
  if constexpr (C == 3)
    f |= kxrcf_half(half_of(um[2], y), half_of(u0[2], y), half_of(up[2], y), half_of(vm[2], y),
                    half_of(v0[2], y), half_of(vp[2], y), left, hthr, hthr_lo);
  return f;
}

// The limiter of the listed troubled cells: (cell, field) on consecutive lanes.
template <int C, int NTH>
__device__ __forceinline__ void limit_listed(SmemPair<C, NTH>& sm, int tid, float gas, float g0, float g1,
                                          float g2, float eps) {
  constexpr int PW = 32 / C;  // cells a warp takes at once
  const float gam[3] = {g0, g1, g2};
  const int lane = tid & 31, f = lane % C, base = min(lane - f, 32 - C), n = sm.ntb;
  for (int k0 = (tid >> 5) * PW; k0 < n; k0 += (NTH / 32) * PW) {  // uniform over the warp
    const int k = k0 + lane / C;
    const bool on = lane < PW * C && k < n;
    const int t = sm.tb[on ? k : k0], e = t >> 1, y = t & 1;
    float U[C], l[C], r[C], d[5] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int c = 0; c < C; ++c) U[c] = at(sm.u[c][0], e, y);
    fld::field<float, C>(gas, U, f, l, r);
#pragma unroll
    for (int c = 0; c < C; ++c) {
      d[0] = fmaf(l[c], at(sm.u[c][0], e - 1, y), d[0]);
      d[1] = fmaf(l[c], U[c], d[1]);
      d[2] = fmaf(l[c], at(sm.u[c][0], e + 1, y), d[2]);
      d[3] = fmaf(l[c], at(sm.u[c][1], e - 1, y), d[3]);
      d[4] = fmaf(l[c], at(sm.u[c][1], e + 1, y), d[4]);
    }
    const float v = fld::to_component<float, C>(
        r, fld::limit_moment(d[0], d[1], d[2], d[3], d[4], gam, eps), f, base);
    if (on) reinterpret_cast<float*>(&sm.vl[f][e])[y] = v;
  }
}

// Step 2.1 of the listed cells into P, the same way.
template <int C, int NTH>
__device__ __forceinline__ void hweno_listed(SmemPair<C, NTH>& sm, int tid, float gas, float g0, float g1,
                                          float g2, float eps, int variant) {
  constexpr int PW = 32 / C;
  const float gam[3] = {g0, g1, g2};
  const int lane = tid & 31, f = lane % C, base = min(lane - f, 32 - C), n = sm.nhw;
  const bool mean = C == 3 && (variant & HWENO_VARIANT_MEAN_EIGEN);
  for (int k0 = (tid >> 5) * PW; k0 < n; k0 += (NTH / 32) * PW) {
    const int k = k0 + lane / C;
    const bool on = lane < PW * C && k < n;
    const int t = sm.hw[on ? k : k0], e = t >> 1, y = t & 1;
    for (int side = 0; side < (mean ? 2 : 1); ++side) {
      float B[C], l[C], r[C], d[6] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
      for (int c = 0; c < C; ++c)
        B[c] = mean ? 0.5f * (at(sm.u[c][0], e - 1 + side, y) + at(sm.u[c][0], e + side, y))
                    : at(sm.u[c][0], e, y);
      fld::field<float, C>(gas, B, f, l, r);
#pragma unroll
      for (int c = 0; c < C; ++c)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          d[j] = fmaf(l[c], at(sm.u[c][0], e - 1 + j, y), d[j]);
          d[3 + j] = fmaf(l[c], at(sm.vl[c], e - 1 + j, y), d[3 + j]);
        }
      float cl, cr;
      fld::hweno(d[0], d[1], d[2], d[3], d[4], d[5], gam, eps, cl, cr);
      if (!mean || side == 0) {
        const float v = fld::to_component<float, C>(r, cl, f, base);
        if (on) reinterpret_cast<float*>(&sm.P[0][f][e])[y] = v;
      }
      if (!mean || side == 1) {
        const float v = fld::to_component<float, C>(r, cr, f, base);
        if (on) reinterpret_cast<float*>(&sm.P[1][f][e])[y] = v;
      }
    }
  }
}

// The same two out of line, for the 128-thread build, whose five CTAs per SM cover a
// call's latency; the others are 3-4 % faster with the work inline (100 instances of
// 40-400 cells, 256 threads: 4.13 -> 3.99 us per stage; 512 of 256-16384, 128 threads:
// 42.3 inline 42.5).
template <int C, int NTH>
__device__ __noinline__ void limit_call(SmemPair<C, NTH>& sm, int tid, float gas, float g0, float g1, float g2,
                                        float eps) {
  limit_listed<C, NTH>(sm, tid, gas, g0, g1, g2, eps);
}
template <int C, int NTH>
__device__ __noinline__ void hweno_call(SmemPair<C, NTH>& sm, int tid, float gas, float g0, float g1, float g2,
                                        float eps, int variant) {
  hweno_listed<C, NTH>(sm, tid, gas, g0, g1, g2, eps, variant);
}

// A tile of 2 (NTH - 6) cells by a CTA of NTH cell threads and the scalar warp
// (s1d::scalar_warp).
template <int C, bool BATCH, int NTH>
__device__ __forceinline__ void stage_tile(Stage1DArgs a, const int tile, SmemPair<C, NTH>& sm) {
  constexpr int T = 2 * SmemPair<C, NTH>::WMAX, NF = C == 3 ? 2 : 1;
  const int tid = threadIdx.x, lane = tid & 31;
  const s1d::TileAt where = s1d::tile_at<float, C, BATCH>(a, tile, T);
  const int n = where.n, base = where.base, Tq = min(T, n - base), W = (Tq + 1) >> 1;
  // the producer of the stage input may still be finishing (programmatic
  // dependent launch): wait for its completion and memory before any read
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (tid >= NTH) {
    s1d::scalar_warp<float, BATCH>(a, tile, where.inst, where.lead, lane, NTH, &sm.alpha, &sm.dt);
    return;
  }
  const float gam[3] = {a.f32[0], a.f32[1], a.f32[2]};
  const float eps = a.f32[3], gas = a.f32[4], inv_dx = a.f32[5];
  const float* __restrict__ w = static_cast<const float*>(a.w);
  // this thread's own cells: slot tid + 2 of both halves
  const int i0 = tid - 1;
  const bool ownx = tid >= 1 && i0 < W, owny = tid >= 1 && W + i0 < Tq;
  const int gx = base + i0, gy = gx + W;
  if (tid == 0) {
    sm.ntb = sm.nhw = 0;
    sm.wmax = 0u;
  }
  // the tile as asynchronous copies: nothing of it passes through registers
  bool mx = false, my = false;
  if (tid < W + 2 * H) {
    int sx, sy;
    if (a.bc == 2) {
      sx = bc_map_wall(base - H + tid, n, &mx);
      sy = bc_map_wall(base + W - H + tid, n, &my);
    } else {
      sx = bc_map(base - H + tid, n, a.bc);
      sy = bc_map(base + W - H + tid, n, a.bc);
    }
    const float *px = w + sx, *py = w + sy;
#pragma unroll
    for (int c = 0; c < C; ++c)
#pragma unroll
      for (int m = 0; m < 2; ++m) {
        copy4(&sm.u[c][m][tid].x, px);
        copy4(&sm.u[c][m][tid].y, py);
        px += n;
        py += n;
      }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
  if (a.stage >= 2) {
    const float* z = static_cast<const float*>(a.u0);
    const float *px = z + gx, *py = z + gy;
#pragma unroll
    for (int c = 0; c < C; ++c)
#pragma unroll
      for (int m = 0; m < 2; ++m) {
        if (ownx) copy4(&sm.z[c][m][tid].x, px);
        if (owny) copy4(&sm.z[c][m][tid].y, py);
        px += n;
        py += n;
      }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
  asm volatile("cp.async.wait_group 1;" ::: "memory");
  if (mx | my) {  // a mirror image behind a wall
#pragma unroll
    for (int c = 0; c < C; ++c)
#pragma unroll
      for (int m = 0; m < 2; ++m) {
        if (mx) sm.u[c][m][tid].x *= mirror_sign(c, m);
        if (my) sm.u[c][m][tid].y *= mirror_sign(c, m);
      }
  }
  bar_sync(kBarCells, NTH);
  // the next stage's CTAs may be scheduled now; they wait for this grid above
  asm volatile("griddepcontrol.launch_dependents;");

  // Step 1: slots 2 .. W+3 on the threads that hold them, 1 and W+4 on two more
  const int e = tid <= W + 1 ? tid + 2 : (tid == W + 2 ? 1 : W + 4);
  float2 um[C], u0[C], up[C], v0[C];
  int flag = 0;
  if (tid < W + 4) {
    float2 vm[C], vp[C];
#pragma unroll
    for (int c = 0; c < C; ++c) {
      um[c] = sm.u[c][0][e - 1];
      u0[c] = sm.u[c][0][e];
      up[c] = sm.u[c][0][e + 1];
      v0[c] = sm.u[c][1][e];
      if (c != 1) {  // (momentum does not enter KXRCF)
        vm[c] = sm.u[c][1][e - 1];
        vp[c] = sm.u[c][1][e + 1];
      }
    }
    if (a.mode != 0) {
      flag = a.mode == 1 ? 3 : 0;
    } else {
      flag = troubled_half<C>(um, u0, up, vm, v0, vp, 0, a.hthr, a.hthr_lo) |
             (troubled_half<C>(um, u0, up, vm, v0, vp, 1, a.hthr, a.hthr_lo) << 1);
    }
    sm.fl[e] = (uint8_t)flag;
    if constexpr (C == 1) {  // one field: the thread that holds the cell limits it
      if (flag & 1) v0[0].x = fld::limit_moment(um[0].x, u0[0].x, up[0].x, vm[0].x, vp[0].x, gam, eps);
      if (flag & 2) v0[0].y = fld::limit_moment(um[0].y, u0[0].y, up[0].y, vm[0].y, vp[0].y, gam, eps);
    }
#pragma unroll
    for (int c = 0; c < C; ++c) sm.vl[c][e] = v0[c];  // (listed cells: replaced below)
    if (C == 3 && flag) {
      int k = atomicAdd(&sm.ntb, __popc(flag));
      if (flag & 1) sm.tb[k++] = (unsigned short)(2 * e);
      if (flag & 2) sm.tb[k] = (unsigned short)(2 * e + 1);
    }
  }
  bar_sync(kBarCells, NTH);
  int hwm = 0;  // halves of this thread's slot whose stencil holds a troubled cell
  const bool any = C == 1 || sm.ntb > 0;  // uniform over the CTA
  if constexpr (C == 1) {
    if (tid < W + 2) hwm = sm.fl[e - 1] | sm.fl[e] | sm.fl[e + 1];
  } else if (any) {
    if constexpr (NTH == 128) limit_call<C, NTH>(sm, tid, gas, gam[0], gam[1], gam[2], eps);
    else limit_listed<C, NTH>(sm, tid, gas, gam[0], gam[1], gam[2], eps);
    if (tid < W + 2) {
      hwm = sm.fl[e - 1] | sm.fl[e] | sm.fl[e + 1];
      if (hwm) {
        int k = atomicAdd(&sm.nhw, __popc(hwm));
        if (hwm & 1) sm.hw[k++] = (unsigned short)(2 * e);
        if (hwm & 2) sm.hw[k] = (unsigned short)(2 * e + 1);
      }
    }
    bar_sync(kBarCells, NTH);
    if constexpr (NTH == 128) hweno_call<C, NTH>(sm, tid, gas, gam[0], gam[1], gam[2], eps, a.variant);
    else hweno_listed<C, NTH>(sm, tid, gas, gam[0], gam[1], gam[2], eps, a.variant);
    bar_sync(kBarCells, NTH);
  }

  // Step 2: the traces and their fluxes, and the interior values' fluxes
  float2 L[C], Rt[C], fL[NF], fR[NF], S[C];  // S: the sum of the interior fluxes
  if (tid < W + 2) {
    float2 gm[C], gp[C], f2[NF], f3[NF];
#pragma unroll
    for (int c = 0; c < C; ++c) {
      if (C == 3 && any) v0[c] = sm.vl[c][e];
      const float2 vm = sm.vl[c][e - 1], vp = sm.vl[c][e + 1];
      p0_pair(um[c], u0[c], up[c], vm, v0[c], vp, L[c], Rt[c], gm[c], gp[c]);
      if constexpr (C == 1) {
        if (hwm & 1) fld::hweno(um[c].x, u0[c].x, up[c].x, vm.x, v0[c].x, vp.x, gam, eps, L[c].x, Rt[c].x);
        if (hwm & 2) fld::hweno(um[c].y, u0[c].y, up[c].y, vm.y, v0[c].y, vp.y, gam, eps, L[c].y, Rt[c].y);
        continue;
      }
      if (hwm & 1) {
        L[c].x = sm.P[0][c][e].x;
        Rt[c].x = sm.P[1][c][e].x;
      }
      if (hwm & 2) {
        L[c].y = sm.P[0][c][e].y;
        Rt[c].y = sm.P[1][c][e].y;
      }
    }
    flux2<C>(gas, gm, f2);
    flux2<C>(gas, gp, f3);
    if constexpr (C == 3) S[0] = add2(gm[1], gp[1]);
#pragma unroll
    for (int k = 0; k < NF; ++k) S[C - NF + k] = add2(f2[k], f3[k]);
    flux2<C>(gas, L, fL);
    flux2<C>(gas, Rt, fR);
#pragma unroll
    for (int c = 0; c < C; ++c) {
      sm.P[0][c][e] = L[c];
      sm.P[1][c][e] = Rt[c];
    }
#pragma unroll
    for (int k = 0; k < NF; ++k) {
      sm.F[0][k][e] = fL[k];
      sm.F[1][k][e] = fR[k];
    }
  }
  // alpha and dt from the scalar warp; a zero dt (t_final reached) is uniform
  // over the grid (the instance), and the stage then writes nothing
  bar_sync(kBarAll, NTH + 32);
  const float alpha = sm.alpha, dt = sm.dt;
  if (a.stage > 0 && !(dt > 0.0f)) return;

  asm volatile("cp.async.wait_group 0;" ::: "memory");  // z: each thread reads its own copies
  // own cells: the Lax-Friedrichs fluxes, F_i, Eq. (odeH), Eq. (RK)
  const float2 mha = bcast2(-0.5f * alpha), half = k2(0.5);
  const float cb = a.stage == 2 ? 0.25f : (float)(2.0 / 3.0);
  float speed = 0.0f;
  unsigned bad = 0u;
  if (ownx) {
    float* out = static_cast<float*>(a.out) + gx;
    float* lim = static_cast<float*>(a.lim_out);
    if (lim) lim += gx;
    float2 nan = make_float2(0.0f, 0.0f);  // 0 while every output is finite
    float2 Uo[C];
#pragma unroll
    for (int c = 0; c < C; ++c) {
      const float2 pr = sm.P[1][c][e - 1], pl = sm.P[0][c][e + 1];
      float2 fl_l, fl_r, fn_l, fn_r;  // fluxes: left neighbour's right trace, own two, right neighbour's left
      if (C == 3 && c == 0) {
        constexpr int m = C == 3 ? 1 : 0;
        fn_l = sm.P[1][m][e - 1]; fl_l = L[m]; fl_r = Rt[m]; fn_r = sm.P[0][m][e + 1];
      } else {
        const int k = C == 3 ? c - 1 : 0;
        fn_l = sm.F[1][k][e - 1]; fl_l = fL[k]; fl_r = fR[k]; fn_r = sm.F[0][k][e + 1];
      }
      const float2 ql = fma2(mha, sub2(L[c], pr), mul2(half, add2(fn_l, fl_l)));
      const float2 qr = fma2(mha, sub2(pl, Rt[c]), mul2(half, add2(fl_r, fn_r)));
      // four-point Gauss-Lobatto F_i; the end points are the cell's own traces
      const float2 F = fma2(k2(5.0 / 12.0), S[c], mul2(k2(1.0 / 12.0), add2(fl_l, fl_r)));
      const float2 Lu = mul2(sub2(ql, qr), bcast2(inv_dx));
      const float2 Lv = mul2(fma2(k2(-0.5), add2(ql, qr), F), bcast2(inv_dx));
      const float2 wu = u0[c], wvm = v0[c];
      const float2 wv = (a.variant & HWENO_VARIANT_RAW_COMBINE) ? sm.u[c][1][e] : wvm;
      float2 ou = Lu, ov = Lv;
      if (a.stage > 0) {
        ou = fma2(bcast2(dt), Lu, wu);
        ov = fma2(bcast2(dt), Lv, wv);
        if (a.stage >= 2) {
          const float2 zu = sm.z[c][0][tid], zv = sm.z[c][1][tid];
          ou = fma2(bcast2(cb), sub2(ou, zu), zu);
          ov = fma2(bcast2(cb), sub2(ov, zv), zv);
        }
      }
      nan = fma2(k2(0.0), ou, fma2(k2(0.0), ov, nan));
      const float2 lv = a.stage == 0 ? wvm : wv;  // rhs mode: the modified moment
      out[0] = ou.x;
      out[n] = ov.x;
      if (owny) {
        out[W] = ou.y;
        out[n + W] = ov.y;
      }
      out += 2 * n;
      if (lim) {
        lim[0] = wu.x;
        lim[n] = lv.x;
        if (owny) {
          lim[W] = wu.y;
          lim[n + W] = lv.y;
        }
        lim += 2 * n;
      }
      Uo[c] = ou;
    }
    if (nan.x != 0.0f || (owny && nan.y != 0.0f)) bad |= ST_NONFINITE;  // (NaN != 0)
    if (a.flags_out) {
      a.flags_out[gx] = flag & 1;
      if (owny) a.flags_out[gy] = flag >> 1;
    }
    if (a.stage > 0) {
#pragma unroll
      for (int y = 0; y < 2; ++y) {
        if (y == 1 && !owny) continue;
        float U[C];
#pragma unroll
        for (int c = 0; c < C; ++c) U[c] = half_of(Uo[c], y);
        const float v = s1d::wave_speed<float, C>(gas, U);
        if (v == v) speed = fmaxf(speed, v);
        else bad |= ST_NONPHYSICAL;
      }
    }
  }
  // the maximum wave speed (non-negative floats order as their bit patterns) into
  // the slot: a batch's instance by each warp, a single instance's tile by one
  // atomic per CTA, so that the 64 slots' queues stay short on large grids
  const unsigned wm = __reduce_max_sync(0xffffffffu, __float_as_uint(speed));
  const int cnt = (ownx ? flag & 1 : 0) + (owny ? flag >> 1 : 0);
  const int wc = any ? __reduce_add_sync(0xffffffffu, cnt) : 0;
  if (bad) atomicOr(&a.sc->status, bad);
  if (lane == 0 && wc) atomicAdd(&a.sc->troubled, (unsigned long long)wc);
  if (!a.a_out) return;
  if (BATCH) {
    if (lane == 0 && wm)
      atomic_max_nonneg(static_cast<double*>(a.a_out) + where.inst, (double)__uint_as_float(wm));
    return;
  }
  if (lane == 0) atomicMax(&sm.wmax, wm);
  bar_sync(kBarCells, NTH);
  if (tid == 0)
    atomic_max_nonneg(static_cast<double*>(a.a_out) + tile % kAlphaSlots, (double)__uint_as_float(sm.wmax));
}

}  // namespace pr
}  // namespace hw
