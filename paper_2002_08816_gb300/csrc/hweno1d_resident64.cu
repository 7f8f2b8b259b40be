// The resident 1D run in FP64: a whole run of third-order TVD Runge-Kutta steps
// (Zhao & Qiu, arXiv:2002.08816, Sec. 2.1, Eq. (odeH), Eq. (RK)) in one
// cooperative launch, every CTA's tile on chip for all stages, the arithmetic
// in the tasks of hweno1d_fp64.cuh.
//
// The FP64 pipe bounds it, so the tiles spread over every SM: tiles of up to
// 26 cells (one warp's width of cells; four warps of tasks) while they cover
// the grid, then equal shares of the grid, two CTAs per SM.
//
// The exchange is that of the FP32 resident run (hweno1d_resident.cu): words
// of 64 bits that carry their stage beside 32 bits of payload, here two for a
// value; the six halo threads of a neighbour poll a CTA's first and last
// three cells, and CTA 0 gathers the wave speeds and publishes alpha.  Alpha
// is only needed after the interface values, which take longer than its two
// L2 round trips.  Every wait is bounded (r.polls): a CTA whose wait runs out
// sets ST_TIMEOUT and leaves, and the others run out too.
//
// Measured (GB300, one pass of set_state, steps, get_state, before: per-stage or
// persistent launches with a cell per thread): 400 cells with shocks, 60 steps
// 9.59 -> 2.87 ms (15.9 us per stage); 65536 cells, 10 steps 2.33 -> 1.19 ms
// (36.8 us per stage alone, the FP64 pipe active 64 % of it; over 2000 steps, with
// shocks formed, 69 -> 67 us per stage).  One CTA of 432 cells per SM instead of two
// of 216: 12 % slower.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "hweno1d_fp64.cuh"
#include "hweno1d_words.cuh"

namespace hw {
namespace {

using f64::Par;
using f64::Smem64;
using s1d::bar_arrive;
using s1d::bar_sync;
using s1d::H;
using s1d::kBarAll;
using s1d::kBarCells;
using s1d::kBarTaken;
using s1d::ldx;

__device__ __forceinline__ void publish(u64* dst, unsigned tag, double v) {
  const u64 b = (u64)__double_as_longlong(v);
  st_relaxed(dst, ((u64)tag << 32) | (b & 0xffffffffull));
  st_relaxed(dst + 1, ((u64)tag << 32) | (b >> 32));
}
__device__ __forceinline__ double value2(u64 lo, u64 hi) {
  return __longlong_as_double((long long)((hi << 32) | (lo & 0xffffffffull)));
}

// The maximum of the ncta <= 32 NE entries (two words each) once all carry
// `tag` (each lane polls up to NE entries, every round's loads in flight
// together); as bit patterns of non-negative doubles.  False after `polls` rounds.
template <int NE>
__device__ __forceinline__ bool gather_max64(const u64* ent, int ncta, unsigned tag, int lane,
                                             double* out, unsigned polls) {
  u64 lo[NE], hi[NE];
#pragma unroll
  for (int j = 0; j < NE; ++j) lo[j] = hi[j] = 0ull;
  bool ok = false;
  for (unsigned it = 0; it < polls && !ok; ++it) {
    bool mine = true;
#pragma unroll
    for (int j = 0; j < NE; ++j) {
      const int k = lane + 32 * j;
      if (k < ncta && tag_of(lo[j]) != tag) lo[j] = ld_relaxed(ent + (size_t)k * kEntStride);
      if (k < ncta && tag_of(hi[j]) != tag) hi[j] = ld_relaxed(ent + (size_t)k * kEntStride + 1);
    }
#pragma unroll
    for (int j = 0; j < NE; ++j)
      if (lane + 32 * j < ncta && (tag_of(lo[j]) != tag || tag_of(hi[j]) != tag)) mine = false;
    ok = __all_sync(0xffffffffu, mine);
  }
  if (!ok) return false;
  u64 m = 0ull;
#pragma unroll
  for (int j = 0; j < NE; ++j)
    if (lane + 32 * j < ncta) {
      const u64 b = (hi[j] << 32) | (lo[j] & 0xffffffffull);
      m = b > m ? b : m;
    }
  *out = __longlong_as_double((long long)f64::warp_max_bits(__longlong_as_double((long long)m)));
  return true;
}

template <int C, int TMAX>
struct SmemRes64 {
  Smem64<C, TMAX> w;
  double u0[C][2][TMAX];  // u^n as limited by stage 1
  // a wait ran out, every thread leaves: set by a halo thread and read after
  // the barrier that opens a stage, or by the scalar warp, between kBarTaken and
  // kBarAll, and read after kBarAll (two flags, so that all threads see the same)
  int abort, abort_alpha;
  unsigned arrived[2];    // warps that have folded their wave speeds in, by stage parity
  u64 red_max[2];
  unsigned trb;
};

constexpr int kEnt = 10;  // entries a scalar-warp lane polls: at most 320 CTAs

template <int C, int TMAX, int NTH>
__global__ void __launch_bounds__(NTH + 32, 2) resident64_kernel(Resident1DArgs r) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  SmemRes64<C, TMAX>& S = *reinterpret_cast<SmemRes64<C, TMAX>*>(smem_raw);
  Smem64<C, TMAX>& sm = S.w;
  const Stage1DArgs& a = r.a;
  const int tid = threadIdx.x, lane = tid & 31;
  const int T = r.tile, n = a.n, ncta = gridDim.x, q = blockIdx.x;
  const int base = q * T;
  const int Tq = min(T, n - base);  // this CTA's cells (the last tile may be short)
  constexpr int NV = 4;             // words per cell and component
  constexpr int HS = 6 * C * NV;
  u64* const hal = r.halo;          // [cta][parity][6 slots][C][NV]

  if (tid == 0) {
    S.abort = S.abort_alpha = 0;
    S.red_max[0] = S.red_max[1] = 0ull;
    S.arrived[0] = S.arrived[1] = 0u;
    S.trb = 0u;
  }
  __syncthreads();

  if (tid >= NTH) {
    // ---- the scalar warp: alpha, dt, the time --------------------------------
    const bool lead = q == 0 && lane == 0;
    const double tf = ldx(&a.sc->t_final);
    double t = ldx(&a.sc->t), rem = ldx(&a.sc->rem), dt = 0.0;
    const unsigned long long steps = ldx(&a.sc->steps);
    unsigned last = 0u;
    int done_steps = 0, s_end = 3 * r.nsteps;
    bool ok = true;
    for (int s = 0; s < 3 * r.nsteps; ++s) {
      const int stage = s % 3 + 1;
      double alpha = 0.0;
      if (s == 0) {
        const u64* p0 = static_cast<const u64*>(r.part0);
        u64 am = 0ull;
        for (int k = lane; k < kAlphaSlots; k += 32) {
          const u64 v = ldx(p0 + k);
          am = v > am ? v : am;
        }
        alpha = __longlong_as_double((long long)f64::warp_max_bits(__longlong_as_double((long long)am)));
      } else if (q == 0) {
        ok = gather_max64<kEnt>(r.entries + (size_t)((s - 1) & 1) * ncta * kEntStride, ncta, (unsigned)s,
                          lane, &alpha, r.polls);
        if (ok && lane == 0) publish(r.alpha_word + 2 * ((s - 1) & 1), (unsigned)s, alpha);
      } else {
        ok = gather_max64<1>(r.alpha_word + 2 * ((s - 1) & 1), 1, (unsigned)s, lane, &alpha, r.polls);
      }
      if (s > 0) {
        // not before the cell threads have read stage s - 1's alpha, dt and flag, or
        // have left (as in the FP32 run)
        __syncwarp();
        bar_sync(kBarTaken, NTH + 32);
        if (S.abort) ok = false;
      }
      if (!ok && lane == 0) {
        atomicOr(&a.sc->status, (unsigned)ST_TIMEOUT);
        S.abort_alpha = 1;
      }
      if (stage == 1) {
        dt = a.cfl_dx / alpha;
        last = 0u;
        if (rem <= 0.0) {
          dt = 0.0;
        } else if (dt >= rem) {
          dt = rem;
          last = 1u;
        }
        if (!(alpha > 0.0) || !isfinite(dt)) dt = 0.0;
      }
      if (lane == 0) {
        sm.alpha = alpha;
        sm.dt = ok ? dt : 0.0;
      }
      bar_arrive(kBarAll, NTH + 32);
      if (!ok || !(dt > 0.0)) {
        s_end = s;
        break;
      }
      if (stage == 3) {
        t = last ? tf : t + dt;
        rem = tf > 0.0 ? tf - t : (double)INFINITY;
        ++done_steps;
      }
    }
    if (ok) bar_sync(kBarTaken, NTH + 32);  // (the last arrival there)
    // alpha of the final state for the next call, as the per-stage launches
    // leave it, once every CTA has published its last stage
    if (q == 0 && ok && s_end > 0) {
      double am = 0.0;
      if (gather_max64<kEnt>(r.entries + (size_t)((s_end - 1) & 1) * ncta * kEntStride, ncta,
                       (unsigned)s_end, lane, &am, r.polls)) {
        double* p0 = static_cast<double*>(r.part0);
        double* p1 = static_cast<double*>(r.part1);
        for (int k = lane; k < kAlphaSlots; k += 32) {
          p0[k] = k == 0 ? am : 0.0;
          p1[k] = 0.0;
        }
      } else if (lane == 0) {
        atomicOr(&a.sc->status, (unsigned)ST_TIMEOUT);
      }
    }
    if (lead) {
      a.sc->t = t;
      a.sc->rem = rem;
      a.sc->rem_f = (float)rem;
      a.sc->dt = dt;
      a.sc->dt_f = (float)dt;
      a.sc->last = last;
      a.sc->steps = steps + (unsigned long long)done_steps;
    }
    return;
  }

  // ---- the cell threads ---------------------------------------------------------
  const Par par = {{a.gam[0], a.gam[1], a.gam[2]}, a.eps, a.gas, a.h, a.thr, a.inv_dx,
                   a.hthr, a.mode, a.variant};
  const double* w = static_cast<const double*>(a.w);
  for (int e = tid; e < Tq + 2 * H; e += NTH) {
    bool mir = false;
    const int g = a.bc == 2 ? bc_map_wall(base - H + e, n, &mir) : bc_map(base - H + e, n, a.bc);
#pragma unroll
    for (int c = 0; c < C; ++c)
#pragma unroll
      for (int m = 0; m < 2; ++m)
        sm.u[0][c][m][e] = mir ? (double)mirror_sign(c, m) * w[(2 * c + m) * n + g] : w[(2 * c + m) * n + g];
  }
  // the six halo threads, on as many warps as there are slots of them
  const int hj = tid < 6 ? tid : -1;
  HaloSrc hs = {0, 0, false};
  if (hj >= 0) hs = halo_source(hj, base, Tq, T, n, a.bc, ncta);
  const unsigned own_warps = (unsigned)((min(Tq, NTH) + 31) / 32);
  unsigned bad = 0u;
  int done = 0, trb = 0, cur = 0;

#pragma unroll 1
  for (int s = 0; s < 3 * r.nsteps; ++s) {
    const int stage = s % 3 + 1;
    double(*u)[2][TMAX + 6] = sm.u[cur];
    double(*un)[2][TMAX + 6] = sm.u[cur ^ 1];
    if (s > 0 && hj >= 0) {  // the halo, from the neighbours' published cells of stage s - 1
      const u64* src = hal + ((size_t)hs.cta * 2 + ((s - 1) & 1)) * HS + hs.slot * (C * NV);
      u64 v[C * NV];
#pragma unroll
      for (int j = 0; j < C * NV; ++j) v[j] = 0ull;
      bool got = false;
      for (unsigned it = 0; it < r.polls && !got; ++it) {
        got = true;
#pragma unroll
        for (int j = 0; j < C * NV; ++j)
          if (tag_of(v[j]) != (unsigned)s) v[j] = ld_relaxed(src + j);
#pragma unroll
        for (int j = 0; j < C * NV; ++j)
          if (tag_of(v[j]) != (unsigned)s) got = false;
      }
      if (!got) {
        atomicOr(&a.sc->status, (unsigned)ST_TIMEOUT);
        S.abort = 1;
      } else {
        const int e = hj < 3 ? hj : Tq + hj;
#pragma unroll
        for (int c = 0; c < C; ++c)
#pragma unroll
          for (int m = 0; m < 2; ++m) {
            const double x = value2(v[NV * c + 2 * m], v[NV * c + 2 * m + 1]);
            u[c][m][e] = hs.mirror ? (double)mirror_sign(c, m) * x : x;
          }
      }
    }
    bar_sync(kBarCells, NTH);
    if (S.abort) {  // leave, past the barriers the scalar warp counts on
      bar_sync(kBarAll, NTH + 32);
      bar_arrive(kBarTaken, NTH + 32);
      break;
    }
    const int mine = f64::step1<C, TMAX, NTH>(sm, u, Tq, tid, par);
    f64::step2<C, TMAX, NTH>(sm, u, Tq, tid, par);
    bar_sync(kBarAll, NTH + 32);  // alpha and dt from the scalar warp
    if (S.abort_alpha) break;
    const double alpha = sm.alpha, dt = sm.dt;
    bar_arrive(kBarTaken, NTH + 32);
    if (!(dt > 0.0)) break;  // t_final reached: uniform over the grid
    trb += mine;
    f64::lax_friedrichs<C, TMAX, NTH>(sm, Tq, tid, alpha);
    // Eq. (odeH) and Eq. (RK): (component, cell)
    const double kd = dt * par.inv_dx;
    const double cb = stage == 2 ? 0.25 : 2.0 / 3.0;
    for (int t = tid; t < C * Tq; t += NTH) {
      const int c = t / Tq, i = t - c * Tq, e = i + H;
      double Gu, Gv;
      f64::rhs_at<C, TMAX>(sm, c, e, Gu, Gv);
      const double wu = u[c][0][e];
      const double wv = (a.variant & HWENO_VARIANT_RAW_COMBINE) ? u[c][1][e] : sm.vl[c][e];
      double ou = fma(kd, Gu, wu), ov = fma(kd, Gv, wv);
      if (stage == 1) {
        S.u0[c][0][i] = wu;
        S.u0[c][1][i] = wv;
      } else {
        ou = rk_combine(cb, S.u0[c][0][i], ou);
        ov = rk_combine(cb, S.u0[c][1][i], ov);
      }
      un[c][0][e] = ou;
      un[c][1][e] = ov;
      if (!is_finite(ou) || !is_finite(ov)) bad |= ST_NONFINITE;
      const int ps = i < 3 ? i : (i >= Tq - 3 ? 3 + i - (Tq - 3) : -1);
      if (ps >= 0) {  // the neighbours' halo
        u64* dst = hal + ((size_t)q * 2 + (s & 1)) * HS + ps * (C * NV) + c * NV;
        publish(dst, (unsigned)(s + 1), ou);
        publish(dst + 2, (unsigned)(s + 1), ov);
      }
    }
    bar_sync(kBarCells, NTH);
    // the wave speed of the output: (cell); the last warp to fold its maximum
    // in publishes the CTA's
    if ((tid >> 5) < (int)own_warps) {
      double sp = 0.0;
      for (int i = tid; i < Tq; i += NTH) {
        double U[C];
#pragma unroll
        for (int c = 0; c < C; ++c) U[c] = un[c][0][i + H];
        const double v = f64::speed_at<C>(par.gas, U);
        if (v == v) sp = fmax(sp, v);
        else bad |= ST_NONPHYSICAL;
      }
      const u64 m = f64::warp_max_bits(sp);
      if (lane == 0) {
        const int g = s & 1;
        atomicMax(&S.red_max[g], m);
        __threadfence_block();
        if (atomicAdd(&S.arrived[g], 1u) == own_warps - 1u) {
          const u64 mm = atomicExch(&S.red_max[g], 0ull);  // read, and reset for stage s + 2
          S.arrived[g] = 0u;
          if (q != r.silent_cta)
            publish(r.entries + ((size_t)g * ncta + q) * kEntStride, (unsigned)(s + 1),
                    __longlong_as_double((long long)mm));
        }
      }
    }
    cur ^= 1;
    ++done;
  }

  // the final state, the status bits and the troubled count
  if (!S.abort && !S.abort_alpha && done > 0) {
    double* out = static_cast<double*>(a.out);
    for (int i = tid; i < Tq; i += NTH)
#pragma unroll
      for (int c = 0; c < C; ++c)
#pragma unroll
        for (int m = 0; m < 2; ++m) out[(2 * c + m) * n + base + i] = sm.u[cur][c][m][i + H];
  }
  if (bad) atomicOr(&a.sc->status, bad);
  if (trb) atomicAdd(&S.trb, (unsigned)trb);
  bar_sync(kBarCells, NTH);
  if (tid == 0 && S.trb) atomicAdd(&a.sc->troubled, (unsigned long long)S.trb);
}

// The two tile shapes, two CTAs of either per SM (one computes while the other
// is at a barrier or waits for its halo): up to 26 cells with four warps of
// tasks, and up to 253 with eight (a tile of fewer cells leaves warps idle).
constexpr int kSmallT = 26, kSmallN = 128, kLargeT = 253, kLargeN = 256, kPerSM = 2;

template <int C, int TMAX, int NTH>
cudaError_t launch_t(const Resident1DArgs& r, int ncta, cudaStream_t s) {
  Resident1DArgs rc = r;
  void* args[] = {&rc};
  const size_t smem = sizeof(SmemRes64<C, TMAX>);
  cudaError_t e = cudaFuncSetAttribute(resident64_kernel<C, TMAX, NTH>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(resident64_kernel<C, TMAX, NTH>, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  if (e != cudaSuccess) return e;
  return cudaLaunchCooperativeKernel((const void*)resident64_kernel<C, TMAX, NTH>, dim3(ncta),
                                     dim3(NTH + 32), args, smem, s);
}

}  // namespace

cudaError_t resident64_geometry(int n, int* tile, int* ncta) {
  *tile = *ncta = 0;
  int dev = 0, nsm = 0, coop = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
  if (e != cudaSuccess) return e;
  if (!coop || n < 6) return cudaSuccess;
  const int slots = std::min(kPerSM * nsm, 32 * kEnt);
  // every tile (the last one too) at least 6 cells, so that the
  // published first and last three cells do not overlap
  auto fits = [&](int t) {
    const int c = (n + t - 1) / t;
    if (c > slots || n - (c - 1) * t < 6) return false;
    *tile = t;
    *ncta = c;
    return true;
  };
  for (int t = n < kSmallT ? n : kSmallT; t >= 6; --t)
    if (fits(t)) return cudaSuccess;
  for (int t = (n + slots - 1) / slots; t <= kLargeT; ++t)
    if (fits(t)) return cudaSuccess;
  return cudaSuccess;
}

size_t resident64_entry_words(int ncta) { return (size_t)2 * ncta * kEntStride + 4; }
size_t resident64_halo_words(int system, int ncta) {
  return (size_t)ncta * 2 * 6 * (system == 0 ? 1 : 3) * 4;
}

cudaError_t launch_resident64(const Resident1DArgs& r, int ncta, double t_final, cudaStream_t s) {
  const cudaError_t e = launch_start_run(r.a.sc, t_final, r.halo, resident64_halo_words(r.a.system, ncta),
                                         r.entries, resident64_entry_words(ncta), s);
  if (e != cudaSuccess) return e;
  if (r.tile <= kSmallT)
    return r.a.system == 0 ? launch_t<1, kSmallT, kSmallN>(r, ncta, s)
                           : launch_t<3, kSmallT, kSmallN>(r, ncta, s);
  return r.a.system == 0 ? launch_t<1, kLargeT, kLargeN>(r, ncta, s)
                         : launch_t<3, kLargeT, kLargeN>(r, ncta, s);
}

}  // namespace hw
