// The words by which the CTAs of a resident 1D run exchange halos and wave
// speeds, and where a tile's ghost cells come from (hweno1d_resident.cu,
// hweno1d_resident64.cu).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "hweno_device.cuh"

namespace hw {

constexpr int kMaxEnt = 10;            // entries a scalar-warp lane polls (ncta <= 320)
constexpr int kEntStride = 16;         // words between two CTAs' entries: one cache line each

typedef unsigned long long u64;
__device__ __forceinline__ u64 ld_relaxed(const u64* p) {
  u64 v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_relaxed(u64* p, u64 v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ u64 tagged(unsigned tag, float v) {
  return ((u64)tag << 32) | (u64)__float_as_uint(v);
}
__device__ __forceinline__ unsigned tag_of(u64 w) { return (unsigned)(w >> 32); }
__device__ __forceinline__ float value_of(u64 w) { return __uint_as_float((unsigned)w); }

// Source of halo slot j (0..2 left, 3..5 right) of the tile of Tq cells from
// base (tiles of T cells; the last one may be shorter): the CTA that owns the
// cell and the slot in that CTA's published cells (0..2 its first three
// cells, 3..5 its last three), and the mirror flag of a reflective ghost.
struct HaloSrc {
  int cta, slot;
  bool mirror;
};
__device__ __forceinline__ HaloSrc halo_source(int j, int base, int Tq, int T, int n, int bc,
                                               int ncta) {
  const int g = j < 3 ? base - 3 + j : base + Tq + (j - 3);
  int src;
  bool mir = false;
  if (bc == 2) src = bc_map_wall(g, n, &mir);
  else src = bc_map(g, n, bc);
  HaloSrc h;
  h.cta = src / T;
  if (h.cta >= ncta) h.cta = ncta - 1;
  const int first = h.cta * T;
  const int last = min(first + T, n);  // one past the owner's last cell
  const int lo = src - first;
  h.slot = lo < 3 ? lo : 3 + (src - (last - 3));
  h.mirror = mir;
  return h;
}

}  // namespace hw
