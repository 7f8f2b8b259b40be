// The arithmetic of one scalar field of the 1D scheme (Zhao & Qiu,
// arXiv:2002.08816, Sec. 2.1) for the kernels that work in tasks of one
// characteristic field (hweno1d_fp64.cuh, hweno1d_pair.cuh): eigenvectors,
// Step 1 and Step 2.1, in R = float or double.
#pragma once

#include "hweno1d_recon.cuh"

namespace hw {
namespace fld {

// Reciprocal and square root: FP32 approximate, FP64 correctly rounded (the
// reciprocal costs 5.4 FP64 instructions, a quotient 8.5).
__device__ __forceinline__ float rcp_of(float x) { return rcp_approx(x); }
__device__ __forceinline__ double rcp_of(double x) { return __drcp_rn(x); }
__device__ __forceinline__ float sqrt_of(float x) { return sqrt_approx(x); }
__device__ __forceinline__ double sqrt_of(double x) { return sqrt(x); }

// One characteristic field of the Jacobian at U: left eigenvector row l, right
// eigenvector column r (Burgers: the identity).
template <typename R, int C>
__device__ __forceinline__ void field(R gas, const R* U, int f, R* l, R* r) {
  if constexpr (C == 1) {
    l[0] = r[0] = R(1);
  } else {
    const R ir = rcp_of(U[0]), mu = U[1] * ir;
    const R mu2 = mu * mu;
    const R p = (gas - R(1)) * fma(R(-0.5) * U[0], mu2, U[2]);
    const R c = sqrt_of(gas * p * ir);
    const R ic = rcp_of(c);
    const R b1 = (gas - R(1)) * ic * ic, b2 = R(0.5) * b1 * mu2;
    if (f == 1) {
      l[0] = R(1) - b2; l[1] = b1 * mu; l[2] = -b1;
      r[0] = R(1); r[1] = mu; r[2] = R(0.5) * mu2;
    } else {
      const R s = f == 0 ? R(1) : R(-1);  // mu - c, mu + c
      const R H = (U[2] + p) * ir;
      l[0] = R(0.5) * fma(s * mu, ic, b2);
      l[1] = R(-0.5) * fma(b1, mu, s * ic);
      l[2] = R(0.5) * b1;
      r[0] = R(1); r[1] = fma(-s, c, mu); r[2] = fma(-s * mu, c, H);
    }
  }
}

// Sum over a cell's fields of r_f[c] x_f, for component c = this lane's own
// place among the cell's C lanes (base: the first of them).
template <typename R, int C>
__device__ __forceinline__ R to_component(const R* r, R x, int f, int base) {
  if constexpr (C == 1) {
    return x;
  } else {
    R t[C], mine[C];
#pragma unroll
    for (int c = 0; c < C; ++c) t[c] = r[c] * x;
#pragma unroll
    for (int g = 0; g < C; ++g) {
#pragma unroll
      for (int c = 0; c < C; ++c) {
        const R v = __shfl_sync(0xffffffffu, t[c], base + g);
        if (c == f) mine[g] = v;
      }
    }
    return mine[0] + mine[1] + mine[2];
  }
}

// Weights3's combination (hweno1d_recon.cuh) with w_0 / gamma_0 formed without
// the division by gamma_0.
template <typename R>
struct Weights {
  R w0g, w1, w2, g1, g2;
  __device__ __forceinline__ Weights(const R* gam, R eps, R b0, R b1, R b2) {
    const R s = R(0.5) * (fabs(b0 - b1) + fabs(b0 - b2));
    const R tau = s * s;
    const R a0 = fma(tau, rcp_of(b0 + eps), R(1));
    const R a1 = gam[1] * fma(tau, rcp_of(b1 + eps), R(1));
    const R a2 = gam[2] * fma(tau, rcp_of(b2 + eps), R(1));
    const R inv = rcp_of(fma(gam[0], a0, a1) + a2);
    w0g = a0 * inv;
    w1 = a1 * inv;
    w2 = a2 * inv;
    g1 = gam[1];
    g2 = gam[2];
  }
  __device__ __forceinline__ R apply(R v0, R v1, R v2) const {
    return fma(w0g, fma(-g2, v2, fma(-g1, v1, v0)), fma(w1, v1, w2 * v2));
  }
};

// The smoothness indicators of the high-degree candidates of Step 1 and Step
// 2.1 as sums of 4 and 5 squares instead of the printed 5 and 8: each is a
// quadratic form without terms mixing the even data (c = u_m - 2 u_0 + u_p, dV
// = v_m - v_p) and the odd ones (dU = u_m - u_p, sV = v_m + v_p, v_0), so an
// exact LDL^T of the two blocks gives it in 10 and 14 operations (the printed
// forms 20 and 37); the even block is the same in both.  Every term is
// positive, and dU^2 and c^2 carry the energy of smooth data.
template <typename R>
__device__ __forceinline__ R even_beta(R c, R dV) {
  const R s = fma(R(110741.0 / 660750.0), c, dV);
  return fma(R(1421461.0 / 1321500.0) * c, c, (R(991125.0 / 112.0) * s) * s);
}

// Step 1 of one field: the modified first moment.
template <typename R>
__device__ __forceinline__ R limit_moment(R um, R u0, R up, R vm, R vp, const R* gam, R eps) {
  const R d1 = u0 - um, d2 = up - u0, dU = um - up, sV = vm + vp, dV = vm - vp;
  const R c = d2 - d1;
  const R s = fma(R(839.0 / 9612.0), dU, sV);
  const R b0 = fma(R(781.0 / 3204.0) * dU, dU, fma(R(144180.0 / 361.0) * s, s, even_beta(c, dV)));
  const Weights<R> w(gam, eps, b0, d1 * d1, d2 * d2);
  return w.apply(fma(R(-5.0 / 76.0), dU, R(-11.0 / 38.0) * sV), R(1.0 / 12.0) * d1, R(1.0 / 12.0) * d2);
}

// p0 by its even and odd parts about x_i: the faces (Step 2.2), and the interior
// Gauss-Lobatto points (Step 2.3), as u_0 plus an increment (the coefficients
// of the averages sum to one), so that each value is rounded once at the size
// of u.  D = u_p - u_m, c = u_m - 2 u_0 + u_p, sV = v_m + v_p, dV = v_m - v_p.
template <typename R>
__device__ __forceinline__ void p0_faces(R u0, R D, R c, R sV, R dV, R v0, R& left, R& right) {
  const R even = fma(R(5.0 / 24.0), c, R(0.75) * dV);
  const R odd = fma(R(19.0 / 216.0), D, fma(R(-31.0 / 108.0), sV, R(241.0 / 54.0) * v0));
  left = u0 + (even - odd);
  right = u0 + (even + odd);
}
template <typename R>
__device__ __forceinline__ void p0_interior(R u0, R D, R c, R sV, R dV, R v0, R& gm, R& gp) {
  constexpr double r5 = 2.2360679774997896964;
  const R even = fma(R(-1.0 / 24.0), c, R(-0.15) * dV);
  const R odd = fma(R(-101.0 / 5400.0 * r5), D, fma(R(841.0 / 13500.0 * r5), sV, R(10289.0 / 6750.0 * r5) * v0));
  gm = u0 + (even - odd);
  gp = u0 + (even + odd);
}

// Step 2.1 of one field: the HWENO values at both interfaces.
template <typename R>
__device__ __forceinline__ void hweno(R um, R u0, R up, R vm, R v0, R vp, const R* gam, R eps, R& left,
                                      R& right) {
  const R d1 = u0 - um, d2 = up - u0, dU = um - up, sV = vm + vp, dV = vm - vp;
  const R c = d2 - d1;
  R p0l, p0r;
  p0_faces(u0, -dU, c, sV, dV, v0, p0l, p0r);
  const R h1 = fma(R(1.0 / 6.0), um, R(5.0 / 6.0) * u0), h2 = fma(R(1.0 / 6.0), up, R(5.0 / 6.0) * u0);
  const R s = fma(R(23124050207.0 / 264871203420.0), dU, sV);
  const R r = fma(R(2632162559.0 / 40053970660.0), dU, fma(R(1155959005.0 / 4005397066.0), sV, v0));
  const R b0 = fma(R(21520059541.0 / 88290401140.0) * dU, dU,
               fma(R(794613610260.0 / 2002698533.0) * s, s,
               fma(R(10013492665.0 / 2916.0) * r, r, even_beta(c, dV))));
  const R v2 = (R(144) * v0) * v0;
  const R e1 = fma(R(12), v0, -d1), e2 = fma(R(12), v0, -d2);
  const Weights<R> w(gam, eps, b0, fma(R(13.0 / 3.0) * e1, e1, v2), fma(R(13.0 / 3.0) * e2, e2, v2));
  left = w.apply(p0l, fma(R(-4), v0, h1), fma(R(-8), v0, h2));
  right = w.apply(p0r, fma(R(8), v0, h1), fma(R(4), v0, h2));
}

}  // namespace fld
}  // namespace hw
