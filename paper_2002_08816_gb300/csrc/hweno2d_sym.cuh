// Generated by gen_hweno2d_coef.py (sym) from the moment conditions of Zhao & Qiu,
// arXiv:2002.08816, Sec. 2.2 Step 5 (exact rationals, printed to 20 digits): the
// linear p0 by parity classes.  Do not edit: rerun the generator.
//
// p0 is equivariant under x -> -x and y -> -y, so its 19 data are folded once
// into four parity classes (p0_classes: 20 sums and differences; even-even 6,
// odd-even 5, even-odd 5, odd-odd 3 entries), and the values at the mirror
// images of one point are sums and differences of four class sums.  Per
// component, with 3 Gauss points the 12 interface and 9 interior values take
// 20 + 68 + 51 operations instead of 353 by the plain maps, with 2 points
// 20 + 42 + 20 instead of 228.  The transposes (_T) run the same steps
// backwards: point adjoints into class sums, into the classes' adjoints, and
// once per component back to the 19 data.
// Measured (GB300, us per pass, plain maps -> classes): 2D Euler 4096 x 4096,
// 4 steps, FP32, 2 points 19971 -> 18746; 250 x 190, 5 steps, FP64, 3 points
// 10893 -> 8555 (the FP64 pipe bounds it); gradient at 512 x 512, 12 steps,
// FP32, 3 points 6614 -> 5820.
//
// T is float, double, or float2 (two components, or points, at once in packed
// FP32: fma.rn.f32x2 with broadcast coefficients).
#pragma once
#ifdef __CUDACC__
#include "hweno2d_coef.cuh"  // hw2_pair
#endif
namespace hw2 {

template <typename T>
__device__ __forceinline__ T add(T a, T b) { return a + b; }
template <typename T>
__device__ __forceinline__ T sub(T a, T b) { return a - b; }
template <typename T>
__device__ __forceinline__ T mul(double c, T a) { return T(c) * a; }
template <typename T>
__device__ __forceinline__ T fma(double c, T a, T b) { return T(c) * a + b; }
#ifdef __CUDACC__
template <>
__device__ __forceinline__ float2 add(float2 a, float2 b) { return __fadd2_rn(a, b); }
template <>
__device__ __forceinline__ float2 sub(float2 a, float2 b) { return __ffma2_rn(hw2_pair(-1.0), b, a); }
template <>
__device__ __forceinline__ float2 mul(double c, float2 a) { return __fmul2_rn(hw2_pair(c), a); }
template <>
__device__ __forceinline__ float2 fma(double c, float2 a, float2 b) { return __ffma2_rn(hw2_pair(c), a, b); }
#endif


template <typename T>
__device__ __forceinline__ void p0_classes(const T* d, T* s) {
  const T g = add(d[8], d[0]), h = add(d[2], d[6]);
  const T e = sub(d[8], d[0]), f = sub(d[2], d[6]);
  s[0] = d[4];
  s[1] = add(d[3], d[5]);
  s[2] = add(d[1], d[7]);
  s[3] = add(g, h);
  s[4] = sub(d[12], d[10]);
  s[5] = sub(d[18], d[14]);
  s[6] = sub(d[5], d[3]);
  s[7] = add(e, f);
  s[8] = d[11];
  s[9] = add(d[10], d[12]);
  s[10] = add(d[9], d[13]);
  s[11] = sub(d[7], d[1]);
  s[12] = sub(e, f);
  s[13] = d[16];
  s[14] = add(d[14], d[18]);
  s[15] = add(d[15], d[17]);
  s[16] = sub(g, h);
  s[17] = sub(d[13], d[9]);
  s[18] = sub(d[17], d[15]);
}

template <typename T>
__device__ __forceinline__ void p0_classes_T(const T* s, T* d) {
  const T g = add(s[3], s[16]), h = sub(s[3], s[16]);
  const T e = add(s[7], s[12]), f = sub(s[7], s[12]);
  d[8] = add(d[8], add(g, e));
  d[0] = add(d[0], sub(g, e));
  d[2] = add(d[2], add(h, f));
  d[6] = add(d[6], sub(h, f));
  d[4] = add(d[4], s[0]);
  d[5] = add(d[5], add(s[1], s[6]));
  d[3] = add(d[3], sub(s[1], s[6]));
  d[7] = add(d[7], add(s[2], s[11]));
  d[1] = add(d[1], sub(s[2], s[11]));
  d[11] = add(d[11], s[8]);
  d[12] = add(d[12], add(s[9], s[4]));
  d[10] = add(d[10], sub(s[9], s[4]));
  d[13] = add(d[13], add(s[10], s[17]));
  d[9] = add(d[9], sub(s[10], s[17]));
  d[16] = add(d[16], s[13]);
  d[18] = add(d[18], add(s[14], s[5]));
  d[14] = add(d[14], sub(s[14], s[5]));
  d[17] = add(d[17], add(s[15], s[18]));
  d[15] = add(d[15], sub(s[15], s[18]));
}

// ---- 2 Gauss points per direction: the x-faces (left, right), the y-faces
// (bottom, top), the interior points

template <typename T>
__device__ __forceinline__ void p0s_xfaces_ng2(const T* s, T* o) {
  {
    const T ee = fma(0.57638888888888888889, s[0], fma(0.20833333333333333333, s[1], fma(0.0034722222222222222222, s[2], fma(-0.75000000000000000000, s[4], mul(-0.020833333333333333333, s[5])))));
    const T oe = fma(0.022727272727272727273, s[6], mul(5.4545454545454545455, s[8]));
    const T eo = fma(-0.032803992567592372983, s[11], fma(0.012028130608117203427, s[12], mul(3.6740471675703457742, s[13])));
    const T oo = fma(-0.034990925405431864516, s[16], fma(0.78729582162221695160, s[17], mul(0.91851179189258644354, s[18])));
    const T p = add(ee, eo), q = sub(ee, eo), r = add(oe, oo), t = sub(oe, oo);
    o[3] = add(p, r); o[1] = sub(p, r); o[2] = add(q, t); o[0] = sub(q, t);
  }
}

template <typename T>
__device__ __forceinline__ void p0s_yfaces_ng2(const T* s, T* o) {
  {
    const T ee = fma(0.57638888888888888889, s[0], fma(0.0034722222222222222222, s[1], fma(0.20833333333333333333, s[2], fma(-0.020833333333333333333, s[4], mul(-0.75000000000000000000, s[5])))));
    const T oe = fma(-0.032803992567592372983, s[6], fma(0.012028130608117203427, s[7], mul(3.6740471675703457742, s[8])));
    const T eo = fma(0.022727272727272727273, s[11], mul(5.4545454545454545455, s[13]));
    const T oo = fma(-0.034990925405431864516, s[16], fma(0.91851179189258644354, s[17], mul(0.78729582162221695160, s[18])));
    const T p = add(ee, eo), q = sub(ee, eo), r = add(oe, oo), t = sub(oe, oo);
    o[3] = add(p, r); o[2] = sub(p, r); o[1] = add(q, t); o[0] = sub(q, t);
  }
}

template <typename T>
__device__ __forceinline__ void p0s_interior_ng2(const T* s, T* o) {
  {
    const T ee = fma(0.98611111111111111111, s[0], fma(0.0034722222222222222222, s[1], fma(0.0034722222222222222222, s[2], fma(-0.020833333333333333333, s[4], mul(-0.020833333333333333333, s[5])))));
    const T oe = fma(-0.0087477313513579661289, s[6], mul(3.6740471675703457742, s[8]));
    const T eo = fma(-0.0087477313513579661289, s[11], mul(3.6740471675703457742, s[13]));
    const T oo = fma(-0.023358585858585858586, s[16], fma(0.53030303030303030303, s[17], mul(0.53030303030303030303, s[18])));
    const T p = add(ee, eo), q = sub(ee, eo), r = add(oe, oo), t = sub(oe, oo);
    o[3] = add(p, r); o[2] = sub(p, r); o[1] = add(q, t); o[0] = sub(q, t);
  }
}

template <typename T>
__device__ __forceinline__ void p0s_xfaces_ng2_T(const T* l, T* s) {
  {
    const T p = add(l[3], l[1]), q = add(l[2], l[0]);
    const T r = sub(l[3], l[1]), t = sub(l[2], l[0]);
    const T ee = add(p, q), eo = sub(p, q), oe = add(r, t), oo = sub(r, t);
    s[0] = fma(0.57638888888888888889, ee, s[0]);
    s[1] = fma(0.20833333333333333333, ee, s[1]);
    s[2] = fma(0.0034722222222222222222, ee, s[2]);
    s[4] = fma(-0.75000000000000000000, ee, s[4]);
    s[5] = fma(-0.020833333333333333333, ee, s[5]);
    s[6] = fma(0.022727272727272727273, oe, s[6]);
    s[8] = fma(5.4545454545454545455, oe, s[8]);
    s[11] = fma(-0.032803992567592372983, eo, s[11]);
    s[12] = fma(0.012028130608117203427, eo, s[12]);
    s[13] = fma(3.6740471675703457742, eo, s[13]);
    s[16] = fma(-0.034990925405431864516, oo, s[16]);
    s[17] = fma(0.78729582162221695160, oo, s[17]);
    s[18] = fma(0.91851179189258644354, oo, s[18]);
  }
}

template <typename T>
__device__ __forceinline__ void p0s_yfaces_ng2_T(const T* l, T* s) {
  {
    const T p = add(l[3], l[2]), q = add(l[1], l[0]);
    const T r = sub(l[3], l[2]), t = sub(l[1], l[0]);
    const T ee = add(p, q), eo = sub(p, q), oe = add(r, t), oo = sub(r, t);
    s[0] = fma(0.57638888888888888889, ee, s[0]);
    s[1] = fma(0.0034722222222222222222, ee, s[1]);
    s[2] = fma(0.20833333333333333333, ee, s[2]);
    s[4] = fma(-0.020833333333333333333, ee, s[4]);
    s[5] = fma(-0.75000000000000000000, ee, s[5]);
    s[6] = fma(-0.032803992567592372983, oe, s[6]);
    s[7] = fma(0.012028130608117203427, oe, s[7]);
    s[8] = fma(3.6740471675703457742, oe, s[8]);
    s[11] = fma(0.022727272727272727273, eo, s[11]);
    s[13] = fma(5.4545454545454545455, eo, s[13]);
    s[16] = fma(-0.034990925405431864516, oo, s[16]);
    s[17] = fma(0.91851179189258644354, oo, s[17]);
    s[18] = fma(0.78729582162221695160, oo, s[18]);
  }
}

template <typename T>
__device__ __forceinline__ void p0s_interior_ng2_T(const T* l, T* s) {
  {
    const T p = add(l[3], l[2]), q = add(l[1], l[0]);
    const T r = sub(l[3], l[2]), t = sub(l[1], l[0]);
    const T ee = add(p, q), eo = sub(p, q), oe = add(r, t), oo = sub(r, t);
    s[0] = fma(0.98611111111111111111, ee, s[0]);
    s[1] = fma(0.0034722222222222222222, ee, s[1]);
    s[2] = fma(0.0034722222222222222222, ee, s[2]);
    s[4] = fma(-0.020833333333333333333, ee, s[4]);
    s[5] = fma(-0.020833333333333333333, ee, s[5]);
    s[6] = fma(-0.0087477313513579661289, oe, s[6]);
    s[8] = fma(3.6740471675703457742, oe, s[8]);
    s[11] = fma(-0.0087477313513579661289, eo, s[11]);
    s[13] = fma(3.6740471675703457742, eo, s[13]);
    s[16] = fma(-0.023358585858585858586, oo, s[16]);
    s[17] = fma(0.53030303030303030303, oo, s[17]);
    s[18] = fma(0.53030303030303030303, oo, s[18]);
  }
}

// ---- 3 Gauss points per direction: the x-faces (left, right), the y-faces
// (bottom, top), the interior points

template <typename T>
__device__ __forceinline__ void p0s_xfaces_ng3(const T* s, T* o) {
  {
    const T ee = fma(0.41527777777777777778, s[0], fma(0.20277777777777777778, s[1], fma(0.084027777777777777778, s[2], fma(0.0027777777777777777778, s[3], fma(-0.75000000000000000000, s[4], mul(-0.33750000000000000000, s[5]))))));
    const T oe = fma(0.0060606060606060606061, s[6], fma(0.0083333333333333333333, s[7], mul(5.4545454545454545455, s[8])));
    const T eo = fma(-0.032274861218395140710, s[11], fma(0.016137430609197570355, s[12], mul(4.6475800154489002622, s[13])));
    const T oo = fma(-0.044011174388720646422, s[16], fma(1.0562681853292955141, s[17], mul(1.1618950038622250656, s[18])));
    const T p = add(ee, eo), q = sub(ee, eo), r = add(oe, oo), t = sub(oe, oo);
    o[5] = add(p, r); o[2] = sub(p, r); o[3] = add(q, t); o[0] = sub(q, t);
  }
  {
    const T ee = fma(0.79340277777777777778, s[0], fma(0.21527777777777777778, s[1], fma(-0.10503472222222222222, s[2], fma(-0.0034722222222222222222, s[3], fma(-0.75000000000000000000, s[4], mul(0.42187500000000000000, s[5]))))));
    const T oe = fma(0.043560606060606060606, s[6], fma(-0.010416666666666666667, s[7], mul(5.4545454545454545455, s[8])));
    o[4] = add(ee, oe); o[1] = sub(ee, oe);
  }
}

template <typename T>
__device__ __forceinline__ void p0s_yfaces_ng3(const T* s, T* o) {
  {
    const T ee = fma(0.41527777777777777778, s[0], fma(0.084027777777777777778, s[1], fma(0.20277777777777777778, s[2], fma(0.0027777777777777777778, s[3], fma(-0.33750000000000000000, s[4], mul(-0.75000000000000000000, s[5]))))));
    const T oe = fma(-0.032274861218395140710, s[6], fma(0.016137430609197570355, s[7], mul(4.6475800154489002622, s[8])));
    const T eo = fma(0.0060606060606060606061, s[11], fma(0.0083333333333333333333, s[12], mul(5.4545454545454545455, s[13])));
    const T oo = fma(-0.044011174388720646422, s[16], fma(1.1618950038622250656, s[17], mul(1.0562681853292955141, s[18])));
    const T p = add(ee, eo), q = sub(ee, eo), r = add(oe, oo), t = sub(oe, oo);
    o[5] = add(p, r); o[3] = sub(p, r); o[2] = add(q, t); o[0] = sub(q, t);
  }
  {
    const T ee = fma(0.79340277777777777778, s[0], fma(-0.10503472222222222222, s[1], fma(0.21527777777777777778, s[2], fma(-0.0034722222222222222222, s[3], fma(0.42187500000000000000, s[4], mul(-0.75000000000000000000, s[5]))))));
    const T eo = fma(0.043560606060606060606, s[11], fma(-0.010416666666666666667, s[12], mul(5.4545454545454545455, s[13])));
    o[4] = add(ee, eo); o[1] = sub(ee, eo);
  }
}

template <typename T>
__device__ __forceinline__ void p0s_interior_ng3(const T* s, T* o) {
  {
    const T ee = fma(0.64611111111111111111, s[0], fma(0.087361111111111111111, s[1], fma(0.087361111111111111111, s[2], fma(0.0011111111111111111111, s[3], fma(-0.33750000000000000000, s[4], mul(-0.33750000000000000000, s[5]))))));
    const T oe = fma(-0.012909944487358056284, s[6], fma(0.0064549722436790281420, s[7], mul(4.6475800154489002622, s[8])));
    const T eo = fma(-0.012909944487358056284, s[11], fma(0.0064549722436790281420, s[12], mul(4.6475800154489002622, s[13])));
    const T oo = fma(-0.037500000000000000000, s[16], fma(0.90000000000000000000, s[17], mul(0.90000000000000000000, s[18])));
    const T p = add(ee, eo), q = sub(ee, eo), r = add(oe, oo), t = sub(oe, oo);
    o[8] = add(p, r); o[6] = sub(p, r); o[2] = add(q, t); o[0] = sub(q, t);
  }
  {
    const T ee = fma(1.0392361111111111111, s[0], fma(-0.10920138888888888889, s[1], fma(0.092361111111111111111, s[2], fma(-0.0013888888888888888889, s[3], fma(0.42187500000000000000, s[4], mul(-0.33750000000000000000, s[5]))))));
    const T eo = fma(0.016137430609197570355, s[11], fma(-0.0080687153045987851775, s[12], mul(4.6475800154489002622, s[13])));
    o[7] = add(ee, eo); o[1] = sub(ee, eo);
  }
  {
    const T ee = fma(1.0392361111111111111, s[0], fma(0.092361111111111111111, s[1], fma(-0.10920138888888888889, s[2], fma(-0.0013888888888888888889, s[3], fma(-0.33750000000000000000, s[4], mul(0.42187500000000000000, s[5]))))));
    const T oe = fma(0.016137430609197570355, s[6], fma(-0.0080687153045987851775, s[7], mul(4.6475800154489002622, s[8])));
    o[5] = add(ee, oe); o[3] = sub(ee, oe);
  }
  {
    const T ee = fma(1.4548611111111111111, s[0], fma(-0.11545138888888888889, s[1], fma(-0.11545138888888888889, s[2], fma(0.0017361111111111111111, s[3], fma(0.42187500000000000000, s[4], mul(0.42187500000000000000, s[5]))))));
    o[4] = ee;
  }
}

template <typename T>
__device__ __forceinline__ void p0s_xfaces_ng3_T(const T* l, T* s) {
  {
    const T p = add(l[5], l[2]), q = add(l[3], l[0]);
    const T r = sub(l[5], l[2]), t = sub(l[3], l[0]);
    const T ee = add(p, q), eo = sub(p, q), oe = add(r, t), oo = sub(r, t);
    s[0] = fma(0.41527777777777777778, ee, s[0]);
    s[1] = fma(0.20277777777777777778, ee, s[1]);
    s[2] = fma(0.084027777777777777778, ee, s[2]);
    s[3] = fma(0.0027777777777777777778, ee, s[3]);
    s[4] = fma(-0.75000000000000000000, ee, s[4]);
    s[5] = fma(-0.33750000000000000000, ee, s[5]);
    s[6] = fma(0.0060606060606060606061, oe, s[6]);
    s[7] = fma(0.0083333333333333333333, oe, s[7]);
    s[8] = fma(5.4545454545454545455, oe, s[8]);
    s[11] = fma(-0.032274861218395140710, eo, s[11]);
    s[12] = fma(0.016137430609197570355, eo, s[12]);
    s[13] = fma(4.6475800154489002622, eo, s[13]);
    s[16] = fma(-0.044011174388720646422, oo, s[16]);
    s[17] = fma(1.0562681853292955141, oo, s[17]);
    s[18] = fma(1.1618950038622250656, oo, s[18]);
  }
  {
    const T ee = add(l[4], l[1]), oe = sub(l[4], l[1]);
    s[0] = fma(0.79340277777777777778, ee, s[0]);
    s[1] = fma(0.21527777777777777778, ee, s[1]);
    s[2] = fma(-0.10503472222222222222, ee, s[2]);
    s[3] = fma(-0.0034722222222222222222, ee, s[3]);
    s[4] = fma(-0.75000000000000000000, ee, s[4]);
    s[5] = fma(0.42187500000000000000, ee, s[5]);
    s[6] = fma(0.043560606060606060606, oe, s[6]);
    s[7] = fma(-0.010416666666666666667, oe, s[7]);
    s[8] = fma(5.4545454545454545455, oe, s[8]);
  }
}

template <typename T>
__device__ __forceinline__ void p0s_yfaces_ng3_T(const T* l, T* s) {
  {
    const T p = add(l[5], l[3]), q = add(l[2], l[0]);
    const T r = sub(l[5], l[3]), t = sub(l[2], l[0]);
    const T ee = add(p, q), eo = sub(p, q), oe = add(r, t), oo = sub(r, t);
    s[0] = fma(0.41527777777777777778, ee, s[0]);
    s[1] = fma(0.084027777777777777778, ee, s[1]);
    s[2] = fma(0.20277777777777777778, ee, s[2]);
    s[3] = fma(0.0027777777777777777778, ee, s[3]);
    s[4] = fma(-0.33750000000000000000, ee, s[4]);
    s[5] = fma(-0.75000000000000000000, ee, s[5]);
    s[6] = fma(-0.032274861218395140710, oe, s[6]);
    s[7] = fma(0.016137430609197570355, oe, s[7]);
    s[8] = fma(4.6475800154489002622, oe, s[8]);
    s[11] = fma(0.0060606060606060606061, eo, s[11]);
    s[12] = fma(0.0083333333333333333333, eo, s[12]);
    s[13] = fma(5.4545454545454545455, eo, s[13]);
    s[16] = fma(-0.044011174388720646422, oo, s[16]);
    s[17] = fma(1.1618950038622250656, oo, s[17]);
    s[18] = fma(1.0562681853292955141, oo, s[18]);
  }
  {
    const T ee = add(l[4], l[1]), eo = sub(l[4], l[1]);
    s[0] = fma(0.79340277777777777778, ee, s[0]);
    s[1] = fma(-0.10503472222222222222, ee, s[1]);
    s[2] = fma(0.21527777777777777778, ee, s[2]);
    s[3] = fma(-0.0034722222222222222222, ee, s[3]);
    s[4] = fma(0.42187500000000000000, ee, s[4]);
    s[5] = fma(-0.75000000000000000000, ee, s[5]);
    s[11] = fma(0.043560606060606060606, eo, s[11]);
    s[12] = fma(-0.010416666666666666667, eo, s[12]);
    s[13] = fma(5.4545454545454545455, eo, s[13]);
  }
}

template <typename T>
__device__ __forceinline__ void p0s_interior_ng3_T(const T* l, T* s) {
  {
    const T p = add(l[8], l[6]), q = add(l[2], l[0]);
    const T r = sub(l[8], l[6]), t = sub(l[2], l[0]);
    const T ee = add(p, q), eo = sub(p, q), oe = add(r, t), oo = sub(r, t);
    s[0] = fma(0.64611111111111111111, ee, s[0]);
    s[1] = fma(0.087361111111111111111, ee, s[1]);
    s[2] = fma(0.087361111111111111111, ee, s[2]);
    s[3] = fma(0.0011111111111111111111, ee, s[3]);
    s[4] = fma(-0.33750000000000000000, ee, s[4]);
    s[5] = fma(-0.33750000000000000000, ee, s[5]);
    s[6] = fma(-0.012909944487358056284, oe, s[6]);
    s[7] = fma(0.0064549722436790281420, oe, s[7]);
    s[8] = fma(4.6475800154489002622, oe, s[8]);
    s[11] = fma(-0.012909944487358056284, eo, s[11]);
    s[12] = fma(0.0064549722436790281420, eo, s[12]);
    s[13] = fma(4.6475800154489002622, eo, s[13]);
    s[16] = fma(-0.037500000000000000000, oo, s[16]);
    s[17] = fma(0.90000000000000000000, oo, s[17]);
    s[18] = fma(0.90000000000000000000, oo, s[18]);
  }
  {
    const T ee = add(l[7], l[1]), eo = sub(l[7], l[1]);
    s[0] = fma(1.0392361111111111111, ee, s[0]);
    s[1] = fma(-0.10920138888888888889, ee, s[1]);
    s[2] = fma(0.092361111111111111111, ee, s[2]);
    s[3] = fma(-0.0013888888888888888889, ee, s[3]);
    s[4] = fma(0.42187500000000000000, ee, s[4]);
    s[5] = fma(-0.33750000000000000000, ee, s[5]);
    s[11] = fma(0.016137430609197570355, eo, s[11]);
    s[12] = fma(-0.0080687153045987851775, eo, s[12]);
    s[13] = fma(4.6475800154489002622, eo, s[13]);
  }
  {
    const T ee = add(l[5], l[3]), oe = sub(l[5], l[3]);
    s[0] = fma(1.0392361111111111111, ee, s[0]);
    s[1] = fma(0.092361111111111111111, ee, s[1]);
    s[2] = fma(-0.10920138888888888889, ee, s[2]);
    s[3] = fma(-0.0013888888888888888889, ee, s[3]);
    s[4] = fma(-0.33750000000000000000, ee, s[4]);
    s[5] = fma(0.42187500000000000000, ee, s[5]);
    s[6] = fma(0.016137430609197570355, oe, s[6]);
    s[7] = fma(-0.0080687153045987851775, oe, s[7]);
    s[8] = fma(4.6475800154489002622, oe, s[8]);
  }
  {
    const T ee = l[4];
    s[0] = fma(1.4548611111111111111, ee, s[0]);
    s[1] = fma(-0.11545138888888888889, ee, s[1]);
    s[2] = fma(-0.11545138888888888889, ee, s[2]);
    s[3] = fma(0.0017361111111111111111, ee, s[3]);
    s[4] = fma(0.42187500000000000000, ee, s[4]);
    s[5] = fma(0.42187500000000000000, ee, s[5]);
  }
}

}  // namespace hw2
