// The 1D contractions of the Q2 cell operators in difference form, for one line of three values in
// fp32 or fp64.  The nodes are {0, 1/2, 1} and the Gauss points 1/2 -+ delta, 1/2 with delta^2 = 3/20,
// so a line of nodal values u has at the outer Gauss points
//   0.4 u1 + 0.3 (u0 + u2) -+ delta (u2 - u0)      (the middle Gauss point is the middle node),
// and 2 delta times the derivatives at the Gauss points of the quadratic through Gauss-point values v
// are -3 v0 + 4 v1 - v2, v2 - v0, v0 - 4 v1 + 3 v2: five additions or multiply-adds per line instead of
// eight products and sums with tabulated constants.  The factor 1 / (2 delta) of every derivative goes
// into the coefficients (both factors of a diffusion term: 5/3).
#pragma once

#include <cuda_runtime.h>

namespace mf {

constexpr double kLineDelta = 0.38729833462074168852;        // sqrt(3/20)
constexpr double kLineDerivScale = 1.2909944487358056284;    // 1 / (2 delta)

// nodes -> Gauss points
template <typename T> __device__ __forceinline__ void line_values(T& u0, const T& u1, T& u2) {
  const T m = T(0.3) * (u0 + u2) + T(0.4) * u1, d = u2 - u0;
  u0 = m - T(kLineDelta) * d;
  u2 = m + T(kLineDelta) * d;
}
// its transpose
template <typename T> __device__ __forceinline__ void line_values_t(T& f0, T& f1, T& f2) {
  const T t = f0 + f2, d = f2 - f0, c = T(0.3) * t;
  f1 = f1 + T(0.4) * t;
  f0 = c - T(kLineDelta) * d;
  f2 = c + T(kLineDelta) * d;
}
// 2 delta times the derivatives at the Gauss points
template <typename T> __device__ __forceinline__ void line_deriv(const T& v0, const T& v1, const T& v2, T& g0, T& g1, T& g2) {
  g1 = v2 - v0;
  const T c = (v0 + v2) - T(2) * v1;
  g0 = g1 - T(2) * c;
  g2 = g1 + T(2) * c;
}
// (r0, r1, r2) += the transpose of that stencil applied to f
template <typename T> __device__ __forceinline__ void line_deriv_t(const T& f0, const T& f1, const T& f2, T& r0, T& r1, T& r2) {
  const T s = (f0 + f2) + f1, e = f2 - f0;
  r0 = (r0 - s) + T(2) * e;
  r1 = r1 - T(4) * e;
  r2 = (r2 + s) + T(2) * e;
}
// one line of a Q1 function: end values -> the three Gauss points
template <typename T> __device__ __forceinline__ void line_q1(const T& p0, const T& p1, T& v0, T& v1, T& v2) {
  const T d = p1 - p0;
  v1 = T(0.5) * (p0 + p1);
  v0 = v1 - T(kLineDelta) * d;
  v2 = v1 + T(kLineDelta) * d;
}
// its transpose with the Gauss weights (5, 8, 5) / 18
template <typename T> __device__ __forceinline__ void line_q1_t(const T& g0, const T& g1, const T& g2, T& o0, T& o1) {
  const T a = T(5.0 / 36.0) * (g0 + g2) + T(8.0 / 36.0) * g1, b = T(kLineDelta * 5.0 / 18.0) * (g2 - g0);
  o0 = a - b;
  o1 = a + b;
}
// Gauss points -> nodes of a test side with values v and derivative fluxes f: the transposed values of
// v + stencil^T f, both transposes sharing their sums and differences
template <typename T>
__device__ __forceinline__ void line_combine_t(const T& f0, const T& f1, const T& f2, T& v0, T& v1, T& v2) {
  const T s = (f0 + f2) + f1, e = f2 - f0;
  const T t = (v0 + v2) + T(4) * e, d = (v2 - v0) + T(2) * s, c = T(0.3) * t;
  v1 = (v1 - T(4) * e) + T(0.4) * t;
  v0 = c - T(kLineDelta) * d;
  v2 = c + T(kLineDelta) * d;
}

// The transposes with the Gauss weights folded into them, for test sides kept without weights: the stencil
// becomes W^-1 stencil^T W (weights (5, 8, 5) / 18), the value transpose S^T W times a factor given by the
// caller's constants k = {0.3 w0, w1, 0.4 w0, delta w0} f.
template <typename T> __device__ __forceinline__ void line_deriv_tw(const T& f0, const T& f1, const T& f2, T& r0, T& r1, T& r2) {
  const T s = (f0 + f2) + T(1.6) * f1, e = f2 - f0;
  r0 = (r0 - s) + T(2) * e;
  r1 = r1 - T(2.5) * e;
  r2 = (r2 + s) + T(2) * e;
}
template <typename T> __device__ __forceinline__ void line_values_tw(const T (&k)[4], T& f0, T& f1, T& f2) {
  const T t = f0 + f2, d = k[3] * (f2 - f0), c = k[0] * t;
  f1 = k[1] * f1 + k[2] * t;
  f0 = c - d;
  f2 = c + d;
}
template <typename T>
__device__ __forceinline__ void line_combine_tw(const T (&k)[4], const T& f0, const T& f1, const T& f2, T& v0, T& v1, T& v2) {
  const T s = (f0 + f2) + T(1.6) * f1, e = f2 - f0;
  const T t = (v0 + v2) + T(4) * e, d = k[3] * ((v2 - v0) + T(2) * s), c = k[0] * t;
  v1 = k[1] * (v1 - T(2.5) * e) + k[2] * t;
  v0 = c - d;
  v2 = c + d;
}

}  // namespace mf
