// Double-float ("dd") arithmetic on the fp32 pipes and the Q2 sum-factorisation sweeps in it, shared
// by the double-float kernels (uniform and octree meshes).  A value is an unnormalised pair of floats
// hi + lo (48-bit significand): Dekker's product through the FMA residual, Knuth's two-sum for the
// high parts (Joldes, Muller and Popescu, ACM TOMS 2017, bound these "double-word" algorithms).
// Doubles enter and leave by bit manipulation, scaled by a power of two chosen by the caller.
#pragma once

#include "ops.h"

namespace mf {
namespace {

struct dd {
  float h, l;
};

// double -> pair of floats for x 2^-bias, by bits (no fp64 instruction: GB300 converts between fp64
// and fp32 at its fp64 rate): hi = the top 24 significand bits (truncated), lo = the remaining 29
// bits rounded once (the high 23 and low 6 bits made floats exactly through the 2^23 offset, joined by
// one FMA), so hi + lo = x 2^-bias to 2^-47 relative.  Magnitudes below 2^-126 after scaling give 0.  bias is the
// exponent of the largest finite input; what Inf and NaN give is covered by the NaN added to their rows.
__device__ __forceinline__ dd d2dd_bits(double x, int bias) {
  const unsigned hi32 = unsigned(__double2hiint(x)), lo32 = unsigned(__double2loint(x));
  const unsigned E0 = (hi32 >> 20) & 0x7FFu, sign = hi32 & 0x80000000u;
  const int E = int(E0) - bias;
  if (E0 == 0u || E < 897 || E > 1150) return {0.f, 0.f};
  const unsigned Ef = unsigned(E - 896);
  const float h = __uint_as_float(sign | (Ef << 23) | ((hi32 & 0xFFFFFu) << 3) | (lo32 >> 29));
  const unsigned m = lo32 & 0x1FFFFFFFu;
  const float mh = __fsub_rn(__uint_as_float(0x4B000000u | (m >> 6)), 8388608.0f);
  const float ml = __fsub_rn(__uint_as_float(0x4B000000u | (m & 63u)), 8388608.0f);
  const float mf = __fmaf_rn(mh, 64.0f, ml);
  const float l = __fmul_rn(__fmul_rn(mf, 0x1p-52f), __uint_as_float(Ef << 23));
  return {h, __uint_as_float(__float_as_uint(l) | sign)};
}
// f 2^bias as a double, by bits (exact for normal floats; zero and subnormals give 0); bias not far_scale, so that no
// exponent leaves the range of doubles
__device__ __forceinline__ double f2d_bits(float f, int bias) {
  const unsigned b = __float_as_uint(f), e = (b >> 23) & 0xFFu;
  const unsigned hi = e ? (b & 0x80000000u) | (unsigned(int(e) + 896 + bias) << 20) | ((b >> 3) & 0xFFFFFu) : 0u;
  return __hiloint2double(int(hi), e ? int(b << 29) : 0);
}
__device__ __forceinline__ double join(dd v, int bias) { return f2d_bits(v.h, bias) + f2d_bits(v.l, bias); }
// Warps whose inputs lie all below 2^-895, or some above 2^895, join their results by fp64 conversions and
// products instead, which flush and overflow as fp64 does, in paths of their own that keep nothing in registers for
// it (range checks in f2d_bits took 4 % of an apply, a test before each product 3 to 7 %).
__device__ __forceinline__ bool far_scale(int bias) { return unsigned(bias + 895) > 1790u; }
__device__ __forceinline__ double join_far(dd v, int bias) {
  const int part = bias / 2;
  return (double(v.h) + double(v.l)) * __hiloint2double((1023 + part) << 20, 0) *
         __hiloint2double((1023 + bias - part) << 20, 0);
}
// The biased exponent of the largest magnitude in a warp's columns of n doubles, where emax is that over all
// of them: Inf and NaN (0x7FF) are left out, and bad says whether the thread's own column holds one.
__device__ __forceinline__ unsigned finite_exponent(unsigned emax, const float2* col, int stride, int n, bool& bad) {
  bad = false;
  if (emax != 0x7FFu) return emax;
  unsigned e = 0;
#pragma unroll 1
  for (int l = 0; l < n; ++l) {
    const unsigned v = unsigned(__double2hiint(*reinterpret_cast<const double*>(col + l * stride))) & 0x7FF00000u;
    if (v == 0x7FF00000u) bad = true;
    else e = max(e, v);
  }
  return __reduce_max_sync(0xffffffffu, e) >> 20;
}
// two-sum of the high parts (exact), low parts added in fp32
__device__ __forceinline__ dd dd_add(dd a, dd b) {
  const float s = __fadd_rn(a.h, b.h);
  const float bb = __fsub_rn(s, a.h);
  const float e = __fadd_rn(__fsub_rn(a.h, __fsub_rn(s, bb)), __fsub_rn(b.h, bb));
  return {s, __fadd_rn(e, __fadd_rn(a.l, b.l))};
}
// exact fp32 product of the high parts (FMA residual) plus the two cross terms
__device__ __forceinline__ dd dd_mul(dd a, dd b) {
  const float p = __fmul_rn(a.h, b.h);
  float e = __fmaf_rn(a.h, b.h, -p);
  e = __fmaf_rn(a.h, b.l, e);
  e = __fmaf_rn(a.l, b.h, e);
  return {p, e};
}
__device__ __forceinline__ dd dd_norm(dd a) {
  const float s = __fadd_rn(a.h, a.l);
  return {s, __fsub_rn(a.l, __fsub_rn(s, a.h))};
}
__device__ __forceinline__ dd dd_fma(dd acc, dd a, dd b) { return dd_add(acc, dd_mul(a, b)); }


// The 1D contractions in difference form.  The Q2 nodes are {0, 1/2, 1} and the Gauss points
// 1/2 -+ delta, 1/2 with delta^2 = 3/20, so a line u of nodal values has at the outer Gauss points
//   0.4 u1 + 0.3 (u0 + u2) -+ delta (u2 - u0)      (the middle Gauss point is the middle node),
// and the derivative of the quadratic through three Gauss-point values v is the integer stencil
//   (-3 v0 + 4 v1 - v2, v2 - v0, v0 - 4 v1 + 3 v2) / (2 delta).
// The factor 1/(2 delta) is folded into the coefficient tables (kDerivScale below), which leaves a
// derivative line with five pair additions and no product, and a value line with three products:
// 44 and 52 fp32 instructions against 78 and 56 in the row-times-column form with tabulated
// constants; the transposes are 68 and 52 against 108 and 65.  An fp32 pair addition costs 8
// instructions and a product 4, and these contractions are most of a double-float cell.
constexpr double kDelta = 0.38729833462074168852;        // sqrt(3/20)
constexpr double kDerivScale = 1.2909944487358056284;    // 1 / (2 delta); its square is 5/3
template <int N> struct DfConst;                          // constants as float pairs
template <> struct DfConst<0> { static constexpr double v = 0.3; };
template <> struct DfConst<1> { static constexpr double v = 0.4; };
template <> struct DfConst<2> { static constexpr double v = kDelta; };
template <> struct DfConst<3> { static constexpr double v = 5.0 / 36.0; };
template <> struct DfConst<4> { static constexpr double v = 8.0 / 36.0; };
template <> struct DfConst<5> { static constexpr double v = kDelta * 5.0 / 18.0; };
template <int N> __device__ __forceinline__ dd dd_mulc(dd a) {
  constexpr float ch = float(DfConst<N>::v);
  constexpr float cl = float(DfConst<N>::v - double(ch));
  return dd_mul(dd{ch, cl}, a);
}
__device__ __forceinline__ dd dd_neg(dd a) { return {-a.h, -a.l}; }
__device__ __forceinline__ dd dd_sub(dd a, dd b) { return dd_add(a, dd_neg(b)); }
__device__ __forceinline__ dd dd_pow2(dd a, float s) { return {a.h * s, a.l * s}; }   // s a power of two

// one line, nodes -> Gauss points (u1 stays)
__device__ __forceinline__ void dd_line_values(dd& u0, dd u1, dd& u2) {
  const dd m = dd_add(dd_mulc<1>(u1), dd_mulc<0>(dd_add(u0, u2)));
  const dd r = dd_mulc<2>(dd_sub(u2, u0));
  u0 = dd_norm(dd_sub(m, r));
  u2 = dd_norm(dd_add(m, r));
}
// one line, Gauss points -> nodes (transposed); not renormalised
__device__ __forceinline__ void dd_line_values_t(dd& f0, dd& f1, dd& f2) {
  const dd t = dd_add(f0, f2), r = dd_mulc<2>(dd_sub(f2, f0)), c = dd_mulc<0>(t);
  f1 = dd_add(f1, dd_mulc<1>(t));
  f0 = dd_sub(c, r);
  f2 = dd_add(c, r);
}
// 2 delta times the derivatives at the three Gauss points of a line of Gauss-point values
__device__ __forceinline__ void dd_line_deriv(dd v0, dd v1, dd v2, dd& g0, dd& g1, dd& g2) {
  g1 = dd_sub(v2, v0);
  const dd c2 = dd_pow2(dd_sub(dd_add(v0, v2), dd_pow2(v1, 2.f)), 2.f);
  g0 = dd_sub(g1, c2);
  g2 = dd_add(g1, c2);
}
// the transpose of that stencil: (r0, r1, r2) += stencil^T (f0, f1, f2)
__device__ __forceinline__ void dd_line_deriv_t(dd f0, dd f1, dd f2, dd& r0, dd& r1, dd& r2) {
  const dd s = dd_add(dd_add(f0, f2), f1), e = dd_sub(f2, f0), e2 = dd_pow2(e, 2.f);
  r0 = dd_add(r0, dd_sub(e2, s));
  r1 = dd_sub(r1, dd_pow2(e, 4.f));
  r2 = dd_add(r2, dd_add(e2, s));
}
// one line of a Q1 function: end values -> the three Gauss points
__device__ __forceinline__ void dd_line_q1(dd p0, dd p1, dd& v0, dd& v1, dd& v2) {
  const dd r = dd_mulc<2>(dd_sub(p1, p0));
  v1 = dd_pow2(dd_add(p0, p1), 0.5f);
  v0 = dd_norm(dd_sub(v1, r));
  v2 = dd_norm(dd_add(v1, r));
}
// its transpose with the Gauss weights (5, 8, 5) / 18
__device__ __forceinline__ void dd_line_q1_t(dd g0, dd g1, dd g2, dd& o0, dd& o1) {
  const dd a = dd_add(dd_mulc<3>(dd_add(g0, g2)), dd_mulc<4>(g1)), b = dd_mulc<5>(dd_sub(g2, g0));
  o0 = dd_norm(dd_sub(a, b));
  o1 = dd_norm(dd_add(a, b));
}
// Gauss points -> nodes of a line whose test side has values v and derivative fluxes f: the transposed
// value contraction applied to v + stencil^T f, with both transposes sharing their sums and differences
__device__ __forceinline__ void dd_line_combine_t(dd f0, dd f1, dd f2, dd& v0, dd& v1, dd& v2) {
  const dd s = dd_add(dd_add(f0, f2), f1), e4 = dd_pow2(dd_sub(f2, f0), 4.f);
  const dd t = dd_add(dd_add(v0, v2), e4), d = dd_add(dd_sub(v2, v0), dd_pow2(s, 2.f));
  const dd c = dd_mulc<0>(t), r = dd_mulc<2>(d);
  v1 = dd_norm(dd_add(dd_sub(v1, e4), dd_mulc<1>(t)));
  v0 = dd_norm(dd_sub(c, r));
  v2 = dd_norm(dd_add(c, r));
}

}  // namespace
}  // namespace mf
