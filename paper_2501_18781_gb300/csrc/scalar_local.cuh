// Local (one cell) action of the scalar operators in collocation form, shared by the apply and the dense
// element-matrix path of the diagonal.  In fp64 the pipe bounds it (16 cycles of an SM per warp instruction), so
// operations count: lines in difference form and Gauss weights inside the transposes (lines.cuh), no products
// with per-point weights.
#pragma once

#include "lines.cuh"
#include "ops.h"

namespace mf {

// Smoothed Heaviside of the interpolated level set (Section 2.3).
template <typename T> __device__ __forceinline__ T heaviside(T phi, int kind, T eps) {
  if (kind == 0) {  // tanh-regularised reading: H = clamp((1 + phi)/2)
    T H = T(0.5) * (T(1) + phi);
    return H < T(0) ? T(0) : (H > T(1) ? T(1) : H);
  }
  // eq. (heaviside) with d = 2 eps atanh(phi)
  const T lim = T(1) - (sizeof(T) == 8 ? T(2.220446049250313e-16) : T(1.1920929e-7));
  T p = phi > lim ? lim : (phi < -lim ? -lim : phi);
  T d = T(2) * eps * atanh(p);
  if (d <= T(-3) * eps) return T(0);
  if (d >= T(3) * eps) return T(1);
  const T pi = T(3.141592653589793);
  return T(0.5) + d / (T(6) * eps) + sin(pi * d / (T(3) * eps)) / (T(2) * pi);
}

// U: nodal values of the cell (overwritten); R: the cell's contribution, at the nodes.
// C: scalar coefficient at the Gauss points (in-kernel phi for MODE 0 reinit).
// POINTS: reinitialisation point by point, which holds two arrays of 27 values instead of three.
template <typename T, int KIND, int MODE, bool BETA, bool TR, bool POINTS = (KIND == K_REINIT && MODE == 0)>
__device__ __forceinline__ void scalar_local(const ScalarArgs<typename Store<T>::type>& A, int64_t cell, T h, T mh2,
                                             const T* C, T* U, T* R) {
  const T eps = T(A.eps);
  auto line = [](int d, int n, int& p0, int& p1, int& p2) {
    p0 = d == 0 ? 3 * n : (d == 1 ? (n % 3) + 9 * (n / 3) : n);
    const int st = d == 0 ? 1 : (d == 1 ? 3 : 9);
    p1 = p0 + st;
    p2 = p1 + st;
  };
#pragma unroll
  for (int d = 0; d < 3; ++d)
#pragma unroll
    for (int n = 0; n < 9; ++n) {
      int p0, p1, p2;
      line(d, n, p0, p1, p2);
      line_values(U[p0], U[p1], U[p2]);
    }
  if constexpr (POINTS) {
    // the normal of every point from the table, or from the level set's gradient there
#pragma unroll
    for (int q = 0; q < 27; ++q) R[q] = T(0);
#pragma unroll
    for (int q = 0; q < 27; ++q) {
      const int qa = q % 3, qb = (q / 3) % 3, qc = q / 9;
      const T w = Tb<T>::W3(q);
      T gx, gy, gz, nx, ny, nz;
      grad_at<T>(U, qa, qb, qc, gx, gy, gz);
      if constexpr (MODE == 0) {
        grad_at<T>(C, qa, qb, qc, nx, ny, nz);
        const T nn = sqrt(nx * nx + ny * ny + nz * nz);
        const T inv = nn < T(1e-12) ? T(0) : T(1) / nn;
        nx *= inv; ny *= inv; nz *= inv;
      } else {
        nx = from_store<T>(__ldg(A.qvec + q * A.ncp + cell));
        ny = from_store<T>(__ldg(A.qvec + (27 + q) * A.ncp + cell));
        nz = from_store<T>(__ldg(A.qvec + (54 + q) * A.ncp + cell));
      }
      const T s = w * (eps * (nx * gx + ny * gy + nz * gz));
      R[q] += w * (mh2 * U[q]);
      add_grad_test<T>(R, qa, qb, qc, s * nx, s * ny, s * nz);
    }
#pragma unroll
    for (int d = 2; d >= 0; --d)
#pragma unroll
      for (int n = 0; n < 9; ++n) {
        int p0, p1, p2;
        line(d, n, p0, p1, p2);
        line_values_t(R[p0], R[p1], R[p2]);
      }
#pragma unroll
    for (int q = 0; q < 27; ++q) R[q] *= h;
  } else {
    // Test side without Gauss weights (the transposes carry them, lines.cuh) and without a factor f that
    // makes the coefficient read per point the flux's own: 5/3 (both derivative factors 1 / (2 delta)),
    // h / (2 delta) with convection.
    T f, fi;
    if constexpr (BETA) {
      f = h * T(kLineDerivScale);
      if constexpr (std::is_same<T, df64>::value) fi = T(1.0 / f.to_double());
      else fi = T(1) / f;
    } else {
      f = KIND == K_MASS ? T(1) : T(5.0 / 3.0);
      fi = KIND == K_MASS ? T(1) : T(0.6);
    }
    const T wm = mh2 * fi;
#pragma unroll
    for (int q = 0; q < 27; ++q) {
      T m = wm;
      if constexpr (KIND == K_HEAT) {  // rho_cp / dt per Gauss point when the heat capacity varies
        if (A.qmass) m = from_store<T>(__ldg(A.qmass + q * A.ncp + cell)) * (h * h * fi);
      }
      R[q] = m * U[q];
    }
    const T kw[4] = {T(0.3 * 5.0 / 18.0), T(8.0 / 18.0), T(0.4 * 5.0 / 18.0), T(kLineDelta * 5.0 / 18.0)};
    const T kx[4] = {kw[0] * (f * h), kw[1] * (f * h), kw[2] * (f * h), kw[3] * (f * h)};
    auto vec = [&](int d, int q) { return from_store<T>(__ldg(A.qvec + (d * 27 + q) * A.ncp + cell)); };
    if constexpr (KIND == K_REINIT) {
      // s = n . grad u, then the fluxes s n
      T S[27];
#pragma unroll
      for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int n = 0; n < 9; ++n) {
          int p0, p1, p2;
          line(d, n, p0, p1, p2);
          T g0, g1, g2;
          line_deriv(U[p0], U[p1], U[p2], g0, g1, g2);
          if (d == 0) {
            S[p0] = vec(d, p0) * g0; S[p1] = vec(d, p1) * g1; S[p2] = vec(d, p2) * g2;
          } else {
            S[p0] += vec(d, p0) * g0; S[p1] += vec(d, p1) * g1; S[p2] += vec(d, p2) * g2;
          }
        }
#pragma unroll
      for (int q = 0; q < 27; ++q) S[q] *= eps;
#pragma unroll
      for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int n = 0; n < 9; ++n) {
          int p0, p1, p2;
          line(d, n, p0, p1, p2);
          const T f0 = S[p0] * vec(d, p0), f1 = S[p1] * vec(d, p1), f2 = S[p2] * vec(d, p2);
          if (d < 2) line_deriv_tw(f0, f1, f2, R[p0], R[p1], R[p2]);
          else line_combine_tw(kw, f0, f1, f2, R[p0], R[p1], R[p2]);
        }
    } else if constexpr (KIND != K_MASS) {
      const T cs = T(5.0 / 3.0) * fi;   // 1 without convection
#pragma unroll
      for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int n = 0; n < 9; ++n) {
          int p[3];
          line(d, n, p[0], p[1], p[2]);
          T g[3], F[3];
          line_deriv(U[p[0]], U[p[1]], U[p[2]], g[0], g[1], g[2]);
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            if constexpr (BETA) {
              F[k] = (cs * C[p[k]]) * g[k];
              const T b = vec(d, p[k]);
              if constexpr (!TR) R[p[k]] += b * g[k];
              else F[k] += b * U[p[k]];
            } else {
              F[k] = C[p[k]] * g[k];
            }
          }
          if (d < 2) line_deriv_tw(F[0], F[1], F[2], R[p[0]], R[p[1]], R[p[2]]);
          else line_combine_tw(kw, F[0], F[1], F[2], R[p[0]], R[p[1]], R[p[2]]);
        }
    }
#pragma unroll
    for (int d = KIND == K_MASS ? 2 : 1; d >= 0; --d)
#pragma unroll
      for (int n = 0; n < 9; ++n) {
        int p0, p1, p2;
        line(d, n, p0, p1, p2);
        line_values_tw(d == 0 ? kx : kw, R[p0], R[p1], R[p2]);
      }
  }
}

}  // namespace mf
