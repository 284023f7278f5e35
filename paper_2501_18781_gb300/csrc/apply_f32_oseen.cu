// fp32 apply of the Oseen operator (Q2 velocity / Q1 pressure, uniform mesh, folded Gauss-point
// coefficients) for the preconditioner's inner iterations.
//
// A block of three warps owns a tile of 8 x 4 x 1 cells; warp C evaluates the test functions of velocity
// component C on axes permuted so that a is its own direction: planes (a, b) with the value terms, the
// diagonal flux along a, the flux along b and the continuity share, then planes (a, c) with the flux along
// c.  The components' Gauss-point values and test sides live in shared memory, so the loops over planes stay
// rolled and the register count low.  One thread per cell held all three components: 255 registers, 8 warps per SM, 31 % of the
// issue slots.  Bound now: L1 accesses and issue (60 and 50 %).  Melt-pool apply at 64^3 164 -> 139 us, at 40^3
// 62.7 (with the separate copy of the Dirichlet rows) -> 39.6 us.
#include "lines.cuh"
#include "ops.h"

namespace mf {

UniformGeom uniform_geom(const mf_dofmap* m);

namespace {

constexpr int kOseenBlocks = 6;   // per SM; 64^3 melt-pool apply with 5 / 6 / 7 / 8 blocks: 136 / 137 / 150 / 150 us (spills)

struct OseenTileArgs {
  const float* src;
  float* dst;
  int64_t nu;        // velocity DoFs per component (pressure block starts at 3 nu)
  const float* cm;   // [tile][27][32] w h^3 (sigma rho + Darcy)
  const float* cv;   // [tile][27][32] (5/3) w h mu
  const float* cb;   // [tile][81][32] w h^2 rho beta / (2 delta)
  const float* nr;   // [tile][81][32] interface normal (melt-pool trace correction)
  float pw[4];       // -h^2 w / (2 delta), by the number of middle coordinates of the point
  float mh2;         // -h^2 / (2 delta)
  int ntx, nty;
};

__device__ __forceinline__ void prefetch_l2(const float* p, unsigned bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// Test side of component C at the warp's cells.  Every pointer is the lane's: sU[27 e + q], pP[q] and pT[q]
// (shared, 32 floats apart), the tables (global, 32 floats apart); sv receives the test side after the
// transposes along c and a, Rp the continuity shares in the order of the permuted axes.  One instance per
// component: all offsets are constants (with run-time strides the addressing doubled the instructions).
template <int C, bool EXT>
__device__ __forceinline__ void oseen_component(const float* sU, const float* pP, const float* pT, float* sv,
                                                const float* __restrict__ cm, const float* __restrict__ cv,
                                                const float* __restrict__ cb, const float* __restrict__ nr, float* Rp) {
  // permuted axes: a = own direction, b and c the others (strides in the 27-array)
  constexpr int sa = C == 0 ? 1 : (C == 1 ? 3 : 9), sb = C == 1 ? 1 : 3, sc = C == 2 ? 1 : 9;
  constexpr int eb = C == 1 ? 0 : 1, ec = C == 2 ? 0 : 2;
  constexpr int oa = 32 * sa, ob = 32 * sb, oc = 32 * sc;
  const float* const uC = sU + 27 * 32 * C;
  const float* const uB = sU + 27 * 32 * eb;
  const float* const uc = sU + 27 * 32 * ec;
  const float* __restrict__ cba = cb + 27 * 32 * C;
  const float* __restrict__ cbb = cb + 27 * 32 * eb;
  const float* __restrict__ cbc = cb + 27 * 32 * ec;
  const float* __restrict__ nA = nr + 27 * 32 * C;
  const float* __restrict__ nB = nr + 27 * 32 * eb;
  const float* __restrict__ nC = nr + 27 * 32 * ec;
#pragma unroll
  for (int n = 0; n < 8; ++n) Rp[n] = 0.f;
#pragma unroll 1
  for (int ic = 0; ic < 3; ++ic) {
    float U[9], c2[9], R[9];
#pragma unroll
    for (int p = 0; p < 9; ++p) {
      const int o = (p % 3) * oa + (p / 3) * ob + ic * oc;
      U[p] = uC[o];
      c2[p] = __ldg(cv + o);
      R[p] = __ldg(cm + o) * U[p];
    }
    float T1[3][2];
#pragma unroll
    for (int n = 0; n < 3; ++n) {
      float g[3], fa[3];
      line_deriv(U[3 * n], U[3 * n + 1], U[3 * n + 2], g[0], g[1], g[2]);
      line_q1_t(g[0], g[1], g[2], T1[n][0], T1[n][1]);
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        const int p = 3 * n + m, o = m * oa + n * ob + ic * oc;
        R[p] += __ldg(cba + o) * g[m];
        fa[m] = 2.f * c2[p] * g[m] + pP[o];
        if (EXT) {
          const float na = __ldg(nA + o);
          fa[m] += pT[o] * na * na;
        }
      }
      line_deriv_t(fa[0], fa[1], fa[2], R[3 * n], R[3 * n + 1], R[3 * n + 2]);
    }
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      float t0, t1;
      line_q1_t(T1[0][m], T1[1][m], T1[2][m], t0, t1);
      const float wc = ic == 1 ? 8.f / 36.f : 5.f / 36.f, xc = float(ic - 1) * float(kLineDelta * 5.0 / 18.0);
      Rp[m] += (wc - xc) * t0;
      Rp[m + 2] += (wc - xc) * t1;
      Rp[m + 4] += (wc + xc) * t0;
      Rp[m + 6] += (wc + xc) * t1;
    }
    float X[9];
#pragma unroll
    for (int n = 0; n < 3; ++n) {
      const float* const q = uB + n * ob + ic * oc;
      line_deriv(q[0], q[oa], q[2 * oa], X[3 * n], X[3 * n + 1], X[3 * n + 2]);
    }
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      float g[3], fb[3];
      line_deriv(U[m], U[m + 3], U[m + 6], g[0], g[1], g[2]);
#pragma unroll
      for (int n = 0; n < 3; ++n) {
        const int p = 3 * n + m, o = m * oa + n * ob + ic * oc;
        R[p] += __ldg(cbb + o) * g[n];
        fb[n] = c2[p] * (g[n] + X[p]);
        if (EXT) fb[n] += pT[o] * __ldg(nA + o) * __ldg(nB + o);
      }
      line_deriv_t(fb[0], fb[1], fb[2], R[m], R[m + 3], R[m + 6]);
    }
#pragma unroll
    for (int p = 0; p < 9; ++p) sv[(p % 3) * oa + (p / 3) * ob + ic * oc] = R[p];
  }
#pragma unroll 1
  for (int ib = 0; ib < 3; ++ib) {
    float X[9], V[9];   // index ia + 3 ic
#pragma unroll
    for (int n = 0; n < 3; ++n) {
      const float* const q = uc + ib * ob + n * oc;
      line_deriv(q[0], q[oa], q[2 * oa], X[3 * n], X[3 * n + 1], X[3 * n + 2]);
    }
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      const float* const q = uC + m * oa + ib * ob;
      float g[3], fc[3];
      line_deriv(q[0], q[oc], q[2 * oc], g[0], g[1], g[2]);
#pragma unroll
      for (int n = 0; n < 3; ++n) {
        const int o = m * oa + ib * ob + n * oc;
        fc[n] = __ldg(cv + o) * (g[n] + X[m + 3 * n]);
        V[m + 3 * n] = sv[o] + __ldg(cbc + o) * g[n];
        if (EXT) fc[n] += pT[o] * __ldg(nA + o) * __ldg(nC + o);
      }
      line_combine_t(fc[0], fc[1], fc[2], V[m], V[m + 3], V[m + 6]);
    }
#pragma unroll
    for (int n = 0; n < 3; ++n) {
      line_values_t(V[3 * n], V[3 * n + 1], V[3 * n + 2]);
#pragma unroll
      for (int m = 0; m < 3; ++m) sv[m * oa + ib * ob + n * oc] = V[3 * n + m];
    }
  }
}

template <bool EXT>
__global__ void __launch_bounds__(96, kOseenBlocks) k_oseen_f32_tiles(const __grid_constant__ OseenTileArgs A, UniformGeom ug) {
  __shared__ float sU[3][27][32], sV[3][27][32];   // values at the Gauss points; each warp's test side
  __shared__ float sP[27][32];             // pressure at the Gauss points; later the continuity shares
  __shared__ float sT[EXT ? 27 : 1][32];   // EXT: t = -2 cv div u
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, xl = lane & 7, yl = lane >> 3;
  const int64_t tile = blockIdx.x;
  const int ncol = A.ntx * A.nty, col = int(tile % ncol), k = int(tile / ncol);
  const int i = (col % A.ntx) * 8 + xl, j = (col / A.ntx) * 4 + yl;
  const bool active = i < ug.nx && j < ug.ny;
  const float* __restrict__ cm = A.cm + tile * (27 * 32) + lane;
  const float* __restrict__ cv = A.cv + tile * (27 * 32) + lane;
  const float* __restrict__ cb = A.cb + tile * (81 * 32) + lane;
  const float* __restrict__ nr = A.nr + (EXT ? tile * (81 * 32) + lane : 0);
  if (lane == 0) {   // the tile's coefficients into L2 while the inputs load
    if (w == 0) {
      prefetch_l2(cm, 27 * 128);
      prefetch_l2(cv, 27 * 128);
    }
    if (w == 1) prefetch_l2(cb, 81 * 128);
    if (EXT && w == 2) prefetch_l2(nr, 81 * 128);
  }
  const int64_t base = active ? 2 * int64_t(i) + ug.sx * (2 * int64_t(j)) + ug.sy * (2 * int64_t(k)) : 0;
  const int64_t px = ug.nx + 1, pxy = px * (ug.ny + 1);
  const int64_t pbase = active ? i + px * (j + (ug.ny + 1) * int64_t(k)) : 0;
  // nodes of the three planes that read as 0 (Dirichlet faces; all of a lane without a cell)
  const uint32_t f = ug.dir_faces;
  const uint32_t side = active ? (((f & 1u) && i == 0) ? 0x049u : 0u) | (((f & 2u) && i == ug.nx - 1) ? 0x124u : 0u) |
                                     (((f & 4u) && j == 0) ? 0x007u : 0u) | (((f & 8u) && j == ug.ny - 1) ? 0x1C0u : 0u)
                               : 0x1FFu;
  const uint32_t off0 = ((f & 16u) && k == 0) ? 0x1FFu : side, off2 = ((f & 32u) && k == ug.nz - 1) ? 0x1FFu : side;
  const uint32_t off = off0 | (side << 9) | (off2 << 18);
  float* const dst = A.dst + w * A.nu + base;
  {
    const float* __restrict__ s = A.src + w * A.nu + base;
    float U[27];
#pragma unroll
    for (int l = 0; l < 27; ++l) U[l] = __ldg(s + (l % 3) + ug.sx * ((l / 3) % 3) + ug.sy * (l / 9));
    float Pn[8];
#pragma unroll
    for (int n = 0; n < 8; ++n) {
      Pn[n] = __ldg(A.src + 3 * A.nu + pbase + (n & 1) + px * ((n >> 1) & 1) + pxy * (n >> 2));
      if (!active) Pn[n] = 0.f;
    }
    if (off) {   // Dirichlet rows return the input
#pragma unroll
      for (int l = 0; l < 27; ++l)
        if ((off >> l) & 1u) {
          if (active) dst[(l % 3) + ug.sx * ((l / 3) % 3) + ug.sy * (l / 9)] = U[l];
          U[l] = 0.f;
        }
    }
#pragma unroll
    for (int n = 0; n < 9; ++n) line_values(U[3 * n], U[3 * n + 1], U[3 * n + 2]);
#pragma unroll
    for (int n = 0; n < 9; ++n) {
      const int p = (n % 3) + 9 * (n / 3);
      line_values(U[p], U[p + 3], U[p + 6]);
    }
#pragma unroll
    for (int p = 0; p < 9; ++p) line_values(U[p], U[p + 9], U[p + 18]);
#pragma unroll
    for (int q = 0; q < 27; ++q) sU[w][q][lane] = U[q];
    // pressure term of the warp's plane qc = w of Gauss points
    const float sg = float(w - 1) * float(kLineDelta);
    float Pz[4], Py[2][3];
#pragma unroll
    for (int n = 0; n < 4; ++n) Pz[n] = 0.5f * (Pn[n] + Pn[n + 4]) + sg * (Pn[n + 4] - Pn[n]);
#pragma unroll
    for (int a = 0; a < 2; ++a) line_q1(Pz[a], Pz[a + 2], Py[a][0], Py[a][1], Py[a][2]);
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      float v[3];
      line_q1(Py[0][b], Py[1][b], v[0], v[1], v[2]);
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const int mid = (a == 1) + (b == 1);
        sP[a + 3 * b + 9 * w][lane] = (w == 1 ? A.pw[mid + 1] : A.pw[mid]) * v[a];
      }
    }
  }
  __syncthreads();
  if (EXT) {   // plane qc = w
    float D[9];
#pragma unroll
    for (int n = 0; n < 3; ++n)
      line_deriv(sU[0][9 * w + 3 * n][lane], sU[0][9 * w + 3 * n + 1][lane], sU[0][9 * w + 3 * n + 2][lane], D[3 * n],
                 D[3 * n + 1], D[3 * n + 2]);
#pragma unroll
    for (int n = 0; n < 3; ++n) {
      float g0, g1, g2;
      line_deriv(sU[1][9 * w + n][lane], sU[1][9 * w + n + 3][lane], sU[1][9 * w + n + 6][lane], g0, g1, g2);
      D[n] += g0;
      D[n + 3] += g1;
      D[n + 6] += g2;
    }
    const float s2 = 2.f * float(w - 1);
#pragma unroll
    for (int p = 0; p < 9; ++p) {
      const float v0 = sU[2][p][lane], v1 = sU[2][p + 9][lane], v2 = sU[2][p + 18][lane];
      const float div = D[p] + ((v2 - v0) + s2 * ((v0 + v2) - 2.f * v1));
      sT[p + 9 * w][lane] = -2.f * __ldg(cv + 32 * (p + 9 * w)) * div;
    }
    __syncthreads();
  }
  float Rp[8];
  float* const sv = &sV[w][0][lane];
  if (w == 0) oseen_component<0, EXT>(&sU[0][0][lane], &sP[0][lane], &sT[0][lane], sv, cm, cv, cb, nr, Rp);
  else if (w == 1) oseen_component<1, EXT>(&sU[0][0][lane], &sP[0][lane], &sT[0][lane], sv, cm, cv, cb, nr, Rp);
  else oseen_component<2, EXT>(&sU[0][0][lane], &sP[0][lane], &sT[0][lane], sv, cm, cv, cb, nr, Rp);
  __syncthreads();   // every warp has read what it needs of sP
  // continuity shares -int psi_n d_C u_C, in the order of the mesh axes
  const int pa = w == 0 ? 1 : (w == 1 ? 2 : 4), pb = w == 1 ? 1 : 2, pc = w == 2 ? 1 : 4;
#pragma unroll
  for (int n = 0; n < 8; ++n) sP[8 * w + (n & 1) * pa + ((n >> 1) & 1) * pb + (n >> 2) * pc][lane] = Rp[n];
  __syncthreads();
  if (active) {
    float* const pd = A.dst + 3 * A.nu + pbase;
    for (int n = w; n < 8; n += 3)
      atomicAdd(pd + (n & 1) + px * ((n >> 1) & 1) + pxy * (n >> 2),
                A.mh2 * ((sP[n][lane] + sP[8 + n][lane]) + sP[16 + n][lane]));
  }
  const uint32_t folded = (xl ? 0x049u : 0u) | (yl ? 0x007u : 0u);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    float R[9];
#pragma unroll
    for (int p = 0; p < 9; ++p) R[p] = active ? sv[32 * (9 * c + p)] : 0.f;
    if (w == 1) {   // the transpose along b is still to do: x for this warp, y for the others
#pragma unroll
      for (int b = 0; b < 3; ++b) line_values_t(R[3 * b], R[3 * b + 1], R[3 * b + 2]);
    } else {
#pragma unroll
      for (int a = 0; a < 3; ++a) line_values_t(R[a], R[a + 3], R[a + 6]);
    }
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const float t = __shfl_down_sync(0xffffffffu, R[3 * b], 1);
      if (xl < 7) R[3 * b + 2] += t;
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float t = __shfl_down_sync(0xffffffffu, (a == 0 && xl > 0) ? 0.f : R[a], 8);
      if (yl < 3) R[a + 6] += t;
    }
    const uint32_t skip = ((off >> (9 * c)) & 0x1FFu) | folded;
    float* const p = dst + ug.sy * c;
#pragma unroll
    for (int l = 0; l < 9; ++l)
      if (!((skip >> l) & 1u)) atomicAdd(p + (l % 3) + ug.sx * (l / 3), R[l]);
  }
}

}  // namespace

mf_status launch_oseen_f32_tables(mf_ctx* ctx, const mf_dofmap* mu, const double* cm64, const double* cv64,
                                  const double* cb64, const double* nr64, float* cm, float* cv, float* cb, float* nr) {
  MF_TRY(launch_tile_table_plain(ctx, mu, cm64, 1, 1.0, cm));
  MF_TRY(launch_tile_table_plain(ctx, mu, cv64, 1, 5.0 / 3.0, cv));
  MF_TRY(launch_tile_table_plain(ctx, mu, cb64, 3, kLineDerivScale, cb));
  return nr ? launch_tile_table_plain(ctx, mu, nr64, 3, 1.0, nr) : MF_OK;
}

mf_status launch_oseen_f32_uniform(mf_ctx* ctx, const mf_dofmap* mu, const float* src, float* dst, const float* cm,
                                   const float* cv, const float* cb, const float* nr) {
  const UniformGeom ug = uniform_geom(mu);
  OseenTileArgs a{};
  a.src = src;
  a.dst = dst;
  a.nu = mu->n_dofs;
  a.cm = cm;
  a.cv = cv;
  a.cb = cb;
  a.nr = nr;
  a.ntx = (ug.nx + 7) / 8;
  a.nty = (ug.ny + 3) / 4;
  const double s = -(ug.h * ug.h) * kLineDerivScale;
  for (int mid = 0; mid < 4; ++mid) {
    double w = s;
    for (int t = 0; t < 3; ++t) w *= t < mid ? 8.0 / 18.0 : 5.0 / 18.0;
    a.pw[mid] = float(w);
  }
  a.mh2 = float(s);
  const unsigned tiles = unsigned(int64_t(a.ntx) * a.nty * ug.nz);
  if (nr) k_oseen_f32_tiles<true><<<tiles, 96, 0, ctx->stream>>>(a, ug);
  else k_oseen_f32_tiles<false><<<tiles, 96, 0, ctx->stream>>>(a, ug);
  ctx->launches++;
  MF_CUDA_TRY(cudaGetLastError());
  return MF_OK;
}

}  // namespace mf
