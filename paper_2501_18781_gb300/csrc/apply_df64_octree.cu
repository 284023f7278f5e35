// Double-float apply of the conservative level-set reinitialisation operator on adaptively refined
// (octree) meshes with hanging-node constraints: (1/dtau) M + eps N_n, N_n(u, v) = int (n.grad u)
// (n.grad v) (Section 2.3 reinitialisation, Appendix B matrix-free evaluation), n the unit normal of
// the level set per Gauss point (the operator's fp64 table, as float pairs).
//
// One thread per leaf, cells in the map's processing order (unconstrained first).  The cell's 27
// values are gathered through the cell map in fp64 (a hanging node as the weighted sum of its
// masters), scaled by one power of two per warp and split into float pairs; values and derivatives
// at the Gauss points run in double-float on the fp32 pipes.  Every flux of this operator is
// s n with s = w eps h (n . grad u).  The values and s live in two shared-memory columns of the thread
// and each phase is a rolled loop over them: planes z = const (n_x d_x u + n_y d_y u), z lines (s),
// planes again (value term and the x and y test parts, over the values), z lines (z test part and
// transpose), slabs of nodes (y and x transposes).  The cell's contributions are joined to doubles and
// added to the free DoFs, hanging ones through the constraint weights.  The blocks of all right-hand
// sides of one range of cells are neighbours in the launch order, so the normals (648 bytes per cell)
// are read from HBM once and from L2 by the other right-hand sides (591 MB instead of 4.0 GB of HBM reads
// for eight of them).  Measured: eight right-hand sides on the base 12 + 3 levels octree 3750 -> 1190 us
// (1.17 ms at 47 % of the issue slots, long-scoreboard stalls on the scattered values).
#include <algorithm>

#include "df_pairs.cuh"

namespace mf {

MF_DEFINE_TABLE_UPLOAD

OctGeom oct_geom(const mf_dofmap* m);

namespace {

constexpr int kOctThreads = 128;

struct DfOctArgs {
  const double* src;
  double* dst;
  int nrhs;           // right-hand sides: block b works on right-hand side b % nrhs
  int64_t ld;         // distance between right-hand sides
  const float2* n;    // [3][27][ncells] unit normal per Gauss point
  int64_t ncells;     // stride of the normal table
  float2 we[27];      // (5/3) w_q eps h0 (h0: edge of a level-0 cell; 5/3: both derivative factors)
  float2 wm[27];      // w_q m h0^3 (m: value coefficient 1 / dtau)
};

constexpr int kOctSmem = 2 * 27 * kOctThreads * int(sizeof(float2));
__device__ __forceinline__ float pow2f_oct(int e) { return __uint_as_float(unsigned(e + 127) << 23); }

__global__ void __launch_bounds__(kOctThreads, 4) k_reinit_df_octree(const __grid_constant__ DfOctArgs A, OctGeom og) {
  extern __shared__ float2 oct_smem[];
  const int t = threadIdx.x;
  float2* const sU = oct_smem + t;
  float2* const sV = oct_smem + 27 * kOctThreads + t;
  auto ld2 = [](const float2* p) { const float2 v = *p; return dd{v.x, v.y}; };
  auto st2 = [](float2* p, dd v) { *p = make_float2(v.h, v.l); };
  auto ldg2 = [](const float2* p) { const float2 v = __ldg(p); return dd{v.x, v.y}; };
  const int rhs = blockIdx.x % A.nrhs;
  const int64_t slot = int64_t(blockIdx.x / A.nrhs) * kOctThreads + t;
  const bool active = slot < og.ncells;
  const int64_t cell = active ? __ldg(og.order + slot) : 0;
  const int lev = active ? __ldg(og.level + cell) : 0;
  const double* __restrict__ src = A.src + rhs * A.ld;
  const int32_t* __restrict__ map = og.cmap + cell;
  const int64_t nc = A.ncells;
  int bias = 0;
  bool bad;   // an Inf or NaN among the cell's inputs
  {
    double X[27];
    uint32_t hanging = 0;
    {
      int32_t id[27];
#pragma unroll
      for (int l = 0; l < 27; ++l) id[l] = __ldg(map + l * og.ncp);
#pragma unroll
      for (int l = 0; l < 27; ++l) {
        X[l] = __ldg(src + max(id[l], 0));
        hanging |= id[l] < 0 ? 1u << l : 0u;
      }
      if (og.dflag) {
#pragma unroll
        for (int l = 0; l < 27; ++l)
          if (id[l] >= 0 && __ldg(og.dflag + id[l])) X[l] = 0.0;
      }
    }
    if (!active) {
      hanging = 0;
#pragma unroll
      for (int l = 0; l < 27; ++l) X[l] = 0.0;
    }
#pragma unroll
    for (int l = 0; l < 27; ++l) *reinterpret_cast<double*>(sU + l * kOctThreads) = X[l];
    unsigned emax = 0;
#pragma unroll
    for (int l = 0; l < 27; ++l)
      if (!((hanging >> l) & 1u)) emax = max(emax, unsigned(__double2hiint(X[l])) & 0x7FF00000u);
    for (uint32_t left = hanging; left; left &= left - 1) {
      const int l = __ffs(left) - 1;
      const int r = -1 - __ldg(map + l * og.ncp);
      double v = 0.0;
      for (int e = __ldg(og.rowptr + r); e < __ldg(og.rowptr + r + 1); ++e) {
        const int32_t m = __ldg(og.cols + e);
        if (!(og.dflag && __ldg(og.dflag + m))) v += __ldg(og.w64 + e) * __ldg(src + m);
      }
      *reinterpret_cast<double*>(sU + l * kOctThreads) = v;
      emax = max(emax, unsigned(__double2hiint(v)) & 0x7FF00000u);
    }
    __syncwarp();
    emax = finite_exponent(__reduce_max_sync(0xffffffffu, emax) >> 20, sU, kOctThreads, 27, bad);
    bias = emax ? int(emax) - 1023 : 0;
  }
#pragma unroll 1
  for (float2* p = sU; p < sU + 27 * kOctThreads; p += 3 * kOctThreads) {
    dd u0 = d2dd_bits(*reinterpret_cast<double*>(p), bias);
    dd u1 = d2dd_bits(*reinterpret_cast<double*>(p + kOctThreads), bias);
    dd u2 = d2dd_bits(*reinterpret_cast<double*>(p + 2 * kOctThreads), bias);
    dd_line_values(u0, u1, u2);
    st2(p, u0);
    st2(p + kOctThreads, u1);
    st2(p + 2 * kOctThreads, u2);
  }
#pragma unroll 1
  for (int n = 0; n < 6; ++n) {   // y lines of the three planes, then z lines
    const int o = n < 3 ? 9 * n : 3 * (n - 3), st = n < 3 ? 3 : 9;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      float2* const p = sU + (o + a) * kOctThreads;
      dd u0 = ld2(p), u2 = ld2(p + 2 * st * kOctThreads);
      dd_line_values(u0, ld2(p + st * kOctThreads), u2);
      st2(p, u0);
      st2(p + 2 * st * kOctThreads, u2);
    }
  }
  const float2* __restrict__ nx = A.n + cell;
  const float2* __restrict__ ny = nx + 27 * nc;
  const float2* __restrict__ nz = ny + 27 * nc;
  // n_x d_x u + n_y d_y u, plane by plane
#pragma unroll 1
  for (int qc = 0; qc < 3; ++qc) {
    const int q0 = 9 * qc;
    dd U[9], S[9];
#pragma unroll
    for (int p = 0; p < 9; ++p) U[p] = ld2(sU + (q0 + p) * kOctThreads);
#pragma unroll
    for (int n = 0; n < 3; ++n) {
      dd g0, g1, g2;
      dd_line_deriv(U[3 * n], U[3 * n + 1], U[3 * n + 2], g0, g1, g2);
      S[3 * n] = dd_mul(ldg2(nx + (q0 + 3 * n) * nc), g0);
      S[3 * n + 1] = dd_mul(ldg2(nx + (q0 + 3 * n + 1) * nc), g1);
      S[3 * n + 2] = dd_mul(ldg2(nx + (q0 + 3 * n + 2) * nc), g2);
    }
#pragma unroll
    for (int n = 0; n < 3; ++n) {
      dd g0, g1, g2;
      dd_line_deriv(U[n], U[n + 3], U[n + 6], g0, g1, g2);
      S[n] = dd_fma(S[n], ldg2(ny + (q0 + n) * nc), g0);
      S[n + 3] = dd_fma(S[n + 3], ldg2(ny + (q0 + n + 3) * nc), g1);
      S[n + 6] = dd_fma(S[n + 6], ldg2(ny + (q0 + n + 6) * nc), g2);
    }
#pragma unroll
    for (int p = 0; p < 9; ++p) st2(sV + (q0 + p) * kOctThreads, S[p]);
  }
  // s = w eps h (n . grad u), z line by z line (h = h0 2^-level, an exact power-of-two scale)
  const float s1 = pow2f_oct(-lev), s3 = pow2f_oct(-3 * lev);
#pragma unroll 1
  for (int p = 0; p < 9; ++p) {
    dd g[3];
    dd_line_deriv(ld2(sU + p * kOctThreads), ld2(sU + (p + 9) * kOctThreads), ld2(sU + (p + 18) * kOctThreads), g[0], g[1],
                  g[2]);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const int q = p + 9 * c;
      const dd ng = dd_norm(dd_fma(ld2(sV + q * kOctThreads), ldg2(nz + q * nc), g[c]));
      st2(sV + q * kOctThreads, dd_norm(dd_pow2(dd_mul(dd{A.we[q].x, A.we[q].y}, ng), s1)));
    }
  }
  // value term and the x and y test parts, plane by plane, over the values
#pragma unroll 1
  for (int qc = 0; qc < 3; ++qc) {
    const int q0 = 9 * qc;
    dd R[9], S[9];
#pragma unroll
    for (int p = 0; p < 9; ++p) {
      S[p] = ld2(sV + (q0 + p) * kOctThreads);
      R[p] = dd_pow2(dd_mul(dd{A.wm[q0 + p].x, A.wm[q0 + p].y}, ld2(sU + (q0 + p) * kOctThreads)), s3);
    }
#pragma unroll
    for (int n = 0; n < 3; ++n) {
      const int p = 3 * n;
      dd_line_deriv_t(dd_mul(S[p], ldg2(nx + (q0 + p) * nc)), dd_mul(S[p + 1], ldg2(nx + (q0 + p + 1) * nc)),
                      dd_mul(S[p + 2], ldg2(nx + (q0 + p + 2) * nc)), R[p], R[p + 1], R[p + 2]);
    }
#pragma unroll
    for (int n = 0; n < 3; ++n)
      dd_line_deriv_t(dd_mul(S[n], ldg2(ny + (q0 + n) * nc)), dd_mul(S[n + 3], ldg2(ny + (q0 + n + 3) * nc)),
                      dd_mul(S[n + 6], ldg2(ny + (q0 + n + 6) * nc)), R[n], R[n + 3], R[n + 6]);
#pragma unroll
    for (int p = 0; p < 9; ++p) st2(sU + (q0 + p) * kOctThreads, dd_norm(R[p]));
  }
#pragma unroll 1
  for (int p = 0; p < 9; ++p) {
    dd f[3], V[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      f[c] = dd_mul(ld2(sV + (p + 9 * c) * kOctThreads), ldg2(nz + (p + 9 * c) * nc));
      V[c] = ld2(sU + (p + 9 * c) * kOctThreads);
    }
    dd_line_combine_t(f[0], f[1], f[2], V[0], V[1], V[2]);
#pragma unroll
    for (int c = 0; c < 3; ++c) st2(sU + (p + 9 * c) * kOctThreads, V[c]);
  }
  if (!active) return;
  double* __restrict__ dst = A.dst + rhs * A.ld;
  const bool far = far_scale(bias);
#pragma unroll 1
  for (int c = 0; c < 3; ++c) {
    dd R[9];
    int32_t id[9];
#pragma unroll
    for (int p = 0; p < 9; ++p) {
      id[p] = __ldg(map + (9 * c + p) * og.ncp);
      R[p] = ld2(sU + (9 * c + p) * kOctThreads);
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      dd_line_values_t(R[a], R[a + 3], R[a + 6]);
      R[a] = dd_norm(R[a]);
      R[a + 3] = dd_norm(R[a + 3]);
      R[a + 6] = dd_norm(R[a + 6]);
    }
#pragma unroll
    for (int b = 0; b < 3; ++b) dd_line_values_t(R[3 * b], R[3 * b + 1], R[3 * b + 2]);
    if (far) {
#pragma unroll
      for (int p = 0; p < 9; ++p) st2(sU + (9 * c + p) * kOctThreads, R[p]);
      continue;
    }
    uint32_t hanging = 0;
#pragma unroll
    for (int p = 0; p < 9; ++p) {
      const double v = join(R[p], bias);
      if (id[p] >= 0) {
        if (!(og.dflag && __ldg(og.dflag + id[p]))) atomicAdd(dst + id[p], v);
      } else {
        hanging |= 1u << p;
        *reinterpret_cast<double*>(sU + (9 * c + p) * kOctThreads) = v;
      }
    }
    for (; hanging; hanging &= hanging - 1) {
      const int p = __ffs(hanging) - 1;
      const double v = *reinterpret_cast<double*>(sU + (9 * c + p) * kOctThreads);
      const int r = -1 - __ldg(map + (9 * c + p) * og.ncp);
      for (int e = __ldg(og.rowptr + r); e < __ldg(og.rowptr + r + 1); ++e) {
        const int32_t m = __ldg(og.cols + e);
        if (!(og.dflag && __ldg(og.dflag + m))) atomicAdd(dst + m, __ldg(og.w64 + e) * v);
      }
    }
  }
  if (bad || far) {   // a NaN into every row of the cell; the test side of a warp with such a scale
#pragma unroll 1
    for (int l = 0; l < 27; ++l) {
      const double v = bad ? __hiloint2double(0x7FF80000, 0) : join_far(ld2(sU + l * kOctThreads), bias);
      const int32_t id = __ldg(map + l * og.ncp);
      if (id >= 0) {
        if (!(og.dflag && __ldg(og.dflag + id))) atomicAdd(dst + id, v);
        continue;
      }
      const int r = -1 - id;
      for (int e = __ldg(og.rowptr + r); e < __ldg(og.rowptr + r + 1); ++e) {
        const int32_t m = __ldg(og.cols + e);
        if (!(og.dflag && __ldg(og.dflag + m))) atomicAdd(dst + m, __ldg(og.w64 + e) * v);
      }
    }
  }
}

}  // namespace

mf_status launch_reinit_df_octree(mf_ctx* ctx, const mf_dofmap* m, const double* src, double* dst, int nrhs,
                                  int64_t ld, const float2* n, double eps, double mass) {
  if (m->uniform || m->degree != 2) return fail(MF_EINVAL, "the double-float octree kernel takes octree Q2 maps");
  MF_CUDA_TRY(upload_tables_here());
  const OctGeom og = oct_geom(m);
  const Tables tb = make_tables();
  DfOctArgs a{};
  a.ld = ld;
  a.n = n;
  a.ncells = m->n_cells;
  const double h0 = m->mesh->h0;
  auto pair = [](double v) {
    const float hi = float(v);
    return make_float2(hi, float(v - double(hi)));
  };
  for (int q = 0; q < 27; ++q) {
    a.we[q] = pair(tb.W3[q] * eps * h0 * (5.0 / 3.0));
    a.wm[q] = pair(tb.W3[q] * mass * h0 * h0 * h0);
  }
  const int64_t nblk = (m->n_cells + kOctThreads - 1) / kOctThreads;
  const int most = int(std::min<int64_t>(nrhs, INT32_MAX / nblk));   // right-hand sides one launch can number
  static bool attrs = false;
  if (!attrs) {
    MF_CUDA_TRY(cudaFuncSetAttribute(k_reinit_df_octree, cudaFuncAttributeMaxDynamicSharedMemorySize, kOctSmem));
    attrs = true;
  }
  for (int r = 0; r < nrhs; r += most) {
    a.nrhs = std::min(most, nrhs - r);
    a.src = src + r * ld;
    a.dst = dst + r * ld;
    k_reinit_df_octree<<<unsigned(nblk * a.nrhs), kOctThreads, kOctSmem, ctx->stream>>>(a, og);
    ctx->launches++;
    MF_CUDA_TRY(cudaGetLastError());
  }
  return MF_OK;
}

}  // namespace mf
