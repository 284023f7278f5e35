// fp32 apply of the conservative level-set reinitialisation operator, (1/dtau) M + eps N_n, to several
// right-hand sides at once on adaptively refined (octree) meshes with hanging-node constraints.
//
// The vectors are interleaved by W = 2, 4 or 8 right-hand sides (one pass in, one pass out), and W
// neighbouring lanes work on one leaf, one right-hand side each.  So a node's values of all right-hand
// sides are one run of 4 W bytes: a gather or an atomic add of a warp touches 32 / W runs instead of 32
// scattered words per right-hand side, and the leaf's node numbers and normals are read once for all of
// them (16-byte loads that the W lanes share).  Dirichlet entries become 0 on the way in and return the
// input on the way out, and the pass out writes every entry, so the output needs no zeroing.  A leaf's two
// tables arrive in shared memory by 16-byte cp.async copies.
//
// Bound: latency of the gathers at 16 warps per SM (ncu: 46 % of the issue slots, long-scoreboard stalls).
// Eight right-hand sides on the base 20 + 3 levels octree (4.8 M DoFs): 1057 us -> 582 us, of it 437 us this
// kernel, 88 us the pass in and 46 us the pass out; L2 atomics fall from 134 M to 31 M sectors and HBM reads
// from 2.0 to 0.8 GB.  Two right-hand sides on a small octree: 109 -> 46 us.
#include <algorithm>

#include <cuda_pipeline.h>

#include "lines.cuh"
#include "ops.h"

namespace mf {



OctGeom oct_geom(const mf_dofmap* m);

namespace {

constexpr int kRhsThreads = 128;
constexpr int kRhsBlocks = 4;   // per SM; 3 / 5 / 6 blocks: 674 / 731 / 854 us (spills from 5 on) against 582 us

template <int W> struct VecOf;
template <> struct VecOf<2> { using type = float2; };
template <> struct VecOf<4> { using type = float4; };
template <> struct VecOf<8> { using type = float4; };

struct RhsArgs {
  const float* in;      // [n][W]
  float* out;           // [n][W], zero on entry
  const int32_t* map;   // per leaf in processing order: 27 node numbers (hanging: -(1 + row)) and the level
  const float* nrm;     // per leaf in processing order: [3][28] unit normal component d along the lines of direction d
  int64_t nslots;
  float we[4];          // (5/3) eps h0 times the weight of a point with 0..3 middle coordinates
  float wm[4];          // m h0^3 times the weight
};

template <int W>
__global__ void __launch_bounds__(256) k_interleave(const float* __restrict__ src, int64_t ld, int nr, int64_t n,
                                                    const uint8_t* __restrict__ dflag, float* __restrict__ in,
                                                    float* __restrict__ out) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const bool off = dflag && dflag[i];
  float v[W];
#pragma unroll
  for (int r = 0; r < W; ++r) v[r] = (r < nr && !off) ? __ldcs(src + r * ld + i) : 0.f;
  using V = typename VecOf<W>::type;
  constexpr int nv = W * 4 / int(sizeof(V));
  const V z{};
#pragma unroll
  for (int k = 0; k < nv; ++k) {
    V t;
    memcpy(&t, v + k * (W / nv), sizeof(V));
    reinterpret_cast<V*>(in)[i * nv + k] = t;
    reinterpret_cast<V*>(out)[i * nv + k] = z;
  }
}

template <int W>
__global__ void __launch_bounds__(256) k_deinterleave(const float* __restrict__ out, const float* __restrict__ src, int64_t ld,
                                                      int nr, int64_t n, const uint8_t* __restrict__ dflag,
                                                      float* __restrict__ dst) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= n) return;
  using V = typename VecOf<W>::type;
  constexpr int nv = W * 4 / int(sizeof(V));
  float v[W];
#pragma unroll
  for (int k = 0; k < nv; ++k) {
    const V t = __ldcs(reinterpret_cast<const V*>(out) + i * nv + k);
    memcpy(v + k * (W / nv), &t, sizeof(V));
  }
  const bool off = dflag && dflag[i];
#pragma unroll
  for (int r = 0; r < W; ++r)
    if (r < nr) __stcs(dst + r * ld + i, off ? __ldg(src + r * ld + i) : v[r]);
}

template <int W>
__global__ void __launch_bounds__(kRhsThreads, kRhsBlocks) k_reinit_octree_rhs(const __grid_constant__ RhsArgs A, OctGeom og) {
  constexpr int L = 32 / W;   // leaves per warp
  __shared__ __align__(16) int32_t sMap[kRhsThreads / 32][L * 28];
  __shared__ __align__(16) float sNrm[kRhsThreads / 32][L * 84];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, r = lane % W, leaf = lane / W;
  const int64_t slot0 = (int64_t(blockIdx.x) * (kRhsThreads / 32) + warp) * L;
  if (slot0 >= A.nslots) return;
  // the warp's leaves are neighbours in both tables: one run of 16-byte copies each
  const int leaves = int(min(int64_t(L), A.nslots - slot0));
  for (int k = lane; k < leaves * 7; k += 32)
    __pipeline_memcpy_async(&sMap[warp][4 * k], A.map + slot0 * 28 + 4 * k, 16);
  __pipeline_commit();
  for (int k = lane; k < leaves * 21; k += 32)
    __pipeline_memcpy_async(&sNrm[warp][4 * k], A.nrm + slot0 * 84 + 4 * k, 16);
  __pipeline_commit();
  __pipeline_wait_prior(1);
  __syncwarp();
  const bool active = leaf < leaves;
  const int32_t* const id = &sMap[warp][(active ? leaf : 0) * 28];
  const float4* const nv = reinterpret_cast<const float4*>(&sNrm[warp][(active ? leaf : 0) * 84]);
  const float* __restrict__ in = A.in + r;
  float U[27];
  bool hanging = false;
#pragma unroll
  for (int k = 0; k < 7; ++k) {
    const int4 v = reinterpret_cast<const int4*>(id)[k];
    const int32_t n[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int l = 4 * k + j;
      if (l >= 27) continue;
      U[l] = __ldg(in + int64_t(max(n[j], 0)) * W);
      hanging |= n[j] < 0;
    }
  }
  if (hanging) {
#pragma unroll
    for (int l = 0; l < 27; ++l) {
      if (id[l] >= 0) continue;
      const int row = -1 - id[l];
      float v = 0.f;
      for (int e = __ldg(og.rowptr + row); e < __ldg(og.rowptr + row + 1); ++e)
        v += __ldg(og.w32 + e) * __ldg(in + int64_t(__ldg(og.cols + e)) * W);
      U[l] = v;
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
  __pipeline_wait_prior(0);
  __syncwarp();
  // four lines share three 16-byte words of a normal component (stored line by line)
  auto lines4 = [&](int d, int c, float* N) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      if (4 * k + 12 * c >= 28) continue;
      const float4 v = nv[7 * d + 3 * c + k];
      N[4 * k] = v.x;
      N[4 * k + 1] = v.y;
      N[4 * k + 2] = v.z;
      N[4 * k + 3] = v.w;
    }
  };
  auto line = [](int d, int n, int& p0, int& p1, int& p2) {
    p0 = d == 0 ? 3 * n : (d == 1 ? (n % 3) + 9 * (n / 3) : n);
    const int st = d == 0 ? 1 : (d == 1 ? 3 : 9);
    p1 = p0 + st;
    p2 = p1 + st;
  };
  // s = w eps h (n . grad u) (h = h0 2^-level), then the value term over U
  float S[27];
#pragma unroll
  for (int d = 0; d < 3; ++d)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      float N[12];
      lines4(d, c, N);
#pragma unroll
      for (int n = 4 * c; n < 4 * c + 4 && n < 9; ++n) {
        int p0, p1, p2;
        line(d, n, p0, p1, p2);
        float g0, g1, g2;
        line_deriv(U[p0], U[p1], U[p2], g0, g1, g2);
        const float* const m = N + 3 * (n - 4 * c);
        S[p0] = (d ? S[p0] : 0.f) + m[0] * g0;
        S[p1] = (d ? S[p1] : 0.f) + m[1] * g1;
        S[p2] = (d ? S[p2] : 0.f) + m[2] * g2;
      }
    }
  const int lev = id[27];
  const float s1 = __uint_as_float(unsigned(127 - lev) << 23), s3 = __uint_as_float(unsigned(127 - 3 * lev) << 23);
  float we[4], wm[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    we[m] = A.we[m] * s1;
    wm[m] = A.wm[m] * s3;
  }
#pragma unroll
  for (int q = 0; q < 27; ++q) {
    const int mid = (q % 3 == 1) + ((q / 3) % 3 == 1) + (q / 9 == 1);
    S[q] *= we[mid];
    U[q] *= wm[mid];
  }
  asm volatile("" ::: "memory");   // read the normals again rather than hold 81 of them in registers
#pragma unroll
  for (int d = 0; d < 3; ++d)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      float N[12];
      lines4(d, c, N);
#pragma unroll
      for (int n = 4 * c; n < 4 * c + 4 && n < 9; ++n) {
        int p0, p1, p2;
        line(d, n, p0, p1, p2);
        const float* const m = N + 3 * (n - 4 * c);
        const float f0 = S[p0] * m[0], f1 = S[p1] * m[1], f2 = S[p2] * m[2];
        if (d < 2) line_deriv_t(f0, f1, f2, U[p0], U[p1], U[p2]);
        else line_combine_t(f0, f1, f2, U[p0], U[p1], U[p2]);
      }
    }
#pragma unroll
  for (int n = 0; n < 9; ++n) {
    const int p = (n % 3) + 9 * (n / 3);
    line_values_t(U[p], U[p + 3], U[p + 6]);
  }
#pragma unroll
  for (int n = 0; n < 9; ++n) line_values_t(U[3 * n], U[3 * n + 1], U[3 * n + 2]);
  if (!active) return;
  asm volatile("" ::: "memory");
  float* __restrict__ out = A.out + r;
#pragma unroll
  for (int k = 0; k < 7; ++k) {
    const int4 v = reinterpret_cast<const int4*>(id)[k];
    const int32_t n[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int l = 4 * k + j;
      if (l < 27 && n[j] >= 0) atomicAdd(out + int64_t(n[j]) * W, U[l]);
    }
  }
  if (hanging) {
#pragma unroll
    for (int l = 0; l < 27; ++l) {
      if (id[l] >= 0) continue;
      const int row = -1 - id[l];
      for (int e = __ldg(og.rowptr + row); e < __ldg(og.rowptr + row + 1); ++e)
        atomicAdd(out + int64_t(__ldg(og.cols + e)) * W, __ldg(og.w32 + e) * U[l]);
    }
  }
}

// node numbers and level, and the fp64 normal table rounded, per leaf in processing order
__global__ void k_rhs_tables(OctGeom og, const double* __restrict__ qvec, int64_t ncp, int32_t* __restrict__ map,
                             float* __restrict__ nrm) {
  const int64_t slot = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (slot >= og.ncells) return;
  const int64_t cell = og.order[slot];
  for (int l = 0; l < 27; ++l) map[slot * 28 + l] = og.cmap[l * og.ncp + cell];
  map[slot * 28 + 27] = og.level[cell];
  for (int d = 0; d < 3; ++d) {
    for (int n = 0; n < 27; ++n) {   // line n / 3 of direction d, point n % 3
      const int line = n / 3, q = d == 0 ? n : (d == 1 ? (line % 3) + 9 * (line / 3) + 3 * (n % 3) : line + 9 * (n % 3));
      nrm[slot * 84 + 28 * d + n] = float(qvec[(27 * d + q) * ncp + cell]);
    }
    nrm[slot * 84 + 28 * d + 27] = 0.f;
  }
}

}  // namespace

mf_status launch_octree_rhs_tables(mf_ctx* ctx, const mf_dofmap* m, const double* qvec64, int32_t* map, float* nrm) {
  const OctGeom og = oct_geom(m);
  k_rhs_tables<<<unsigned((m->n_cells + 127) / 128), 128, 0, ctx->stream>>>(og, qvec64, m->n_cells, map, nrm);
  ctx->launches++;
  MF_CUDA_TRY(cudaGetLastError());
  return MF_OK;
}

template <int W>
static mf_status launch_w(mf_ctx* ctx, const mf_dofmap* m, const float* src, float* dst, int nr, int64_t ld, RhsArgs a,
                          float* work) {
  const OctGeom og = oct_geom(m);
  const int64_t n = m->n_dofs;
  float *in = work, *out = work + n * W;
  a.in = in;
  a.out = out;
  const unsigned gb = unsigned((n + 255) / 256);
  k_interleave<W><<<gb, 256, 0, ctx->stream>>>(src, ld, nr, n, og.dflag, in, out);
  ctx->launches++;
  MF_CUDA_TRY(cudaGetLastError());
  const int64_t warps = (a.nslots + 32 / W - 1) / (32 / W);
  k_reinit_octree_rhs<W><<<unsigned((warps + kRhsThreads / 32 - 1) / (kRhsThreads / 32)), kRhsThreads, 0, ctx->stream>>>(a, og);
  ctx->launches++;
  MF_CUDA_TRY(cudaGetLastError());
  k_deinterleave<W><<<gb, 256, 0, ctx->stream>>>(out, src, ld, nr, n, og.dflag, dst);
  ctx->launches++;
  MF_CUDA_TRY(cudaGetLastError());
  return MF_OK;
}

mf_status launch_reinit_f32_octree_rhs(mf_ctx* ctx, const mf_dofmap* m, const float* src, float* dst, int nr, int64_t ld,
                                       const int32_t* map, const float* nrm, double eps, double mass, float* work) {
  if (nr < 2 || nr > 8) return fail(MF_EINVAL, "two to eight right-hand sides");
  RhsArgs a{};
  a.map = map;
  a.nrm = nrm;
  a.nslots = m->n_cells;
  const double h0 = m->mesh->h0;
  for (int mid = 0; mid < 4; ++mid) {
    double w = 1.0;
    for (int t = 0; t < 3; ++t) w *= t < mid ? 8.0 / 18.0 : 5.0 / 18.0;
    a.we[mid] = float(w * eps * h0 * (5.0 / 3.0));
    a.wm[mid] = float(w * mass * h0 * h0 * h0);
  }
  if (nr == 2) return launch_w<2>(ctx, m, src, dst, nr, ld, a, work);
  if (nr <= 4) return launch_w<4>(ctx, m, src, dst, nr, ld, a, work);
  return launch_w<8>(ctx, m, src, dst, nr, ld, a, work);
}

}  // namespace mf
