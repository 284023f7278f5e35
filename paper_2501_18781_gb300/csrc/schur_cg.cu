// The Schur complement solve of the Oseen block-triangular preconditioner in one launch: Jacobi-
// preconditioned CG on the assembled 125-point pressure stencil, fp32 vectors, fp64 scalars.
//
// Run as separate kernels, a step was four launches on vectors that fit in L2 (40^3 cells: 69 k rows, 33 us
// per step in the launch list of a melt-pool step), and the steps after convergence still launched.  Here
// one cooperative grid holds the whole iteration, one block of 1024 threads per SM, with two grid barriers
// per step: the stencil is applied to z, which the barrier after the vector update has just made visible, and
// s = S~ p follows from s = S~ z + beta s, so the direction needs no barrier of its own.  p . s is summed as
// it stands: formed from z . S~ z as in the single-reduction CG it loses digits, which moved the
// outer iteration's count.  Every block adds the per-block partial sums in the same order, so all blocks
// hold the same scalars and the result does not depend on timing.  A barrier gives up after one second
// of %globaltimer and sets a flag.
// Bound: latency of the barriers and of the two dependent passes, 16 us per step at 40^3 (325 us per
// call; 303 with the block sums in fewer bits and two partial sums per row and thread); the 40^3 step's Schur
// solves went from 30 to 9.1 ms.  The fp64 scalars are one thread's work:
// divisions in all 32 warps took 8 us per step, the fp64 sums over all of them 5 us.
#include <cuda_fp16.h>

#include <cstring>

#include "grid_barrier.cuh"
#include "ops.h"

namespace mf {
namespace {

constexpr int kThreads = 1024;

struct SchurArgs {
  const __half* S;      // scaled fp16 tiled layout of stencil_at
  const float* scale;
  const float* dinv;
  const double* b;     // right-hand side
  float *x, *r, *z, *p, *s;
  double* zout;        // -x in fp64
  double* part;        // partial sums: [2][grid] (r.r, r.z), then [grid] (p.s)
  double* steps;       // step counter over all solves
  unsigned* bar;
  double tol2;
  int nx, ny, nz, maxit;
};

// Words K0 .. K0 + K - 1 (8 entries each) of stencil row i times v, in five partial sums (error of a row of 125
// against 64 bits, of the sum of magnitudes: 1.2e-8 rms, with two 1.7e-8; eight cost 1 % of a 64^3 step); w: the
// row's first word (words 32 apart, the scaled fp16 tiled layout of stencil_at).  Entries toward nodes outside the
// grid are 0, and their loads are clamped into it; v changes during the launch: plain loads.
template <int K0, int K>
__device__ __forceinline__ float stencil_words(const SchurArgs& A, const uint4* w, const float* v, int i) {
  const int px = A.nx + 1, pxy = px * (A.ny + 1);
  const int ix = i % px, iy = (i / px) % (A.ny + 1), iz = i / pxy;
  int ox[5], oy[5], oz[5];
#pragma unroll
  for (int d = 0; d < 5; ++d) {
    ox[d] = min(max(ix + d - 2, 0), A.nx);
    oy[d] = px * min(max(iy + d - 2, 0), A.ny);
    oz[d] = pxy * min(max(iz + d - 2, 0), A.nz);
  }
  float s[5] = {0.f, 0.f, 0.f, 0.f, 0.f};   // by x offset
#pragma unroll
  for (int c = 0; c < K / 4; ++c) {
    uint4 q[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) q[k] = w[32 * (4 * c + k)];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint32_t pair[4] = {q[k].x, q[k].y, q[k].z, q[k].w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        __half2 h2;
        memcpy(&h2, &pair[j], 4);
        const float2 f = __half22float2(h2);
        const int o = 8 * (K0 + 4 * c + k) + 2 * j;
        if (o < 125) s[o % 5] = fmaf(f.x, v[ox[o % 5] + oy[(o / 5) % 5] + oz[o / 25]], s[o % 5]);
        if (o + 1 < 125)
          s[(o + 1) % 5] = fmaf(f.y, v[ox[(o + 1) % 5] + oy[((o + 1) / 5) % 5] + oz[(o + 1) / 25]], s[(o + 1) % 5]);
      }
    }
  }
  return ((s[0] + s[1]) + (s[2] + s[3])) + s[4];
}

// PARTS threads share a row (warp by warp, so that every thread's entries are known at compile time).  With two
// or four a block has one run of rows (start()), whose coefficients stay in shared memory for the whole solve.
template <int PARTS>
__global__ void __launch_bounds__(kThreads, 1) k_schur_cg(const SchurArgs A) {
  extern __shared__ uint4 coef[];
  __shared__ double tot[2];
  __shared__ float2 sh[2][kThreads / PARTS];
  __shared__ float coef_s;   // beta, then alpha
  __shared__ bool done;
  __shared__ float ssum[PARTS > 1 ? PARTS : 1][kThreads / PARTS];
  constexpr int kRows = kThreads / PARTS, kWords = 16 / PARTS;   // rows of a block at a time, words of a thread
  constexpr bool CACHED = PARTS > 1;
  const int np = (A.nx + 1) * (A.ny + 1) * (A.nz + 1);
  const int part = threadIdx.x / kRows, local = threadIdx.x % kRows;
  const unsigned G = gridDim.x;
  // rows of this block: consecutive runs of kRows
  const int first = blockIdx.x * kRows, step = int(G) * kRows;
  const int t0 = first + int(threadIdx.x);
  const bool own = threadIdx.x < kRows;   // the thread that keeps the row's vectors
  auto words = [&](int i) { return reinterpret_cast<const uint4*>(A.S + stencil_at(0, i)); };
  if (CACHED) {
    const uint4* const g = words(first);   // kRows is a multiple of 32: the rows are consecutive tiles
    const int n = (min(kRows, np - first) + 31) / 32 * 512;
    for (int q = threadIdx.x; q < n; q += kThreads) coef[q] = __ldg(g + q);
    __syncthreads();
  }
  // p = z + beta p, s = S~ z + beta s (so s = S~ p) on the block's rows, and the thread's share of p . s
  auto apply = [&](int k, float be, Dot2f& aps) {
    for (int i0 = first; i0 < np; i0 += step) {
      const int i = i0 + local;
      float w = 0.f;
      if (i < np) {
        const uint4* const q = (CACHED ? coef + (local >> 5) * 512 + (local & 31) : words(i)) + 32 * kWords * part;
        if (PARTS == 1) w = stencil_words<0, kWords>(A, q, A.z, i);
        else if (part == 0) w = stencil_words<0, kWords>(A, q, A.z, i);
        else if (part == 1) w = stencil_words<kWords % 16, kWords>(A, q, A.z, i);
        else if (part == 2) w = stencil_words<2 * kWords % 16, kWords>(A, q, A.z, i);
        else w = stencil_words<3 * kWords % 16, kWords>(A, q, A.z, i);
      }
      if (PARTS > 1) {
        ssum[part][local] = w;
        __syncthreads();
        if (own) {
          w = ssum[0][local];
#pragma unroll
          for (int j = 1; j < PARTS; ++j) w += ssum[j][local];
        }
      }
      if (own && i < np) {
        w *= A.scale[i];
        const float p = k ? A.z[i] + be * A.p[i] : A.z[i], t = k ? w + be * A.s[i] : w;
        A.p[i] = p;
        A.s[i] = t;
        aps.add(p, t);
      }
      if (PARTS > 1) __syncthreads();
    }
  };
  Dot2f arr, arz;
  if (own)
    for (int i = t0; i < np; i += step) {
      const float r = float(A.b[i]), z = A.dinv[i] * r;
      A.r[i] = r;
      A.z[i] = z;
      A.x[i] = 0.f;
      arr.add(r, r);
      arz.add(r, z);
    }
  double rz = 1.0, stop = 0.0;   // thread 0 of every block: fp64 divisions by one thread, not by 32 warps
  int k = 0;
  for (; k < A.maxit; ++k) {
    const Dot2f v2[2] = {arr, arz};
    block_partials<2, kRows>(v2, sh, A.part, G);
    if (!grid_barrier(A.bar, G, 2 * k + 1)) return;
    grid_totals(A.part, 2, G, tot);
    if (threadIdx.x == 0) {
      if (k == 0) stop = A.tol2 * tot[0];
      done = tot[0] <= stop;   // converged, or a zero right-hand side
      coef_s = float(k ? tot[1] / rz : 0.0);
      rz = tot[1];
    }
    __syncthreads();
    if (done) break;
    Dot2f v1[1];
    apply(k, coef_s, v1[0]);
    block_partials<1, kRows>(v1, sh, A.part + 2 * int64_t(G), G);
    if (!grid_barrier(A.bar, G, 2 * k + 2)) return;
    grid_totals(A.part + 2 * int64_t(G), 1, G, tot);
    if (threadIdx.x == 0) {
      done = !(tot[0] > 0.0);   // a breakdown: x stays as it is
      coef_s = float(rz / tot[0]);
    }
    __syncthreads();
    if (done) break;
    const float al = coef_s;
    arr = Dot2f();
    arz = Dot2f();
    if (own)
      for (int i = t0; i < np; i += step) {
        const float r = A.r[i] - al * A.s[i], z = A.dinv[i] * r;
        A.x[i] += al * A.p[i];
        A.r[i] = r;
        A.z[i] = z;
        arr.add(r, r);
        arz.add(r, z);
      }
  }
  if (own)
    for (int i = t0; i < np; i += step) A.zout[i] = -double(A.x[i]);
  if (blockIdx.x == 0 && threadIdx.x == 0) *A.steps += double(k);
}

// PARTS > 1 only where the grid holds all rows at once
template <int PARTS> cudaError_t start(mf_ctx* ctx, SchurArgs& a, int64_t np) {
  constexpr int rows = kThreads / PARTS;
  const int64_t want = (np + rows - 1) / rows;
  const unsigned grid = unsigned(want < ctx->sm_count ? want : ctx->sm_count);
  const size_t bytes = PARTS > 1 ? size_t(rows) * 256 : 0;   // 128 or 64 KB
  const void* const k = reinterpret_cast<const void*>(k_schur_cg<PARTS>);
  if (bytes) {
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(bytes));
    if (e != cudaSuccess) return e;
  }
  const cudaError_t e = cudaMemsetAsync(a.bar, 0, sizeof(unsigned), ctx->stream);
  if (e != cudaSuccess) return e;
  void* args[] = {&a};
  return cudaLaunchCooperativeKernel(k, dim3(grid), dim3(kThreads), args, bytes, ctx->stream);
}

}  // namespace

// zout = -x and x = S~^-1 b by at most maxit steps from 0, to ||r|| <= sqrt(tol2) ||b||.  work: 4 n_p
// floats (r, z, p, s).
mf_status launch_schur_cg(mf_ctx* ctx, const void* S, const float* scale, const float* dinv, const double* b, float* x,
                          float* work, double* zout, int nx, int ny, int nz, int maxit, double tol2, double* steps) {
  const int64_t np = int64_t(nx + 1) * (ny + 1) * (nz + 1);
  SchurArgs a{};
  a.S = static_cast<const __half*>(S);
  a.scale = scale;
  a.dinv = dinv;
  a.b = b;
  a.x = x;
  a.r = work;
  a.z = work + np;
  a.p = work + 2 * np;
  a.s = work + 3 * np;
  a.zout = zout;
  a.part = ctx->scratch.as<double>();
  a.steps = steps;
  a.bar = ctx->counters.as<unsigned>() + kBarrierCounter;
  a.tol2 = tol2;
  a.nx = nx;
  a.ny = ny;
  a.nz = nz;
  a.maxit = maxit;
  // as many threads per row as the grid has to spare
  const int64_t threads = int64_t(ctx->sm_count) * kThreads;
  MF_CUDA_TRY(4 * np <= threads ? start<4>(ctx, a, np) : (2 * np <= threads ? start<2>(ctx, a, np) : start<1>(ctx, a, np)));
  ctx->launches++;
  return MF_OK;
}

// MF_ETIMEOUT (once) if the barrier of a cooperative launch gave up
mf_status grid_barrier_take_error(mf_ctx* ctx) {
  unsigned timed_out = 0u;
  unsigned* const d = ctx->counters.as<unsigned>() + kBarrierCounter + 1;
  MF_CUDA_TRY(cudaMemcpyAsync(&timed_out, d, sizeof timed_out, cudaMemcpyDeviceToHost, ctx->stream));
  MF_CUDA_TRY(cudaStreamSynchronize(ctx->stream));
  if (!timed_out) return MF_OK;
  MF_CUDA_TRY(cudaMemsetAsync(d, 0, sizeof timed_out, ctx->stream));
  return fail(MF_ETIMEOUT, "a grid barrier of a solver kernel timed out");
}

}  // namespace mf
