// Device-side pieces of the deterministic reductions (internal): block sums, compensated fp32
// dot products, and the finishing step that the last block of a reduction runs.
#pragma once

#include "vec.cuh"

namespace mf {
namespace {

// Sums over a block of kRedThreads threads.  GB300's fp64 pipe takes 16 cycles of an SM per warp
// instruction, so a shuffle tree over every warp (five adds each) costs more than the data of a small
// vector: the threads' values go to shared memory, and one warp per value adds eight of them per lane
// before its shuffles (13 fp64 adds instead of 43; a 257 k element fp32 dot 14.7 -> 8.8 us with the grid cut
// to the vector and 16-byte loads, the fp32 multidot of 5 vectors of 1.6 M 19.9 -> 12.1 us).  N values share the barrier; value k is summed by warp
// k in a fixed order and given to put(k, sum) by its first lane.  Every thread of the block calls this.
__device__ __forceinline__ double (*red_area1())[kRedThreads] {   // one area for every instance in a kernel
  __shared__ double sh[1][kRedThreads];
  return sh;
}
__device__ __forceinline__ double (*red_area())[kRedThreads] {
  __shared__ double sh[kRedThreads / 32][kRedThreads];
  return sh;
}
template <int N, typename F> __device__ __forceinline__ void block_sums(const double (&v)[N], F&& put) {
  static_assert(N <= kRedThreads / 32, "one warp per value");
  double(*sh)[kRedThreads] = N == 1 ? red_area1() : red_area();
#pragma unroll
  for (int k = 0; k < N; ++k) sh[k][threadIdx.x] = v[k];
  __syncthreads();
  if (threadIdx.x < 32 * N) {
    const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double s = sh[k][lane];
#pragma unroll
    for (int j = 1; j < kRedThreads / 32; ++j) s += sh[k][lane + 32 * j];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) put(k, s);
  }
  __syncthreads();
}
__device__ __forceinline__ double block_sum(double v) {
  double s = 0.0;
  const double a[1] = {v};
  block_sums<1>(a, [&](int, double t) { s = t; });
  return s;  // valid in thread 0
}

// fp32 data: GB300's fp64 pipe (1/64 of the fp32 rate) cannot keep up with HBM if every
// element is converted and accumulated in fp64 (a conversion and an fp64 FMA per 4-byte
// element).  Within a thread, fp32 products and sums are therefore carried as unevaluated
// pairs of floats: the product error by an FMA (a*b = p + e exactly) and the sum error by
// Knuth's two-sum, i.e. the compensated dot product of Ogita, Rump and Oishi ("Accurate sum
// and dot product", SIAM J. Sci. Comput. 26, 2005), whose result is as accurate as a dot
// product evaluated in twice the working precision.  Partials leave the thread as
// double(s) + double(c) and are reduced in fp64.
struct Dot2f {
  float s = 0.0f, c = 0.0f;
  __device__ __forceinline__ void add(float a, float b) {
    const float p = a * b;
    const float e = fmaf(a, b, -p);
    const float t = s + p;
    const float z = t - s;
    c += ((s - (t - z)) + (p - z)) + e;
    s = t;
  }
  // the sum of both pairs
  __device__ __forceinline__ void merge(float os, float oc) {
    const float t = s + os;
    const float z = t - s;
    c += oc + ((s - (t - z)) + (os - z));
    s = t;
  }
  __device__ __forceinline__ void merge(const Dot2f& o) { merge(o.s, o.c); }
  // lane 0: the sum over the warp (pairs of floats: no fp64 instruction)
  __device__ __forceinline__ void warp_sum() {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
      merge(__shfl_down_sync(0xffffffffu, s, o), __shfl_down_sync(0xffffffffu, c, o));
  }
  __device__ __forceinline__ double value() const { return double(s) + double(c); }
};

// The same for pairs: summed over each warp as pairs, then the warps' sums in fp64.
template <int N, typename F> __device__ __forceinline__ void block_sums(Dot2f (&v)[N], F&& put) {
  static_assert(N <= kRedThreads / 32, "one warp per value");
  __shared__ double sh[N][kRedThreads / 32];
#pragma unroll
  for (int k = 0; k < N; ++k) v[k].warp_sum();
  if ((threadIdx.x & 31) == 0)
#pragma unroll
    for (int k = 0; k < N; ++k) sh[k][threadIdx.x >> 5] = v[k].value();
  __syncthreads();
  if (threadIdx.x < 32 * N) {
    const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double s = lane < kRedThreads / 32 ? sh[k][lane] : 0.0;
#pragma unroll
    for (int o = kRedThreads / 64; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) put(k, s);
  }
  __syncthreads();
}

// What the sum of a row of g partials feeds (row r; mode 0: out[r] = sum; 1: pAp and alpha;
// 2: rr, rz (second row), beta; 3: rz and beta; 4: rr and rz; 5: rr).  count: one arrival
// counter per row (zero between launches); NULL when a separate k_finish launch does the sum.
struct Finish {
  double* out;
  int mode;
  double* S;
  unsigned* count;
};

// Sums row r of the partials in a fixed order (so results are reproducible bit for bit) and
// applies the mode.  The loads go to L2: in the fused form other blocks of the same launch
// wrote the partials.
__device__ void finish_row(const double* part, int g, int r, const Finish& f) {
  const double* pr = part + int64_t(r) * 2 * g;
  double s = 0.0;
  for (int i = threadIdx.x; i < g; i += blockDim.x) s += __ldcg(pr + i);
  s = block_sum(s);
  double s2 = 0.0;
  if (f.mode == 2 || f.mode == 4) {
    for (int i = threadIdx.x; i < g; i += blockDim.x) s2 += __ldcg(pr + g + i);
    s2 = block_sum(s2);
  }
  if (threadIdx.x == 0) {
    double* Sr = f.S ? f.S + r * S_NSCAL : nullptr;
    if (f.mode == 0) f.out[r] = s;
    else if (f.mode == 1) {
      Sr[S_PAP] = s;
      Sr[S_ALPHA] = (Sr[S_ACTIVE] != 0.0 && s != 0.0) ? Sr[S_RZ] / s : 0.0;
    } else if (f.mode == 2 || f.mode == 3) {
      const double rz = f.mode == 2 ? s2 : s;
      if (f.mode == 2) Sr[S_RR] = s;
      Sr[S_RZN] = rz;
      Sr[S_BETA] = (Sr[S_ACTIVE] != 0.0 && Sr[S_RZ] != 0.0) ? rz / Sr[S_RZ] : 0.0;
      Sr[S_RZ] = rz;
    } else if (f.mode == 4) {
      Sr[S_RR] = s;
      Sr[S_RZ] = s2;
    } else if (f.mode == 5) {
      Sr[S_RR] = s;
    }
  }
}

// Called by every thread after thread 0 stored the block's partials of row blockIdx.y: the last
// block of the row to arrive sums the row (finish_row) and resets the counter for the next launch.
__device__ __forceinline__ void finish_if_last(const double* part, const Finish& f) {
  if (!f.count) return;
  __shared__ unsigned last;
  __threadfence();  // this block's partials are visible device-wide before it is counted
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(f.count + blockIdx.y, 1u) == gridDim.x - 1 ? 1u : 0u;
  __syncthreads();
  if (!last) return;
  __threadfence();
  finish_row(part, gridDim.x, blockIdx.y, f);
  if (threadIdx.x == 0) f.count[blockIdx.y] = 0u;
}

}  // namespace
}  // namespace mf
