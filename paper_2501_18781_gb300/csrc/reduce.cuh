// Device-side pieces of the deterministic reductions (internal): block sums, compensated fp32
// dot products, and the finishing step that the last block of a reduction runs.
#pragma once

#include "vec.cuh"

namespace mf {
namespace {

// Sums over a block of kRedThreads threads, in fp64.  GB300's fp64 pipe takes 16 cycles of an SM per warp
// instruction, so a shuffle tree over every warp (five adds each) costs more than the data of a small
// vector: the threads' values go to shared memory, and one warp per value adds eight of them per lane
// before its shuffles (13 fp64 adds instead of 43).  N values share the barrier; value k is summed by warp
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
  __device__ __forceinline__ double value() const { return double(s) + double(c); }
};

// A sum of pairs, exact beyond fp64: the high parts and then the low parts are added without error, what both
// leave goes to a third float (72 bits).  Adding pairs as pairs loses bits against fp64 (sums of squares of
// 4,096 to 1.6 M elements: 9e-16 of the sum; this way, as with every pair converted, 2e-16), and converting every
// pair costs three fp64 instructions.  A sum past the largest float is an fp64 number: s is then Inf and c, l are
// its bits.
struct Sum3f {
  float s, c, l;
  Sum3f() = default;
  __device__ __forceinline__ explicit Sum3f(const Dot2f& a) : s(a.s), c(a.c), l(0.f) {}
  __device__ __forceinline__ void add(const Dot2f& a) { add(a.s, a.c, 0.f); }
  __device__ __forceinline__ void add(const Sum3f& a) { add(a.s, a.c, a.l); }
  __device__ __forceinline__ void add(float os, float oc, float ol) {
    const float t = s + os, z = t - s, d = (s - (t - z)) + (os - z);
    const float u = c + oc, y = u - c, e = (c - (u - y)) + (oc - y);
    const float v = u + d, x = v - u, f = (u - (v - x)) + (d - x);
    s = t;
    c = v;
    l = (l + ol) + (e + f);
  }
  __device__ __forceinline__ bool in_range() const { return fabsf(s) <= 3.402823466e38f; }
  __device__ __forceinline__ double value() const {
    return in_range() ? double(s) + (double(c) + double(l)) : __hiloint2double(__float_as_int(c), __float_as_int(l));
  }
};
// fp64 sum of the N pairs or triples that load(0 .. N - 1) gives
template <int N, typename L> __device__ __forceinline__ double exact_sum(L&& load) {
  Sum3f t(load(0));
#pragma unroll
  for (int k = 1; k < N; ++k) t.add(load(k));
  if (t.in_range()) return t.value();
  double v = 0.0;
#pragma unroll 1
  for (int k = 0; k < N; ++k) v += load(k).value();
  return v;
}
// a thread's N accumulators in one
template <int N, typename A> __device__ __forceinline__ Sum3f thread_sum(const A (&a)[N]) {
  Sum3f t(a[0]);
#pragma unroll
  for (int k = 1; k < N; ++k) t.add(a[k]);
  if (!t.in_range()) {
    double v = 0.0;
#pragma unroll
    for (int k = 0; k < N; ++k) v += a[k].value();
    t.s = __int_as_float(0x7F800000);
    t.c = __int_as_float(__double2hiint(v));
    t.l = __int_as_float(__double2loint(v));
  }
  return t;
}
// The block sums of pairs or triples: one warp per value adds eight threads' per lane exactly, then in fp64 (10 fp64
// instructions per value).  The areas serve every instance in a kernel.
template <typename P, int ROWS> __device__ __forceinline__ P (*exact_area())[kRedThreads] {
  __shared__ __align__(16) char sh[ROWS * kRedThreads * sizeof(P)];
  return reinterpret_cast<P(*)[kRedThreads]>(sh);
}
template <int N, typename P, typename F> __device__ __forceinline__ void block_sums_exact(const P (&v)[N], F&& put) {
  static_assert(N <= kRedThreads / 32, "one warp per value");
  P(*sh)[kRedThreads] = N <= 2 ? exact_area<P, 2>() : exact_area<P, kRedThreads / 32>();
#pragma unroll
  for (int k = 0; k < N; ++k) sh[k][threadIdx.x] = v[k];
  __syncthreads();
  if (threadIdx.x < 32 * N) {
    const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double s = exact_sum<kRedThreads / 32>([&](int j) { return sh[k][lane + 32 * j]; });
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
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
