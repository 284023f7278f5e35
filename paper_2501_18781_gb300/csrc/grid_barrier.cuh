// Device-side pieces of the cooperative solver kernels (internal): a bounded barrier over the grid and the
// reduction of values over it.
#pragma once

#include "reduce.cuh"

namespace mf {
namespace {

// Barrier over the whole (co-resident) grid; bar = {arrivals, timed out}, the arrivals zeroed before the launch
// and never reset in it, so an arrival needs no answer and the blocks wait for the count itself.  (A last
// block that resets the count and publishes a generation adds a round trip to L2: with that and the sums
// below read one after another, the 16^3 Jacobi-CG took 5.5 ms instead of 4.4, the Schur solve of a 40^3
// step 362 us instead of 303.  Polling every block's sum in place of a count is slower still: 5.7 ms,
// 437 us.)  nth counts the launch's barriers from 1.  The release of the
// arrivals and the acquire of the count order the blocks' global memory accesses.  A block that waits for
// one second of %globaltimer sets the flag and gives up.
__device__ __forceinline__ unsigned load_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ bool grid_barrier(unsigned* bar, unsigned nblocks, unsigned nth) {
  __shared__ bool ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    ok = true;
    const unsigned target = nblocks * nth;
    asm volatile("red.add.release.gpu.global.u32 [%0], 1;" ::"l"(bar) : "memory");
    unsigned long long t0 = 0;
    for (unsigned spins = 0; int(load_acquire(bar) - target) < 0; ++spins) {
      if ((spins & 1023u) != 1023u) continue;
      unsigned long long t;
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
      if (!t0) t0 = t;
      if (t - t0 > 1000000000ull || load_acquire(bar + 1)) {
        atomicExch(bar + 1, 1u);
        ok = false;
        break;
      }
    }
  }
  __syncthreads();
  return ok;
}

// Fixed-order sums of N arrays of the blocks' partial sums, value w to tot[w], the same in every block: one warp
// per array, with the loads of up to 160 blocks in flight together.  Every thread of the block calls this.
__device__ __forceinline__ void grid_totals(const double* part, int n, unsigned nblocks, double* tot) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (w < n) {
    const double* const q = part + w * int64_t(nblocks);
    double v[5], s = 0.0;
#pragma unroll
    for (int j = 0; j < 5; ++j) v[j] = lane + 32u * j < nblocks ? __ldcg(q + lane + 32 * j) : 0.0;
#pragma unroll
    for (int j = 0; j < 5; ++j) s += v[j];
    for (unsigned k = lane + 160; k < nblocks; k += 32) s += __ldcg(q + k);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) tot[w] = s;
  }
  __syncthreads();
}

// Block sums of N values of the first ROWS threads, value k to part[k * stride + blockIdx.x]: one warp per value
// adds ROWS / 32 pairs per lane exactly, then in fp64.  (fp64 adds cost 16 cycles of the SM per warp
// instruction: a tree of them over the block's 32 warps took longer than the step's stencil.)
template <int N, int ROWS>
__device__ __forceinline__ void block_partials(const Dot2f (&v)[N], float2 (*sh)[ROWS], double* part, int64_t stride) {
  if (threadIdx.x < ROWS)
#pragma unroll
    for (int k = 0; k < N; ++k) sh[k][threadIdx.x] = make_float2(v[k].s, v[k].c);
  __syncthreads();
  if (threadIdx.x < 32 * N) {
    const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double s = 0.0;
#pragma unroll 1
    for (int j = lane; j < ROWS; j += 256)
      s += exact_sum<8>([&](int i) {
        const float2 p = sh[k][j + 32 * i];
        Dot2f a;
        a.s = p.x;
        a.c = p.y;
        return a;
      });
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) part[k * stride + blockIdx.x] = s;
  }
}

}  // namespace
}  // namespace mf
