// Device-side pieces of the cooperative solver kernels (internal): a bounded barrier over the grid and the
// reduction of a value over it.
#pragma once

#include "reduce.cuh"

namespace mf {
namespace {

// Barrier over the whole (co-resident) grid; bar = {arrived, generation, timed out}.  The release of the
// arrival and the acquire of the new generation order the blocks' global memory accesses.
__device__ __forceinline__ unsigned load_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ bool grid_barrier(unsigned* bar, unsigned nblocks) {
  __shared__ bool ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    ok = true;
    const unsigned gen = load_acquire(bar + 1);
    unsigned before;
    asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(before) : "l"(bar) : "memory");
    if (before == nblocks - 1) {
      bar[0] = 0u;
      asm volatile("red.add.release.gpu.global.u32 [%0], 1;" ::"l"(bar + 1) : "memory");
    } else {
      unsigned long long t0 = 0;
      for (unsigned spins = 0; load_acquire(bar + 1) == gen; ++spins) {
        if ((spins & 1023u) != 1023u) continue;
        unsigned long long t;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        if (!t0) t0 = t;
        if (t - t0 > 1000000000ull || load_acquire(bar + 2)) {
          atomicExch(bar + 2, 1u);
          ok = false;
          break;
        }
      }
    }
  }
  __syncthreads();
  return ok;
}

// Block sums of N values, value k to part[k * stride + blockIdx.x].  Pairs of floats down to one value per
// warp: fp64 adds cost 16 cycles of the SM per warp instruction (a tree of them over the block's 32 warps
// took longer than the step's stencil).
template <int N> __device__ __forceinline__ void block_partials(Dot2f (&v)[N], double (*sh)[32], double* part, int64_t stride) {
#pragma unroll
  for (int k = 0; k < N; ++k) v[k].warp_sum();
  if ((threadIdx.x & 31) == 0)
#pragma unroll
    for (int k = 0; k < N; ++k) sh[k][threadIdx.x >> 5] = v[k].value();
  __syncthreads();
  if (threadIdx.x < 32 * N) {
    const int k = threadIdx.x >> 5;
    double s = sh[k][threadIdx.x & 31];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) part[k * stride + blockIdx.x] = s;
  }
}

}  // namespace
}  // namespace mf
