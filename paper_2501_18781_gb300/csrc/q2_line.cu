// Q2 Helmholtz and heat applies on small uniform meshes, and the whole Jacobi-CG solve on them in one launch.
//
// Where one thread per cell would leave most SMs idle, nine threads work on a cell: each takes one line of
// three values per direction, in difference form (lines.cuh), and the lines of the next direction are read
// from shared memory.  The test side is kept without Gauss weights, which the transposes carry in their
// constants, so a point costs one product per flux.  88 fp64 operations per thread instead of 123 with the
// dense 3 x 3 contractions; the fp64 pipe (16 cycles of an SM per warp instruction) bounds it together with
// the latency of the seven phases.  16^3 cells in fp64, with the launch that zeroes the result: 18.4 -> 14.3 us.
#include <algorithm>

#include "grid_barrier.cuh"
#include "lines.cuh"
#include "ops.h"

namespace mf {

UniformGeom uniform_geom(const mf_dofmap* m);

namespace {

// cells of a block of 9 * CPB (rounded up to warps) threads
template <int CPB> constexpr int line_threads() { return (9 * CPB + 31) / 32 * 32; }

template <typename T> struct LineArgs {
  const T* coef;    // [27][ncells] scalar coefficient at the Gauss points
  T wm;             // value coefficient m h^2 3/5 (the common factor h 5/3 is in kx)
  T k[4], kx[4];    // constants of the weighted transposes; kx with the factor h 5/3
  int64_t ncells;
};

template <typename T> LineArgs<T> line_args(const mf_dofmap* m, const T* coef, double mass) {
  LineArgs<T> a{};
  const double h = m->mesh->h0, w0 = 5.0 / 18.0, w1 = 8.0 / 18.0, k[4] = {0.3 * w0, w1, 0.4 * w0, kLineDelta * w0};
  a.coef = coef;
  a.wm = T(mass * h * h * 0.6);
  for (int n = 0; n < 4; ++n) {
    a.k[n] = T(k[n]);
    a.kx[n] = T(k[n] * h * (5.0 / 3.0));
  }
  a.ncells = m->n_cells;
  return a;
}

// A cell's first node, the Dirichlet nodes of the z line through local node (i, j) and of the x line through
// (y, z) = (i, j), as bits.  (DoF indices fit 32 bits, so cell numbers do.)
struct LineCell {
  int64_t base;
  uint32_t zdir, xdir;
};
__device__ __forceinline__ LineCell line_cell(const UniformGeom& g, int cell, int i, int j) {
  LineCell c;
  const int row = cell / g.nx, cx = cell - row * g.nx, cz = row / g.ny, cy = row - cz * g.ny;
  c.base = 2 * cx + g.sx * (2 * cy) + g.sy * (2 * cz);
  c.zdir = c.xdir = 0u;
  const uint32_t f = g.dir_faces;
  if (f) {
    const bool side = ((f & 1u) && cx == 0 && i == 0) || ((f & 2u) && cx == g.nx - 1 && i == 2) ||
                      ((f & 4u) && cy == 0 && j == 0) || ((f & 8u) && cy == g.ny - 1 && j == 2);
    c.zdir = side ? 7u : 0u;
    if ((f & 16u) && cz == 0) c.zdir |= 1u;
    if ((f & 32u) && cz == g.nz - 1) c.zdir |= 4u;
    if (((f & 4u) && cy == 0 && i == 0) || ((f & 8u) && cy == g.ny - 1 && i == 2) || ((f & 16u) && cz == 0 && j == 0) ||
        ((f & 32u) && cz == g.nz - 1 && j == 2))
      c.xdir = 7u;
    else
      c.xdir = (((f & 1u) && cx == 0) ? 1u : 0u) | (((f & 2u) && cx == g.nx - 1) ? 4u : 0u);
  }
  return c;
}

// The coefficients of a thread's x, y and z lines of Gauss points.
template <typename T> struct LineCoef {
  T x[3], y[3], z[3];
};
template <typename T>
__device__ __forceinline__ LineCoef<T> line_coef(const LineArgs<T>& A, int cell, bool on, int i, int j) {
  LineCoef<T> c;
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    c.x[q] = on ? __ldg(A.coef + (q + 3 * i + 9 * j) * A.ncells + cell) : T(0);
    c.y[q] = on ? __ldg(A.coef + (i + 3 * q + 9 * j) * A.ncells + cell) : T(0);
    c.z[q] = on ? __ldg(A.coef + (i + 3 * j + 9 * q) * A.ncells + cell) : T(0);
  }
  return c;
}

// One cell per nine threads (slot = the cell's place in the block, (i, j) the thread's in the cell; on = a
// cell is there).  load(z): the value of node (i, j, z), 0 at Dirichlet nodes; add(x, v): adds v to node
// (x, i, j).  Every thread of the block calls this.
template <typename T, typename Load, typename Add>
__device__ __forceinline__ void line_apply(const LineArgs<T>& A, const LineCoef<T>& C, bool on, bool in_block, int i, int j,
                                           T* u, T* v, Load&& load, Add&& add) {
  T a0 = T(0), a1 = T(0), a2 = T(0);
  if (on) {
    a0 = load(0);
    a1 = load(1);
    a2 = load(2);
  }
  line_values(a0, a1, a2);
  T* const uz = u + i + 3 * j;          // z line through (i, j): stride 9
  T* const uy = u + i + 9 * j;          // y line through x = i, z = j: stride 3
  T* const ux = u + 3 * i + 9 * j;      // x line through y = i, z = j: stride 1
  T* const vz = v + i + 3 * j;
  T* const vy = v + i + 9 * j;
  T* const vx = v + 3 * i + 9 * j;
  if (in_block) {
    uz[0] = a0;
    uz[9] = a1;
    uz[18] = a2;
  }
  __syncthreads();
  if (in_block) {
    T b0 = uy[0], b2 = uy[6];
    line_values(b0, uy[3], b2);
    uy[0] = b0;
    uy[6] = b2;
  }
  __syncthreads();
  if (in_block) {
    T b0 = ux[0], b1 = ux[1], b2 = ux[2], g0, g1, g2;
    line_values(b0, b1, b2);
    ux[0] = b0;
    ux[2] = b2;
    T r0 = A.wm * b0, r1 = A.wm * b1, r2 = A.wm * b2;
    line_deriv(b0, b1, b2, g0, g1, g2);
    line_deriv_tw(C.x[0] * g0, C.x[1] * g1, C.x[2] * g2, r0, r1, r2);
    vx[0] = r0;
    vx[1] = r1;
    vx[2] = r2;
  }
  __syncthreads();
  if (in_block) {
    T g0, g1, g2, r0 = vy[0], r1 = vy[3], r2 = vy[6];
    line_deriv(uy[0], uy[3], uy[6], g0, g1, g2);
    line_deriv_tw(C.y[0] * g0, C.y[1] * g1, C.y[2] * g2, r0, r1, r2);
    vy[0] = r0;
    vy[3] = r1;
    vy[6] = r2;
  }
  __syncthreads();
  if (in_block) {
    T g0, g1, g2, r0 = vz[0], r1 = vz[9], r2 = vz[18];
    line_deriv(uz[0], uz[9], uz[18], g0, g1, g2);
    line_combine_tw(A.k, C.z[0] * g0, C.z[1] * g1, C.z[2] * g2, r0, r1, r2);
    vz[0] = r0;
    vz[9] = r1;
    vz[18] = r2;
  }
  __syncthreads();
  if (in_block) {
    T r0 = vy[0], r1 = vy[3], r2 = vy[6];
    line_values_tw(A.k, r0, r1, r2);
    vy[0] = r0;
    vy[3] = r1;
    vy[6] = r2;
  }
  __syncthreads();
  if (on) {
    T r0 = vx[0], r1 = vx[1], r2 = vx[2];
    line_values_tw(A.kx, r0, r1, r2);
    add(0, r0);
    add(1, r1);
    add(2, r2);
  }
}

constexpr int kCells = 14;   // per block of 128 threads

template <typename T>
__global__ void __launch_bounds__(line_threads<kCells>()) k_q2_line(const __grid_constant__ LineArgs<T> A, UniformGeom g,
                                                                    const T* __restrict__ src, T* __restrict__ dst) {
  __shared__ T su[kCells][27], sv[kCells][27];
  const int slot = threadIdx.x / 9, r = threadIdx.x % 9, i = r % 3, j = r / 3;
  const bool in_block = slot < kCells;
  const int cell = int(blockIdx.x) * kCells + slot;
  const bool on = in_block && cell < A.ncells;
  const LineCell c = line_cell(g, on ? cell : 0, i, j);
  const T* const s = src + c.base + i + g.sx * j;
  T* const d = dst + c.base + g.sx * i + g.sy * j;
  line_apply<T>(
      A, line_coef(A, cell, on, i, j), on, in_block, i, j, su[in_block ? slot : 0], sv[in_block ? slot : 0],
      [&](int z) { return ((c.zdir >> z) & 1u) ? T(0) : __ldg(s + g.sy * z); },
      [&](int x, T v) {
        if (!((c.xdir >> x) & 1u)) atomicAdd(d + x, v);
      });
}

// Jacobi-CG with the line apply: one cooperative grid, two barriers per step.  The direction p = z + beta
// p_old is formed where it is read (by the cells that gather it and by the row that stores it, into the
// other of two buffers), and p . A p is summed over the cells, so a step is
//   cells: Ap += A_cell p, p . A_cell p          barrier
//   rows:  p, x, r, z, r . r, r . z, Ap = 0      barrier
// 16^3 cells, 255 steps: 10.7 -> 4.6 ms; each of the five kernels of a step had paid a launch and a drained grid.
constexpr int kCgCells = 28, kCgThreads = kRedThreads;   // 252 of 256 threads work on cells

struct LineCgArgs {
  LineArgs<double> line;
  double *x, *r, *z, *p[2], *Ap;   // p[0] holds the first direction
  const double* dinv;
  const int32_t* dir;              // Dirichlet rows: A p = p there
  int64_t n, ndir;
  double tol2;
  int maxit;
  bool stop_indefinite;            // stop at p . A p <= 0
  double* S;                       // scalars of cg_init_scalars: r.r and r.z of the start
  double* steps;
  double* part;                    // partial sums: [grid] (p . A p), then [2][2][grid] (r.r, r.z by parity)
  unsigned* bar;
};

// SINGLE: every thread has one cell for the whole solve, whose place and coefficients stay in registers
template <bool SINGLE>
__global__ void __launch_bounds__(kCgThreads, 1) k_q2_line_cg(const __grid_constant__ LineCgArgs A, UniformGeom g) {
  __shared__ double su[kCgCells][27], sv[kCgCells][27], sp[kCgCells][27];
  __shared__ double tot[2], sbeta, salpha;
  __shared__ bool done;
  const unsigned G = gridDim.x;
  const int slot = threadIdx.x / 9, t9 = threadIdx.x % 9, i = t9 % 3, j = t9 / 3;
  const bool in_block = slot < kCgCells;
  const int64_t t0 = int64_t(blockIdx.x) * kCgThreads + threadIdx.x, st = int64_t(G) * kCgThreads;
  const int ncells = int(A.line.ncells), cell0 = int(blockIdx.x) * kCgCells + slot;
  const bool on0 = in_block && cell0 < ncells;
  const LineCell first = line_cell(g, on0 ? cell0 : 0, i, j);
  const LineCoef<double> coef0 = line_coef(A.line, cell0, on0, i, j);
  const double rr0 = A.S[S_RR];
  double rz = A.S[S_RZ], rr = rr0;   // thread 0
  if (threadIdx.x == 0) {
    sbeta = 0.0;
    done = false;
  }
  __syncthreads();
  int k = 0;
  for (; k < A.maxit; ++k) {
    // p = z + beta p_old, except the first direction, which is there already
    const double beta = sbeta;
    const double* const po = A.p[(k + 1) & 1];
    double* const pn = A.p[k & 1];
    auto direction = [&](int64_t row) { return k ? A.z[row] + beta * po[row] : pn[row]; };
    double acc = 0.0;
    for (int c0 = int(blockIdx.x) * kCgCells; c0 < ncells; c0 += int(G) * kCgCells) {
      const int cell = c0 + slot;
      const bool on = in_block && cell < ncells;
      const LineCell c = SINGLE ? first : line_cell(g, on ? cell : 0, i, j);
      const int64_t row = c.base + i + g.sx * j;
      const int64_t out = c.base + g.sx * i + g.sy * j;
      double* const keep = sp[in_block ? slot : 0];
      line_apply<double>(
          A.line, SINGLE ? coef0 : line_coef(A.line, cell, on, i, j), on, in_block, i, j, su[in_block ? slot : 0],
          sv[in_block ? slot : 0],
          [&](int z) {
            const double v = ((c.zdir >> z) & 1u) ? 0.0 : direction(row + g.sy * z);
            keep[i + 3 * j + 9 * z] = v;
            return v;
          },
          [&](int x, double v) {
            if (!((c.xdir >> x) & 1u)) {
              acc = fma(keep[x + 3 * i + 9 * j], v, acc);
              atomicAdd(A.Ap + out + x, v);
            }
          });
      __syncthreads();   // the next cells overwrite the shared lines
    }
    for (int64_t q = t0; q < A.ndir; q += st) {
      const int64_t row = A.dir[q];
      const double v = direction(row);
      A.Ap[row] = v;
      acc = fma(v, v, acc);
    }
    {
      const double v1[1] = {acc};
      block_sums<1>(v1, [&](int, double s) { A.part[blockIdx.x] = s; });
    }
    if (!grid_barrier(A.bar, G, 2 * k + 1)) return;
    grid_totals(A.part, 1, G, tot);
    if (threadIdx.x == 0) salpha = tot[0] != 0.0 ? rz / tot[0] : 0.0;
    __syncthreads();
    const double alpha = salpha;
    double v2[2] = {0.0, 0.0};
    for (int64_t q = t0; q < A.n; q += st) {
      const double p = direction(q);
      if (k) pn[q] = p;
      A.x[q] += alpha * p;
      const double r = A.r[q] - alpha * A.Ap[q];
      A.Ap[q] = 0.0;
      A.r[q] = r;
      v2[0] = fma(r, r, v2[0]);
      const double z = A.dinv[q] * r;
      A.z[q] = z;
      v2[1] = fma(r, z, v2[1]);
    }
    double* const pr = A.part + (1 + 2 * (k & 1)) * int64_t(G);
    block_sums<2>(v2, [&](int w, double s) { pr[w * int64_t(G) + blockIdx.x] = s; });
    const double pap = tot[0];
    if (!grid_barrier(A.bar, G, 2 * k + 2)) return;
    grid_totals(pr, 2, G, tot);
    if (threadIdx.x == 0) {
      rr = tot[0];
      sbeta = rz != 0.0 ? tot[1] / rz : 0.0;
      rz = tot[1];
      done = rr <= A.tol2 * rr0 || !isfinite(rr) || (A.stop_indefinite && !(pap > 0.0));
    }
    __syncthreads();
    if (done) {
      ++k;
      break;
    }
  }
  if (t0 == 0) {
    A.S[S_RR] = rr;
    A.S[S_RZ] = rz;
    A.S[S_ACTIVE] = done ? 0.0 : 1.0;
    A.steps[0] = double(k);
  }
}

}  // namespace

template <typename T>
mf_status launch_q2_line(mf_ctx* ctx, const mf_dofmap* m, const T* src, T* dst, const T* coef, double mass) {
  if (m->degree != 2 || !m->uniform) return fail(MF_EINVAL, "the line kernel takes uniform Q2 maps");
  const int64_t nb = (m->n_cells + kCells - 1) / kCells;
  k_q2_line<T><<<unsigned(nb), line_threads<kCells>(), 0, ctx->stream>>>(line_args<T>(m, coef, mass), uniform_geom(m), src,
                                                                         dst);
  ctx->launches++;
  MF_CUDA_TRY(cudaGetLastError());
  return MF_OK;
}
template mf_status launch_q2_line<double>(mf_ctx*, const mf_dofmap*, const double*, double*, const double*, double);
template mf_status launch_q2_line<float>(mf_ctx*, const mf_dofmap*, const float*, float*, const float*, double);

// Five rounds of the grid: with more cells per group of threads the eight warps per SM that the barriers
// allow cost more than the launches of the separate kernels.  One launch against those kernels replayed as
// a graph, ms per Helmholtz solve: 20^3 cells 8.5 / 11.9, 28^3 27.2 / 27.4, 32^3 39.5 / 38.3, 36^3 58.7 / 54.6,
// 44^3 130 / 108.
int64_t q2_line_cg_cells(const mf_ctx* ctx) { return int64_t(5) * kCgCells * ctx->sm_count; }

mf_status launch_q2_line_cg(mf_ctx* ctx, const mf_dofmap* m, const double* coef, double mass, const double* dinv, double* x,
                            double* r, double* z, double* p, double* p2, double* Ap, double tol, int maxit,
                            bool stop_indefinite, double* S, double* steps) {
  if (!dinv) return fail(MF_EINVAL, "the one-launch CG is Jacobi-preconditioned");
  LineCgArgs a{};
  a.line = line_args<double>(m, coef, mass);
  a.x = x;
  a.r = r;
  a.z = z;
  a.p[0] = p;
  a.p[1] = p2;
  a.Ap = Ap;
  a.dinv = dinv;
  a.dir = m->d_dir_list.as<int32_t>();
  a.n = m->n_dofs;
  a.ndir = int64_t(m->dirichlet_list.size());
  a.tol2 = tol * tol;
  a.maxit = maxit;
  a.stop_indefinite = stop_indefinite;
  a.S = S;
  a.steps = steps;
  a.part = ctx->scratch.as<double>();
  a.bar = ctx->counters.as<unsigned>() + kBarrierCounter;
  UniformGeom g = uniform_geom(m);
  const int64_t want = std::max<int64_t>((m->n_cells + kCgCells - 1) / kCgCells, 1);
  const unsigned grid = unsigned(std::min<int64_t>(want, ctx->sm_count));
  MF_CUDA_TRY(cudaMemsetAsync(a.bar, 0, sizeof(unsigned), ctx->stream));
  MF_CUDA_TRY(cudaMemsetAsync(Ap, 0, sizeof(double) * a.n, ctx->stream));
  void* args[] = {&a, &g};
  const void* const k = want <= grid ? reinterpret_cast<const void*>(k_q2_line_cg<true>)
                                     : reinterpret_cast<const void*>(k_q2_line_cg<false>);
  MF_CUDA_TRY(cudaLaunchCooperativeKernel(k, dim3(grid), dim3(kCgThreads), args, 0, ctx->stream));
  ctx->launches++;
  return MF_OK;
}

}  // namespace mf
