// fp32 apply of the scalar Q2 operators on uniform meshes (Helmholtz, heat, heat with convection and
// its transpose), coefficients tabulated per Gauss point.
//
// A warp owns a column of 8 x 4 cells in x and y (one cell per lane) and marches up it in z.  The nodes
// of a cell's top plane are the bottom nodes of the next one, so each layer loads and interpolates two
// planes of nodes instead of three, and on the test side the top plane is carried on, in registers,
// before its x and y transposes: each layer transposes, folds and scatters two planes.  Faces shared
// inside the warp are folded by shuffles, and a node is added to memory once per warp.
//
// The coefficient tables are stored per tile of 8 x 4 x 1 cells as [q][lane], weights and powers of h
// folded in: a warp reads 128 consecutive bytes per Gauss point at constant offsets from one address,
// also on boxes whose extents are not multiples of the tile (lanes without a cell hold zeros).  The loads of
// a layer run one layer ahead by cp.async.
//
// Bound: instruction issue (71 % of the slots while an SM is busy).  1010 warp instructions per layer of 32
// cells against 2108 of the one-thread-per-cell kernel: the difference form of the contractions (lines.cuh),
// the shared planes, and one address per table instead of 27.  125 x 97 x 111 heat apply 109 -> 75.5 us
// (8 of them the zeroing of the output), 96^3 61 -> 39 us.
#include <algorithm>

#include <cuda_pipeline.h>

#include "lines.cuh"
#include "ops.h"

namespace mf {

MF_DEFINE_TABLE_UPLOAD

UniformGeom uniform_geom(const mf_dofmap* m);

namespace {

// one warp per block: the marches end at different times, and a block's resources are free as soon as its
// warp ends (125 x 97 x 111 heat apply, four layers per march: 77.7 us with four warps per block, 75.5 so)
constexpr int kTileThreads = 32;
constexpr int kTileBlocks = 16;   // resident blocks per SM: 128 registers; 20 blocks at 96 registers spill (102 us)
// with convection 12 blocks of 168 registers, so that the loads of the 81 coefficients run ahead of their use
// (64^3 transpose apply: 63 us with 16 blocks, 37.0 with 12, 37.8 with 10)
constexpr int kConvBlocks = 12;

struct TileArgs {
  const float* src;
  float* dst;
  int64_t ld;        // distance between right-hand sides, one per blockIdx.y
  const float* c;    // [tile][27][32] (5/3) w_q h c_q
  const float* b;    // convection: [tile][81][32] w_q h^2 rho_cp beta_d / (2 delta)
  const float* m;    // QM: [tile][27][32] w_q h^3 m_q
  float wm[4];       // m h^3 times the weight of a point with 0..3 middle coordinates
  int ntx, nty, march;
};

template <bool CONV, bool TR, bool QM>
__global__ void __launch_bounds__(kTileThreads, CONV ? kConvBlocks : kTileBlocks) k_scalar_f32_march(const __grid_constant__ TileArgs A, UniformGeom ug) {
  const int lane = threadIdx.x & 31, xl = lane & 7, yl = lane >> 3;
  const int wid = blockIdx.x * (kTileThreads / 32) + (threadIdx.x >> 5);
  const int ncol = A.ntx * A.nty, col = wid % ncol, k0 = (wid / ncol) * A.march, k1 = min(k0 + A.march, ug.nz);
  if (k0 >= k1) return;
  const int i = (col % A.ntx) * 8 + xl, j = (col / A.ntx) * 4 + yl;
  const bool active = i < ug.nx && j < ug.ny;
  const int64_t base = active ? 2 * int64_t(i) + ug.sx * (2 * int64_t(j)) : 0;
  // nodes of a plane z = const: those read as 0 (Dirichlet faces; all of a lane without a cell) and
  // those that another lane adds to memory
  const uint32_t f = ug.dir_faces;
  const uint32_t side = active ? (((f & 1u) && i == 0) ? 0x049u : 0u) | (((f & 2u) && i == ug.nx - 1) ? 0x124u : 0u) |
                                     (((f & 4u) && j == 0) ? 0x007u : 0u) | (((f & 8u) && j == ug.ny - 1) ? 0x1C0u : 0u)
                               : 0x1FFu;
  const uint32_t folded = (xl ? 0x049u : 0u) | (yl ? 0x007u : 0u);
  auto plane_mask = [&](int zc) {
    return ((f & 16u) && zc == 0) || ((f & 32u) && zc == 2 * ug.nz) ? 0x1FFu : side;
  };
  const float* __restrict__ s = A.src + int64_t(blockIdx.y) * A.ld + base;
  float* __restrict__ d = A.dst + int64_t(blockIdx.y) * A.ld + base;
  // The loads of a layer run one layer ahead, by cp.async: the 18 new nodes into the lane's own slots, the
  // tile's coefficients into one of two buffers of the warp.
  __shared__ __align__(16) float sNode[kTileThreads / 32][18][32];
  __shared__ __align__(16) float sCoef[kTileThreads / 32][2][27 * 32];
  float* const sN = &sNode[threadIdx.x >> 5][0][lane];
  float* const sC = &sCoef[threadIdx.x >> 5][0][0];
  auto fetch = [&](int k) {
    const float* __restrict__ p = s + ug.sy * (2 * k + 1);
#pragma unroll
    for (int l = 0; l < 18; ++l)
      __pipeline_memcpy_async(sN + 32 * l, p + (l % 3) + ug.sx * ((l / 3) % 3) + (l < 9 ? 0 : ug.sy), 4);
    const float* __restrict__ c = A.c + (int64_t(k) * ncol + col) * (27 * 32);
    float* const o = sC + (k & 1) * (27 * 32);
#pragma unroll
    for (int n = 0; n < 7; ++n)
      if (n < 6 || lane < 24) __pipeline_memcpy_async(o + 4 * (lane + 32 * n), c + 4 * (lane + 32 * n), 16);
    if (CONV) {   // the convection coefficients into L2 (10 KB per tile; 23 x 31 x 17 cells: 13.8 us without, 10.5 with)
      const char* const pb = reinterpret_cast<const char*>(A.b + (int64_t(k) * ncol + col) * (81 * 32)) + 128 * lane;
#pragma unroll
      for (int n = 0; n < 3; ++n)
        if (n < 2 || lane < 17) asm volatile("prefetch.global.L2 [%0];" ::"l"(pb + 4096 * n));
    }
    __pipeline_commit();
  };
  // one plane of nodes (raw values in P): Dirichlet rows return the input and read as 0, then the
  // interpolation to the Gauss points in x and y
  auto enter_plane = [&](int zc, float* P) {
    const uint32_t off = plane_mask(zc);
    if (off) {
#pragma unroll
      for (int l = 0; l < 9; ++l)
        if ((off >> l) & 1u) {
          if (active) d[ug.sy * zc + (l % 3) + ug.sx * (l / 3)] = P[l];
          P[l] = 0.f;
        }
    }
#pragma unroll
    for (int b = 0; b < 3; ++b) line_values(P[3 * b], P[3 * b + 1], P[3 * b + 2]);
#pragma unroll
    for (int a = 0; a < 3; ++a) line_values(P[a], P[a + 3], P[a + 6]);
  };
  // one plane of the test side to its nodes: transposes, folding, scatter
  auto store_plane = [&](int zc, float* R) {
#pragma unroll
    for (int a = 0; a < 3; ++a) line_values_t(R[a], R[a + 3], R[a + 6]);
#pragma unroll
    for (int b = 0; b < 3; ++b) line_values_t(R[3 * b], R[3 * b + 1], R[3 * b + 2]);
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const float w = __shfl_down_sync(0xffffffffu, R[3 * b], 1);
      if (xl < 7) R[3 * b + 2] += w;
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float w = __shfl_down_sync(0xffffffffu, (a == 0 && xl > 0) ? 0.f : R[a], 8);
      if (yl < 3) R[a + 6] += w;
    }
    const uint32_t skip = plane_mask(zc) | folded;
    float* __restrict__ p = d + ug.sy * zc;
#pragma unroll
    for (int l = 0; l < 9; ++l)
      if (!((skip >> l) & 1u)) atomicAdd(p + (l % 3) + ug.sx * (l / 3), R[l]);
  };
  float B[9], Rc[9];
  fetch(k0);
#pragma unroll
  for (int l = 0; l < 9; ++l) B[l] = __ldg(s + ug.sy * (2 * k0) + (l % 3) + ug.sx * (l / 3));
  enter_plane(2 * k0, B);
#pragma unroll
  for (int l = 0; l < 9; ++l) Rc[l] = 0.f;
#pragma unroll 1
  for (int k = k0; k < k1; ++k) {
    const int64_t tile = int64_t(k) * ncol + col;
    const float* const tc = sC + (k & 1) * (27 * 32) + lane;
    const float* __restrict__ tb = A.b + tile * (81 * 32) + lane;
    const float* __restrict__ tm = A.m + tile * (27 * 32) + lane;
    float U[27], R[27];
    __pipeline_wait_prior(0);
    __syncwarp();
#pragma unroll
    for (int l = 0; l < 18; ++l) U[9 + l] = sN[32 * l];
    if (k + 1 < k1) fetch(k + 1);
    enter_plane(2 * k + 1, U + 9);
    enter_plane(2 * k + 2, U + 18);
#pragma unroll
    for (int p = 0; p < 9; ++p) {
      U[p] = B[p];
      B[p] = U[18 + p];
      line_values(U[p], U[9 + p], U[18 + p]);
    }
#pragma unroll
    for (int q = 0; q < 27; ++q) {
      const int mid = (q % 3 == 1) + ((q / 3) % 3 == 1) + (q / 9 == 1);
      R[q] = (QM ? __ldg(tm + 32 * q) : A.wm[mid]) * U[q];
    }
#pragma unroll
    for (int dir = 0; dir < 2; ++dir)
#pragma unroll
      for (int n = 0; n < 9; ++n) {
        const int st = dir ? 3 : 1, p0 = dir ? (n % 3) + 9 * (n / 3) : 3 * n, p1 = p0 + st, p2 = p1 + st;
        float g0, g1, g2;
        line_deriv(U[p0], U[p1], U[p2], g0, g1, g2);
        float f0 = tc[32 * p0] * g0, f1 = tc[32 * p1] * g1, f2 = tc[32 * p2] * g2;
        if (CONV) {
          const float b0 = __ldg(tb + 32 * (27 * dir + p0)), b1 = __ldg(tb + 32 * (27 * dir + p1)),
                      b2 = __ldg(tb + 32 * (27 * dir + p2));
          if (TR) {
            f0 += b0 * U[p0];
            f1 += b1 * U[p1];
            f2 += b2 * U[p2];
          } else {
            R[p0] += b0 * g0;
            R[p1] += b1 * g1;
            R[p2] += b2 * g2;
          }
        }
        line_deriv_t(f0, f1, f2, R[p0], R[p1], R[p2]);
      }
#pragma unroll
    for (int p = 0; p < 9; ++p) {
      float g0, g1, g2;
      line_deriv(U[p], U[p + 9], U[p + 18], g0, g1, g2);
      float f0 = tc[32 * p] * g0, f1 = tc[32 * (p + 9)] * g1, f2 = tc[32 * (p + 18)] * g2;
      if (CONV) {
        const float b0 = __ldg(tb + 32 * (54 + p)), b1 = __ldg(tb + 32 * (63 + p)), b2 = __ldg(tb + 32 * (72 + p));
        if (TR) {
          f0 += b0 * U[p];
          f1 += b1 * U[p + 9];
          f2 += b2 * U[p + 18];
        } else {
          R[p] += b0 * g0;
          R[p + 9] += b1 * g1;
          R[p + 18] += b2 * g2;
        }
      }
      line_combine_t(f0, f1, f2, R[p], R[p + 9], R[p + 18]);
      R[p] += Rc[p];
      Rc[p] = R[p + 18];
    }
    store_plane(2 * k, R);
    store_plane(2 * k + 1, R + 9);
  }
  store_plane(2 * k1, Rc);
}

// [rows][27][ncells] table -> [tile][27 rows][32] times s (and w_q); lanes without a cell 0
template <bool WEIGHTED>
__global__ void k_tile_table(const double* __restrict__ c, int rows, double s, float* __restrict__ out, int ntx, int nty,
                             UniformGeom ug) {
  const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  const int64_t nc = int64_t(ug.nx) * ug.ny * ug.nz;
  if (t >= int64_t(ntx) * nty * ug.nz * 32) return;
  const int lane = int(t & 31);
  const int64_t tile = t >> 5;
  const int col = int(tile % (ntx * nty)), k = int(tile / (ntx * nty));
  const int i = (col % ntx) * 8 + (lane & 7), j = (col / ntx) * 4 + (lane >> 3);
  const bool active = i < ug.nx && j < ug.ny;
  const int64_t cell = i + int64_t(ug.nx) * (j + int64_t(ug.ny) * k);
  for (int r = 0; r < 27 * rows; ++r)
    out[(tile * (27 * rows) + r) * 32 + lane] = active ? float(c[r * nc + cell] * (WEIGHTED ? cW364[r % 27] * s : s)) : 0.f;
}

int64_t tile_count(const UniformGeom& ug) { return int64_t((ug.nx + 7) / 8) * ((ug.ny + 3) / 4) * ug.nz; }

}  // namespace

int64_t tile_table_floats(const mf_dofmap* m, int rows) { return tile_count(uniform_geom(m)) * 27 * rows * 32; }

// which: 0 diffusion coefficient, 1 rho_cp beta (three components), 2 value coefficient
mf_status launch_tile_table(mf_ctx* ctx, const mf_dofmap* m, int which, const double* c, float* out) {
  MF_CUDA_TRY(upload_tables_here());
  const UniformGeom ug = uniform_geom(m);
  const double h = ug.h, s = which == 0 ? h * (5.0 / 3.0) : (which == 1 ? h * h * kLineDerivScale : h * h * h);
  const int64_t n = tile_count(ug) * 32;
  k_tile_table<true><<<unsigned((n + 255) / 256), 256, 0, ctx->stream>>>(c, which == 1 ? 3 : 1, s, out, (ug.nx + 7) / 8,
                                                                         (ug.ny + 3) / 4, ug);
  ctx->launches++;
  MF_CUDA_TRY(cudaGetLastError());
  return MF_OK;
}

mf_status launch_tile_table_plain(mf_ctx* ctx, const mf_dofmap* m, const double* c, int rows, double scale, float* out) {
  const UniformGeom ug = uniform_geom(m);
  const int64_t n = tile_count(ug) * 32;
  k_tile_table<false><<<unsigned((n + 255) / 256), 256, 0, ctx->stream>>>(c, rows, scale, out, (ug.nx + 7) / 8,
                                                                          (ug.ny + 3) / 4, ug);
  ctx->launches++;
  MF_CUDA_TRY(cudaGetLastError());
  return MF_OK;
}

// Whether this kernel, rather than the one-thread-per-cell kernel, serves an apply to nrhs right-hand sides.  Lanes
// without a cell cost it more (their nodes are masked plane by plane, and both kernels' warps are 8 x 4 columns):
// up to 9 of 16 lanes with a cell the general kernel is the faster one on large meshes (us, marching / general: 3 x
// 200 x 40 cells 9.2 / 6.6, 9 x 100 x 100 17.4 / 12.2, 1 x 1 x 4000 17.8 / 9.4; at three in four lanes they meet).
// But it takes the right-hand sides one after another and leaves Dirichlet rows to a launch of their own (2 us):
// below three tiles per SM (six with Dirichlet rows) it serves only what has neither (eight right-hand sides, 17^3
// cells: 9.7 / 16.7; one, 4^3 cells with Dirichlet rows: 6.2 / 8.2, without: 6.2 / 6.2; 2 x 40 x 40 with: 5.1 / 5.8).
bool march_serves(const mf_ctx* ctx, const mf_dofmap* m, int nrhs) {
  if (!m->uniform) return false;
  const UniformGeom ug = uniform_geom(m);
  const int64_t ncol = int64_t((ug.nx + 7) / 8) * ((ug.ny + 3) / 4);
  if (16 * int64_t(ug.nx) * ug.ny > 9 * 32 * ncol) return true;
  const bool rows = !m->dirichlet_list.empty();
  return ncol * ug.nz < (rows ? 6 : 3) * int64_t(ctx->sm_count) && (nrhs > 1 || rows);
}

mf_status launch_scalar_f32_uniform(mf_ctx* ctx, const mf_dofmap* m, const float* src, float* dst, int nrhs, int64_t ld,
                                    const float* c, const float* b, const float* qm, double mass, bool transpose) {
  const UniformGeom ug = uniform_geom(m);
  TileArgs a{};
  a.src = src;
  a.dst = dst;
  a.ld = ld;
  a.c = c;
  a.b = b;
  a.m = qm;
  a.ntx = (ug.nx + 7) / 8;
  a.nty = (ug.ny + 3) / 4;
  for (int mid = 0; mid < 4; ++mid) {
    double w = mass * ug.h * ug.h * ug.h;
    for (int t = 0; t < 3; ++t) w *= t < mid ? 8.0 / 18.0 : 5.0 / 18.0;
    a.wm[mid] = float(w);
  }
  const int64_t ncol = int64_t(a.ntx) * a.nty;
  const int64_t resident = int64_t(ctx->sm_count) * (b ? kConvBlocks : kTileBlocks) * (kTileThreads / 32);
  // Layers per march: long marches share more planes (125 x 97 x 111: 93, 81, 77, 75.5, 76, 78, 84 us with 1,
  // 2, 3, 4, 6, 8, 12 layers), but the warps must go round the resident ones about twice, or the slowest SM
  // finishes alone (one round of 19 layers: 86 us; 96^3 is fastest at 6 layers, 40^3 at 1).
  a.march = int(std::min<int64_t>(6, std::max<int64_t>(1, 4 * ncol * ug.nz * nrhs / (7 * resident))));
  const int64_t warps = ncol * ((ug.nz + a.march - 1) / a.march);
  const dim3 grid(unsigned((warps + kTileThreads / 32 - 1) / (kTileThreads / 32)), unsigned(nrhs));
  if (!b && qm)
    k_scalar_f32_march<false, false, true><<<grid, kTileThreads, 0, ctx->stream>>>(a, ug);
  else if (!b)
    k_scalar_f32_march<false, false, false><<<grid, kTileThreads, 0, ctx->stream>>>(a, ug);
  else if (transpose && qm)
    k_scalar_f32_march<true, true, true><<<grid, kTileThreads, 0, ctx->stream>>>(a, ug);
  else if (transpose)
    k_scalar_f32_march<true, true, false><<<grid, kTileThreads, 0, ctx->stream>>>(a, ug);
  else if (qm)
    k_scalar_f32_march<true, false, true><<<grid, kTileThreads, 0, ctx->stream>>>(a, ug);
  else
    k_scalar_f32_march<true, false, false><<<grid, kTileThreads, 0, ctx->stream>>>(a, ug);
  ctx->launches++;
  MF_CUDA_TRY(cudaGetLastError());
  return MF_OK;
}

}  // namespace mf
