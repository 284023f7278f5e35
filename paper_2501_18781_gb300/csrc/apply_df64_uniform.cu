// Double-float applies on uniform meshes (Section 2.3 coefficients, Appendix B matrix-free evaluation).  First the
// scalar Q2 operators: Helmholtz and the implicit heat step, without or with convection (also transposed, and
// then also with a value coefficient per Gauss point), the conductivity (or a(phi)) tabulated per Gauss point; then
// the Oseen operator, without and with the melt-pool terms.
//
// Vectors stay fp64 in HBM; in the kernel every value is a pair of floats hi + lo (48-bit
// significand) and every operation is an error-free fp32 transformation on the fp32 pipes, which
// GB300 runs at 64 times its fp64 rate (Dekker's product through the FMA residual, Knuth's two-sum;
// Joldes, Muller and Popescu, ACM TOMS 2017, bound these "double-word" algorithms).  Pairs are
// carried unnormalised through each contraction (|lo| a few ulp(hi) at most) and renormalised at its
// end; the error of a sum stays below a few 2^-47 (|a| + |b|), so results agree with the fp64 apply
// to a few 1e-14 of |A||u| componentwise.  Doubles enter and leave the kernel by bit manipulation
// (GB300 converts between fp64 and fp32 only at its fp64 rate), scaled by one power of two per warp so
// that the warp's largest input lies in [1, 2): any fp64 magnitude is kept to 47 bits relative to that
// largest finite input of the warp's 8 x 4 cells; inputs more than 2^126 below it count as zero, and the rows
// of a cell with an Inf or NaN among its inputs get a NaN.
//
// One thread per cell in 8 x 4 x 4 bricks; the cell's values and test side live in the thread's own
// columns of shared memory and every phase is a short rolled loop over them.  No thread of the scalar
// kernel reads another thread's column: no barrier is needed.
#include "df_pairs.cuh"

namespace mf {

MF_DEFINE_TABLE_UPLOAD

UniformGeom uniform_geom(const mf_dofmap* m);

namespace {

struct DfArgs {
  const double* src;
  double* dst;
  int64_t ld;         // distance between right-hand sides, one per blockIdx.y
  const float2* c;    // [27][ncells] pairs of (5/3) w_q h c_q (c: conductivity or a(phi) at Gauss point q)
  const float2* b;    // convection: [3][27][ncells] pairs of w_q h^2 rho_cp beta_d / (2 delta), or NULL
  const float2* m;    // QM: [27][ncells] pairs of w_q h^3 m_q (m_q = rho_cp,q / dt) in place of wm
  int64_t ncells;
  float2 wm[27];      // w_q m h^3 (m: value coefficient)
};

__device__ __forceinline__ dd shfl_down_dd(dd v, int d) {
  return {__shfl_down_sync(0xffffffffu, v.h, d), __shfl_down_sync(0xffffffffu, v.l, d)};
}

// Scatter-add of one slab z = const of 9 nodes per cell of a warp of the 8 x 4 x 4 brick (dst at the
// slab's first node): the faces shared by x and y neighbours inside the warp are folded by shuffles on
// the pairs (all lanes share one scale), then every node is added to memory once per warp as a double (not
// for a far_scale).  Every lane calls this; inactive lanes pass zeros.
__device__ __forceinline__ void scatter_dd_slab(double* __restrict__ dst, int64_t sx, uint32_t dmask, dd* R, bool active,
                                                int bias) {
  const int xl = threadIdx.x & 7, yl = (threadIdx.x >> 3) & 3;
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    dd w = shfl_down_dd(R[3 * b], 1);
    if (xl == 7) w = dd{0.f, 0.f};
    R[3 * b + 2] = dd_add(R[3 * b + 2], w);
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    dd w = shfl_down_dd((a == 0 && xl > 0) ? dd{0.f, 0.f} : R[a], 8);
    if (yl == 3) w = dd{0.f, 0.f};
    R[a + 6] = dd_add(R[a + 6], w);
  }
  if (!active) return;
#pragma unroll
  for (int l = 0; l < 9; ++l) {
    const int a = l % 3, b = l / 3;
    if ((a == 0 && xl > 0) || (b == 0 && yl > 0) || ((dmask >> l) & 1u)) continue;
    atomicAdd(dst + a + sx * b, join(R[l], bias));
  }
}
// What scatter_dd_slab leaves: the test side of a cell of a warp whose scale is far (col, slots STRIDE apart; dst
// at the cell's first node), and a NaN into every row of a cell with an Inf or NaN among its inputs.
template <int STRIDE>
__device__ __forceinline__ void scatter_rare(double* __restrict__ dst, int64_t sx, int64_t sy, uint32_t dmask,
                                             const float2* col, int bias, bool bad) {
#pragma unroll 1
  for (int l = 0; l < 27; ++l) {
    const float2 v = col[l * STRIDE];
    if (!((dmask >> l) & 1u))
      atomicAdd(dst + l % 3 + sx * ((l / 3) % 3) + sy * (l / 9),
                bad ? __hiloint2double(0x7FF80000, 0) : join_far(dd{v.x, v.y}, bias));
  }
}

constexpr int kThreads = 128;
constexpr int kLineSmem = 2 * 27 * kThreads * int(sizeof(float2));

// One thread per cell; its 27 value pairs and 27 test-side pairs live in two shared-memory columns
// (float2 slots, 8-byte accesses), so every phase is a short rolled loop over the columns:
//   gather and x lines, y lines, z lines                   nodes -> Gauss points
//   planes z = const: value term, y and x fluxes           -> test side V of the plane
//   z lines: z fluxes, then the z transpose of V + D_z^T F
//   slabs of nodes z = const: y and x transposes, warp folding, scatter
// Bound: fp32 instruction issue, 9.4k instructions per 32 cells at 75 % of the issue slots (ncu).  The
// unrolled form with the values in registers held 198 KB of instructions (12.4k per 32 cells, with
// convection 15.4k; 2 to 6 instruction-fetch stalls per issue) and spilled at its 96 registers.  Measured:
// 128^3 heat apply 1039 -> 653 us, 64^3 transposed convective apply 336 -> 131 us.  Unrolling the z lines
// three times costs 692 us, every loop 891 us (instruction fetch again).  Four blocks per SM is what the
// 432 bytes of shared memory per thread allow.
template <bool CONV, bool TR, bool QM>
__global__ void __launch_bounds__(kThreads, 4) k_scalar_df_uniform(const __grid_constant__ DfArgs A, UniformGeom ug) {
  extern __shared__ float2 df_smem[];
  int i, j, k;
  const bool active = brick_cell(ug, i, j, k);
  const int t = threadIdx.x;
  float2* const sU = df_smem + t;                    // slot q at sU[q * kThreads]
  float2* const sV = df_smem + 27 * kThreads + t;
  auto ld2 = [](const float2* p) { const float2 v = *p; return dd{v.x, v.y}; };
  auto st2 = [](float2* p, dd v) { *p = make_float2(v.h, v.l); };
  auto ldg2 = [](const float2* p) { const float2 v = __ldg(p); return dd{v.x, v.y}; };
  const int64_t cell = active ? i + int64_t(ug.nx) * (j + int64_t(ug.ny) * k) : 0;
  const int64_t base = active ? 2 * int64_t(i) + ug.sx * (2 * int64_t(j)) + ug.sy * (2 * int64_t(k)) : 0;
  const uint32_t dmask = active ? dirichlet_mask(ug, i, j, k) : 0u;
  const int64_t nc = A.ncells;
  // L2 prefetch of the coefficient rows while the inputs load and the sweeps run, one 32-byte sector per
  // brick row and table row by the row's lanes (128^3: 684 -> 653 us; both halves of the row's 64 bytes
  // 657 us, the convection rows as well 657 us and no gain for the convective operator)
  if (j < ug.ny && k < ug.nz) {
    const int lx = t & 7;
    const float2* const p = A.c + (int64_t(i - lx) + int64_t(ug.nx) * (j + int64_t(ug.ny) * k));
#pragma unroll 1
    for (int q = lx; q < 27; q += 8) asm volatile("prefetch.global.L2 [%0];" ::"l"(p + q * nc));
  }
  int bias = 0;
  bool bad;   // an Inf or NaN among the cell's inputs
  {
    // gather (Dirichlet nodes and lanes without a cell read as 0); right-hand side blockIdx.y
    const double* __restrict__ s = A.src + int64_t(blockIdx.y) * A.ld + base;
    double X[27];
#pragma unroll
    for (int l = 0; l < 27; ++l) {
      const int a = l % 3, b = (l / 3) % 3, c = l / 9;
      X[l] = __ldg(s + a + ug.sx * b + ug.sy * c);
    }
    const uint32_t off = active ? dmask : 0x7FFFFFFu;
    if (off) {
#pragma unroll
      for (int l = 0; l < 27; ++l)
        if ((off >> l) & 1u) X[l] = 0.0;
    }
    // one power-of-two scale per warp (its 8 x 4 cells share faces folded below): the largest
    // input maps to [1, 2)
    unsigned emax = 0;
#pragma unroll
    for (int l = 0; l < 27; ++l) emax = max(emax, unsigned(__double2hiint(X[l])) & 0x7FF00000u);
#pragma unroll
    for (int l = 0; l < 27; ++l) *reinterpret_cast<double*>(sU + l * kThreads) = X[l];
    emax = finite_exponent(__reduce_max_sync(0xffffffffu, emax) >> 20, sU, kThreads, 27, bad);
    bias = emax ? int(emax) - 1023 : 0;
  }
#pragma unroll 1
  for (float2* p = sU; p < sU + 27 * kThreads; p += 3 * kThreads) {
    dd u0 = d2dd_bits(*reinterpret_cast<double*>(p), bias);
    dd u1 = d2dd_bits(*reinterpret_cast<double*>(p + kThreads), bias);
    dd u2 = d2dd_bits(*reinterpret_cast<double*>(p + 2 * kThreads), bias);
    dd_line_values(u0, u1, u2);
    st2(p, u0);
    st2(p + kThreads, u1);
    st2(p + 2 * kThreads, u2);
  }
#pragma unroll 1
  for (int qc = 0; qc < 3; ++qc) {
    float2* const p = sU + 9 * qc * kThreads;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      dd u0 = ld2(p + a * kThreads), u2 = ld2(p + (a + 6) * kThreads);
      dd_line_values(u0, ld2(p + (a + 3) * kThreads), u2);
      st2(p + a * kThreads, u0);
      st2(p + (a + 6) * kThreads, u2);
    }
  }
#pragma unroll 1
  for (int p3 = 0; p3 < 9; p3 += 3) {
    float2* const p = sU + p3 * kThreads;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      dd u0 = ld2(p + a * kThreads), u2 = ld2(p + (a + 18) * kThreads);
      dd_line_values(u0, ld2(p + (a + 9) * kThreads), u2);
      st2(p + a * kThreads, u0);
      st2(p + (a + 18) * kThreads, u2);
    }
  }
  const float2* __restrict__ gc = A.c + cell;
  const float2* __restrict__ gb = A.b + cell;
  const float2* __restrict__ gm = A.m + cell;
#pragma unroll 1
  for (int qc = 0; qc < 3; ++qc) {
    const int q0 = 9 * qc;
    dd U[9], C[9], R[9];
#pragma unroll
    for (int p = 0; p < 9; ++p) {
      C[p] = ldg2(gc + (q0 + p) * nc);
      U[p] = ld2(sU + (q0 + p) * kThreads);
    }
#pragma unroll
    for (int p = 0; p < 9; ++p)
      R[p] = dd_mul(QM ? ldg2(gm + (q0 + p) * nc) : dd{A.wm[q0 + p].x, A.wm[q0 + p].y}, U[p]);
#pragma unroll
    for (int dir = 1; dir >= 0; --dir) {
      const int st = dir ? 3 : 1;
#pragma unroll
      for (int n = 0; n < 3; ++n) {
        const int p0 = dir ? n : 3 * n, p1 = p0 + st, p2 = p1 + st;
        dd g0, g1, g2;
        dd_line_deriv(U[p0], U[p1], U[p2], g0, g1, g2);
        dd f0 = dd_mul(C[p0], g0), f1 = dd_mul(C[p1], g1), f2 = dd_mul(C[p2], g2);
        if (CONV) {
          const float2* __restrict__ bd = gb + (27 * dir + q0) * nc;
          const dd b0 = ldg2(bd + p0 * nc), b1 = ldg2(bd + p1 * nc), b2 = ldg2(bd + p2 * nc);
          if (TR) {
            f0 = dd_fma(f0, b0, U[p0]);
            f1 = dd_fma(f1, b1, U[p1]);
            f2 = dd_fma(f2, b2, U[p2]);
          } else {
            R[p0] = dd_fma(R[p0], b0, g0);
            R[p1] = dd_fma(R[p1], b1, g1);
            R[p2] = dd_fma(R[p2], b2, g2);
          }
        }
        dd_line_deriv_t(f0, f1, f2, R[p0], R[p1], R[p2]);
      }
    }
#pragma unroll
    for (int p = 0; p < 9; ++p) st2(sV + (q0 + p) * kThreads, dd_norm(R[p]));
  }
#pragma unroll 1
  for (int p = 0; p < 9; ++p) {
    dd C[3], U[3], V[3], B[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      C[c] = ldg2(gc + (p + 9 * c) * nc);
      if (CONV) B[c] = ldg2(gb + (54 + p + 9 * c) * nc);
      U[c] = ld2(sU + (p + 9 * c) * kThreads);
      V[c] = ld2(sV + (p + 9 * c) * kThreads);
    }
    dd g0, g1, g2;
    dd_line_deriv(U[0], U[1], U[2], g0, g1, g2);
    dd f0 = dd_mul(C[0], g0), f1 = dd_mul(C[1], g1), f2 = dd_mul(C[2], g2);
    if (CONV && TR) {
      f0 = dd_fma(f0, B[0], U[0]);
      f1 = dd_fma(f1, B[1], U[1]);
      f2 = dd_fma(f2, B[2], U[2]);
    } else if (CONV) {
      V[0] = dd_fma(V[0], B[0], g0);
      V[1] = dd_fma(V[1], B[1], g1);
      V[2] = dd_fma(V[2], B[2], g2);
    }
    dd_line_combine_t(f0, f1, f2, V[0], V[1], V[2]);
#pragma unroll
    for (int c = 0; c < 3; ++c) st2(sV + (p + 9 * c) * kThreads, V[c]);
  }
  double* __restrict__ d = A.dst + int64_t(blockIdx.y) * A.ld + base;
  const bool far = far_scale(bias);
#pragma unroll 1
  for (int c = 0; c < 3; ++c) {
    dd R[9];
#pragma unroll
    for (int p = 0; p < 9; ++p) R[p] = ld2(sV + (9 * c + p) * kThreads);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      dd_line_values_t(R[a], R[a + 3], R[a + 6]);
      R[a] = dd_norm(R[a]);
      R[a + 3] = dd_norm(R[a + 3]);
      R[a + 6] = dd_norm(R[a + 6]);
    }
#pragma unroll
    for (int b = 0; b < 3; ++b) dd_line_values_t(R[3 * b], R[3 * b + 1], R[3 * b + 2]);
    if (!active) {
#pragma unroll
      for (int p = 0; p < 9; ++p) R[p] = dd{0.f, 0.f};
    }
    if (far) {
#pragma unroll
      for (int p = 0; p < 9; ++p) st2(sV + (9 * c + p) * kThreads, R[p]);
    } else {
      scatter_dd_slab(d + ug.sy * c, ug.sx, (dmask >> (9 * c)) & 0x1FFu, R, active, bias);
    }
  }
  if (active && (far || bad)) scatter_rare<kThreads>(d, ug.sx, ug.sy, dmask, sV, bias, bad);
}

// ---------------------------------------------------------------------------------------------
// Double-float Oseen apply (Q2 velocity / Q1 pressure, uniform mesh, folded Gauss-point coefficients
// as float pairs).  A block of three warps owns an 8 x 4 x 1 brick of 32 cells; warp C evaluates the
// test functions of velocity component C for the brick's cells, reading the other components'
// Gauss-point values (for the symmetric part of the stress) from shared memory.  Velocity and pressure
// inputs are scaled by their own powers of two (the block's largest finite velocity / pressure input in
// [1, 2); a field that is zero in the block takes the other's); velocity fluxes and value terms are rescaled
// by an exact power of two so that every velocity test term is accumulated in the larger of the two scales.
//
// All three warps run one code path on permuted axes: a = the warp's own component direction C, b
// and c the other two.  Planes (a, b) first: value terms, the diagonal flux along a (with the
// pressure), the flux along b, whose other half d_a u_b lies in the plane, and the continuity share of
// d_a u_a.  Then planes (a, c): the flux along c with its half d_a u_c, the transpose along c of the
// whole test side, and the value transpose along a.  So each derivative is taken by whole lines, and the
// rolled loops over planes keep the three warps inside a short instruction body.
// Bound: fp32 instruction issue at 12 warps per SM (48 KB of shared memory per block).  45.9k instead of
// 72.9k instructions per 32 cells at 63 % instead of 46 % of the issue slots: 64^3 1105 -> 505 us (539 with tables over cells,
// whose rows took 64-bit address arithmetic; per tile they share the offsets of the shared arrays, and one
// instruction per table fetches a tile into L2).

struct DfOseenArgs {
  const double* src;
  double* dst;
  int64_t nu;              // velocity DoFs per component (pressure block starts at 3 nu)
  // per tile of 8 x 4 x 1 cells as [q][lane]; lanes without a cell 0
  const float2* cm;        // [tile][27][32] w h^3 sigma rho (+ Darcy)
  const float2* cv;        // [tile][27][32] (5/3) w h mu
  const float2* cb;        // [tile][81][32] w h^2 rho beta / (2 delta)
  const float2* nr;        // melt-pool trace correction: interface normal per Gauss point, [tile][81][32]
  float2 pw[27];           // -h^2 w_q / (2 delta): pressure term of the gradient test
  float2 mh2;              // -h^2 / (2 delta): continuity rows
};

__device__ __forceinline__ void prefetch_l2(const float2* p, unsigned bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

__device__ __forceinline__ float pow2f(int e) {  // 2^e for e in [-126, 127]; 0 below
  return e < -126 ? 0.f : __uint_as_float(unsigned(min(e, 127) + 127) << 23);
}

// EXT: the melt-pool trace correction -2 mu (div u) n (x) n : grad v adds t n_C n_d to the flux of
// component C in direction d, t = -2 cv div u, formed once per Gauss point (the Darcy term sits in cm)
template <bool EXT> constexpr int kOseenSmem = int(sizeof(float2)) * 32 * 27 * (EXT ? 8 : 7);

template <bool EXT>
__global__ void __launch_bounds__(96, 4) k_oseen_df_uniform(const __grid_constant__ DfOseenArgs A, UniformGeom ug) {
  extern __shared__ float2 df_smem[];
  __shared__ int sE[3];
  __shared__ unsigned sBad[4];   // cells with an Inf or NaN among the component's inputs, among the pressures
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float2* const sU = df_smem + lane;                    // component e, point q at sU[(27 e + q) * 32]
  float2* const sV = df_smem + 81 * 32 + w * 27 * 32 + lane;
  float2* const sP = df_smem + 162 * 32 + lane;         // pressure term at the Gauss points (output scale)
  float2* const sT = df_smem + 189 * 32 + lane;         // EXT: t
  auto ld2 = [](const float2* p) { const float2 v = *p; return dd{v.x, v.y}; };
  auto st2 = [](float2* p, dd v) { *p = make_float2(v.h, v.l); };
  auto ldg2 = [](const float2* p) { const float2 v = __ldg(p); return dd{v.x, v.y}; };
  const int nbx = (ug.nx + 7) >> 3, nby = (ug.ny + 3) >> 2;
  const int blk = blockIdx.x;
  const int i = (blk % nbx) * 8 + (lane & 7), j = ((blk / nbx) % nby) * 4 + (lane >> 3), k = blk / (nbx * nby);
  const bool active = i < ug.nx && j < ug.ny;
  const int64_t base = active ? 2 * int64_t(i) + ug.sx * (2 * int64_t(j)) + ug.sy * (2 * int64_t(k)) : 0;
  const uint32_t dmask = active ? dirichlet_mask(ug, i, j, k) : 0u;
  const int64_t px = ug.nx + 1, pxy = px * (ug.ny + 1);
  const int64_t pbase = active ? i + px * (j + (ug.ny + 1) * int64_t(k)) : 0;
  // the tile's coefficients, addressed by the offsets of the shared arrays
  const float2* __restrict__ const tm = A.cm + int64_t(blk) * (27 * 32) + lane;
  const float2* __restrict__ const tv = A.cv + int64_t(blk) * (27 * 32) + lane;
  const float2* __restrict__ const tb = A.cb + int64_t(blk) * (81 * 32) + lane;
  const float2* __restrict__ const tn = A.nr + int64_t(blk) * (81 * 32) + lane;
  // into L2 while the inputs load and the sweeps run
  if (lane == 0) {
    constexpr unsigned kRow = 32 * sizeof(float2);
    if (w == 0) {
      prefetch_l2(tv, 27 * kRow);
      prefetch_l2(tm, 27 * kRow);
    } else if (w == 1) {
      prefetch_l2(tb, 81 * kRow);
    } else if (EXT) {
      prefetch_l2(tn, 81 * kRow);
    }
  }
  // raw inputs: this warp's velocity component (Dirichlet nodes and lanes without a cell read as 0)
  // and the cell's 8 pressures
  double Pn[8];
  unsigned eu = 0, ep = 0;
  {
    double X[27];
#pragma unroll
    for (int l = 0; l < 27; ++l) {
      const int a = l % 3, bb = (l / 3) % 3, c = l / 9;
      X[l] = __ldg(A.src + w * A.nu + base + a + ug.sx * bb + ug.sy * c);
    }
#pragma unroll
    for (int n = 0; n < 8; ++n) {
      Pn[n] = __ldg(A.src + 3 * A.nu + pbase + (n & 1) + px * ((n >> 1) & 1) + pxy * (n >> 2));
      if (!active) Pn[n] = 0.0;
      ep = max(ep, unsigned(__double2hiint(Pn[n])) & 0x7FF00000u);
    }
    const uint32_t off = active ? dmask : 0x7FFFFFFu;
    if (off) {
#pragma unroll
      for (int l = 0; l < 27; ++l)
        if ((off >> l) & 1u) X[l] = 0.0;
    }
#pragma unroll
    for (int l = 0; l < 27; ++l) {
      eu = max(eu, unsigned(__double2hiint(X[l])) & 0x7FF00000u);
      *reinterpret_cast<double*>(sU + (27 * w + l) * 32) = X[l];
    }
  }
  bool bad_u, bad_p = false;
  eu = finite_exponent(__reduce_max_sync(0xffffffffu, eu) >> 20, sU + 27 * w * 32, 32, 27, bad_u);
  ep = __reduce_max_sync(0xffffffffu, ep) >> 20;   // the same cells in every warp
  if (ep == 0x7FFu) {
    ep = 0;
#pragma unroll
    for (int n = 0; n < 8; ++n) {
      const unsigned e = unsigned(__double2hiint(Pn[n])) & 0x7FF00000u;
      if (e == 0x7FF00000u) bad_p = true;
      else ep = max(ep, e);
    }
    ep = __reduce_max_sync(0xffffffffu, ep) >> 20;
  }
  const unsigned cells_u = __ballot_sync(0xffffffffu, bad_u), cells_p = __ballot_sync(0xffffffffu, bad_p);
  if (lane == 0) {
    sE[w] = int(eu);
    sBad[w] = cells_u;
    if (w == 0) sBad[3] = cells_p;
  }
  __syncthreads();
  const int em = max(sE[0], max(sE[1], sE[2]));
  // (a field that is zero in the whole block takes the other's scale: with 2^0 it would hide small values)
  const int exp_u = em ? em : int(ep), exp_p = ep ? int(ep) : em;
  const int bias_u = exp_u ? exp_u - 1023 : 0, bias_p = exp_p ? exp_p - 1023 : 0;
  const int bias_out = max(bias_u, bias_p);
  const float su = pow2f(bias_u - bias_out);   // velocity terms into the output scale
  {
    float2* const p0 = sU + 27 * w * 32;
#pragma unroll 1
    for (float2* p = p0; p < p0 + 27 * 32; p += 3 * 32) {
      dd u0 = d2dd_bits(*reinterpret_cast<double*>(p), bias_u);
      dd u1 = d2dd_bits(*reinterpret_cast<double*>(p + 32), bias_u);
      dd u2 = d2dd_bits(*reinterpret_cast<double*>(p + 64), bias_u);
      dd_line_values(u0, u1, u2);
      st2(p, u0);
      st2(p + 32, u1);
      st2(p + 64, u2);
    }
#pragma unroll 1
    for (int n = 0; n < 6; ++n) {   // y lines of the three planes, then z lines
      const int o = n < 3 ? 9 * n : 3 * (n - 3), st = n < 3 ? 3 : 9;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        float2* const p = p0 + (o + a) * 32;
        dd u0 = ld2(p), u2 = ld2(p + 2 * st * 32);
        dd_line_values(u0, ld2(p + st * 32), u2);
        st2(p, u0);
        st2(p + 2 * st * 32, u2);
      }
    }
    // pressure term -h^2 w_q p(x_q) / (2 delta) at the warp's plane qc = w of Gauss points
    const float sp = pow2f(bias_p - bias_out);
    const float sg = w == 0 ? -1.f : (w == 1 ? 0.f : 1.f);
    dd Pz[4];
#pragma unroll
    for (int n = 0; n < 4; ++n) {
      const dd q0 = d2dd_bits(Pn[n], bias_p), q1 = d2dd_bits(Pn[n + 4], bias_p);
      Pz[n] = dd_norm(dd_add(dd_pow2(dd_add(q0, q1), 0.5f), dd_mulc<2>(dd_pow2(dd_sub(q1, q0), sg))));
    }
    dd Py[2][3];
#pragma unroll
    for (int a = 0; a < 2; ++a) dd_line_q1(Pz[a], Pz[a + 2], Py[a][0], Py[a][1], Py[a][2]);
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      dd v[3];
      dd_line_q1(Py[0][b], Py[1][b], v[0], v[1], v[2]);
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const int q = a + 3 * b + 9 * w;
        st2(sP + q * 32, dd_pow2(dd_norm(dd_mul(dd{A.pw[q].x, A.pw[q].y}, v[a])), sp));
      }
    }
  }
  __syncthreads();
  if (EXT) {
    // t = -2 cv div u at the warp's plane qc = w
    const float sg = 2.f * float(w - 1);
    dd D[9];
#pragma unroll
    for (int n = 0; n < 3; ++n) {
      const float2* const p = sU + (9 * w + 3 * n) * 32;
      dd_line_deriv(ld2(p), ld2(p + 32), ld2(p + 64), D[3 * n], D[3 * n + 1], D[3 * n + 2]);
    }
#pragma unroll
    for (int n = 0; n < 3; ++n) {
      const float2* const p = sU + (27 + 9 * w + n) * 32;
      dd g0, g1, g2;
      dd_line_deriv(ld2(p), ld2(p + 96), ld2(p + 192), g0, g1, g2);
      D[n] = dd_add(D[n], g0);
      D[n + 3] = dd_add(D[n + 3], g1);
      D[n + 6] = dd_add(D[n + 6], g2);
    }
#pragma unroll
    for (int p = 0; p < 9; ++p) {
      const float2* const z = sU + (54 + p) * 32;
      const dd v0 = ld2(z), v1 = ld2(z + 9 * 32), v2 = ld2(z + 18 * 32);
      const dd cc = dd_sub(dd_add(v0, v2), dd_pow2(v1, 2.f));
      const dd div = dd_norm(dd_add(D[p], dd_add(dd_sub(v2, v0), dd_pow2(cc, sg))));
      const dd cv = ldg2(tv + (p + 9 * w) * 32);
      st2(sT + (p + 9 * w) * 32, dd_norm(dd_pow2(dd_mul(cv, div), -2.f)));
    }
    __syncthreads();
  }
  // permuted axes: a = own direction, b and c the others (strides in the 27-array)
  const int sa = w == 0 ? 1 : (w == 1 ? 3 : 9), sb = w == 1 ? 1 : 3, sc = w == 2 ? 1 : 9;
  const int eb = w == 1 ? 0 : 1, ec = w == 2 ? 0 : 2;
  const int na = sa * 32, nb = sb * 32, ncc = sc * 32;
  const float2* const uC = sU + 27 * w * 32;
  dd Rp[8];
#pragma unroll
  for (int n = 0; n < 8; ++n) Rp[n] = dd{0.f, 0.f};
#pragma unroll 1
  for (int ic = 0; ic < 3; ++ic) {
    const int o = ic * sc * 32;
    const float2* __restrict__ gm = tm + o;
    const float2* __restrict__ gv = tv + o;
    const float2* __restrict__ ga = tb + 27 * 32 * w + o;
    const float2* __restrict__ gb = tb + 27 * 32 * eb + o;
    dd U[9], R[9], cv[9];
#pragma unroll
    for (int p = 0; p < 9; ++p) {
      cv[p] = ldg2(gv + (p % 3) * na + (p / 3) * nb);
      U[p] = ld2(uC + o + ((p % 3) * sa + (p / 3) * sb) * 32);
    }
#pragma unroll
    for (int p = 0; p < 9; ++p) R[p] = dd_mul(ldg2(gm + (p % 3) * na + (p / 3) * nb), U[p]);
    // own direction: convection, continuity and the diagonal flux 2 cv d_a u_a + p
    dd fa[9], T1[3][2];
#pragma unroll
    for (int n = 0; n < 3; ++n) {
      dd g[3];
      dd_line_deriv(U[3 * n], U[3 * n + 1], U[3 * n + 2], g[0], g[1], g[2]);
      dd_line_q1_t(g[0], g[1], g[2], T1[n][0], T1[n][1]);
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        const int p = 3 * n + m;
        R[p] = dd_fma(R[p], ldg2(ga + m * na + n * nb), g[m]);
        fa[p] = dd_add(dd_pow2(dd_mul(cv[p], g[m]), 2.f * su), ld2(sP + o + (m * sa + n * sb) * 32));
      }
    }
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      dd t0, t1;
      dd_line_q1_t(T1[0][m], T1[1][m], T1[2][m], t0, t1);
      // weights of the c direction: w_c (1/2 -+ x_c)
      const dd w0{ic == 1 ? 8.f / 36.f : float(5.0 / 36.0), ic == 1 ? float(8.0 / 36.0 - double(8.f / 36.f))
                                                                   : float(5.0 / 36.0 - double(float(5.0 / 36.0)))};
      const float sx = ic == 1 ? 0.f : (ic == 0 ? -1.f : 1.f);
      const dd h0 = dd_mul(w0, t0), h1 = dd_mul(w0, t1);
      const dd x0 = dd_pow2(dd_mulc<5>(t0), sx), x1 = dd_pow2(dd_mulc<5>(t1), sx);
      Rp[m] = dd_add(Rp[m], dd_sub(h0, x0));
      Rp[m + 2] = dd_add(Rp[m + 2], dd_sub(h1, x1));
      Rp[m + 4] = dd_add(Rp[m + 4], dd_add(h0, x0));
      Rp[m + 6] = dd_add(Rp[m + 6], dd_add(h1, x1));
    }
    // b direction: cv (d_b u_a + d_a u_b)
    dd fb[9];
    {
      const float2* const uB = sU + 27 * eb * 32 + o;
#pragma unroll
      for (int n = 0; n < 3; ++n) {
        const float2* const q = uB + n * sb * 32;
        dd_line_deriv(ld2(q), ld2(q + sa * 32), ld2(q + 2 * sa * 32), fb[3 * n], fb[3 * n + 1], fb[3 * n + 2]);
      }
    }
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      dd g[3];
      dd_line_deriv(U[m], U[m + 3], U[m + 6], g[0], g[1], g[2]);
#pragma unroll
      for (int n = 0; n < 3; ++n) {
        const int p = 3 * n + m;
        R[p] = dd_pow2(dd_fma(R[p], ldg2(gb + m * na + n * nb), g[n]), su);
        fb[p] = dd_pow2(dd_mul(cv[p], dd_add(g[n], fb[p])), su);
      }
    }
    if (EXT) {
#pragma unroll
      for (int p = 0; p < 9; ++p) {
        const int on = o + (p % 3) * na + (p / 3) * nb;
        const dd nA = ldg2(tn + 27 * 32 * w + on), nB = ldg2(tn + 27 * 32 * eb + on);
        const dd tA = dd_mul(dd_pow2(ld2(sT + o + ((p % 3) * sa + (p / 3) * sb) * 32), su), nA);
        fa[p] = dd_fma(fa[p], tA, nA);
        fb[p] = dd_fma(fb[p], tA, nB);
      }
    }
#pragma unroll
    for (int n = 0; n < 3; ++n) {
      dd_line_deriv_t(fa[3 * n], fa[3 * n + 1], fa[3 * n + 2], R[3 * n], R[3 * n + 1], R[3 * n + 2]);
    }
#pragma unroll
    for (int m = 0; m < 3; ++m) dd_line_deriv_t(fb[m], fb[m + 3], fb[m + 6], R[m], R[m + 3], R[m + 6]);
#pragma unroll
    for (int p = 0; p < 9; ++p) st2(sV + o + ((p % 3) * sa + (p / 3) * sb) * 32, dd_norm(R[p]));
  }
  if (active) {
    // continuity rows -int psi_n d_C u_C: this component's share, in the velocity scale
    const dd mh2{A.mh2.x, A.mh2.y};
    const int64_t pa = w == 0 ? 1 : (w == 1 ? px : pxy), pb = w == 1 ? 1 : px, pc = w == 2 ? 1 : pxy;
    double* const pd = A.dst + 3 * A.nu + pbase;
    if (__builtin_expect(far_scale(bias_u), 0)) {
#pragma unroll
      for (int n = 0; n < 8; ++n)
        atomicAdd(pd + (n & 1) * pa + ((n >> 1) & 1) * pb + (n >> 2) * pc,
                  join_far(dd_mul(mh2, dd_norm(Rp[n])), bias_u));
    } else {
#pragma unroll
      for (int n = 0; n < 8; ++n)
        atomicAdd(pd + (n & 1) * pa + ((n >> 1) & 1) * pb + (n >> 2) * pc, join(dd_mul(mh2, dd_norm(Rp[n])), bias_u));
    }
    if (__builtin_expect(((sBad[0] | sBad[1] | sBad[2]) >> lane) & 1u, 0))
#pragma unroll 1
      for (int n = 0; n < 8; ++n)
        atomicAdd(pd + (n & 1) * pa + ((n >> 1) & 1) * pb + (n >> 2) * pc, __hiloint2double(0x7FF80000, 0));
  }
  // planes (a, c): flux along c, transposes along c and a
#pragma unroll 1
  for (int ib = 0; ib < 3; ++ib) {
    const int o = ib * sb * 32;
    dd X[9], V[9];   // index ia + 3 ic
    const float2* const uc = sU + 27 * ec * 32 + o;
#pragma unroll
    for (int n = 0; n < 3; ++n) {
      const float2* const q = uc + n * sc * 32;
      dd_line_deriv(ld2(q), ld2(q + sa * 32), ld2(q + 2 * sa * 32), X[3 * n], X[3 * n + 1], X[3 * n + 2]);
    }
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      const int om = o + m * sa * 32;
      dd g[3], f[3];
      dd_line_deriv(ld2(uC + om), ld2(uC + om + sc * 32), ld2(uC + om + 2 * sc * 32), g[0], g[1], g[2]);
#pragma unroll
      for (int n = 0; n < 3; ++n) {
        const int p = m + 3 * n;
        f[n] = dd_pow2(dd_mul(ldg2(tv + om + n * ncc), dd_add(g[n], X[p])), su);
        V[p] = dd_add(ld2(sV + om + n * sc * 32), dd_pow2(dd_mul(ldg2(tb + 27 * 32 * ec + om + n * ncc), g[n]), su));
        if (EXT) {
          const dd nA = ldg2(tn + 27 * 32 * w + om + n * ncc), nC = ldg2(tn + 27 * 32 * ec + om + n * ncc);
          f[n] = dd_fma(f[n], dd_mul(dd_pow2(ld2(sT + om + n * sc * 32), su), nA), nC);
        }
      }
      dd_line_combine_t(f[0], f[1], f[2], V[m], V[m + 3], V[m + 6]);
    }
#pragma unroll
    for (int n = 0; n < 3; ++n) {
      dd_line_values_t(V[3 * n], V[3 * n + 1], V[3 * n + 2]);
#pragma unroll
      for (int m = 0; m < 3; ++m) st2(sV + o + (m * sa + n * sc) * 32, dd_norm(V[3 * n + m]));
    }
  }
  double* __restrict__ d = A.dst + w * A.nu + base;
  const bool far = far_scale(bias_out);
#pragma unroll 1
  for (int c = 0; c < 3; ++c) {
    dd R[9];
#pragma unroll
    for (int p = 0; p < 9; ++p) R[p] = ld2(sV + (9 * c + p) * 32);
    if (w == 1) {   // b = x
#pragma unroll
      for (int b = 0; b < 3; ++b) dd_line_values_t(R[3 * b], R[3 * b + 1], R[3 * b + 2]);
    } else {        // b = y
#pragma unroll
      for (int a = 0; a < 3; ++a) dd_line_values_t(R[a], R[a + 3], R[a + 6]);
    }
    if (!active) {
#pragma unroll
      for (int p = 0; p < 9; ++p) R[p] = dd{0.f, 0.f};
    }
    if (__builtin_expect(far, 0)) {
#pragma unroll
      for (int p = 0; p < 9; ++p) st2(sV + (9 * c + p) * 32, R[p]);
    } else {
      scatter_dd_slab(d + ug.sy * c, ug.sx, (dmask >> (9 * c)) & 0x1FFu, R, active, bias_out);
    }
  }
  const bool bad = ((sBad[0] | sBad[1] | sBad[2] | sBad[3]) >> lane) & 1u;
  if (__builtin_expect(active && (far || bad), 0)) scatter_rare<32>(d, ug.sx, ug.sy, dmask, sV, bias_out, bad);
}

// s c as float pairs
__global__ void k_split_plain(const double* __restrict__ c, int64_t n, double s, float2* out) {
  const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (t >= n) return;
  const double v = c[t] * s;
  const float hi = __double2float_rn(v);
  out[t] = make_float2(hi, __double2float_rn(v - double(hi)));
}

// s c of a [rows][ncells] table as float pairs, per tile of 8 x 4 x 1 cells: [tile][rows][32]
__global__ void k_split_tiles(const double* __restrict__ c, int rows, double s, float2* __restrict__ out, int ntx, int nty,
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
  for (int r = 0; r < rows; ++r) {
    const double v = active ? c[r * nc + cell] * s : 0.0;
    const float hi = __double2float_rn(v);
    out[(tile * rows + r) * 32 + lane] = make_float2(hi, __double2float_rn(v - double(hi)));
  }
}

// w_q s c_q of a Gauss-point table ([27][ncells] or [3][27][ncells]) as float pairs
__global__ void k_split_weighted(const double* __restrict__ c, int64_t n, int64_t ncells, double s, float2* out) {
  const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (t >= n) return;
  const double v = c[t] * cW364[int((t / ncells) % 27)] * s;
  const float hi = __double2float_rn(v);
  out[t] = make_float2(hi, __double2float_rn(v - double(hi)));
}

}  // namespace

static mf_status launch_split_weighted(mf_ctx* ctx, const mf_dofmap* m, const double* c, int rows, double scale,
                                       float2* out) {
  MF_CUDA_TRY(upload_tables_here());
  const int64_t n = rows * m->n_cells;
  k_split_weighted<<<unsigned((n + 255) / 256), 256, 0, ctx->stream>>>(c, n, m->n_cells, scale, out);
  ctx->launches++;
  MF_CUDA_TRY(cudaGetLastError());
  return MF_OK;
}

// both derivative factors 1 / (2 delta) of the diffusion term: 5/3
mf_status launch_df_coef_split(mf_ctx* ctx, const mf_dofmap* m, const double* qcoef64, float2* out) {
  return launch_split_weighted(ctx, m, qcoef64, 27, m->mesh->h0 * (5.0 / 3.0), out);
}

mf_status launch_df_vec_split(mf_ctx* ctx, const mf_dofmap* m, const double* qvec64, float2* out) {
  return launch_split_weighted(ctx, m, qvec64, 81, m->mesh->h0 * m->mesh->h0 * kDerivScale, out);
}

mf_status launch_df_mass_split(mf_ctx* ctx, const mf_dofmap* m, const double* qmass64, float2* out) {
  const double h = m->mesh->h0;
  return launch_split_weighted(ctx, m, qmass64, 27, h * h * h, out);
}

mf_status launch_scalar_df_uniform(mf_ctx* ctx, const mf_dofmap* m, const double* src, double* dst, int nrhs, int64_t ld,
                                   const float2* c, const float2* b, const float2* qm, double mass, bool transpose) {
  MF_CUDA_TRY(upload_tables_here());
  if (qm && !b) return fail(MF_EINVAL, "a value coefficient per Gauss point needs the convective kernel");
  static bool attrs = false;
  if (!attrs) {
    for (auto f : {k_scalar_df_uniform<false, false, false>, k_scalar_df_uniform<true, false, false>,
                   k_scalar_df_uniform<true, true, false>, k_scalar_df_uniform<true, false, true>,
                   k_scalar_df_uniform<true, true, true>})
      MF_CUDA_TRY(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kLineSmem));
    attrs = true;
  }
  const Tables tb = make_tables();
  DfArgs a{};
  a.src = src;
  a.dst = dst;
  a.ld = ld;
  a.c = c;
  a.b = b;
  a.m = qm;
  a.ncells = m->n_cells;
  const double h = m->mesh->h0;
  for (int q = 0; q < 27; ++q) {
    const double v = tb.W3[q] * mass * h * h * h;
    a.wm[q].x = float(v);
    a.wm[q].y = float(v - double(a.wm[q].x));
  }
  const UniformGeom ug = uniform_geom(m);
  const dim3 grid(brick_blocks(ug.nx, ug.ny, ug.nz), nrhs);
  if (!b)
    k_scalar_df_uniform<false, false, false><<<grid, kThreads, kLineSmem, ctx->stream>>>(a, ug);
  else if (transpose && qm)
    k_scalar_df_uniform<true, true, true><<<grid, kThreads, kLineSmem, ctx->stream>>>(a, ug);
  else if (transpose)
    k_scalar_df_uniform<true, true, false><<<grid, kThreads, kLineSmem, ctx->stream>>>(a, ug);
  else if (qm)
    k_scalar_df_uniform<true, false, true><<<grid, kThreads, kLineSmem, ctx->stream>>>(a, ug);
  else
    k_scalar_df_uniform<true, false, false><<<grid, kThreads, kLineSmem, ctx->stream>>>(a, ug);
  ctx->launches++;
  MF_CUDA_TRY(cudaGetLastError());
  return MF_OK;
}

mf_status launch_split_pairs(mf_ctx* ctx, const double* c, int64_t n, double scale, float2* out) {
  k_split_plain<<<unsigned((n + 255) / 256), 256, 0, ctx->stream>>>(c, n, scale, out);
  ctx->launches++;
  MF_CUDA_TRY(cudaGetLastError());
  return MF_OK;
}

static mf_status launch_split_tiles(mf_ctx* ctx, const mf_dofmap* m, const double* c, int rows, double scale, float2* out) {
  const UniformGeom ug = uniform_geom(m);
  const int ntx = (ug.nx + 7) / 8, nty = (ug.ny + 3) / 4;
  const int64_t n = int64_t(ntx) * nty * ug.nz * 32;
  k_split_tiles<<<unsigned((n + 127) / 128), 128, 0, ctx->stream>>>(c, rows, scale, out, ntx, nty, ug);
  ctx->launches++;
  MF_CUDA_TRY(cudaGetLastError());
  return MF_OK;
}

// cv carries both derivative factors 1 / (2 delta) of the viscous term, cb the one of the convection; nr64, nr:
// the interface normals, or NULL
mf_status launch_oseen_df_split(mf_ctx* ctx, const mf_dofmap* mu, const double* cm64, const double* cv64,
                                const double* cb64, const double* nr64, float2* cm, float2* cv, float2* cb, float2* nr) {
  MF_TRY(launch_split_tiles(ctx, mu, cm64, 27, 1.0, cm));
  MF_TRY(launch_split_tiles(ctx, mu, cv64, 27, 5.0 / 3.0, cv));
  MF_TRY(launch_split_tiles(ctx, mu, cb64, 81, kDerivScale, cb));
  return nr64 ? launch_split_tiles(ctx, mu, nr64, 81, 1.0, nr) : MF_OK;
}

mf_status launch_oseen_df_uniform(mf_ctx* ctx, const mf_dofmap* mu, const double* src, double* dst, const float2* cm,
                                  const float2* cv, const float2* cb, const float2* nr) {
  MF_CUDA_TRY(upload_tables_here());
  static bool attrs = false;
  if (!attrs) {
    MF_CUDA_TRY(cudaFuncSetAttribute(k_oseen_df_uniform<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     kOseenSmem<false>));
    MF_CUDA_TRY(cudaFuncSetAttribute(k_oseen_df_uniform<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     kOseenSmem<true>));
    attrs = true;
  }
  const Tables tb = make_tables();
  DfOseenArgs a{};
  a.src = src;
  a.dst = dst;
  a.nu = mu->n_dofs;
  a.cm = cm;
  a.cv = cv;
  a.cb = cb;
  a.nr = nr;
  const double h = mu->mesh->h0;
  auto pair = [](double v) {
    const float hi = float(v);
    return make_float2(hi, float(v - double(hi)));
  };
  for (int q = 0; q < 27; ++q) a.pw[q] = pair(-(h * h) * tb.W3[q] * kDerivScale);
  a.mh2 = pair(-(h * h) * kDerivScale);
  const UniformGeom ug = uniform_geom(mu);
  const int nb = ((ug.nx + 7) / 8) * ((ug.ny + 3) / 4) * ug.nz;
  if (nr)
    k_oseen_df_uniform<true><<<nb, 96, kOseenSmem<true>, ctx->stream>>>(a, ug);
  else
    k_oseen_df_uniform<false><<<nb, 96, kOseenSmem<false>, ctx->stream>>>(a, ug);
  ctx->launches++;
  MF_CUDA_TRY(cudaGetLastError());
  return MF_OK;
}

}  // namespace mf
