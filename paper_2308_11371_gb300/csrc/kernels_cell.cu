// Cell-level kernels of the hot path.
//
// * cell_gemv: per-cell dense operators assembled from the ROM (Eq. 43).
// * grouped_gemm: Y = sum_k c_k (A_k X), one principal operator A_k serving
//   every cell's column (Remark 7; Eq. 46a with separate outputs).
// * gram_solve: Eq. 46b with diagonal-pivoted Cholesky.
// * grad: adjoint compliance gradient -w^T dK_s/dr_s u.
#include <algorithm>
#include <type_traits>

#include "common.cuh"

namespace fetidp {

namespace {

inline int ceil_div(long long a, long long b) { return (int)((a + b - 1) / b); }

// ---- K_rr^(s) R for many vectors as a sparse product (Eq. 46b, mixed path)
// Every cell has the same sparsity pattern, so K_rr^(s) (remaining DOF, local (i, d) order) is
// stored in ELL form: one column table [slot][row] shared by all cells and FP32 values
// [cell][slot][row] (row fastest, so a warp's 32 rows read 128 contiguous bytes per slot), rounded
// once per setup from the FP64 K_s.

constexpr int kSpVB = 16;   // vectors per block
constexpr int kSpLd = 20;   // shared row stride (floats): 16 vectors + 4, conflict-free 16-byte reads
// One block per (cell, rhs, chunk of kSpVB vectors), cell slowest: the vectors of the chunk are
// staged transposed ([dof][vector]) in shared memory, each thread owns rows and accumulates the
// chunk's kSpVB products in registers (four 16-byte shared reads per 16 FMAs per slot).
__global__ void __launch_bounds__(256) krr_spmm_f32_kernel(const int* __restrict__ ecol, const float* __restrict__ eval,
                                                           int nnz, int nr, int nrhs, int nchunk,
                                                           const float* __restrict__ u, long long u_rs, int u_cs,
                                                           float* __restrict__ y, long long y_rs, int y_cs, int nvec,
                                                           long long ext) {
  extern __shared__ __align__(16) float uss[];   // [nr][kSpLd]
  const int chunk = (int)(blockIdx.x % nchunk);
  const long long rest = blockIdx.x / nchunk;
  const int rhs = (int)(rest % nrhs);
  const long long cell = rest / nrhs;
  const int v0 = chunk * kSpVB, vb = min(kSpVB, nvec - v0);
  const long long base = rhs * u_rs + cell * u_cs;
  for (int t = threadIdx.x; t < kSpVB * nr; t += blockDim.x) {
    const int v = t / nr, q = t - v * nr;
    float x = 0.f;
    if (v < vb && FD_INB(base + (long long)(v0 + v) * nr + q, ext, 205)) x = u[base + (long long)(v0 + v) * nr + q];
    uss[q * kSpLd + v] = x;
  }
  __syncthreads();
  const float* ev = eval + cell * (long long)nnz * nr;
  const long long ybase = rhs * y_rs + cell * y_cs;
  for (int r = threadIdx.x; r < nr; r += blockDim.x) {
    float acc[kSpVB];
#pragma unroll
    for (int v = 0; v < kSpVB; ++v) acc[v] = 0.f;
    // eight slots' (column, value) pairs are loaded before any of them is used
    for (int sl0 = 0; sl0 < nnz; sl0 += 8) {
      int cc[8];
      float aa[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int sl = sl0 + u;
        cc[u] = sl < nnz ? __ldg(ecol + (long long)sl * nr + r) : 0;
        aa[u] = sl < nnz ? __ldcs(ev + (long long)sl * nr + r) : 0.f;
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const float4* xs = reinterpret_cast<const float4*>(uss + cc[u] * kSpLd);
        const float a = aa[u];
#pragma unroll
        for (int v4 = 0; v4 < kSpVB / 4; ++v4) {
          const float4 x = xs[v4];
          acc[4 * v4] = fmaf(a, x.x, acc[4 * v4]);
          acc[4 * v4 + 1] = fmaf(a, x.y, acc[4 * v4 + 1]);
          acc[4 * v4 + 2] = fmaf(a, x.z, acc[4 * v4 + 2]);
          acc[4 * v4 + 3] = fmaf(a, x.w, acc[4 * v4 + 3]);
        }
      }
    }
#pragma unroll
    for (int v = 0; v < kSpVB; ++v)
      if (v < vb && FD_INB(ybase + (long long)(v0 + v) * nr + r, ext, 206)) y[ybase + (long long)(v0 + v) * nr + r] = acc[v];
  }
}

// The same product for the nodal pattern of K_rr (every node's D rows share their neighbour
// nodes): one thread per node, so each 16-byte shared read of a neighbour component's vectors feeds
// D rows, and the warp's lanes read consecutive nodes' neighbours (regular, conflict-free
// addresses).  The D slots of neighbour k (D * n_r values, shared by the cell's (rhs, chunk)
// blocks through L2) are staged in shared memory by cp.async one neighbour ahead.
__device__ __forceinline__ void cp_async4(float* dst, const float* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(src) : "memory");
}
template <int D>
__global__ void __launch_bounds__(352, 2) krr_spmm_nodal_f32_kernel(
    const int* __restrict__ nbr, const float* __restrict__ eval, int nnz, int nr, int nrhs, int nchunk,
    const float* __restrict__ u, long long u_rs, int u_cs, float* __restrict__ y, long long y_rs, int y_cs, int nvec,
    long long ext) {
  extern __shared__ __align__(16) float uss[];   // [nr][kSpLd], then two slot buffers [D * nr]
  float* evs = uss + (size_t)nr * kSpLd;
  const int chunk = (int)(blockIdx.x % nchunk);
  const long long rest = blockIdx.x / nchunk;
  const int rhs = (int)(rest % nrhs);
  const long long cell = rest / nrhs;
  const int v0 = chunk * kSpVB, vb = min(kSpVB, nvec - v0);
  const long long base = rhs * u_rs + cell * u_cs;
  const int nnode = nr / D, nk = nnz / D, sl = D * nr;
  const float* ev = eval + cell * (long long)nnz * nr;
  // the chunk's vectors, transposed into [dof][vector], and neighbour 0's slots: asynchronous copies
  for (int t = threadIdx.x; t < kSpVB * nr; t += blockDim.x) {
    const int v = t / nr, q = t - v * nr;
    if (v < vb && FD_INB(base + (long long)(v0 + v) * nr + q, ext, 207))
      cp_async4(uss + q * kSpLd + v, u + base + (long long)(v0 + v) * nr + q);
    else
      uss[q * kSpLd + v] = 0.f;
  }
  for (int t = threadIdx.x; t < sl; t += blockDim.x) cp_async4(evs + t, ev + t);   // neighbour 0
  asm volatile("cp.async.commit_group;\n" ::: "memory");
  const long long ybase = rhs * y_rs + cell * y_cs;
  const int n = threadIdx.x;                      // one node per thread (the host launches >= nnode threads)
  const bool live = n < nnode;
  float acc[D][kSpVB];
#pragma unroll
  for (int a = 0; a < D; ++a)
#pragma unroll
    for (int v = 0; v < kSpVB; ++v) acc[a][v] = 0.f;
  int m_next = live ? __ldg(nbr + n) : 0;
  for (int k = 0; k < nk; ++k) {
    if (k + 1 < nk) {
      const float* src = ev + (long long)(k + 1) * sl;
      float* dst = evs + ((k + 1) & 1) * sl;
      for (int t = threadIdx.x; t < sl; t += blockDim.x) cp_async4(dst + t, src + t);
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    __syncthreads();                              // neighbour k's slots (and the vectors) are in place
    const int m = m_next;
    if (live && k + 1 < nk) m_next = __ldg(nbr + (long long)(k + 1) * nnode + n);
    if (live) {
      const float* e = evs + (k & 1) * sl;
#pragma unroll
      for (int cq = 0; cq < D; ++cq) {
        float av[D];
#pragma unroll
        for (int a = 0; a < D; ++a) av[a] = e[cq * nr + D * n + a];
        const float4* xs = reinterpret_cast<const float4*>(uss + (D * m + cq) * kSpLd);
#pragma unroll
        for (int v4 = 0; v4 < kSpVB / 4; ++v4) {
          const float4 x = xs[v4];
#pragma unroll
          for (int a = 0; a < D; ++a) {
            acc[a][4 * v4] = fmaf(av[a], x.x, acc[a][4 * v4]);
            acc[a][4 * v4 + 1] = fmaf(av[a], x.y, acc[a][4 * v4 + 1]);
            acc[a][4 * v4 + 2] = fmaf(av[a], x.z, acc[a][4 * v4 + 2]);
            acc[a][4 * v4 + 3] = fmaf(av[a], x.w, acc[a][4 * v4 + 3]);
          }
        }
      }
    }
    __syncthreads();                              // buffer k & 1 is refilled at step k + 1
  }
  if (!live) return;
#pragma unroll
  for (int v = 0; v < kSpVB; ++v)
#pragma unroll
    for (int a = 0; a < D; ++a) {
      const long long o = ybase + (long long)(v0 + v) * nr + D * n + a;
      if (v < vb && FD_INB(o, ext, 208)) y[o] = acc[a][v];
    }
}

// Per-cell dense operators in FP64: y[rhs][cell][i] = alpha sum_j M_cell[j ld + i] x[rhs][cell][j] + beta y,
// i < nout, j < nin -- the stored rows multiply x (M^T x; M x for the symmetric operators).
//
// Bound: GB300 issues two FP64 FMAs per clock and SM, and every 8-byte entry takes MR of them, so the
// kernel is FP64-bound for every MR (5.0 TB/s of operator at MR = 1).  What matters is that all SMs have
// the same share of FMAs and that nothing else uses the FP64 pipe: a CTA takes TI outputs of one cell
// (32, or all of a narrower operator), its threads are S interleaved slices of the stored rows, a thread
// keeps the MR sums of one output in registers, so a warp reads 256 consecutive bytes of a row, x comes
// as shared-memory broadcasts, and only S - 1 additions per output are outside the FMA chain.  One CTA
// per 32 outputs also gives 20 CTAs per 6^3 cell where a lattice has few cells.  The kernel it replaces
// (one CTA per cell, a warp per row, five shuffle-adds per row and RHS) took 679 us per launch of this
// class on 32 cells of n_d = 630 with 6 RHS, this one 96 us; the three products of an F_ring application
// on 256 such cells took 1.90 ms and take 1.15 ms (FP64 bound 1.04 ms).
constexpr int kMaxRhsGemv = 8;
constexpr int kGemvThreads = 256;
template <int MR>
__global__ void __launch_bounds__(kGemvThreads) cell_gemvt_kernel(const double* __restrict__ mats, long long mstride,
                                                                  int ld, int nout, int nin, int TI, int S,
                                                                  const double* __restrict__ x, long long x_rs,
                                                                  int x_cs, double* __restrict__ y, long long y_rs,
                                                                  int y_cs, double alpha, double beta, int ntile) {
  extern __shared__ __align__(16) double gvs[];   // x as [nin][MR]; then the slice sums [S][TI][MR]
  constexpr int U = MR <= 2 ? 8 : 4;              // entries loaded ahead of their FMAs
  const long long cell = blockIdx.x / ntile;
  const int i0 = (int)(blockIdx.x - cell * ntile) * TI;
  const double* xc = x + cell * x_cs;
#pragma unroll
  for (int r = 0; r < MR; ++r)
    for (int j = threadIdx.x; j < nin; j += blockDim.x) gvs[j * MR + r] = xc[r * x_rs + j];
  __syncthreads();
  const int il = threadIdx.x % TI, sl = threadIdx.x / TI;
  const bool live = sl < S && i0 + il < nout;
  double acc[MR];
#pragma unroll
  for (int r = 0; r < MR; ++r) acc[r] = 0.0;
  if (live) {
    const double* M = mats + cell * mstride + i0 + il;
    int j = sl;
    for (; j + (U - 1) * S < nin; j += U * S) {
      double mv[U];
#pragma unroll
      for (int u = 0; u < U; ++u) mv[u] = __ldcs(M + (long long)(j + u * S) * ld);
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int r = 0; r < MR; ++r) acc[r] = fma(mv[u], gvs[(j + u * S) * MR + r], acc[r]);
    }
    for (; j < nin; j += S) {
      const double mv = __ldcs(M + (long long)j * ld);
#pragma unroll
      for (int r = 0; r < MR; ++r) acc[r] = fma(mv, gvs[j * MR + r], acc[r]);
    }
  }
  __syncthreads();                                // x is no longer read
  if (sl < S)
#pragma unroll
    for (int r = 0; r < MR; ++r) gvs[(sl * TI + il) * MR + r] = acc[r];
  __syncthreads();
  for (int t = threadIdx.x; t < TI * MR; t += blockDim.x) {
    const int r = t / TI, i = t - r * TI;
    if (i0 + i >= nout) continue;
    double s = gvs[i * MR + r];
    for (int q = 1; q < S; ++q) s += gvs[(q * TI + i) * MR + r];
    double* dst = y + r * y_rs + cell * y_cs + i0 + i;
    *dst = (beta == 0.0) ? alpha * s : alpha * s + beta * (*dst);
  }
}

// Narrow per-cell operators with a compile-time column count MC (n_p: 8 in 2D, 24 in 3D): one
// thread per (cell, row); the row's MC entries arrive as 16-byte loads issued before any use, so
// each thread waits for memory once.  Rows must be 16-byte aligned (ld and the base even).
template <int MC>
__global__ void cell_gemv_narrow_fixed(const double* __restrict__ mats, long long mstride, int ld, int mrows,
                                       const double* __restrict__ x, long long x_rs, int x_cs,
                                       double* __restrict__ y, long long y_rs, int y_cs, double alpha,
                                       double beta, int nrhs, long long ncell) {
  const int total = (int)(ncell * mrows);             // < 2^31, checked by the host
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
    const int cell = t / mrows;
    const int row = t - cell * mrows;
    const double2* Mr = reinterpret_cast<const double2*>(mats + (long long)cell * mstride + (long long)row * ld);
    double mv[MC];
#pragma unroll
    for (int q = 0; q < MC / 2; ++q) {
      const double2 v = Mr[q];
      mv[2 * q] = v.x;
      mv[2 * q + 1] = v.y;
    }
    for (int r = 0; r < nrhs; ++r) {
      const double* xc = x + r * x_rs + (long long)cell * x_cs;
      double acc = 0.0;
#pragma unroll
      for (int q = 0; q < MC; ++q) acc = fma(mv[q], xc[q], acc);
      double* dst = y + r * y_rs + (long long)cell * y_cs + row;
      *dst = (beta == 0.0) ? alpha * acc : alpha * acc + beta * (*dst);
    }
  }
}

// Narrow per-cell operators (at most 32 columns, e.g. the n_r x n_p prolongations): one thread
// per (cell, row), so consecutive threads read consecutive rows; x entries are shared by the
// threads of a cell (cache broadcast).
__global__ void cell_gemv_narrow_kernel(const double* __restrict__ mats, long long mstride, int ld,
                                        int mrows, int mcols, const double* __restrict__ x, long long x_rs,
                                        int x_cs, double* __restrict__ y, long long y_rs, int y_cs,
                                        double alpha, double beta, int nrhs, long long ncell) {
  const long long total = ncell * mrows;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const long long cell = t / mrows;
    const int row = (int)(t - cell * mrows);
    const double* Mr = mats + cell * mstride + (long long)row * ld;
    for (int r0 = 0; r0 < nrhs; r0 += kMaxRhsGemv) {
      const int rb = min(kMaxRhsGemv, nrhs - r0);
      double acc[kMaxRhsGemv];
#pragma unroll
      for (int r = 0; r < kMaxRhsGemv; ++r) acc[r] = 0.0;
      for (int q = 0; q < mcols; ++q) {
        const double mv = Mr[q];
#pragma unroll
        for (int r = 0; r < kMaxRhsGemv; ++r)
          if (r < rb) acc[r] += mv * x[(r0 + r) * x_rs + cell * x_cs + q];
      }
#pragma unroll
      for (int r = 0; r < kMaxRhsGemv; ++r) {
        if (r < rb) {
          double* dst = y + (r0 + r) * y_rs + cell * y_cs + row;
          *dst = (beta == 0.0) ? alpha * acc[r] : alpha * acc[r] + beta * (*dst);
        }
      }
    }
  }
}

// ---- assembled per-cell ROM operators in FP32 (mixed path, large cells)
// F_dd_ring^(s) = sum_k delta_k F_dd^(sigma_k) and S_dd_ring^(s) = sum_k alpha_k S_dd^(sigma_k)
// (Eqs. 43, 48, 49) formed once per setup.  Applying the principal form costs 2 N_rb n_d^2 flops
// per column (three BF16 products with the hi/lo split); the assembled operator costs 4 n_d^2
// bytes per cell, shared by the cell's m columns.  At n_d = 630 the streamed operator is the
// cheaper of the two on GB300, and it is HBM-bound.

// out[cell][r][c] (FP32; ldo entries per row, in blocks of blkw columns whose rows follow each other, or
// plain rows when blkw = 0) = sum_k coef[cell][k] src[k][(r0 + r) * ld + c0 + c].
// A thread owns one entry (r, c): its NRBM principal values sit in registers and are reused for
// kCombCells cells, whose coefficients are staged in shared memory (FP32 arithmetic).
constexpr int kCombCells = 32;
// symT > 0: the output is the packed symmetric tile form (upper-triangle 32 x 32 tiles of a
// symT x symT tile grid, sym_tile_offset) and entries below the diagonal tiles are not written.
__host__ __device__ inline long long sym_tile_index(int I, int J, int T) {
  return (long long)I * T - (long long)I * (I - 1) / 2 + (J - I);
}
// element (r, c) of a 32 x 32 tile: quad c / 4 of row r at float4 slot 32 (c / 4) + r, so a warp
// whose lane r loads quad k reads 512 contiguous bytes
__host__ __device__ inline int sym_in_tile(int r, int c) { return (((c >> 2) * 32 + r) << 2) + (c & 3); }
template <int NRBM>
__global__ void __launch_bounds__(256) rom_combine_f32_kernel(const double* __restrict__ src, long long kstride,
                                                              int ld, int r0, int c0, int rows, int cols,
                                                              const double* __restrict__ coef, int nrb,
                                                              long long ncell, float* __restrict__ out, int ldo,
                                                              int blkw, int symT) {
  __shared__ float cs[kCombCells][NRBM];
  const long long per = (long long)rows * cols;
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const int r_ = t < per ? (int)(t / cols) : 0, c_ = t < per ? (int)(t - (long long)r_ * cols) : 0;
  const bool live = t < per && (symT == 0 || (r_ >> 5) <= (c_ >> 5));
  const int r = r_, cc = c_;
  const long long cell_stride = symT ? 1024LL * symT * (symT + 1) / 2 : (long long)rows * ldo;
  const long long eoff = symT ? 1024LL * sym_tile_index(r >> 5, cc >> 5, symT) + sym_in_tile(r & 31, cc & 31)
                         : blkw ? (long long)(cc / blkw) * blkw * rows +
                                      (long long)r * min(blkw, ldo - cc / blkw * blkw) + cc % blkw
                                : (long long)r * ldo + cc;
  float p[NRBM];
#pragma unroll
  for (int k = 0; k < NRBM; ++k)
    p[k] = (live && k < nrb) ? (float)src[k * kstride + (long long)(r0 + r) * ld + c0 + cc] : 0.f;
  for (long long cell0 = (long long)blockIdx.y * kCombCells; cell0 < ncell; cell0 += (long long)gridDim.y * kCombCells) {
    const int nc = (int)min((long long)kCombCells, ncell - cell0);
    __syncthreads();
    for (int q = threadIdx.x; q < kCombCells * NRBM; q += blockDim.x) {
      const int ci = q / NRBM, k = q - ci * NRBM;
      cs[ci][k] = (ci < nc && k < nrb) ? (float)coef[(cell0 + ci) * nrb + k] : 0.f;
    }
    __syncthreads();
    if (!live) continue;
    for (int ci = 0; ci < nc; ++ci) {
      float acc = 0.f;
#pragma unroll
      for (int k = 0; k < NRBM; ++k) acc = fmaf(cs[ci][k], p[k], acc);
      out[(cell0 + ci) * cell_stride + eoff] = acc;
    }
  }
}

// y[rhs][cell][0..nout) = alpha M[cell]^T x[rhs][cell][0..nin) + beta y for per-cell FP32 matrices M[cell] of
// nin stored rows: row j of M multiplies x_j (M x for the symmetric F_dd_ring and S_dd_ring).  Bound: HBM --
// every entry is read once and feeds MR FMAs.  The operator is stored in blocks of at most 128 outputs,
// each block's rows in sequence, so one warp (a CTA of its own) streams one block of one cell contiguously;
// a lane owns V outputs and copies its own 4 V bytes of every row into its own slots of a shared-memory
// ring, kRing rows ahead of the FMAs, without any synchronisation beyond its own cp.async groups.  24 KB in
// flight per warp (the 16-byte register loads it replaces kept 4 KB, and waited for each batch) need few
// warps per SM, and the unit of work, a block, is a fifth of a 6^3 cell: lattices of a few hundred cells
// fill the SMs evenly.  Copy groups of 16 rows: a wait costs a warp about as much as the FMAs of 4 rows (32
// cells, 6 RHS: 48.6, 33.5, 28 us with groups of 4, 8, 16).  With fewer than two warps per SM the lanes own
// 2 or 1 outputs instead of 4 (24 cells: 17 us against 24; 32 cells: 22 against 28).
// x comes interleaved by RHS in FP32 ([j][P], gathered or packed that way), read as 16-byte broadcasts.
// Every output is one chain of FMAs over ascending j, as before.
// Measured, n_d = 630, before and now: 2,048 cells, 6 RHS 657 -> 502 us (6.7 TB/s of operator and vectors);
// 864 cells, 1 RHS 249 -> 210 us; 256 cells, 6 RHS 110 -> 78 us; 50 cells, 3 RHS 100 -> 22 us.
constexpr int kMaxRhsF32 = 8;
constexpr int kRing = 48, kRingG = 16;            // rows in flight, rows per copy group
template <int MR, int P, int V, typename TO>
__global__ void __launch_bounds__(32) cell_gemm_f32_kernel(const float* __restrict__ mats, int ldm, int nout, int nin,
                                                           int W, int nb, const float* __restrict__ xf, int xcs,
                                                           TO* __restrict__ y, long long y_rs, int y_cs,
                                                           double alpha, double beta, int nrhs) {
  extern __shared__ __align__(16) float gsm[];    // x [nin][P], padded to 16 bytes; then the ring
  constexpr int NG = kRing / kRingG;
  const int lane = threadIdx.x;
  const long long cell = blockIdx.x / nb;
  const int b = (int)(blockIdx.x - cell * nb);
  const int xn = (nin * P + 3) >> 2;              // 16-byte pieces of x
  const int w = min(W, ldm - b * W);              // the block's row stride
  const bool live = V * lane < w;
  // lanes past the block's width copy and compute its first outputs again (nothing is stored for them)
  const float* M = mats + cell * (long long)nin * ldm + (long long)b * W * nin + (live ? V * lane : 0);
  float* ring = gsm + 4 * xn + lane * V;
  auto copy = [](float* dst, const float* src, auto bytes) {
    constexpr int B = decltype(bytes)::value;
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    if (B == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(d), "l"(src), "n"(B) : "memory");
  };
  for (int t = lane; t < xn; t += 32)
    copy(gsm + 4 * t, xf + cell * xcs + 4 * t, std::integral_constant<int, 16>());
  asm volatile("cp.async.commit_group;\n" ::: "memory");
  auto issue = [&](int j0) {                      // rows j0 .. j0 + kRingG - 1 into their slots
    const float* src = M + (long long)j0 * w;
    float* dst = ring + (j0 % kRing) * 32 * V;
    if (j0 + kRingG <= nin) {
#pragma unroll
      for (int u = 0; u < kRingG; ++u) copy(dst + u * 32 * V, src + (long long)u * w, std::integral_constant<int, 4 * V>());
    } else {
      for (int u = 0; j0 + u < nin; ++u) copy(dst + u * 32 * V, src + (long long)u * w, std::integral_constant<int, 4 * V>());
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
#pragma unroll
  for (int g = 0; g < NG; ++g) issue(g * kRingG);
  asm volatile("cp.async.wait_group %0;\n" ::"n"(NG) : "memory");
  __syncwarp();                                   // every lane's part of x is in place
  float acc[V][MR];
#pragma unroll
  for (int a = 0; a < V; ++a)
#pragma unroll
    for (int q = 0; q < MR; ++q) acc[a][q] = 0.f;
  auto row = [&](const float* m, const float* x) {
    float mv[V], xv[P];
    if constexpr (V == 4) {
      const float4 t = *reinterpret_cast<const float4*>(m);
      mv[0] = t.x; mv[1] = t.y; mv[2] = t.z; mv[3] = t.w;
    } else if constexpr (V == 2) {
      const float2 t = *reinterpret_cast<const float2*>(m);
      mv[0] = t.x; mv[1] = t.y;
    } else {
      mv[0] = *m;
    }
    if constexpr (P >= 4) {
#pragma unroll
      for (int q = 0; q < P; q += 4) {
        const float4 t = *reinterpret_cast<const float4*>(x + q);
        xv[q] = t.x; xv[q + 1] = t.y; xv[q + 2] = t.z; xv[q + 3] = t.w;
      }
    } else {
#pragma unroll
      for (int q = 0; q < P; ++q) xv[q] = x[q];
    }
#pragma unroll
    for (int a = 0; a < V; ++a)
#pragma unroll
      for (int q = 0; q < MR; ++q) acc[a][q] = fmaf(mv[a], xv[q], acc[a][q]);
  };
  for (int j0 = 0; j0 < nin; j0 += kRingG) {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(NG - 1) : "memory");
    const float* m = ring + (j0 % kRing) * 32 * V;
    const float* x = gsm + j0 * P;
    if (j0 + kRingG <= nin) {
#pragma unroll
      for (int u = 0; u < kRingG; ++u) row(m + u * 32 * V, x + u * P);
    } else {
      for (int u = 0; j0 + u < nin; ++u) row(m + u * 32 * V, x + u * P);
    }
    issue(j0 + kRing);                            // the slots just read
  }
  if (!live) return;
  const int r0 = b * W + V * lane;
#pragma unroll
  for (int a = 0; a < V; ++a) {
    if (r0 + a >= nout) continue;
#pragma unroll
    for (int q = 0; q < MR; ++q) {
      if (q >= nrhs) break;
      TO* dst = y + q * y_rs + cell * y_cs + r0 + a;
      if constexpr (sizeof(TO) == 4) *dst = acc[a][q];   // alpha = 1, beta = 0
      else *dst = (beta == 0.0) ? alpha * (double)acc[a][q] : alpha * (double)acc[a][q] + beta * (*dst);
    }
  }
}

// y = alpha M x + beta y for the SYMMETRIC per-cell operators stored as packed upper-triangle tiles
// (32 x 32, T tile rows, sym_in_tile layout): every stored tile (I, J), I < J, is read from memory
// once and used twice, y_I += M_IJ x_J and y_J += M_IJ^T x_I; a diagonal tile gives y_I += M_II x_I.
// One CTA per cell with T'/2 warps (T' = T rounded up to even).  The off-diagonal tiles are visited
// in the T' - 1 rounds of the circle schedule -- in each round the warps hold disjoint block pairs,
// so every y block has one writer per round and the summation order is fixed (deterministic, no
// atomics) -- then the diagonal tiles.  A warp loads its tile with lane r owning row r (eight
// 16-byte loads of 512 contiguous bytes) and the next round's tile while it computes; the column
// products read the tile transposed through a 32 x 33 shared buffer.  x and y are staged in
// shared memory in FP32 ([row][8] and [row][9]), up to eight RHS at a time.
__device__ __forceinline__ bool sym_round_pair(int round, int w, int Tp, int T, int& I, int& J) {
  int a, b;
  if (w == 0) {
    a = round;
    b = Tp - 1;
  } else {
    a = (round + w) % (Tp - 1);
    b = (round - w + (Tp - 1)) % (Tp - 1);
  }
  I = min(a, b);
  J = max(a, b);
  return J < T;                                   // block T of an odd T is the empty pad block
}
__global__ void __launch_bounds__(320, 2) cell_symv_f32_kernel(const float* __restrict__ mats, int T, int n,
                                                               const double* __restrict__ x, long long x_rs,
                                                               int x_cs, double* __restrict__ y, long long y_rs,
                                                               int y_cs, double alpha, double beta, int nrhs) {
  extern __shared__ __align__(16) float symsm[];
  const int NP = T * 32;
  float* xs = symsm;                              // [NP][8]
  float* ys = xs + (size_t)NP * 8;                // [NP][9]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  float* tb = ys + (size_t)NP * 9 + (size_t)warp * 32 * 33;
  const int Tp = (T + 1) & ~1;
  const long long cell = blockIdx.x;
  const float4* Mc = reinterpret_cast<const float4*>(mats + cell * 1024LL * T * (T + 1) / 2);
  const int nrounds = Tp - 1;
  for (int rb0 = 0; rb0 < nrhs; rb0 += 8) {
    const int rb = min(8, nrhs - rb0);
    __syncthreads();
    for (int t = tid; t < NP * 8; t += blockDim.x) {
      const int q = t / NP, j = t - q * NP;
      xs[j * 8 + q] = (q < rb && j < n) ? (float)x[(rb0 + q) * x_rs + cell * x_cs + j] : 0.f;
    }
    for (int t = tid; t < NP * 9; t += blockDim.x) ys[t] = 0.f;
    __syncthreads();
    // rounds 0 .. nrounds-1: off-diagonal pairs; round nrounds + s: diagonal tiles w + s * nw
    int I, J;
    bool have = nrounds > 0 ? sym_round_pair(0, warp, Tp, T, I, J) : false;
    float4 m[8];
    if (have)
#pragma unroll
      for (int k = 0; k < 8; ++k) m[k] = __ldcs(Mc + sym_tile_index(I, J, T) * 256 + k * 32 + lane);
    const int ndiag_steps = (T + nw - 1) / nw;
    for (int step = 0; step < nrounds + ndiag_steps; ++step) {
      // the next step's tile, loaded before this one is used
      int In = 0, Jn = 0;
      bool have_n = false;
      if (step + 1 < nrounds) have_n = sym_round_pair(step + 1, warp, Tp, T, In, Jn);
      else if (step + 1 < nrounds + ndiag_steps) {
        In = Jn = warp + (step + 1 - nrounds) * nw;
        have_n = In < T;
      }
      float4 mn[8];
      if (have_n)
#pragma unroll
        for (int k = 0; k < 8; ++k) mn[k] = __ldcs(Mc + sym_tile_index(In, Jn, T) * 256 + k * 32 + lane);
      if (have) {
        // y_I[lane] += sum_c M[lane][c] x_J[c]
        float ar[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        const float4* xJ = reinterpret_cast<const float4*>(xs + (size_t)J * 32 * 8);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const float mv[4] = {m[k].x, m[k].y, m[k].z, m[k].w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float4 x0 = xJ[(4 * k + e) * 2], x1 = xJ[(4 * k + e) * 2 + 1];
            ar[0] = fmaf(mv[e], x0.x, ar[0]);
            ar[1] = fmaf(mv[e], x0.y, ar[1]);
            ar[2] = fmaf(mv[e], x0.z, ar[2]);
            ar[3] = fmaf(mv[e], x0.w, ar[3]);
            ar[4] = fmaf(mv[e], x1.x, ar[4]);
            ar[5] = fmaf(mv[e], x1.y, ar[5]);
            ar[6] = fmaf(mv[e], x1.z, ar[6]);
            ar[7] = fmaf(mv[e], x1.w, ar[7]);
          }
        }
        float* yI = ys + (size_t)(I * 32 + lane) * 9;
#pragma unroll
        for (int q = 0; q < 8; ++q) yI[q] += ar[q];
        if (I != J) {
          // y_J[lane] += sum_r M[r][lane] x_I[r], column lane of the tile through the buffer
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            tb[lane * 33 + 4 * k] = m[k].x;
            tb[lane * 33 + 4 * k + 1] = m[k].y;
            tb[lane * 33 + 4 * k + 2] = m[k].z;
            tb[lane * 33 + 4 * k + 3] = m[k].w;
          }
          __syncwarp();
          float ac[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
          const float4* xI = reinterpret_cast<const float4*>(xs + (size_t)I * 32 * 8);
#pragma unroll 8
          for (int r = 0; r < 32; ++r) {
            const float tv = tb[r * 33 + lane];
            const float4 x0 = xI[r * 2], x1 = xI[r * 2 + 1];
            ac[0] = fmaf(tv, x0.x, ac[0]);
            ac[1] = fmaf(tv, x0.y, ac[1]);
            ac[2] = fmaf(tv, x0.z, ac[2]);
            ac[3] = fmaf(tv, x0.w, ac[3]);
            ac[4] = fmaf(tv, x1.x, ac[4]);
            ac[5] = fmaf(tv, x1.y, ac[5]);
            ac[6] = fmaf(tv, x1.z, ac[6]);
            ac[7] = fmaf(tv, x1.w, ac[7]);
          }
          __syncwarp();                           // the buffer is rewritten by the next tile
          float* yJ = ys + (size_t)(J * 32 + lane) * 9;
#pragma unroll
          for (int q = 0; q < 8; ++q) yJ[q] += ac[q];
        }
      }
      __syncthreads();                            // this round's y blocks are complete
      have = have_n;
      I = In;
      J = Jn;
#pragma unroll
      for (int k = 0; k < 8; ++k) m[k] = mn[k];
    }
    const bool plain = alpha == 1.0, overwrite = beta == 0.0;
    for (int t = tid; t < n * 8; t += blockDim.x) {
      const int q = t / n, r = t - q * n;
      if (q >= rb) continue;
      double* dst = y + (rb0 + q) * y_rs + cell * y_cs + r;
      const double v = plain ? (double)ys[r * 9 + q] : alpha * (double)ys[r * 9 + q];
      *dst = overwrite ? v : v + beta * (*dst);
    }
  }
}

// Coarse restriction and prolongation of the inner iterations (the coarse term of Eq. 48) with the
// FP32 copy of U_dp_ring (the dual rows of U_rp_ring), [cell][n_d][NP] row-major:
//   udp_t:  cp[rhs][cell][p] = sum_d U[d][p] g[rhs][cell][d]
//   udp_n:  y[rhs][cell][d]  = y[rhs][cell][d] + sum_p U[d][p] cp[rhs][cell][p]
// Bound: HBM (U once, the vectors).  The sum over d keeps its order: RG = 256 / (NP / 4) interleaved chains of
// FMAs, then their sums in sequence.  udp_t runs one CTA per cell, a thread four consecutive p of one chain
// (its first rows loaded before x is staged), MR sums each, the chains added through shared memory; where
// every chain has one row (n_d <= RG, 2D cells up to 17^2 elements) it is one thread per (cell, p) and no
// barrier.  udp_n is one thread per (cell, d) for the RHS of a chunk.
// 2,048 cells of n_d = 630 and 6 RHS: udp_t 100 -> 32 us, udp_n 100 -> 49; 864 cells, 1 RHS: 37 -> 12 and 41 -> 13;
// 4,096 cells of n_d = 120, 1 RHS: 58 -> 20 and 23 -> 6.5 us.
template <int NP, int MR, int P>
__global__ void __launch_bounds__(256) udp_t_f32_kernel(const float* __restrict__ U, int nd, XfLayout xf,
                                                        double* __restrict__ cp, long long c_rs, int c_cs,
                                                        int nrhs) {
  constexpr int G = NP / 4;          // 16-byte groups per row
  constexpr int RG = 256 / G;        // row groups
  constexpr int UB = 8;              // rows loaded ahead of their FMAs, the first batch ahead of the staging
  extern __shared__ __align__(16) float smu[];   // gs[nd][P] (16-byte padded), red[RG * G][4 MR]
  float* gs = smu;
  float* red = smu + (((size_t)nd * P + 3) & ~(size_t)3);
  const long long cell = blockIdx.x;
  const int tid = threadIdx.x;
  const int grp = tid % G, rg = tid / G;
  const float4* Uc = reinterpret_cast<const float4*>(U + cell * (long long)nd * NP) + grp;
  float4 u[UB];
#pragma unroll
  for (int k = 0; k < UB; ++k)
    u[k] = rg < RG && rg + k * RG < nd ? __ldcs(Uc + (long long)(rg + k * RG) * G) : make_float4(0.f, 0.f, 0.f, 0.f);
  const float* xc = xf.p + cell * xf.cs;
  if (xf.ds == P) {
#pragma unroll 4
    for (int t = tid; t < (nd * P + 3) / 4; t += blockDim.x)
      reinterpret_cast<float4*>(gs)[t] = __ldg(reinterpret_cast<const float4*>(xc) + t);
  } else {
    for (int t = tid; t < nd * P; t += blockDim.x) gs[t] = t % P < nrhs ? xc[t / P * xf.ds + t % P * xf.rs] : 0.f;
  }
  __syncthreads();
  float acc[4][MR];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int q = 0; q < MR; ++q) acc[a][q] = 0.f;
  if (rg < RG) {
    for (int d0 = rg; d0 < nd; d0 += UB * RG) {
      if (d0 != rg)
#pragma unroll
        for (int k = 0; k < UB; ++k)
          u[k] = d0 + k * RG < nd ? __ldcs(Uc + (long long)(d0 + k * RG) * G) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int k = 0; k < UB; ++k) {
        const int d = d0 + k * RG;
        if (d >= nd) break;
        const float uv[4] = {u[k].x, u[k].y, u[k].z, u[k].w};
        const float* x = gs + d * P;
#pragma unroll
        for (int q = 0; q < MR; ++q) {
          const float xq = x[q];
#pragma unroll
          for (int a = 0; a < 4; ++a) acc[a][q] = fmaf(uv[a], xq, acc[a][q]);
        }
      }
    }
    float* rd = red + (size_t)(rg * G + grp) * 4 * MR;
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int q = 0; q < MR; ++q) rd[a * MR + q] = acc[a][q];
  }
  __syncthreads();
  for (int o = tid; o < NP * MR; o += blockDim.x) {
    const int p = o / MR, q = o - p * MR;
    float sum = 0.f;
#pragma unroll 14
    for (int k = 0; k < RG; ++k) sum += red[(size_t)(k * G + (p >> 2)) * 4 * MR + (p & 3) * MR + q];
    if (q < nrhs) cp[q * c_rs + cell * c_cs + p] = fd_widen(sum);
  }
}

template <int NP>
__global__ void __launch_bounds__(128) udp_t_short_f32_kernel(const float* __restrict__ U, int nd, XfLayout xf,
                                                              double* __restrict__ cp, long long c_rs, int c_cs,
                                                              int nrhs, long long ncell) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long cell = t / NP;
  const int p = (int)(t - cell * NP);
  if (cell >= ncell) return;
  const float* Uc = U + cell * (long long)nd * NP + p;
  for (int q = 0; q < nrhs; ++q) {
    const float* x = xf.p + cell * xf.cs + q * xf.rs;
    float tot = 0.f;
    int d = 0;
    for (; d + 8 <= nd; d += 8) {
      float u[8], v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        u[k] = __ldg(Uc + (d + k) * NP);
        v[k] = __ldg(x + (d + k) * xf.ds);
      }
#pragma unroll
      for (int k = 0; k < 8; ++k) tot = __fadd_rn(tot, __fmul_rn(u[k], v[k]));   // a chain's sum is its one product
    }
    for (; d < nd; ++d) tot = __fadd_rn(tot, __fmul_rn(__ldg(Uc + d * NP), __ldg(x + d * xf.ds)));
    cp[q * c_rs + cell * c_cs + p] = fd_widen(tot);
  }
}

// With cvt, mul and fma on the FP64 pipe the epilogue bound the kernel (111 of 101-120 us at 2,048 cells and 6
// RHS): the sums are widened by integer instructions and one FP64 addition is left.  cp comes rounded to
// FP32, [cell][NP][8] (broadcast reads); yin is the FP32 or FP64 vector the product is added to.
template <int NP, int MR, typename TI>
__global__ void __launch_bounds__(128) udp_n_f32_kernel(const float* __restrict__ U, int nd,
                                                        const float* __restrict__ cpf, const TI* yin,
                                                        long long yi_rs, int yi_cs, double* y, long long y_rs,
                                                        int y_cs, int nrhs, long long ncell) {
  constexpr int G = NP / 4;
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long cell = t / nd;
  const int d = (int)(t - cell * nd);
  if (cell >= ncell) return;
  const float4* Uc = reinterpret_cast<const float4*>(U + t * NP);
  float4 u[G];
#pragma unroll
  for (int gq = 0; gq < G; ++gq) u[gq] = __ldcs(Uc + gq);
  TI y0[MR];
#pragma unroll
  for (int q = 0; q < MR; ++q) y0[q] = yin[min(q, nrhs - 1) * yi_rs + cell * yi_cs + d];
  const float4* cc = reinterpret_cast<const float4*>(cpf + cell * NP * 8);
  float acc[MR];
#pragma unroll
  for (int q = 0; q < MR; ++q) acc[q] = 0.f;
#pragma unroll
  for (int gq = 0; gq < G; ++gq) {
    const float uv[4] = {u[gq].x, u[gq].y, u[gq].z, u[gq].w};
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const float4 x0 = __ldg(cc + 2 * (4 * gq + a)), x1 = MR > 4 ? __ldg(cc + 2 * (4 * gq + a) + 1) : x0;
      const float xv[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
#pragma unroll
      for (int q = 0; q < MR; ++q) acc[q] = fmaf(uv[a], xv[q], acc[q]);
    }
  }
#pragma unroll
  for (int q = 0; q < MR; ++q)
    if (q < nrhs) y[q * y_rs + cell * y_cs + d] = fd_widen(acc[q]) + fd_load(y0[q]);
}

// Grouped FP64 GEMM, 64 x TN output tile per block (256 threads, 4 x TN/16 per thread), K chunks of 16.
// Bound: the FP64 pipe (2 FMA per clock and SM; 1 FMA per output and k), so a launch needs blocks on
// every SM and little padding: TN is the narrowest of 16, 32, 64 that holds the columns (32 columns on a
// 64-wide tile are half padding) and separate outputs take one principal per blockIdx.z.  With one block
// per tile running the principals one after the other, the 16 local bases of 32 cells of 6^3 elements
// and 6 RHS kept 48 blocks busy for 17 ms; they take 6.2 ms now (FP64 bound 4.9 ms).
constexpr int GT = 64, GK = 16;
template <int TN>
__global__ void __launch_bounds__(256) grouped_gemm_kernel(
    const double* __restrict__ A, long long a_stride_k, int lda, int M, int K, int nk,
    const double* __restrict__ X, long long x_rs, int x_cs, double* __restrict__ Y, long long y_rs,
    int y_cs, const double* __restrict__ coef, double alpha, double beta, long long ncell, int nrhs,
    bool separate, long long y_k_stride) {
  constexpr int NJ = TN / 16;
  __shared__ double As[GK][GT + 1];
  __shared__ double Xs[GK][TN + 1];
  const long long ncols = ncell * nrhs;
  const long long col0 = (long long)blockIdx.x * TN;
  const int m0 = blockIdx.y * GT;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;   // 16 x 16 threads
  const int kb = separate ? blockIdx.z : 0, ke = separate ? kb + 1 : nk;
  double tot[4][NJ];
  for (int i = 0; i < 4; ++i)
    for (int j = 0; j < NJ; ++j) tot[i][j] = 0.0;
  for (int k = kb; k < ke; ++k) {
    const double* Ak = A + k * a_stride_k;
    double acc[4][NJ];
    for (int i = 0; i < 4; ++i)
      for (int j = 0; j < NJ; ++j) acc[i][j] = 0.0;
    for (int kk0 = 0; kk0 < K; kk0 += GK) {
      for (int t = threadIdx.x; t < GK * GT; t += 256) {
        const int r = t / GK, q = t - r * GK;     // A: row r, k q  (q fastest -> coalesced rows)
        const int gm = m0 + r, gk = kk0 + q;
        As[q][r] = (gm < M && gk < K) ? Ak[(size_t)gm * lda + gk] : 0.0;
      }
      for (int t = threadIdx.x; t < GK * TN; t += 256) {
        const int r = t / GK, q = t - r * GK, gk = kk0 + q;
        const long long gc = col0 + r;            // X: column r, k q
        double xv = 0.0;
        if (gc < ncols && gk < K) {
          const int rhs = (int)(gc / ncell);
          const long long cell = gc - (long long)rhs * ncell;
          xv = X[rhs * x_rs + cell * x_cs + gk];
        }
        Xs[q][r] = xv;
      }
      __syncthreads();
#pragma unroll
      for (int q = 0; q < GK; ++q) {
        double a[4], b[NJ];
        for (int i = 0; i < 4; ++i) a[i] = As[q][ty + 16 * i];
        for (int j = 0; j < NJ; ++j) b[j] = Xs[q][tx + 16 * j];
        for (int i = 0; i < 4; ++i)
          for (int j = 0; j < NJ; ++j) acc[i][j] += a[i] * b[j];
      }
      __syncthreads();
    }
    if (separate) {
      for (int j = 0; j < NJ; ++j) {
        const long long gc = col0 + tx + 16 * j;
        if (gc >= ncols) continue;
        const int rhs = (int)(gc / ncell);
        const long long cell = gc - (long long)rhs * ncell;
        double* yc = Y + k * y_k_stride + rhs * y_rs + cell * y_cs;
        for (int i = 0; i < 4; ++i) {
          const int gm = m0 + ty + 16 * i;
          if (gm < M) yc[gm] = alpha * acc[i][j];
        }
      }
    } else {
      for (int j = 0; j < NJ; ++j) {
        const long long gc = col0 + tx + 16 * j;
        double cf = 1.0;
        if (coef != nullptr && gc < ncols) {
          const long long cell = gc % ncell;
          cf = coef[cell * nk + k];
        }
        for (int i = 0; i < 4; ++i) tot[i][j] += cf * acc[i][j];
      }
    }
  }
  if (!separate) {
    for (int j = 0; j < NJ; ++j) {
      const long long gc = col0 + tx + 16 * j;
      if (gc >= ncols) continue;
      const int rhs = (int)(gc / ncell);
      const long long cell = gc - (long long)rhs * ncell;
      double* yc = Y + rhs * y_rs + cell * y_cs;
      for (int i = 0; i < 4; ++i) {
        const int gm = m0 + ty + 16 * i;
        if (gm < M) yc[gm] = (beta == 0.0) ? alpha * tot[i][j] : alpha * tot[i][j] + beta * yc[gm];
      }
    }
  }
}

// One operator against every column, Y[col][m] = sum_k A[m][k] X[col][k] (the Eq. 42 traces), K summed
// in one chain of FMAs per output as the tiled kernel does: the traces of nearly dependent principal
// fields are solved by a pivoted Gram solve that amplifies a change of summation order by ~1e7, so K is
// not split.  The FP64 pipe takes 64 cycles per warp instruction and sub-partition, so a T x T tile of
// T^2 threads with one output each already keeps it busy (two 8-byte shared reads per FMA are hidden),
// and small tiles spread few outputs over all SMs: 288 traces of 32 cells were 5 blocks of 64 x 64 and
// 92 ms, now 4.4 ms (one chain of 77,760 FMAs: 2.4 ms); of 256 cells 94 ms, now 9.9 ms (FP64 bound 9.1).
constexpr int kTraceK = 32, kTraceLd = 33;   // row stride: a warp's 16 (or 8) rows hit different banks
template <int T>
__global__ void __launch_bounds__(T * T) trace_gemm_kernel(const double* __restrict__ A, int lda, int M, int K,
                                                           const double* __restrict__ X, long long x_cs,
                                                           double* __restrict__ Y, long long y_cs, long long ncols,
                                                           int mtiles) {
  __shared__ double As[2][T][kTraceLd], Xs[2][T][kTraceLd];
  // row tiles fastest; all tiles on blockIdx.x, whose range does not limit the number of cells
  const long long ct = blockIdx.x / mtiles, col0 = ct * T;
  const int m0 = (int)(blockIdx.x - ct * mtiles) * T;
  const int tx = threadIdx.x % T, ty = threadIdx.x / T;
  auto load = [&](int buf, int k0) {
    for (int t = threadIdx.x; t < 2 * T * kTraceK; t += T * T) {
      const int q = t % kTraceK, row = (t / kTraceK) % T, gk = k0 + q;
      const bool isx = t >= T * kTraceK;
      const long long g = isx ? col0 + row : m0 + row;
      const bool in = gk < K && g < (isx ? ncols : (long long)M);
      const double* src = isx ? X + (in ? g * x_cs + gk : 0) : A + (in ? g * lda + gk : 0);
      const unsigned d = (unsigned)__cvta_generic_to_shared(isx ? &Xs[buf][row][q] : &As[buf][row][q]);
      asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(d), "l"(src), "r"(in ? 8 : 0) : "memory");
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  double acc = 0.0;
  load(0, 0);
  for (int k0 = 0, buf = 0; k0 < K; k0 += kTraceK, buf ^= 1) {
    if (k0 + kTraceK < K) {
      load(buf ^ 1, k0 + kTraceK);
      asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kTraceK; ++q) acc = fma(As[buf][ty][q], Xs[buf][tx][q], acc);
    __syncthreads();                              // this buffer is refilled by the next iteration's load
  }
  if (m0 + ty < M && col0 + tx < ncols) Y[(col0 + tx) * y_cs + m0 + ty] = acc;
}

// Eq. 46b for one (rhs, cell) per warp.
//  1. G = R^T (K R) and h = R^T v.  G is formed in 32 x 32 blocks (upper blocks only, then
//     mirrored): lane r owns row r of the block.  Chunks of 32 entries of the basis vectors are
//     staged in shared memory, the R rows with a padded stride (each lane reads its own row,
//     conflict-free) and the K R chunk transposed with 16-byte rows (all lanes read the same
//     address: broadcast, four values per load).  Products in the basis type, chunk sums in FP64.
//  2. Diagonal-pivoted Cholesky, right-looking: each step takes the largest remaining Schur
//     diagonal (lowest index on ties), stops when it is not above drop_rel * max diag(G), stores
//     the scaled pivot column as the next column of L and applies the rank-1 update (lanes own
//     matrix columns, so the row-major updates are conflict-free).
//  3. L y = h(piv), L^T c(piv) = y (column-oriented, lane-parallel), c = 0 off the pivots,
//     and x = R c.
// Scratch per warp (doubles): S (nrb x (nrb + 1)), h, y, c, pivot column (nrb each), nrb pivot
// ints (in nrb doubles), 2 scalars, two v chunks (2 x 32), then one region shared by the two
// buffers of the two staging tiles (32 rows x kGramLd values of the basis type each; phase 1)
// and L (nrb x (nrb + 1); phase 2), padded to an even count.
constexpr int kMaxRb = 64;
constexpr int kGramQ = 32;     // basis-vector entries per staged chunk
constexpr int kGramLd = 36;    // row stride of a staged tile (16-byte rows, 4-bank row offset)
__host__ __device__ inline int gram_warp_head(int nrb) {
  const int fixed = nrb * (nrb + 1) + 5 * nrb + 2 + 2 * kGramQ;
  return fixed + (fixed & 1);   // the shared region starts 16-byte aligned
}
__host__ __device__ inline int gram_warp_doubles(int nrb, int tb_bytes) {
  const int tiles = (2 * 2 * kGramQ * kGramLd * tb_bytes + 7) / 8;
  const int lmat = nrb * (nrb + 1);
  const int tot = gram_warp_head(nrb) + (tiles > lmat ? tiles : lmat);
  return tot + (tot & 1);
}

// One element (4 or 8 bytes) global -> shared without waiting; zero-filled when !valid.
template <typename TB>
__device__ __forceinline__ void cp_async_elem(TB* dst, const TB* src, bool valid) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  const int n = valid ? (int)sizeof(TB) : 0;
  if (sizeof(TB) == 8)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(d), "l"(src), "r"(n) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(d), "l"(src), "r"(n) : "memory");
}

__device__ __forceinline__ void load4(const float* p, float (&o)[4]) {
  const float4 t = *reinterpret_cast<const float4*>(p);
  o[0] = t.x; o[1] = t.y; o[2] = t.z; o[3] = t.w;
}
__device__ __forceinline__ void load4(const double* p, double (&o)[4]) {
  const double2 t0 = *reinterpret_cast<const double2*>(p);
  const double2 t1 = *reinterpret_cast<const double2*>(p + 2);
  o[0] = t0.x; o[1] = t0.y; o[2] = t1.x; o[3] = t1.y;
}

// Diagonal-pivoted Cholesky solve of one symmetric nrb x nrb system by one warp, on the warp's
// shared scratch (row stride ld = nrb + 1): S holds G (overwritten), hs the right-hand side; the
// coefficients land in cs (0 off the pivots).  Each step takes the largest remaining Schur
// diagonal (lowest index on ties) and stops when it is not above drop_rel * max diag(G); the
// scaled pivot column is the next column of L and the rank-1 update runs with lanes over columns.
// Then L y = h(piv), L^T c(piv) = y, column-oriented and lane-parallel.
__device__ void warp_pivoted_gram_solve(double* S, double* Lc, const double* hs, double* ys, double* cs,
                                        double* colv, int* piv, int nrb, int ld, double drop_rel, int lane) {
  double dmax = 0.0;
  for (int i = 0; i < nrb; ++i) dmax = fmax(dmax, S[i * ld + i]);
  unsigned long long used = 0ull;                   // identical in every lane
  int np = 0;
  while (np < nrb) {
    // largest remaining Schur diagonal, lowest index on ties (lane-parallel, then a warp argmax)
    int jb = -1;
    double best = 0.0;
    for (int i = lane; i < nrb; i += 32) {
      if ((used >> i) & 1ull) continue;
      const double dv = S[i * ld + i];
      if (jb < 0 || dv > best) { best = dv; jb = i; }
    }
    for (int o = 16; o > 0; o >>= 1) {
      const double ob = __shfl_xor_sync(0xffffffffu, best, o);
      const int oj = __shfl_xor_sync(0xffffffffu, jb, o);
      if (oj >= 0 && (jb < 0 || ob > best || (ob == best && oj < jb))) { best = ob; jb = oj; }
    }
    if (jb < 0 || !(best > drop_rel * dmax)) break;   // uniform across the warp
    used |= 1ull << jb;
    if (lane == 0) piv[np] = jb;
    const double inv = 1.0 / sqrt(best);
    for (int i = lane; i < nrb; i += 32) {
      const double cv = S[i * ld + jb] * inv;
      colv[i] = cv;
      Lc[np * ld + i] = cv;
    }
    __syncwarp();
    for (int i = 0; i < nrb; ++i) {                    // lanes own columns j
      if ((used >> i) & 1ull) continue;                // pivoted rows are not read again
      const double ci = colv[i];
      for (int j = lane; j < nrb; j += 32) S[i * ld + j] -= ci * colv[j];
    }
    ++np;
    __syncwarp();
  }

  for (int i = lane; i < nrb; i += 32) { ys[i] = hs[i]; cs[i] = 0.0; }
  __syncwarp();
  for (int a = 0; a < np; ++a) {                       // forward: column a of L
    const int pa = piv[a];
    const double ya = ys[pa] / Lc[a * ld + pa];
    __syncwarp();
    for (int r = a + 1 + lane; r < np; r += 32) ys[piv[r]] -= Lc[a * ld + piv[r]] * ya;
    if (lane == 0) colv[a] = ya;                       // y in pivot order
    __syncwarp();
  }
  for (int a = np - 1; a >= 0; --a) {                  // backward: row a of L^T = column a of L
    const int pa = piv[a];
    const double ca = colv[a] / Lc[a * ld + pa];
    __syncwarp();
    for (int r = lane; r < a; r += 32) colv[r] -= Lc[r * ld + pa] * ca;
    if (lane == 0) cs[pa] = ca;
    __syncwarp();
  }
}

// The same diagonal-pivoted Cholesky solve by a whole CTA (nthreads threads, all of them calling):
// warp 0 picks the pivot, every thread forms part of the pivot column and of the rank-1 update,
// which touches only the upper triangle of the unpivoted rows and columns (S stays symmetric there;
// each entry receives the same FP64 operations in the same order as in the warp solve, and the
// pivot's scale is one rsqrt instead of a square root and a division, the step's latency on
// GB300's FP64 unit).  The substitutions run on warp 0.  sh holds a double and an int of
// block-shared scratch.  nthreads is a multiple of 64 and nrb <= 64.
__device__ void block_pivoted_gram_solve(double* S, double* Lc, const double* hs, double* ys, double* cs,
                                         double* colv, int* piv, double* sh_inv, int* sh_jb, int nrb, int ld,
                                         double drop_rel, int tid, int nthreads) {
  const int lane = tid & 31, warp = tid >> 5;
  double dmax = 0.0;                                 // needed by warp 0 only
  if (warp == 0) {
    for (int i = lane; i < nrb; i += 32) dmax = fmax(dmax, S[i * ld + i]);
    for (int o = 16; o > 0; o >>= 1) dmax = fmax(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
  }
  unsigned long long used = 0ull;                   // identical in every thread
  int np = 0;
  while (np < nrb) {
    if (warp == 0) {
      int jb = -1;
      double best = 0.0;
      for (int i = lane; i < nrb; i += 32) {
        if ((used >> i) & 1ull) continue;
        const double dv = S[i * ld + i];
        if (jb < 0 || dv > best) { best = dv; jb = i; }
      }
      for (int o = 16; o > 0; o >>= 1) {
        const double ob = __shfl_xor_sync(0xffffffffu, best, o);
        const int oj = __shfl_xor_sync(0xffffffffu, jb, o);
        if (oj >= 0 && (jb < 0 || ob > best || (ob == best && oj < jb))) { best = ob; jb = oj; }
      }
      if (lane == 0) {
        const bool take = jb >= 0 && best > drop_rel * dmax;
        *sh_jb = take ? jb : -1;
        if (take) { *sh_inv = rsqrt(best); piv[np] = jb; }   // one call on the pivot chain
      }
    }
    __syncthreads();
    const int jb = *sh_jb;
    if (jb < 0) break;                                 // uniform across the block
    const double inv = *sh_inv;
    used |= 1ull << jb;
    for (int i = tid; i < nrb; i += nthreads) {
      const double cv = S[min(i, jb) * ld + max(i, jb)] * inv;
      colv[i] = cv;
      Lc[np * ld + i] = cv;
    }
    __syncthreads();
    // nrb <= 64 and nthreads a multiple of 64: the thread's column j is fixed, its rows step by
    // nthreads / 64 up to the diagonal
    {
      const int j = tid & 63, rs = nthreads >> 6;
      if (j < nrb && !((used >> j) & 1ull)) {
        const double cj = colv[j];
        for (int i = tid >> 6; i <= j; i += rs)
          if (!((used >> i) & 1ull)) S[i * ld + j] -= colv[i] * cj;
      }
    }
    ++np;
    __syncthreads();
  }
  if (warp != 0) return;
  for (int i = lane; i < nrb; i += 32) { ys[i] = hs[i]; cs[i] = 0.0; }
  __syncwarp();
  for (int a = 0; a < np; ++a) {
    const int pa = piv[a];
    const double ya = ys[pa] / Lc[a * ld + pa];
    __syncwarp();
    for (int r = a + 1 + lane; r < np; r += 32) ys[piv[r]] -= Lc[a * ld + piv[r]] * ya;
    if (lane == 0) colv[a] = ya;
    __syncwarp();
  }
  for (int a = np - 1; a >= 0; --a) {
    const int pa = piv[a];
    const double ca = colv[a] / Lc[a * ld + pa];
    __syncwarp();
    for (int r = lane; r < a; r += 32) colv[r] -= Lc[r * ld + pa] * ca;
    if (lane == 0) cs[pa] = ca;
    __syncwarp();
  }
}

// s + c += x with Neumaier's compensation (c collects the rounding error of every addition)
template <typename T>
__device__ __forceinline__ void neumaier_add(T& s, T& c, T x) {
  if (sizeof(T) == 8) {   // FP64 sums need no compensation at these lengths
    s += x;
    return;
  }
  const T t = s + x;
  c += (fabs(s) >= fabs(x)) ? ((s - t) + x) : ((x - t) + s);
  s = t;
}

// Eq. 46b in FP32 for one (rhs, cell) per block of 256 threads: G = R^T (K R) and h = R^T v from
// 32-entry chunks of the basis staged in shared memory, each thread a strided 4 x 4 tile of G
// (rows ti + 16a, columns tj + 16b: a broadcast read of R and a conflict-free read of K R per
// product), FP32 chunk sums accumulated with Neumaier's compensation; then warp 0 runs the same
// diagonal-pivoted Cholesky solve as the warp kernel, and all threads form x = R c.
constexpr int kGbQ = 32;
constexpr int kGbLd = 36;   // 16-byte rows; a warp's 16 distinct K R rows take the minimum two wavefronts
// The two staging stages of R, K R and v (filled by cp.async one chunk ahead) live inside the L
// factor's region, used only after the Gram matrix is complete: a 64-basis block needs 74 KB and
// three blocks fit an SM.
__host__ __device__ inline size_t gram_block_stage_floats(int nrb) { return 2 * (size_t)nrb * kGbLd + kGbQ; }
__host__ __device__ inline size_t gram_block_smem(int nrb) {
  const size_t ld = (size_t)nrb + 1;
  const size_t stage = 2 * sizeof(float) * gram_block_stage_floats(nrb);
  const size_t lc = sizeof(double) * nrb * ld;
  return sizeof(double) * (nrb * ld + 6 * (size_t)nrb + 2) + (stage > lc ? stage : lc);
}
__global__ void __launch_bounds__(256, 3) gram_block_f32_kernel(const float* __restrict__ R, const float* __restrict__ KR,
                                                             const double* __restrict__ v, long long v_rs, int v_cs,
                                                             double* __restrict__ x, long long x_rs, int x_cs, int nr,
                                                             int nrb, long long ncell, double drop_rel) {
  extern __shared__ __align__(16) double gbsm[];
  const int ld = nrb + 1;
  double* S = gbsm;                                  // [nrb][ld]
  double* hs = S + (size_t)nrb * ld;
  double* ys = hs + nrb;
  double* cs = ys + nrb;
  double* colv = cs + nrb;
  int* piv = reinterpret_cast<int*>(colv + nrb);     // nrb ints in 2 nrb doubles of room
  double* sh_inv = colv + 3 * nrb;
  int* sh_jb = reinterpret_cast<int*>(sh_inv + 1);
  double* Lc = sh_inv + 2;                           // [nrb][ld], after the Gram matrix is formed
  float* stage0 = reinterpret_cast<float*>(Lc);      // two staging stages while it is formed
  const size_t stage_f = gram_block_stage_floats(nrb);
  const long long col = blockIdx.x;                  // rhs * ncell + cell
  const int rhs = (int)(col / ncell);
  const long long cell = col - (long long)rhs * ncell;
  const float* Rc = R + col * (long long)nrb * nr;
  const float* KRc = KR + col * (long long)nrb * nr;
  const double* vc = v + rhs * v_rs + cell * v_cs;
  const int tid = threadIdx.x, ti = tid >> 4, tj = tid & 15;
  float acc[4][4], cmp[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) { acc[a][b] = 0.f; cmp[a][b] = 0.f; }
  float hacc = 0.f, hcmp = 0.f;
  // chunk k of R and K R goes to stage k & 1 by cp.async (zero-filled past n_r), one chunk ahead
  auto issue = [&](int q0, float* st) {
    float* Rs_ = st;
    float* Ks_ = st + (size_t)nrb * kGbLd;
    for (int t = tid; t < nrb * kGbQ; t += blockDim.x) {
      const int i = t / kGbQ, qq = t - i * kGbQ, q = q0 + qq;
      const bool in = q < nr;
      cp_async_elem(Rs_ + i * kGbLd + qq, Rc + (size_t)i * nr + (in ? q : 0), in);
      cp_async_elem(Ks_ + i * kGbLd + qq, KRc + (size_t)i * nr + (in ? q : 0), in);
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  const int nchunk = (nr + kGbQ - 1) / kGbQ;
  issue(0, stage0);
  float part[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) part[a][b] = 0.f;
  float hp = 0.f;
  for (int ck = 0; ck < nchunk; ++ck) {
    const int q0 = ck * kGbQ;
    float* Rs = stage0 + (ck & 1) * stage_f;
    float* Ks = Rs + (size_t)nrb * kGbLd;
    float* vs = Ks + (size_t)nrb * kGbLd;
    if (ck + 1 < nchunk) {
      issue(q0 + kGbQ, stage0 + ((ck + 1) & 1) * stage_f);
      asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    }
    if (tid < kGbQ) vs[tid] = q0 + tid < nr ? (float)vc[q0 + tid] : 0.f;
    __syncthreads();                                  // chunk ck (and its v) is in place
#pragma unroll 2
    for (int qq = 0; qq < kGbQ; qq += 4) {
      float4 rv[4], kv[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const int i = ti + 16 * a, j = tj + 16 * a;
        rv[a] = i < nrb ? *reinterpret_cast<const float4*>(Rs + i * kGbLd + qq) : make_float4(0.f, 0.f, 0.f, 0.f);
        kv[a] = j < nrb ? *reinterpret_cast<const float4*>(Ks + j * kGbLd + qq) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          float p = part[a][b];
          p = fmaf(rv[a].x, kv[b].x, p);
          p = fmaf(rv[a].y, kv[b].y, p);
          p = fmaf(rv[a].z, kv[b].z, p);
          p = fmaf(rv[a].w, kv[b].w, p);
          part[a][b] = p;
        }
    }
    if (tid < nrb)
      for (int qq = 0; qq < kGbQ; ++qq) hp = fmaf(Rs[tid * kGbLd + qq], vs[qq], hp);
    // the partial sums of two chunks (64 terms) are added with Neumaier's compensation
    if ((ck & 1) || ck + 1 == nchunk) {
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          neumaier_add(acc[a][b], cmp[a][b], part[a][b]);
          part[a][b] = 0.f;
        }
      if (tid < nrb) neumaier_add(hacc, hcmp, hp);
      hp = 0.f;
    }
    __syncthreads();                                  // stage ck & 1 is refilled at chunk ck + 2
  }
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int i = ti + 16 * a, j = tj + 16 * b;
      if (i < nrb && j < nrb && i <= j) S[i * ld + j] = (double)acc[a][b] + (double)cmp[a][b];
    }
  if (tid < nrb) hs[tid] = (double)hacc + (double)hcmp;
  __syncthreads();
  for (int t = tid; t < nrb * nrb; t += blockDim.x) {   // the upper triangle, mirrored
    const int i = t / nrb, j = t - (t / nrb) * nrb;
    if (i > j) S[i * ld + j] = S[j * ld + i];
  }
  __syncthreads();
  block_pivoted_gram_solve(S, Lc, hs, ys, cs, colv, piv, sh_inv, sh_jb, nrb, ld, drop_rel, tid, blockDim.x);
  __syncthreads();
  float* csf = reinterpret_cast<float*>(ys);         // the coefficients in FP32, converted once
  if (tid < nrb) csf[tid] = (float)cs[tid];
  __syncthreads();
  double* xc = x + rhs * x_rs + cell * x_cs;
  for (int q = tid; q < nr; q += blockDim.x) {
    float sx = 0.f;
#pragma unroll 8
    for (int i = 0; i < nrb; ++i) sx = fmaf(csf[i], Rc[(size_t)i * nr + q], sx);
    xc[q] = (double)sx;
  }
}

template <typename TB>
__global__ void gram_warp_kernel(const TB* __restrict__ R, const TB* __restrict__ KR,
                                 const double* __restrict__ v, long long v_rs, int v_cs,
                                 double* __restrict__ x, long long x_rs, int x_cs, int nr, int nrb,
                                 long long ncell, int nrhs, double drop_rel) {
  extern __shared__ double gwsm[];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const long long col = (long long)blockIdx.x * (blockDim.x >> 5) + wib;
  if (col >= ncell * nrhs) return;                  // the whole warp leaves together
  const int ld = nrb + 1;
  double* S = gwsm + (size_t)wib * gram_warp_doubles(nrb, (int)sizeof(TB));
  double* hs = S + nrb * ld;
  double* ys = hs + nrb;
  double* cs = ys + nrb;
  double* colv = cs + nrb;
  int* piv = reinterpret_cast<int*>(colv + nrb);
  double* sc = colv + 2 * nrb;
  double* vq = sc + 2;                              // [2][32]: v chunks
  double* region = S + gram_warp_head(nrb);
  TB* Rs = reinterpret_cast<TB*>(region);           // phase 1: [2][32 rows][kGramLd]
  TB* Ks = Rs + 2 * kGramQ * kGramLd;               // phase 1: [2][32 rows][kGramLd]
  double* Lc = region;                              // phase 2: column a of L at Lc[a * ld + i]
  const int rhs = (int)(col / ncell);
  const long long cell = col - (long long)rhs * ncell;
  const TB* Rc = R + col * (long long)nrb * nr;
  const TB* KRc = KR + col * (long long)nrb * nr;
  const double* vc = v + rhs * v_rs + cell * v_cs;
  const int nchunk = (nr + kGramQ - 1) / kGramQ;

  // ---- 1. G (upper blocks) and h.  Rows of R and K R are staged chunk by chunk (row-major,
  // lane = entry q, one async copy per element), the next chunk in flight while this one is
  // used.  Lane j accumulates column j of the block: per row i and 4 entries one broadcast
  // 16-byte read of R and 4 FMAs against the lane's own K R values.
  for (int ib = 0; ib < nrb; ib += 32) {
    const int ni = min(32, nrb - ib);
    for (int jb = ib; jb < nrb; jb += 32) {
      const int nj = min(32, nrb - jb);
      const bool diag = (jb == ib);
      // chunk sums in the basis type, accumulated over chunks with Neumaier compensation (as
      // accurate as FP64 chunk sums, with no FP64 pipe work in the FP32 path)
      TB gacc[32], gcmp[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) { gacc[i] = TB(0); gcmp[i] = TB(0); }
      TB hacc = TB(0), hcmp = TB(0);
      auto stage = [&](int buf, int ch) {
        const int q = ch * kGramQ + lane;
        const bool in = q < nr;
        TB* rs = Rs + buf * kGramQ * kGramLd;
        TB* ks = Ks + buf * kGramQ * kGramLd;
        for (int r = 0; r < 32; ++r) {
          cp_async_elem(rs + r * kGramLd + lane, Rc + (size_t)(ib + (r < ni ? r : 0)) * nr + (in ? q : 0),
                        in && r < ni);
          cp_async_elem(ks + r * kGramLd + lane, KRc + (size_t)(jb + (r < nj ? r : 0)) * nr + (in ? q : 0),
                        in && r < nj);
        }
        if (diag) vq[buf * kGramQ + lane] = in ? vc[q] : 0.0;
        asm volatile("cp.async.commit_group;\n" ::: "memory");
      };
      __syncwarp();
      stage(0, 0);
      for (int ch = 0; ch < nchunk; ++ch) {
        const int buf = ch & 1;
        if (ch + 1 < nchunk) {
          stage(buf ^ 1, ch + 1);
          asm volatile("cp.async.wait_group 1;\n" ::: "memory");
        } else {
          asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        }
        __syncwarp();
        const TB* rs = Rs + buf * kGramQ * kGramLd;
        const TB* ks = Ks + buf * kGramQ * kGramLd;
        TB acc[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) acc[i] = TB(0);
#pragma unroll
        for (int q = 0; q < kGramQ; q += 4) {
          TB k4[4];
          load4(ks + lane * kGramLd + q, k4);
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            TB r4[4];
            load4(rs + i * kGramLd + q, r4);   // broadcast
            acc[i] = fma(r4[0], k4[0], acc[i]);
            acc[i] = fma(r4[1], k4[1], acc[i]);
            acc[i] = fma(r4[2], k4[2], acc[i]);
            acc[i] = fma(r4[3], k4[3], acc[i]);
          }
        }
#pragma unroll
        for (int i = 0; i < 32; ++i) neumaier_add(gacc[i], gcmp[i], acc[i]);
        if (diag) {   // h_i, lane i
          TB hsum = TB(0);
          for (int q = 0; q < kGramQ; ++q) hsum += rs[lane * kGramLd + q] * (TB)vq[buf * kGramQ + q];
          neumaier_add(hacc, hcmp, hsum);
        }
        __syncwarp();   // this buffer is refilled by the next stage call
      }
      if (lane < nj) {
#pragma unroll
        for (int i = 0; i < 32; ++i)
          if (i < ni && (!diag || i <= lane)) S[(ib + i) * ld + jb + lane] = (double)gacc[i] + (double)gcmp[i];
      }
      if (diag && lane < ni) hs[ib + lane] = (double)hacc + (double)hcmp;
    }
  }
  __syncwarp();
  for (int t = lane; t < nrb * nrb; t += 32) {      // mirror the upper triangle
    const int i = t / nrb, j = t - (t / nrb) * nrb;
    if (i > j) S[i * ld + j] = S[j * ld + i];
  }
  __syncwarp();

  warp_pivoted_gram_solve(S, Lc, hs, ys, cs, colv, piv, nrb, ld, drop_rel, lane);
  __syncwarp();
  double* xc = x + rhs * x_rs + cell * x_cs;
  for (int q = lane; q < nr; q += 32) {
    TB sx = TB(0);
    for (int i = 0; i < nrb; ++i) sx += (TB)cs[i] * Rc[(size_t)i * nr + q];
    xc[q] = (double)sx;
  }
}

// The two Eq. 42 systems of every cell from its traces Y[cell] = [A upper (npair), b (nrb),
// M upper (npair)]: pi solves A pi = b, delta solves M delta = dvec (shared right-hand side).
// One warp per (cell, system); same pivoted solve as Eq. 46b.
__global__ void gram_direct_kernel(const double* __restrict__ Y, int ntab, int nrb,
                                   const double* __restrict__ dvec, double* __restrict__ pi,
                                   double* __restrict__ delta, long long ncell, double drop_rel) {
  extern __shared__ double gdsm[];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const long long task = (long long)blockIdx.x * (blockDim.x >> 5) + wib;
  if (task >= 2 * ncell) return;                    // the whole warp leaves together
  const long long cell = task >> 1;
  const int sys = (int)(task & 1);                  // 0: pi, 1: delta
  const int ld = nrb + 1;
  const int per = 2 * nrb * ld + 6 * nrb;
  double* S = gdsm + (size_t)wib * (per + (per & 1));
  double* Lc = S + nrb * ld;
  double* hs = Lc + nrb * ld;
  double* ys = hs + nrb;
  double* cs = ys + nrb;
  double* colv = cs + nrb;
  int* piv = reinterpret_cast<int*>(colv + nrb);
  const int npair = nrb * (nrb + 1) / 2;
  const double* y = Y + cell * ntab;
  const double* g = y + (sys == 0 ? 0 : npair + nrb);
  for (int p = lane; p < npair; p += 32) {
    int i = 0, rem = p;
    while (rem >= nrb - i) { rem -= nrb - i; ++i; }
    const int j = i + rem;
    S[i * ld + j] = g[p];
    S[j * ld + i] = g[p];
  }
  for (int i = lane; i < nrb; i += 32) hs[i] = (sys == 0) ? y[npair + i] : dvec[i];
  __syncwarp();
  warp_pivoted_gram_solve(S, Lc, hs, ys, cs, colv, piv, nrb, ld, drop_rel, lane);
  __syncwarp();
  double* out = (sys == 0 ? pi : delta) + cell * nrb;
  for (int i = lane; i < nrb; i += 32) out[i] = cs[i];
}

// g[rhs][cell] = - sum_e sum_gp w G(w)^T dC_hat/dr G(u), one block per (rhs, cell).
template <int D>
__global__ void grad_kernel(Geo g, const double* __restrict__ r_cell, long long ncell, int n,
                            const double* __restrict__ u, const double* __restrict__ w, long long u_rs,
                            double* __restrict__ out, long long out_rs, double wq, double inv_h) {
  extern __shared__ double sm[];
  constexpr int NA = 1 << D;
  constexpr int NI = D * D;
  const long long col = blockIdx.x;
  const int rhs = (int)(col / ncell);
  const long long cell = col - (long long)rhs * ncell;   // cell within this launch's lattice
  const double* uc = u + rhs * u_rs + cell * n;
  const double* wc = w + rhs * u_rs + cell * n;
  double* us = sm;
  double* ws = sm + n;
  for (int t = threadIdx.x; t < n; t += blockDim.x) { us[t] = uc[t]; ws[t] = wc[t]; }
  __syncthreads();
  const int e = g.e;
  const int nel = e * e * (D == 3 ? e : 1);
  const int cx = (int)(cell % g.nc[0]);
  const int cy = (int)((cell / g.nc[0]) % g.nc[1]);
  const int cz = (int)(cell / ((long long)g.nc[0] * g.nc[1]));
  double acc = 0.0;
  for (int t = threadIdx.x; t < nel * NA; t += blockDim.x) {
    const int el = t / NA, gp = t - el * NA;
    const int ex = el % e, ey = (el / e) % e, ez = el / (e * e);
    double eta[3], xi[3], J[3][3];
    gauss_point(g, cx, cy, cz, ex, ey, ez, gp, eta, xi);
    macro_jacobian(g, xi, J);
    const double dE = youngs_dr(g, strut_distance(g, eta), r_cell[cell]);
    if (dE == 0.0) continue;
    double C[45];
    chat_upper(D, g.nu, J, dE, C);
    double tq[D];
    for (int k = 0; k < D; ++k) tq[k] = gauss_t((gp >> k) & 1);
    double Gu[NI], Gw[NI];
    for (int I = 0; I < NI; ++I) { Gu[I] = 0.0; Gw[I] = 0.0; }
    for (int A = 0; A < NA; ++A) {
      const int ax = A & 1, ay = (A >> 1) & 1, az = (A >> 2) & 1;
      const int node = (ex + ax) + (e + 1) * ((ey + ay) + (e + 1) * (D == 3 ? (ez + az) : 0));
      for (int a = 0; a < D; ++a) {
        double dn = inv_h;
        for (int k = 0; k < D; ++k) {
          const int off = (A >> k) & 1;
          if (k == a) dn *= off ? 1.0 : -1.0;
          else dn *= off ? tq[k] : 1.0 - tq[k];
        }
        for (int i = 0; i < D; ++i) {
          Gu[i * D + a] += us[node * D + i] * dn;
          Gw[i * D + a] += ws[node * D + i] * dn;
        }
      }
    }
    int q = 0;
    double s = 0.0;
    for (int I = 0; I < NI; ++I)
      for (int Jx = I; Jx < NI; ++Jx) {
        const double cij = C[q++];
        s += cij * Gw[I] * Gu[Jx];
        if (Jx != I) s += cij * Gw[Jx] * Gu[I];
      }
    acc += wq * s;
  }
  // block reduction in fixed order
  __shared__ double red[32];
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) red[wid] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) s += red[k];
    out[rhs * out_rs + cell] = -s;
  }
}

}  // namespace

// K_rr^(s) times nvec FP32 vectors per (rhs, cell) column (the local ROM bases of the mixed path).
fetidp_status k_krr_apply_f32(Ctx& c, const float* u, long long u_rs, int u_cs, float* y, long long y_rs,
                              int y_cs, int nvec, int nrhs, long long ext) {
  const int nchunk = (nvec + kSpVB - 1) / kSpVB;
  const size_t smem = (size_t)c.nr * kSpLd * sizeof(float);
  // algorithmic work: one FMA per stored entry and vector; bytes: the values once per cell, the
  // vectors in and out
  ProfScope ps(c, FETIDP_K_MULTI_K, 2.0 * (double)c.N * nrhs * nvec * c.krr_nnz * c.nr,
               4.0 * (double)c.N * c.krr_nnz * c.nr + 8.0 * (double)c.N * nrhs * nvec * c.nr);
  const int nnode = c.nr / c.d;
  const size_t smem_n = smem + sizeof(float) * 2 * (size_t)c.d * c.nr;
  if (c.krr_nbr && nnode <= 352 && smem_n <= 113 * 1024) {
    const int threads = (nnode + 31) / 32 * 32;
    if (c.d == 3) {
      cudaFuncSetAttribute(krr_spmm_nodal_f32_kernel<3>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_n);
      krr_spmm_nodal_f32_kernel<3><<<(unsigned)(c.N * nrhs * nchunk), threads, smem_n, c.stream>>>(
          c.krr_nbr, c.krr_val, c.krr_nnz, c.nr, nrhs, nchunk, u, u_rs, u_cs, y, y_rs, y_cs, nvec, ext);
    } else {
      cudaFuncSetAttribute(krr_spmm_nodal_f32_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_n);
      krr_spmm_nodal_f32_kernel<2><<<(unsigned)(c.N * nrhs * nchunk), threads, smem_n, c.stream>>>(
          c.krr_nbr, c.krr_val, c.krr_nnz, c.nr, nrhs, nchunk, u, u_rs, u_cs, y, y_rs, y_cs, nvec, ext);
    }
  } else {
    cudaFuncSetAttribute(krr_spmm_f32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    krr_spmm_f32_kernel<<<(unsigned)(c.N * nrhs * nchunk), 256, smem, c.stream>>>(
        c.krr_col, c.krr_val, c.krr_nnz, c.nr, nrhs, nchunk, u, u_rs, u_cs, y, y_rs, y_cs, nvec, ext);
  }
  FD_CHECK_LAUNCH();
  return FETIDP_OK;
}

fetidp_status k_rom_combine_f32(Ctx& c, const double* src, long long kstride, int ld, int r0, int c0, int rows,
                                int cols, const double* coef, float* out, int ldo, int blkw, int symT) {
  if (c.nrb > 64) { set_error("n_rb above 64"); return FETIDP_EINVAL; }
  const long long per = (long long)rows * cols;
  long long gy = (c.N + kCombCells - 1) / kCombCells;
  if (gy > 64) gy = 64;
  const dim3 grid((unsigned)((per + 255) / 256), (unsigned)gy);
  ProfScope ps(c, FETIDP_K_SETUP, 2.0 * c.nrb * per * (double)c.N, 4.0 * per * (double)c.N);
  if (c.nrb <= 16)
    rom_combine_f32_kernel<16><<<grid, 256, 0, c.stream>>>(src, kstride, ld, r0, c0, rows, cols, coef, c.nrb, c.N, out, ldo,
                                                             blkw, symT);
  else if (c.nrb <= 32)
    rom_combine_f32_kernel<32><<<grid, 256, 0, c.stream>>>(src, kstride, ld, r0, c0, rows, cols, coef, c.nrb, c.N, out, ldo,
                                                             blkw, symT);
  else
    rom_combine_f32_kernel<64><<<grid, 256, 0, c.stream>>>(src, kstride, ld, r0, c0, rows, cols, coef, c.nrb, c.N, out, ldo,
                                                             blkw, symT);
  FD_CHECK_LAUNCH();
  return FETIDP_OK;
}

template <int MR, int P, int V, typename TO>
static fetidp_status gemm_f32_launch(Ctx& c, const float* mats, int ldm, int nout, int nin, const float* xf, TO* y,
                                     long long y_rs, int y_cs, double alpha, double beta, int nrhs) {
  const int W = gemm_block_width(nout, c.N), nb = ceil_div(nout, W);
  const size_t smem = 16 * ((size_t)(nin * P + 3) / 4) + 4 * (size_t)kRing * 32 * V;
  cudaFuncSetAttribute(cell_gemm_f32_kernel<MR, P, V, TO>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  cell_gemm_f32_kernel<MR, P, V, TO><<<(unsigned)(c.N * nb), 32, smem, c.stream>>>(
      mats, ldm, nout, nin, W, nb, xf, c.xf_cs(nin), y, y_rs, y_cs, alpha, beta, nrhs);
  FD_CHECK_LAUNCH();
  return FETIDP_OK;
}

template <typename TO>
static fetidp_status cell_gemm_f32(Ctx& c, const float* mats, int ldm, int nout, int nin, const float* xf, TO* y,
                                   long long y_rs, int y_cs, double alpha, double beta, int nrhs) {
  // algorithmic bytes: the operators once (padded rows as stored), the vectors in (FP32) and out
  ProfScope ps(c, FETIDP_K_ASM_OP, 2.0 * nout * nin * (double)c.N * nrhs,
               4.0 * c.N * (double)nin * ldm + c.N * (double)nrhs * ((double)sizeof(TO) * nout + 4.0 * nin));
  if (nout < 1 || nin < 1 || nout > 1024 || ldm % 4 != 0 || ldm < nout ||
      (size_t)nin * kMaxRhsF32 * sizeof(float) > 200 * 1024 || (reinterpret_cast<uintptr_t>(mats) & 15) != 0) {
    set_error("FP32 cell operators: at most 1024 outputs, rows padded to 16 bytes");
    return FETIDP_EINVAL;
  }
  for (int r0 = 0; r0 < nrhs; r0 += kMaxRhsF32) {
    const float* x = xf + (r0 / kMaxRhsF32) * (long long)c.N * c.xf_cs(nin);
    TO* yr = y + r0 * y_rs;
    const int mr = std::min(kMaxRhsF32, nrhs - r0);
    fetidp_status st = FETIDP_EINVAL;
    // P: the interleave of the context's RHS count; MR: RHS computed (>= those of this chunk)
    const int V = gemm_lane_outputs(nout, c.N);
#define FD_GEMM(MR, P)                                                                              \
  st = V == 4   ? gemm_f32_launch<MR, P, 4>(c, mats, ldm, nout, nin, x, yr, y_rs, y_cs, alpha, beta, mr) \
       : V == 2 ? gemm_f32_launch<MR, P, 2>(c, mats, ldm, nout, nin, x, yr, y_rs, y_cs, alpha, beta, mr) \
                : gemm_f32_launch<MR, P, 1>(c, mats, ldm, nout, nin, x, yr, y_rs, y_cs, alpha, beta, mr)
    if (c.xf_P == 1) FD_GEMM(1, 1);
    else if (c.xf_P == 2) FD_GEMM(2, 2);
    else if (c.xf_P == 4) { if (mr == 3) FD_GEMM(3, 4); else FD_GEMM(4, 4); }
    else if (mr <= 5) FD_GEMM(5, 8);
    else if (mr == 6) FD_GEMM(6, 8);
    else FD_GEMM(8, 8);
#undef FD_GEMM
    FD_TRY(st);
  }
  return FETIDP_OK;
}

fetidp_status k_cell_gemm_f32(Ctx& c, const float* mats, int ldm, int nout, int nin, const float* xf, CellVec y,
                              double alpha, double beta, int nrhs) {
  return cell_gemm_f32(c, mats, ldm, nout, nin, xf, y.p, y.rs, y.cs, alpha, beta, nrhs);
}

// The FP32 sums as they are.
fetidp_status k_cell_gemm_f32_out(Ctx& c, const float* mats, int ldm, int nout, int nin, const float* xf,
                                  const FCellVec& y, int nrhs) {
  return cell_gemm_f32(c, mats, ldm, nout, nin, xf, y.p, y.rs, y.cs, 1.0, 0.0, nrhs);
}

fetidp_status k_cell_symv_f32(Ctx& c, const float* mats, CCellVec x, CellVec y, double alpha, double beta,
                              int nrhs) {
  const int T = c.sym_T, n = c.nd;
  const long long ntile = (long long)T * (T + 1) / 2;
  // algorithmic bytes: the packed operator once, the FP64 vectors in and out
  ProfScope ps(c, FETIDP_K_ASM_OP, 2.0 * n * n * (double)c.N * nrhs,
               4096.0 * ntile * c.N + 8.0 * c.N * (double)nrhs * 2.0 * n);
  const int nw = (T + 1) / 2;
  if (T < 1 || n > 32 * T || nw > 10 || (reinterpret_cast<uintptr_t>(mats) & 15) != 0) {
    set_error("packed FP32 cell operators: at most 20 tile rows");
    return FETIDP_EINVAL;
  }
  const size_t smem = sizeof(float) * ((size_t)T * 32 * 17 + (size_t)nw * 32 * 33);
  cudaFuncSetAttribute(cell_symv_f32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  cell_symv_f32_kernel<<<(unsigned)c.N, 32 * nw, smem, c.stream>>>(mats, T, n, x.p, x.rs, x.cs, y.p, y.rs, y.cs,
                                                                   alpha, beta, nrhs);
  FD_CHECK_LAUNCH();
  return FETIDP_OK;
}

// x in an FP32 layout (the gather's, or packed)
fetidp_status k_udp_t_f32(Ctx& c, const XfLayout& xf, CellVec y, int nrhs) {
  const int nd = c.nd, np = c.np;
  if (!c.Udp_f || (np != 8 && np != 24) || nd < 1) { set_error("FP32 U_dp needs n_p of 8 or 24"); return FETIDP_EINVAL; }
  ProfScope ps(c, FETIDP_K_CELL_GEMV, 2.0 * nd * np * (double)c.N * nrhs,
               4.0 * c.N * nd * np + 8.0 * c.N * nrhs * np + 4.0 * c.N * nrhs * nd);
  const int G = np / 4, RG = 256 / G;
  for (int r0 = 0; r0 < nrhs; r0 += 8) {
    XfLayout x = xf;
    x.p += (r0 >> 3) * xf.chs;
    const int mr = std::min(8, nrhs - r0);
    double* o = y.p + r0 * y.rs;
    if (nd <= RG) {
      const unsigned grid = (unsigned)ceil_div(c.N * np, 128);
      if (np == 8) udp_t_short_f32_kernel<8><<<grid, 128, 0, c.stream>>>(c.Udp_f, nd, x, o, y.rs, y.cs, mr, c.N);
      else udp_t_short_f32_kernel<24><<<grid, 128, 0, c.stream>>>(c.Udp_f, nd, x, o, y.rs, y.cs, mr, c.N);
      FD_CHECK_LAUNCH();
      continue;
    }
    // P: the interleave x has, or is staged with; MR >= the chunk's RHS
    const int P = xf.ds == 8 || xf.ds == 4 || xf.ds == 2 ? xf.ds : mr == 1 ? 1 : 8;
#define FD_UDPT(NP, MR, P)                                                                                       \
  do {                                                                                                           \
    const size_t smem = sizeof(float) * ((((size_t)nd * P + 3) & ~(size_t)3) + (size_t)RG * G * 4 * MR);          \
    if (smem > 227 * 1024) { set_error("FP32 U_dp: n_d too large"); return FETIDP_EINVAL; }                       \
    cudaFuncSetAttribute(udp_t_f32_kernel<NP, MR, P>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);    \
    udp_t_f32_kernel<NP, MR, P><<<(unsigned)c.N, 256, smem, c.stream>>>(c.Udp_f, nd, x, o, y.rs, y.cs, mr);       \
  } while (0)
#define FD_UDPT_NP(NP)                          \
  do {                                          \
    if (P == 1) FD_UDPT(NP, 1, 1);              \
    else if (P == 2) FD_UDPT(NP, 2, 2);         \
    else if (P == 4) FD_UDPT(NP, 4, 4);         \
    else if (mr <= 6) FD_UDPT(NP, 6, 8);        \
    else FD_UDPT(NP, 8, 8);                     \
  } while (0)
    if (np == 8) FD_UDPT_NP(8);
    else FD_UDPT_NP(24);
#undef FD_UDPT_NP
#undef FD_UDPT
    FD_CHECK_LAUNCH();
  }
  return FETIDP_OK;
}

// y = yf + U_dp x (yf FP32) or y += U_dp x (yf null); xf: x rounded to FP32, [chunk][cell][n_p][8]
fetidp_status k_udp_n_f32(Ctx& c, const float* cpf, const FCellVec* yf, CellVec y, int nrhs) {
  const int nd = c.nd, np = c.np;
  if (!c.Udp_f || (np != 8 && np != 24) || nd < 1) { set_error("FP32 U_dp needs n_p of 8 or 24"); return FETIDP_EINVAL; }
  ProfScope ps(c, FETIDP_K_CELL_GEMV, 2.0 * nd * np * (double)c.N * nrhs,
               4.0 * c.N * nd * np + 8.0 * c.N * nrhs * (nd + np) + (yf ? 4.0 : 8.0) * c.N * nrhs * nd);
  const unsigned grid = (unsigned)ceil_div(c.N * nd, 128);
  for (int r0 = 0; r0 < nrhs; r0 += 8) {
    const int mr = std::min(8, nrhs - r0);
    const float* x = cpf + (r0 >> 3) * c.N * np * 8;
    double* o = y.p + r0 * y.rs;
#define FD_UDPN(NP, MR)                                                                                          \
  do {                                                                                                           \
    if (yf)                                                                                                      \
      udp_n_f32_kernel<NP, MR, float><<<grid, 128, 0, c.stream>>>(c.Udp_f, nd, x, yf->p + r0 * yf->rs, yf->rs, yf->cs, \
                                                                  o, y.rs, y.cs, mr, c.N);                       \
    else                                                                                                         \
      udp_n_f32_kernel<NP, MR, double><<<grid, 128, 0, c.stream>>>(c.Udp_f, nd, x, o, y.rs, y.cs, o, y.rs, y.cs, mr, c.N); \
  } while (0)
#define FD_UDPN_NP(NP)          \
  do {                          \
    if (mr == 1) FD_UDPN(NP, 1); \
    else if (mr <= 3) FD_UDPN(NP, 3); \
    else if (mr <= 6) FD_UDPN(NP, 6); \
    else FD_UDPN(NP, 8);        \
  } while (0)
    if (np == 8) FD_UDPN_NP(8);
    else FD_UDPN_NP(24);
#undef FD_UDPN_NP
#undef FD_UDPN
    FD_CHECK_LAUNCH();
  }
  return FETIDP_OK;
}

fetidp_status k_cell_gemv_strided(Ctx& c, const double* mats, long long mstride, int ld, int mrows,
                                  int mcols, CCellVec x, CellVec y, double alpha, double beta,
                                  int nrhs) {
  ProfScope ps(c, FETIDP_K_CELL_GEMV, 2.0 * mrows * mcols * (double)c.N * nrhs,
               8.0 * c.N * ((double)mrows * mcols + (double)nrhs * (mrows + mcols)));
  const bool aligned16 = (ld % 2 == 0) && (mstride % 2 == 0) && ((reinterpret_cast<uintptr_t>(mats) & 15) == 0);
  if ((mcols == 8 || mcols == 24) && aligned16 && c.N * mrows < (1LL << 31)) {
    const long long total = c.N * mrows;
    long long grid = (total + 255) / 256;
    if (grid > 152LL * 32) grid = 152LL * 32;
    if (mcols == 8)
      cell_gemv_narrow_fixed<8><<<(unsigned)grid, 256, 0, c.stream>>>(mats, mstride, ld, mrows, x.p, x.rs, x.cs, y.p,
                                                                     y.rs, y.cs, alpha, beta, nrhs, c.N);
    else
      cell_gemv_narrow_fixed<24><<<(unsigned)grid, 256, 0, c.stream>>>(mats, mstride, ld, mrows, x.p, x.rs, x.cs,
                                                                      y.p, y.rs, y.cs, alpha, beta, nrhs, c.N);
    FD_CHECK_LAUNCH();
    return FETIDP_OK;
  }
  if (mcols <= 32) {
    const long long total = c.N * mrows;
    long long grid = (total + 255) / 256;
    if (grid > 152LL * 16) grid = 152LL * 16;
    cell_gemv_narrow_kernel<<<(unsigned)grid, 256, 0, c.stream>>>(mats, mstride, ld, mrows, mcols, x.p, x.rs,
                                                                 x.cs, y.p, y.rs, y.cs, alpha, beta, nrhs, c.N);
    FD_CHECK_LAUNCH();
    return FETIDP_OK;
  }
  set_error("narrow per-cell operators: at most 32 columns");
  return FETIDP_EINVAL;
}

template <int MR>
static fetidp_status gemvt_launch(Ctx& c, const double* mats, long long mstride, int ld, int nout, int nin, CCellVec x,
                                  CellVec y, double alpha, double beta, long long ncell, int tile) {
  const int TI = std::min(nout, tile), S = kGemvThreads / TI, ntile = ceil_div(nout, TI);
  const size_t smem = sizeof(double) * MR * (size_t)std::max(nin, S * TI);
  if (smem > 227 * 1024) { set_error("per-cell operators: too many columns for shared memory"); return FETIDP_EINVAL; }
  cudaFuncSetAttribute(cell_gemvt_kernel<MR>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  cell_gemvt_kernel<MR><<<(unsigned)(ncell * ntile), kGemvThreads, smem, c.stream>>>(
      mats, mstride, ld, nout, nin, TI, S, x.p, x.rs, x.cs, y.p, y.rs, y.cs, alpha, beta, ntile);
  FD_CHECK_LAUNCH();
  return FETIDP_OK;
}

static fetidp_status gemvt(Ctx& c, const double* mats, long long mstride, int ld, int nout, int nin, CCellVec x,
                           CellVec y, double alpha, double beta, int nrhs, long long ncell, int tile) {
  // RHS per launch: eight, fewer where their x would not fit shared memory
  const int most = (int)std::max<long long>(1, std::min<long long>(kMaxRhsGemv, 227 * 1024 / (8LL * nin)));
  for (int r0 = 0; r0 < nrhs; r0 += most) {
    const CCellVec xr{x.p + r0 * x.rs, x.rs, x.cs};
    const CellVec yr{y.p + r0 * y.rs, y.rs, y.cs};
    switch (std::min(most, nrhs - r0)) {
      case 1: FD_TRY(gemvt_launch<1>(c, mats, mstride, ld, nout, nin, xr, yr, alpha, beta, ncell, tile)); break;
      case 2: FD_TRY(gemvt_launch<2>(c, mats, mstride, ld, nout, nin, xr, yr, alpha, beta, ncell, tile)); break;
      case 3: FD_TRY(gemvt_launch<3>(c, mats, mstride, ld, nout, nin, xr, yr, alpha, beta, ncell, tile)); break;
      case 4: FD_TRY(gemvt_launch<4>(c, mats, mstride, ld, nout, nin, xr, yr, alpha, beta, ncell, tile)); break;
      case 5: FD_TRY(gemvt_launch<5>(c, mats, mstride, ld, nout, nin, xr, yr, alpha, beta, ncell, tile)); break;
      case 6: FD_TRY(gemvt_launch<6>(c, mats, mstride, ld, nout, nin, xr, yr, alpha, beta, ncell, tile)); break;
      case 7: FD_TRY(gemvt_launch<7>(c, mats, mstride, ld, nout, nin, xr, yr, alpha, beta, ncell, tile)); break;
      default: FD_TRY(gemvt_launch<8>(c, mats, mstride, ld, nout, nin, xr, yr, alpha, beta, ncell, tile)); break;
    }
  }
  return FETIDP_OK;
}

fetidp_status k_cell_gemvt(Ctx& c, const double* mats, long long mstride, int ld, int nout, int nin, CCellVec x,
                           CellVec y, double alpha, double beta, int nrhs) {
  ProfScope ps(c, FETIDP_K_CELL_GEMV, 2.0 * nout * nin * (double)c.N * nrhs,
               8.0 * c.N * ((double)nout * nin + (double)nrhs * (nout + nin)));
  return gemvt(c, mats, mstride, ld, nout, nin, x, y, alpha, beta, nrhs, c.N, 32);
}

// Tiles of 8 outputs: one matrix of at most 1,024 columns then spreads over up to 128 SMs, each thread with a
// chain of at most 32 loads.
fetidp_status k_dense_symv(Ctx& c, const double* S, int n, const double* b, long long b_rs, double* x, long long x_rs,
                           int nrhs) {
  return gemvt(c, S, 0, n, n, n, CCellVec{b, b_rs, 0}, CellVec{x, x_rs, 0}, 1.0, 0.0, nrhs, 1, 8);
}

fetidp_status k_grouped_gemm(Ctx& c, const double* A, long long a_stride_k, int lda, int M, int K,
                             CCellVec X, CellVec Y, const double* coef, double alpha, double beta,
                             int nrhs, bool separate, long long y_k_stride) {
  const int nk = c.nrb;
  const long long ncell = c.N;
  const long long ncols = ncell * nrhs;
  ProfScope ps(c, FETIDP_K_GROUPED_GEMM, 2.0 * M * K * nk * (double)ncols,
               8.0 * ((double)nk * M * K + (double)ncols * K + (double)ncols * M * (separate ? nk : 1)));
  const int TN = ncols <= 16 ? 16 : ncols <= 32 ? 32 : 64;
  const dim3 grid((unsigned)ceil_div(ncols, TN), (unsigned)ceil_div(M, GT), (unsigned)(separate ? nk : 1));
#define FD_GROUPED(T)                                                                                              \
  grouped_gemm_kernel<T><<<grid, 256, 0, c.stream>>>(A, a_stride_k, lda, M, K, nk, X.p, X.rs, X.cs, Y.p, Y.rs, Y.cs, \
                                                     coef, alpha, beta, ncell, nrhs, separate, y_k_stride)
  if (TN == 16) FD_GROUPED(16);
  else if (TN == 32) FD_GROUPED(32);
  else FD_GROUPED(64);
#undef FD_GROUPED
  FD_CHECK_LAUNCH();
  return FETIDP_OK;
}

fetidp_status k_trace_gemm(Ctx& c, const double* A, int lda, int M, int K, const double* X, int x_cs, long long ncols,
                           double* Y, int y_cs) {
  if (M <= 0 || ncols <= 0) return FETIDP_OK;
  ProfScope ps(c, FETIDP_K_TRACES, 2.0 * M * (double)K * ncols, 8.0 * ((double)M * K + (double)ncols * (K + M)));
  // 16 x 16 outputs per block; 8 x 8 while those blocks do not cover the SMs twice over
  const bool small = (long long)ceil_div(M, 16) * ceil_div(ncols, 16) < 2 * 152;
  const int T = small ? 8 : 16;
  const int mtiles = ceil_div(M, T);
  const long long grid = mtiles * ((ncols + T - 1) / T);
  if (grid >= (1LL << 31)) { set_error("trace contraction: too many blocks for one launch"); return FETIDP_EINVAL; }
  if (small) trace_gemm_kernel<8><<<(unsigned)grid, 64, 0, c.stream>>>(A, lda, M, K, X, x_cs, Y, y_cs, ncols, mtiles);
  else trace_gemm_kernel<16><<<(unsigned)grid, 256, 0, c.stream>>>(A, lda, M, K, X, x_cs, Y, y_cs, ncols, mtiles);
  FD_CHECK_LAUNCH();
  return FETIDP_OK;
}

template <typename TB>
static fetidp_status gram_solve_t(Ctx& c, const TB* R, const TB* KR, CCellVec v, CellVec x, int nrhs,
                                  double drop_rel, int len = -1) {
  if (len < 0) len = c.nr;
  if (c.nrb > kMaxRb) {
    set_error("n_rb above 64 is not supported by the Gram solve");
    return FETIDP_EINVAL;
  }
  const long long cols = c.N * nrhs;
  ProfScope ps(c, FETIDP_K_GRAM, cols * 2.0 * len * (c.nrb * (c.nrb + 1) / 2.0 + 2.0 * c.nrb),
               cols * (double)sizeof(TB) * (2.0 * c.nrb * len) + cols * 16.0 * len);
  const size_t per_warp = (size_t)gram_warp_doubles(c.nrb, (int)sizeof(TB)) * sizeof(double);
  int wpb = (int)std::min<size_t>(8, (200 * 1024) / per_warp);
  if (wpb < 1) wpb = 1;
  const size_t smem = per_warp * wpb;
  cudaFuncSetAttribute(gram_warp_kernel<TB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  gram_warp_kernel<TB><<<(unsigned)ceil_div(cols, wpb), 32 * wpb, smem, c.stream>>>(
      R, KR, v.p, v.rs, v.cs, x.p, x.rs, x.cs, len, c.nrb, c.N, nrhs, drop_rel);
  FD_CHECK_LAUNCH();
  return FETIDP_OK;
}

fetidp_status k_gram_solve(Ctx& c, const double* R, const double* KR, CCellVec v, CellVec x,
                           int nrhs, int len) {
  return gram_solve_t<double>(c, R, KR, v, x, nrhs, 1e-12, len);
}

fetidp_status k_gram_solve_f32(Ctx& c, const float* R, const float* KR, CCellVec v, CellVec x,
                               int nrhs, long long r_ext) {
  (void)r_ext;
  if (c.nrb > kMaxRb) {
    set_error("n_rb above 64 is not supported by the Gram solve");
    return FETIDP_EINVAL;
  }
  const long long cols = c.N * nrhs;
  ProfScope ps(c, FETIDP_K_GRAM, cols * 2.0 * c.nr * ((double)c.nrb * c.nrb + c.nrb) + cols * 2.0 * c.nr * c.nrb,
               cols * 4.0 * (2.0 * c.nrb * c.nr) + cols * 16.0 * c.nr);
  const size_t smem = gram_block_smem(c.nrb);
  cudaFuncSetAttribute(gram_block_f32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  gram_block_f32_kernel<<<(unsigned)cols, 256, smem, c.stream>>>(R, KR, v.p, v.rs, v.cs, x.p, x.rs, x.cs, c.nr,
                                                                  c.nrb, c.N, c.opt.gram_drop_mixed);
  FD_CHECK_LAUNCH();
  return FETIDP_OK;
}

fetidp_status k_grad(Ctx& c, const double* u, const double* w, double* g) {
  const double h = 1.0 / c.e;
  const double wq = pow(0.5 * h, c.d);
  const size_t smem = 2 * (size_t)c.n * sizeof(double);
  for (const LatticeSpan& ls : c.lat) {   // one launch per lattice: its own geometry and radii
    const dim3 grid((unsigned)(ls.ncell * c.m));
    const long long off = ls.cell0 * c.n;
    if (c.d == 2)
      grad_kernel<2><<<grid, 256, smem, c.stream>>>(ls.geo, c.r_dev + ls.cell0, ls.ncell, c.n, u + off, w + off,
                                                    c.N * c.n, g + ls.cell0, c.N, wq, 1.0 / h);
    else
      grad_kernel<3><<<grid, 256, smem, c.stream>>>(ls.geo, c.r_dev + ls.cell0, ls.ncell, c.n, u + off, w + off,
                                                    c.N * c.n, g + ls.cell0, c.N, wq, 1.0 / h);
    FD_CHECK_LAUNCH();
  }
  FD_CHECK_LAUNCH();
  return FETIDP_OK;
}

FD_DEFINE_CHECK(fd_check_cell)

fetidp_status k_gram_direct(Ctx& c, const double* Y, int ntab, const double* dvec, double* pi, double* delta,
                           double drop_rel) {
  const int nrb = c.nrb, ld = nrb + 1;
  const int per = 2 * nrb * ld + 6 * nrb;
  const size_t per_warp = (size_t)(per + (per & 1)) * sizeof(double);
  int wpb = (int)std::min<size_t>(8, (200 * 1024) / per_warp);
  if (wpb < 1) wpb = 1;
  const size_t smem = per_warp * wpb;
  cudaFuncSetAttribute(gram_direct_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  gram_direct_kernel<<<(unsigned)ceil_div(2 * c.N, wpb), 32 * wpb, smem, c.stream>>>(Y, ntab, nrb, dvec, pi, delta,
                                                                                      c.N, drop_rel);
  FD_CHECK_LAUNCH();
  return FETIDP_OK;
}

}  // namespace fetidp
