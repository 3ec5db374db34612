// Cell stiffness K_s (Eq. 5a through Eq. 52): snapshots of C_hat, the sparse FP64 K_s of every cell,
// its products with vectors, and the FP32 copy of K_rr for the mixed path's local ROM.
//
// Every cell has the same node graph, so K_s is stored in block-ELL form over it: node n (local
// (i, d, p) order) has up to 3^d neighbour nodes, listed in local order; value (n, k, c, a) couples
// component a of n with component c of its k-th neighbour, at ((cell nk + k) d^2 + c d + a) nn + n, so
// that a warp of consecutive nodes reads consecutive doubles.
//
// Why sparse and not matrix-free: GB300 issues two FP64 FMAs per clock and SM, and K_s is used for
// every RHS of every outer iteration and, in the FP64 path, for n_rb vectors per local ROM solve.  A
// product costs 62 k FMAs per 6^3 cell and vector; the matrix-free loop (gradients, C_hat and
// transposed gradients at 1,728 Gauss points, butterfly sums) issued about a million FP64 instructions.
// On 864 cells and 3 RHS a product takes 0.34 ms (FP64 bound 0.27 ms), the loop took 4.12 ms; the n_rb = 16
// vectors of 6 RHS on 32 cells 0.5 ms against 7 ms.  Assembling K_s costs 0.85 M FMAs per cell once per
// setup (2.7 ms for 864 cells), from the isotropic form
//   K_(Ai)(Bj) = lam Q_ij + mu Q_ji + mu d_ij tr Q,  Q = sum_gp s g_A g_B^T,  g_A = J^-T grad N_A,
// s = w E det J: nine FMAs per node pair and Gauss point.
#include <algorithm>
#include <cmath>
#include <vector>

#include "common.cuh"

namespace fetidp {

namespace {

inline int ceil_div(long long a, long long b) { return (int)((a + b - 1) / b); }

// C_hat at every Gauss point (the greedy's snapshots) and, component-major per cell, the d^2 entries
// of J^-1 and s = w E det J of the point: gpd[cell][d^2 + 1][npt].
__global__ void snapshot_kernel(Geo g, const double* __restrict__ r_cell, long long ncell,
                                int nelem, int ngp, int nc, double wq, double* __restrict__ snap,
                                double* __restrict__ gpd) {
  const long long total = ncell * nelem * ngp;
  const int npt = nelem * ngp, dd = g.dim * g.dim;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const long long cell = t / (nelem * ngp);
    const int rem = (int)(t - cell * nelem * ngp);
    const int el = rem / ngp, gp = rem - el * ngp;
    const int cx = (int)(cell % g.nc[0]);
    const int cy = (int)((cell / g.nc[0]) % g.nc[1]);
    const int cz = (int)(cell / ((long long)g.nc[0] * g.nc[1]));
    const int ex = el % g.e, ey = (el / g.e) % g.e, ez = el / (g.e * g.e);
    double eta[3], xi[3], J[3][3];
    gauss_point(g, cx, cy, cz, ex, ey, ez, gp, eta, xi);
    macro_jacobian(g, xi, J);
    const double E = youngs(g, strut_distance(g, eta), r_cell[cell]);
    double out[45];
    chat_upper(g.dim, g.nu, J, E, out);
    double* dst = snap + cell * (long long)nelem * ngp * nc + (long long)rem * nc;
    for (int k = 0; k < nc; ++k) dst[k] = out[k];
    double Ji[3][3];
    const double det = jacobian_inverse(g.dim, J, Ji);
    double* o = gpd + cell * (long long)(dd + 1) * npt + rem;
    for (int a = 0; a < g.dim; ++a)
      for (int k = 0; k < g.dim; ++k) o[(long long)(a * g.dim + k) * npt] = Ji[a][k];
    o[(long long)dd * npt] = wq * E * det;
  }
}

template <int D>
struct Elem {
  static constexpr int NA = 1 << D;              // nodes and Gauss points of an element
  static constexpr int NP = NA * (NA + 1) / 2;   // node pairs A <= B
  static constexpr int EB = D == 3 ? 8 : 32;     // elements per block of the element-matrix kernel
};
__host__ __device__ inline int pair_index(int A, int B, int NA) { return A * NA - A * (A - 1) / 2 + (B - A); }

// Upper node-pair blocks of the element matrices, Ke[cell][el][pair][d * d], EB elements per block: the
// physical shape gradients of the block's Gauss points in shared memory, then one thread per (element,
// node pair).  FP64-bound: 9 FMAs per pair and point against 6 shared reads.
template <int D>
__global__ void __launch_bounds__(320) element_pairs_kernel(const double* __restrict__ gpd, int nelem, int nblk,
                                                            double inv_h, double lam, double mu,
                                                            double* __restrict__ Ke) {
  constexpr int NA = Elem<D>::NA, NP = Elem<D>::NP, EB = Elem<D>::EB, DD = D * D;
  __shared__ double dns[NA][NA][D];               // [gp][A][a], reference gradients
  __shared__ double gs[EB][NA][NA][D];            // [element][gp][A][k], physical gradients
  __shared__ double ss[EB][NA];
  const long long cell = blockIdx.x / nblk;
  const int e0 = (int)(blockIdx.x - cell * nblk) * EB, ne = min(EB, nelem - e0), npt = nelem * NA;
  for (int t = threadIdx.x; t < NA * NA * D; t += blockDim.x) {
    const int a = t % D, A = (t / D) % NA, gp = t / (D * NA);
    double v = inv_h;
    for (int q = 0; q < D; ++q) {
      const int off = (A >> q) & 1;
      const double tq = gauss_t((gp >> q) & 1);
      v *= q == a ? (off ? 1.0 : -1.0) : (off ? tq : 1.0 - tq);
    }
    dns[gp][A][a] = v;
  }
  __syncthreads();
  const double* gc = gpd + cell * (long long)(DD + 1) * npt + (long long)e0 * NA;
  for (int t = threadIdx.x; t < ne * NA * NA; t += blockDim.x) {
    const int A = t % NA, pt = t / NA, gp = pt % NA, el = pt / NA;
#pragma unroll
    for (int k = 0; k < D; ++k) {
      double v = 0.0;
#pragma unroll
      for (int a = 0; a < D; ++a) v = fma(dns[gp][A][a], gc[(long long)(a * D + k) * npt + pt], v);
      gs[el][gp][A][k] = v;
    }
    if (A == 0) ss[el][gp] = gc[(long long)DD * npt + pt];
  }
  __syncthreads();
  for (int t = threadIdx.x; t < ne * NP; t += blockDim.x) {
    const int el = t / NP;
    int A = 0, rem = t - el * NP;
    while (rem >= NA - A) { rem -= NA - A; ++A; }
    const int B = A + rem;
    double Q[D][D];
#pragma unroll
    for (int i = 0; i < D; ++i)
#pragma unroll
      for (int j = 0; j < D; ++j) Q[i][j] = 0.0;
#pragma unroll 2
    for (int gp = 0; gp < NA; ++gp) {
      const double s = ss[el][gp];
#pragma unroll
      for (int i = 0; i < D; ++i) {
        const double ga = s * gs[el][gp][A][i];
#pragma unroll
        for (int j = 0; j < D; ++j) Q[i][j] = fma(ga, gs[el][gp][B][j], Q[i][j]);
      }
    }
    double tr = 0.0;
#pragma unroll
    for (int i = 0; i < D; ++i) tr += Q[i][i];
    double* o = Ke + ((cell * nelem + e0 + el) * NP + (t - el * NP)) * DD;
#pragma unroll
    for (int i = 0; i < D; ++i)
#pragma unroll
      for (int j = 0; j < D; ++j) o[i * D + j] = lam * Q[i][j] + mu * Q[j][i] + (i == j ? mu * tr : 0.0);
  }
}

// Block-ELL values from the element pairs: one thread per (cell, slot k, node n) sums the at most 2^d
// elements that hold both nodes, in element order (deterministic, no atomics).
template <int D>
__global__ void stiffness_gather_kernel(const double* __restrict__ Ke, const int* __restrict__ nbr,
                                        const int* __restrict__ nat, int e, int nk, int nn, long long ncell,
                                        double* __restrict__ val) {
  constexpr int NA = Elem<D>::NA, NP = Elem<D>::NP, DD = D * D;
  const int n1 = e + 1, nelem = D == 3 ? e * e * e : e * e;
  const long long per = (long long)nk * nn;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < ncell * per;
       t += (long long)gridDim.x * blockDim.x) {
    const long long cell = t / per;
    const int kn = (int)(t - cell * per), k = kn / nn, n = kn - k * nn;
    double v[DD];
#pragma unroll
    for (int q = 0; q < DD; ++q) v[q] = 0.0;
    const int m = nbr[kn];
    if (m >= 0) {
      const int a0 = nat[n], b0 = nat[m];
      const int na[3] = {a0 % n1, (a0 / n1) % n1, D == 3 ? a0 / (n1 * n1) : 0};
      const int nb[3] = {b0 % n1, (b0 / n1) % n1, D == 3 ? b0 / (n1 * n1) : 0};
      int lo[3], hi[3];                           // elements holding both nodes, per axis
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        lo[q] = q < D ? max(0, max(na[q], nb[q]) - 1) : 0;
        hi[q] = q < D ? min(e - 1, min(na[q], nb[q])) : 0;
      }
      for (int ez = lo[2]; ez <= hi[2]; ++ez)
        for (int ey = lo[1]; ey <= hi[1]; ++ey)
          for (int ex = lo[0]; ex <= hi[0]; ++ex) {
            const int el = ex + e * (ey + e * ez);
            const int A = (na[0] - ex) + 2 * (na[1] - ey) + (D == 3 ? 4 * (na[2] - ez) : 0);
            const int B = (nb[0] - ex) + 2 * (nb[1] - ey) + (D == 3 ? 4 * (nb[2] - ez) : 0);
            const bool up = A <= B;
            const double* p = Ke + ((cell * nelem + el) * NP + pair_index(up ? A : B, up ? B : A, NA)) * DD;
#pragma unroll
            for (int c = 0; c < D; ++c)
#pragma unroll
              for (int a = 0; a < D; ++a) v[c * D + a] += up ? p[a * D + c] : p[c * D + a];
          }
    }
#pragma unroll
    for (int q = 0; q < DD; ++q) val[((cell * nk + k) * DD + q) * nn + n] = v[q];
  }
}

// FP32 ELL copy of K_rr for the mixed path's local ROM products: krr[cell][d k + c][d n + a].
template <int D>
__global__ void krr_from_stiffness_kernel(const double* __restrict__ val, int nk, int nn, const int* __restrict__ nbr,
                                          int nnz, int nr, long long ncell, float* __restrict__ krr) {
  const long long per = (long long)nnz * nr;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < ncell * per;
       t += (long long)gridDim.x * blockDim.x) {
    const long long cell = t / per;
    const int r = (int)(t - cell * per), sl = r / nr, row = r - sl * nr;
    const int k = sl / D, c = sl - k * D, n = row / D, a = row - n * D;
    const int m = nbr[k * nn + n];
    krr[t] = (m >= 0 && m < nr / D) ? (float)val[((cell * nk + k) * (D * D) + c * D + a) * nn + n] : 0.f;
  }
}

// y = K_s u for MR vectors per thread, one thread per (cell, row node): nine (four in 2D) values and d
// vector entries per neighbour and vector feed d^2 MR FMAs, so the FP64 pipe is what bounds it (values
// cost 8 bytes per MR FMAs).  The values of a cell are read once per group of MR vectors (from L2 after
// the first), u through L1: a warp's neighbours are nearly consecutive nodes.  Rows stop at nrow nodes
// and columns at ncol nodes (K_rr and K_ii are leading blocks of the local order).
struct KView {
  double* r;           // the first nsplit nodes of a vector
  double* p;           // the remaining nodes (the corners), when kept elsewhere
  long long rs, prs;   // RHS strides
  long long cs, pcs;   // cell strides
  int len;             // distance of a cell's vectors from each other
};
template <int D, int MR>
__global__ void __launch_bounds__(64) stiffness_apply_kernel(const double* __restrict__ val,
                                                             const int* __restrict__ nbr, const int* __restrict__ cnt,
                                                             const int* __restrict__ nat, int nk, int nn, int nrow,
                                                             int ncol, int nsplit, KView U, KView Y, int nvec, int ntot,
                                                             int ntile, int nchunk) {
  constexpr int DD = D * D;
  const int chunk = blockIdx.x % nchunk;
  const long long rest = blockIdx.x / nchunk;
  const long long cell = rest / ntile;
  const int n = (int)(rest - cell * ntile) * 64 + threadIdx.x;
  const int nc = min(n, nn - 1);
  const int kmax = __reduce_max_sync(0xffffffffu, n < nrow ? cnt[nc] : 0);
  const double *ur[MR], *up[MR];
#pragma unroll
  for (int r = 0; r < MR; ++r) {
    const int v = min(chunk * MR + r, ntot - 1), rhs = v / nvec, vq = v - rhs * nvec;
    ur[r] = U.r + rhs * U.rs + cell * U.cs + (long long)vq * U.len;
    up[r] = U.p + rhs * U.prs + cell * U.pcs;
  }
  double acc[D][MR];
#pragma unroll
  for (int a = 0; a < D; ++a)
#pragma unroll
    for (int r = 0; r < MR; ++r) acc[a][r] = 0.0;
  const double* vc = val + cell * (long long)nk * DD * nn + nc;
  for (int k = 0; k < kmax; ++k) {
    const int m = nbr[k * nn + nc];
    double kv[DD];
#pragma unroll
    for (int q = 0; q < DD; ++q) kv[q] = __ldg(vc + (long long)(k * DD + q) * nn);
    if (m < 0 || m >= ncol) continue;
    const bool rem = m < nsplit;
    const int off = D * (rem ? (nat ? nat[m] : m) : m - nsplit);
#pragma unroll
    for (int r = 0; r < MR; ++r) {
      const double* u = (rem ? ur[r] : up[r]) + off;
#pragma unroll
      for (int c = 0; c < D; ++c) {
        const double x = u[c];
#pragma unroll
        for (int a = 0; a < D; ++a) acc[a][r] = fma(kv[c * D + a], x, acc[a][r]);
      }
    }
  }
  if (n >= nrow) return;
  const bool rem = n < nsplit;
  const int off = D * (rem ? (nat ? nat[n] : n) : n - nsplit);
#pragma unroll
  for (int r = 0; r < MR; ++r) {
    const int v = chunk * MR + r;
    if (v >= ntot) break;
    const int rhs = v / nvec, vq = v - rhs * nvec;
    double* o = rem ? Y.r + rhs * Y.rs + cell * Y.cs + (long long)vq * Y.len + off
                    : Y.p + rhs * Y.prs + cell * Y.pcs + off;
#pragma unroll
    for (int a = 0; a < D; ++a) o[a] = acc[a][r];
  }
}

template <int D, int MR>
void apply_launch(Ctx& c, const KView& u, const KView& y, bool natural, int nrow, int ncol, int nsplit, int nvec,
                  int ntot) {
  const int ntile = ceil_div(nrow, 64), nchunk = ceil_div(ntot, MR);
  stiffness_apply_kernel<D, MR><<<(unsigned)(c.N * ntile * nchunk), 64, 0, c.stream>>>(
      c.K_val, c.K_nbr, c.K_cnt, natural ? c.K_nat : nullptr, c.K_nk, c.n / D, nrow, ncol, nsplit, u, y, nvec, ntot,
      ntile, nchunk);
}

template <int D>
fetidp_status apply_dispatch(Ctx& c, const KView& u, const KView& y, bool natural, int nrow, int ncol, int nsplit,
                             int nvec, int ntot) {
  // groups of at most eight vectors, as even as possible (an absent vector of the last group is computed twice)
  const int MR = ceil_div(ntot, ceil_div(ntot, 8));
  if (c.N * (long long)ceil_div(nrow, 64) * ceil_div(ntot, MR) >= (1LL << 31)) {
    set_error("cell stiffness: too many blocks for one launch");
    return FETIDP_EINVAL;
  }
  switch (MR) {
    case 1: apply_launch<D, 1>(c, u, y, natural, nrow, ncol, nsplit, nvec, ntot); break;
    case 2: apply_launch<D, 2>(c, u, y, natural, nrow, ncol, nsplit, nvec, ntot); break;
    case 3: apply_launch<D, 3>(c, u, y, natural, nrow, ncol, nsplit, nvec, ntot); break;
    case 4: apply_launch<D, 4>(c, u, y, natural, nrow, ncol, nsplit, nvec, ntot); break;
    case 5: apply_launch<D, 5>(c, u, y, natural, nrow, ncol, nsplit, nvec, ntot); break;
    case 6: apply_launch<D, 6>(c, u, y, natural, nrow, ncol, nsplit, nvec, ntot); break;
    case 7: apply_launch<D, 7>(c, u, y, natural, nrow, ncol, nsplit, nvec, ntot); break;
    default: apply_launch<D, 8>(c, u, y, natural, nrow, ncol, nsplit, nvec, ntot); break;
  }
  FD_CHECK_LAUNCH();
  return FETIDP_OK;
}

fetidp_status apply(Ctx& c, const KView& u, const KView& y, bool natural, int nrow, int ncol, int nsplit, int nvec,
                    int nrhs) {
  const int ntot = nvec * nrhs, dd = c.d * c.d;
  const double pairs = std::pow(3.0 * c.e + 1.0, c.d);   // coupled node pairs of a cell
  ProfScope ps(c, FETIDP_K_APPLY_K, 2.0 * dd * pairs * c.N * ntot,
               8.0 * c.N * (dd * pairs + (double)ntot * c.d * (nrow + ncol)));
  return c.d == 2 ? apply_dispatch<2>(c, u, y, natural, nrow, ncol, nsplit, nvec, ntot)
                  : apply_dispatch<3>(c, u, y, natural, nrow, ncol, nsplit, nvec, ntot);
}

// Element matrices of a chunk of cells at a time: 0.56 MB per 6^3 cell would double the setup's memory
constexpr size_t kPairBytes = (size_t)256 << 20;

template <int D>
fetidp_status assemble(Ctx& c, const double* gpd) {
  constexpr int NP = Elem<D>::NP, DD = D * D;
  const int nn = c.n / D;
  const size_t cell_pairs = (size_t)c.nelem * NP * DD;
  const long long chunk = std::max<long long>(1, std::min<long long>(c.N, kPairBytes / (sizeof(double) * cell_pairs)));
  const double lam = c.geo.nu / ((1.0 + c.geo.nu) * (1.0 - 2.0 * c.geo.nu)), mu = 1.0 / (2.0 * (1.0 + c.geo.nu));
  double* Ke = nullptr;
  FD_TRY(tmp_alloc(c, reinterpret_cast<void**>(&Ke), sizeof(double) * cell_pairs * chunk));
  const int nblk = ceil_div(c.nelem, Elem<D>::EB), threads = (Elem<D>::EB * NP + 31) / 32 * 32;
  const long long npt = (long long)c.nelem * c.ngp;
  cudaError_t e = cudaSuccess;
  for (long long c0 = 0; c0 < c.N && e == cudaSuccess; c0 += chunk) {
    const long long nc = std::min(chunk, c.N - c0);
    element_pairs_kernel<D><<<(unsigned)(nc * nblk), threads, 0, c.stream>>>(gpd + c0 * (DD + 1) * npt, c.nelem, nblk,
                                                                             (double)c.e, lam, mu, Ke);
    count_launch();
    const long long work = nc * c.K_nk * nn;
    stiffness_gather_kernel<D><<<(int)std::min<long long>((work + 127) / 128, 152LL * 64), 128, 0, c.stream>>>(
        Ke, c.K_nbr, c.K_nat, c.e, c.K_nk, nn, nc, c.K_val + (size_t)c0 * c.K_nk * DD * nn);
    count_launch();
    e = cudaPeekAtLastError();
  }
  tmp_free(c, Ke);
  if (e != cudaSuccess) {
    set_error(std::string("kernel launch: ") + cudaGetErrorString(cudaGetLastError()));
    return FETIDP_ECUDA;
  }
  return FETIDP_OK;
}

}  // namespace

// Snapshots of every cell and the sparse K_s from the same Gauss-point data.
fetidp_status k_snapshots(Ctx& c) {
  const int d = c.d, dd = d * d, nn = c.n / d;
  double* gpd = nullptr;
  const size_t npt = (size_t)c.nelem * c.ngp;
  FD_TRY(tmp_alloc(c, reinterpret_cast<void**>(&gpd), sizeof(double) * c.N * (dd + 1) * npt));
  fetidp_status st = FETIDP_OK;
  {
    ProfScope ps(c, FETIDP_K_SETUP, 0.0, (double)c.N * c.nsnap * 8.0);
    const double wq = std::pow(0.5 / c.e, d);
    const long long total = c.N * c.nelem * c.ngp;
    const int grid = (int)std::min<long long>(ceil_div(total, 256), 152 * 32);
    for (const LatticeSpan& ls : c.lat) {   // one launch per lattice: its own geometry and radii
      snapshot_kernel<<<grid, 256, 0, c.stream>>>(ls.geo, c.r_dev + ls.cell0, ls.ncell, c.nelem, c.ngp, c.nc, wq,
                                                  c.snap + ls.cell0 * c.nsnap, gpd + ls.cell0 * (dd + 1) * npt);
      count_launch();
    }
    if (cudaPeekAtLastError() != cudaSuccess) {
      set_error(std::string("kernel launch: ") + cudaGetErrorString(cudaGetLastError()));
      st = FETIDP_ECUDA;
    }
  }
  if (st == FETIDP_OK) st = dalloc_t(c, &c.K_val, (size_t)c.N * c.K_nk * dd * nn);
  if (st == FETIDP_OK) {
    ProfScope ps(c, FETIDP_K_SETUP, 0.0, 8.0 * (double)c.N * c.K_nk * dd * nn);
    st = d == 2 ? assemble<2>(c, gpd) : assemble<3>(c, gpd);
  }
  tmp_free(c, gpd);
  return st;
}

// The FP32 copy of K_rr in ELL form (mixed path); nnz slots per row.
fetidp_status k_krr_f32(Ctx& c) {
  FD_TRY(dalloc_t(c, &c.krr_val, (size_t)c.N * c.krr_nnz * c.nr));
  ProfScope ps(c, FETIDP_K_SETUP, 0.0, 12.0 * (double)c.N * c.krr_nnz * c.nr);
  const long long work = c.N * (long long)c.krr_nnz * c.nr;
  const int grid = (int)std::min<long long>((work + 255) / 256, 152LL * 64);
  if (c.d == 2)
    krr_from_stiffness_kernel<2><<<grid, 256, 0, c.stream>>>(c.K_val, c.K_nk, c.n / 2, c.K_nbr, c.krr_nnz, c.nr, c.N,
                                                             c.krr_val);
  else
    krr_from_stiffness_kernel<3><<<grid, 256, 0, c.stream>>>(c.K_val, c.K_nk, c.n / 3, c.K_nbr, c.krr_nnz, c.nr, c.N,
                                                             c.krr_val);
  FD_CHECK_LAUNCH();
  return FETIDP_OK;
}

// y = K_s u, column (rhs, cell) holding nvec vectors of len entries in local (i, d, p) order; len < n takes
// the leading len x len block (K_rr, K_ii).
fetidp_status k_apply_K(Ctx& c, CCellVec u, CellVec y, int nvec, int nrhs, int len) {
  const int nodes = len / c.d;
  const KView U{const_cast<double*>(u.p), nullptr, u.rs, 0, u.cs, 0, len}, Y{y.p, nullptr, y.rs, 0, y.cs, 0, len};
  return apply(c, U, Y, false, nodes, nodes, nodes, nvec, nrhs);
}

// y = K_s u in natural node order.
fetidp_status k_apply_K_natural(Ctx& c, CCellVec u, CellVec y, int nrhs) {
  const int nodes = c.n / c.d;
  const KView U{const_cast<double*>(u.p), nullptr, u.rs, 0, u.cs, 0, c.n}, Y{y.p, nullptr, y.rs, 0, y.cs, 0, c.n};
  return apply(c, U, Y, true, nodes, nodes, nodes, 1, nrhs);
}

// The same with the remaining DOF and the corner DOF of u and of y in separate buffers.
fetidp_status k_apply_K_split(Ctx& c, CCellVec ur, CCellVec up, CellVec yr, CellVec yp, int nrhs) {
  const int nodes = c.n / c.d;
  const KView U{const_cast<double*>(ur.p), const_cast<double*>(up.p), ur.rs, up.rs, ur.cs, up.cs, 0};
  const KView Y{yr.p, yp.p, yr.rs, yp.rs, yr.cs, yp.cs, 0};
  return apply(c, U, Y, false, nodes, nodes, c.nr / c.d, 1, nrhs);
}

}  // namespace fetidp
