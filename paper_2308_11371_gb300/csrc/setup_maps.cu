// Index maps and loads of the setup phase, built on the GPU: the multiplier maps (Eqs. 14-15), the
// corner maps (Eq. 18) and the right-hand side of Eq. 16 (Eq. 5b).
//
// Multiplier rows are numbered by global node (lexicographic, x fastest), so a node's first row is an
// exclusive sum of the row counts before it: one pass sums blocks of nodes, one block sums the sums, and
// the third pass scans its nodes again and writes their rows, every entry with one writer.  On the host
// the same loops took 7 ms for the 64 x 64 lattice of 16^2 elements (1 M nodes) and 2 ms for its loads,
// most of it starting threads and pageable uploads, before any kernel could start; whole set-up and solve
// on a GB300: 86.7 -> 76.9 ms there, 14.1 -> 12.1 ms for 4 x 4 cells of 8^2.
#include <algorithm>
#include <vector>

#include "common.cuh"

namespace fetidp {

namespace {

constexpr int kNodeBlock = 256, kNodeItems = 8;   // nodes per scan block: 256 threads x 8 consecutive nodes

struct LatNodes {
  int d, e, nd, nn1;
  int nc[3];
  long long gd[3], nodes;        // global grid
  long long cell0, clamp_coord;  // first cell; coordinate of the clamped plane
  int clamp_axis;
  long long row0, simple0, other0;   // rows before this lattice: all, in the first and second part of the order
};

// Owner cells of a node per axis (at most two), how many cells share it, and whether it is clamped.
// Returns the number of multiplier node rows (times d components), 0 off the interface.
__device__ __forceinline__ int node_rows(const LatNodes& L, long long t, int g[3], int cand[3][2], int nca[3],
                                         int& mult, bool& clamped) {
  g[0] = (int)(t % L.gd[0]);
  g[1] = (int)((t / L.gd[0]) % L.gd[1]);
  g[2] = (int)(t / (L.gd[0] * L.gd[1]));
  int on = 0;
  mult = 1;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    cand[k][0] = cand[k][1] = 0;
    nca[k] = 1;
    if (k >= L.d) continue;
    const int q = g[k] / L.e;
    if (g[k] - q * L.e == 0) {
      ++on;
      nca[k] = 0;
      if (q - 1 >= 0) cand[k][nca[k]++] = q - 1;
      if (q < L.nc[k]) cand[k][nca[k]++] = q;
    } else {
      cand[k][0] = q;
    }
    mult *= nca[k];
  }
  if (on == 0 || on == L.d) { mult = 0; return 0; }   // cell interior or lattice vertex (primal)
  clamped = g[L.clamp_axis] == L.clamp_coord;
  return clamped ? mult : mult - 1;
}

__device__ __forceinline__ long long block_exclusive(long long v, long long* sh, long long& total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  long long x = v;
  for (int o = 1; o < 32; o <<= 1) {
    const long long y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) sh[w] = x;
  __syncthreads();
  long long before = 0;
  total = 0;
  for (int k = 0; k < (int)(blockDim.x >> 5); ++k) {
    if (k < w) before += sh[k];
    total += sh[k];
  }
  __syncthreads();
  return before + x - v;
}

// Node rows of a thread's nodes: low half all rows, high half those of nodes with at most one row per
// component off the clamped plane (n <= 1: D is a number there).
__device__ __forceinline__ long long thread_rows(const LatNodes& L, long long t0) {
  long long s = 0;
  for (int k = 0; k < kNodeItems; ++k) {
    if (t0 + k >= L.nodes) break;
    int g[3], cand[3][2], nca[3], mult;
    bool clamped = false;
    const int r = node_rows(L, t0 + k, g, cand, nca, mult, clamped);
    s += r + ((clamped || mult <= 2) ? (long long)r << 32 : 0);
  }
  return s;
}

__global__ void __launch_bounds__(kNodeBlock) node_sum_kernel(LatNodes L, long long* __restrict__ sums) {
  __shared__ long long sh[kNodeBlock / 32];
  long long total;
  block_exclusive(thread_rows(L, ((long long)blockIdx.x * kNodeBlock + threadIdx.x) * kNodeItems), sh, total);
  if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

__global__ void __launch_bounds__(1024) node_scan_kernel(long long* __restrict__ sums, int n) {
  __shared__ long long sh[32];
  long long carry = 0;
  for (int b = 0; b < n; b += 1024) {
    const int i = b + threadIdx.x;
    const long long v = i < n ? sums[i] : 0;
    long long total;
    const long long ex = block_exclusive(v, sh, total);
    if (i < n) sums[i] = carry + ex;
    carry += total;
  }
}

__global__ void __launch_bounds__(kNodeBlock) node_fill_kernel(LatNodes L, const long long* __restrict__ sums,
                                                               const int* __restrict__ dual_pos,
                                                               int* __restrict__ gath, int* __restrict__ scat,
                                                               int* __restrict__ dinfo, int* __restrict__ order) {
  __shared__ long long sh[kNodeBlock / 32];
  const long long t0 = ((long long)blockIdx.x * kNodeBlock + threadIdx.x) * kNodeItems;
  long long total;
  long long at = sums[blockIdx.x] + block_exclusive(thread_rows(L, t0), sh, total);
  for (int k = 0; k < kNodeItems; ++k) {
    if (t0 + k >= L.nodes) break;
    int g[3], cand[3][2], nca[3], mult;
    bool clamped = false;
    const int rows = node_rows(L, t0 + k, g, cand, nca, mult, clamped);
    if (mult == 0) continue;
    const bool simple = clamped || mult <= 2;
    const long long all = at & 0xffffffffll, sb = at >> 32;
    const long long r0 = L.row0 + all * L.d;                                        // first row of the node
    const long long o0 = simple ? L.simple0 + sb * L.d : L.other0 + (all - sb) * L.d;   // its place in the order
    at += rows + (simple ? (long long)rows << 32 : 0);
    // the copies, by ascending cell
    long long prev = 0;
    int p = 0;
    for (int iz = 0; iz < nca[2]; ++iz)
      for (int iy = 0; iy < nca[1]; ++iy)
        for (int ix = 0; ix < nca[0]; ++ix, ++p) {
          const int cx = cand[0][ix], cy = cand[1][iy], cz = cand[2][iz];
          const long long s = L.cell0 + cx + (long long)L.nc[0] * (cy + (long long)L.nc[1] * cz);
          const int lx = g[0] - cx * L.e, ly = g[1] - cy * L.e, lz = L.d == 3 ? g[2] - cz * L.e : 0;
          const long long j0 = s * L.nd + (long long)dual_pos[lx + L.nn1 * (ly + L.nn1 * lz)] * L.d;
          for (int comp = 0; comp < L.d; ++comp) {
            const long long j = j0 + comp;
            if (clamped) {
              const long long r = r0 + (long long)p * L.d + comp;
              reinterpret_cast<int2*>(gath)[j] = make_int2((int)(r + 1), 0);
              reinterpret_cast<int2*>(scat)[r] = make_int2((int)(j + 1), 0);
              dinfo[r] = 0;
              if (order) order[o0 + (long long)p * L.d + comp] = (int)r;
            } else {
              // rows p - 1 (this copy second) and p (first)
              const int before = p > 0 ? -(int)(r0 + (long long)(p - 1) * L.d + comp + 1) : 0;
              const int after = p + 1 < mult ? (int)(r0 + (long long)p * L.d + comp + 1) : 0;
              reinterpret_cast<int2*>(gath)[j] = p > 0 ? make_int2(before, after) : make_int2(after, 0);
              if (p > 0) {
                const long long r = r0 + (long long)(p - 1) * L.d + comp;
                reinterpret_cast<int2*>(scat)[r] = make_int2((int)(prev + comp + 1), -(int)(j + 1));
                dinfo[r] = ((mult - 1) << 8) | (p - 1);
                if (order) order[o0 + (long long)(p - 1) * L.d + comp] = (int)r;
              }
            }
          }
          prev = j0;
        }
  }
}

struct LatVerts {
  int d, ncorner;
  int nc[3], vd[3], vf[3];       // cells, vertices, free vertices per axis
  int lo[3];                     // first free vertex per axis (1 on the clamped axis at side 0)
  long long cell0, V0, nfree;
};

// Free vertex number (lexicographic over the free vertices) or -1.
__device__ __forceinline__ int vertex_number(const LatVerts& V, const int v[3]) {
  long long n = 0, stride = 1;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int q = v[k] - V.lo[k];
    if (q < 0 || q >= V.vf[k]) return -1;
    n += q * stride;
    stride *= V.vf[k];
  }
  return (int)(V.V0 + n);
}

__global__ void corner_map_kernel(LatVerts V, long long ncell, int* __restrict__ corner_v) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < ncell * V.ncorner;
       t += (long long)gridDim.x * blockDim.x) {
    const long long s = t / V.ncorner;
    const int k = (int)(t - s * V.ncorner);
    const int v[3] = {(int)(s % V.nc[0]) + (k & 1), (int)((s / V.nc[0]) % V.nc[1]) + ((k >> 1) & 1),
                      V.d == 3 ? (int)(s / ((long long)V.nc[0] * V.nc[1])) + ((k >> 2) & 1) : 0};
    corner_v[V.cell0 * V.ncorner + t] = vertex_number(V, v);
  }
}

__global__ void vertex_cells_kernel(LatVerts V, int* __restrict__ vert_cells) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < V.nfree;
       t += (long long)gridDim.x * blockDim.x) {
    const int v[3] = {(int)(t % V.vf[0]) + V.lo[0], (int)((t / V.vf[0]) % V.vf[1]) + V.lo[1],
                      (int)(t / ((long long)V.vf[0] * V.vf[1])) + V.lo[2]};
    int* out = vert_cells + (V.V0 + t) * V.ncorner;
    int n = 0;
    for (int oz = V.d == 3 ? 1 : 0; oz >= 0; --oz)      // ascending cells: the vertex is a high corner first
      for (int oy = 1; oy >= 0; --oy)
        for (int ox = 1; ox >= 0; --ox) {
          const int cx = v[0] - ox, cy = v[1] - oy, cz = v[2] - oz;
          if (cx < 0 || cx >= V.nc[0] || cy < 0 || cy >= V.nc[1] || cz < 0 || cz >= V.nc[2]) continue;
          const long long s = V.cell0 + cx + (long long)V.nc[0] * (cy + (long long)V.nc[1] * cz);
          out[n++] = (int)(s * V.ncorner + ox + 2 * oy + 4 * oz);
        }
    for (; n < V.ncorner; ++n) out[n] = -1;
  }
}

// f^(s) of one traction load case (Eq. 5b) for the cells on the loaded face: one thread per (face cell, face
// node of the cell) sums the at most 2^(d-1) face elements at the node, in element order.
__global__ void traction_kernel(Geo g, int nr, int np, const int* __restrict__ iperm, int ax, int side, double dx,
                                double dy, double dz, long long cell0, double* __restrict__ rhs,
                                double* __restrict__ fpc) {
  const int d = g.dim, e = g.e, nn1 = e + 1;
  int tang[2] = {0, 0}, nt = 0;
  for (int k = 0; k < d; ++k)
    if (k != ax) tang[nt++] = k;
  const bool two = nt == 2;
  const int n0 = g.nc[tang[0]], n1 = two ? g.nc[tang[1]] : 1;
  const int fnode = two ? nn1 * nn1 : nn1;
  const double h = 1.0 / e;
  double hw = 1.0;
  for (int k = 0; k + 1 < d; ++k) hw *= 0.5 * h;
  const double dir[3] = {dx, dy, dz};
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < (long long)n0 * n1 * fnode;
       t += (long long)gridDim.x * blockDim.x) {
    const long long fc = t / fnode;
    const int fn = (int)(t - fc * fnode);
    int cc[3] = {0, 0, 0}, nd3[3] = {0, 0, 0};
    cc[ax] = side ? g.nc[ax] - 1 : 0;
    cc[tang[0]] = (int)(fc % n0);
    if (two) cc[tang[1]] = (int)(fc / n0);
    nd3[ax] = side ? e : 0;
    nd3[tang[0]] = fn % nn1;
    if (two) nd3[tang[1]] = fn / nn1;
    double f = 0.0;
    for (int b1 = two ? 1 : 0; b1 >= 0; --b1)        // the node is the element's high node first
      for (int b0 = 1; b0 >= 0; --b0) {
        const int e0 = nd3[tang[0]] - b0, e1 = two ? nd3[tang[1]] - b1 : 0;
        if (e0 < 0 || e0 >= e || e1 < 0 || e1 >= (two ? e : 1)) continue;
        for (int fg = 0; fg < (1 << (d - 1)); ++fg) {
          double tq[3] = {0.0, 0.0, 0.0};
          tq[ax] = side ? 1.0 : 0.0;
          for (int q = 0; q < nt; ++q) tq[tang[q]] = gauss_t((fg >> q) & 1);
          int ec[3] = {0, 0, 0};
          ec[ax] = side ? e - 1 : 0;
          ec[tang[0]] = e0;
          if (two) ec[tang[1]] = e1;
          double xi[3] = {0.0, 0.0, 0.0}, J[3][3];
          for (int k = 0; k < d; ++k) xi[k] = cc[k] + (ec[k] + tq[k]) * h;
          macro_jacobian(g, xi, J);
          double meas;
          if (d == 2) {
            meas = sqrt(J[0][tang[0]] * J[0][tang[0]] + J[1][tang[0]] * J[1][tang[0]]);
          } else {
            const double a[3] = {J[0][tang[0]], J[1][tang[0]], J[2][tang[0]]};
            const double b[3] = {J[0][tang[1]], J[1][tang[1]], J[2][tang[1]]};
            const double cr[3] = {a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]};
            meas = sqrt(cr[0] * cr[0] + cr[1] * cr[1] + cr[2] * cr[2]);
          }
          double Nv = b0 ? tq[tang[0]] : 1.0 - tq[tang[0]];
          if (two) Nv *= b1 ? tq[tang[1]] : 1.0 - tq[tang[1]];
          f += hw * meas * Nv;
        }
      }
    const long long s = cell0 + cc[0] + (long long)g.nc[0] * (cc[1] + (long long)g.nc[1] * cc[2]);
    const int node = nd3[0] + nn1 * (nd3[1] + (d == 3 ? nn1 * nd3[2] : 0));
    for (int i = 0; i < d; ++i) {
      const int li = iperm[node * d + i];
      if (li < nr) rhs[s * nr + li] = f * dir[i];
      else fpc[s * np + (li - nr)] = f * dir[i];
    }
  }
}

inline unsigned grid_of(long long work, int threads) {
  return (unsigned)std::max<long long>(1, std::min<long long>((work + threads - 1) / threads, 152LL * 32));
}

}  // namespace

// Rows, row order and corner maps of every lattice; fills c.L, c.nV, c.nP, the lattices' offsets and the maps.
fetidp_status k_build_maps(Ctx& c, const int* dual_pos_dev) {
  const int d = c.d, e = c.e;
  // counts: copies of interface nodes less their free nodes (one row per copy pair, per copy if clamped)
  long long L = 0, nV = 0, other = 0;
  std::vector<LatNodes> nodes(c.lat.size());
  std::vector<LatVerts> verts(c.lat.size());
  for (size_t b = 0; b < c.lat.size(); ++b) {
    LatticeSpan& ls = c.lat[b];
    LatNodes& G = nodes[b];
    LatVerts& V = verts[b];
    G = LatNodes{};
    V = LatVerts{};
    G.d = V.d = d;
    G.e = e;
    G.nd = c.nd;
    G.nn1 = e + 1;
    V.ncorner = c.ncorner;
    G.cell0 = V.cell0 = ls.cell0;
    G.clamp_axis = ls.clamp_axis;
    long long interior = ls.ncell, nvert = 1, plane = 1, plane_vert = 1;
    G.nodes = 1;
    V.nfree = 1;
    for (int k = 0; k < 3; ++k) {
      const int nc = ls.geo.nc[k];
      G.nc[k] = V.nc[k] = nc;
      G.gd[k] = k < d ? (long long)nc * e + 1 : 1;
      V.vd[k] = V.vf[k] = k < d ? nc + 1 : 1;
      G.nodes *= G.gd[k];
      nvert *= V.vd[k];
      if (k < d) interior *= e - 1;
      if (k < d && k != ls.clamp_axis) { plane *= G.gd[k]; plane_vert *= V.vd[k]; }
      if (k == ls.clamp_axis) {
        V.vf[k] -= 1;
        V.lo[k] = ls.clamp_side ? 0 : 1;
      }
      V.nfree *= V.vf[k];
    }
    G.clamp_coord = ls.clamp_side ? G.gd[ls.clamp_axis] - 1 : 0;
    const long long iface = G.nodes - interior - nvert;
    ls.L0 = L;
    ls.nL = ls.ncell * c.nd - d * (iface - (plane - plane_vert));
    ls.V0 = V.V0 = nV;
    ls.nV = V.nfree;
    G.row0 = L;
    long long many = 0;   // rows of nodes with three rows per component: interior cell edges in 3D
    if (d == 3)
      for (int a = 0; a < 3; ++a) {
        const int p = (a + 1) % 3, q = (a + 2) % 3;
        many += 3LL * d * (G.nc[p] - 1) * (G.nc[q] - 1) * G.nc[a] * (e - 1);
      }
    G.simple0 = L - other;   // rows of the first part so far
    G.other0 = other;        // + all rows of the first part, below
    L += ls.nL;
    nV += ls.nV;
    other += many;
  }
  c.L = L;
  c.nV = (int)nV;
  c.nP = nV * d;
  FD_TRY(dalloc_t(c, &c.gath, (size_t)c.N * c.nd * 2));
  FD_TRY(dalloc_t(c, &c.scat, 2 * (size_t)std::max(L, 1LL)));
  FD_TRY(dalloc_t(c, &c.dinfo, (size_t)std::max(L, 1LL)));
  if (d == 3) FD_TRY(dalloc_t(c, &c.row_order, (size_t)std::max(L, 1LL)));
  FD_TRY(dalloc_t(c, &c.corner_v, (size_t)c.N * c.ncorner));
  FD_TRY(dalloc_t(c, &c.vert_cells, (size_t)std::max(nV, 1LL) * c.ncorner));
  long long most = 1;
  for (const LatNodes& G : nodes) most = std::max(most, (G.nodes + kNodeBlock * kNodeItems - 1) / (kNodeBlock * kNodeItems));
  long long* sums = nullptr;
  FD_TRY(tmp_alloc(c, reinterpret_cast<void**>(&sums), sizeof(long long) * most));
  ProfScope ps(c, FETIDP_K_SETUP, 0.0, 16.0 * (double)c.N * c.nd + 12.0 * (double)L);
  for (size_t b = 0; b < c.lat.size(); ++b) {
    LatNodes G = nodes[b];
    G.other0 += L - other;
    const unsigned nb = (unsigned)((G.nodes + kNodeBlock * kNodeItems - 1) / (kNodeBlock * kNodeItems));
    node_sum_kernel<<<nb, kNodeBlock, 0, c.stream>>>(G, sums);
    count_launch();
    node_scan_kernel<<<1, 1024, 0, c.stream>>>(sums, (int)nb);
    count_launch();
    node_fill_kernel<<<nb, kNodeBlock, 0, c.stream>>>(G, sums, dual_pos_dev, c.gath, c.scat, c.dinfo, c.row_order);
    count_launch();
    const LatVerts& V = verts[b];
    corner_map_kernel<<<grid_of(c.lat[b].ncell * c.ncorner, 256), 256, 0, c.stream>>>(V, c.lat[b].ncell, c.corner_v);
    count_launch();
    vertex_cells_kernel<<<grid_of(V.nfree, 256), 256, 0, c.stream>>>(V, c.vert_cells);
    count_launch();
  }
  tmp_free(c, sums);
  if (cudaPeekAtLastError() != cudaSuccess) {
    set_error(std::string("kernel launch: ") + cudaGetErrorString(cudaGetLastError()));
    return FETIDP_ECUDA;
  }
  return FETIDP_OK;
}

// rhs = (f_R, f_P, 0) of every load case and each cell's own corner loads.
fetidp_status k_build_loads(Ctx& c, const fetidp_problem* probs) {
  const int d = c.d, m = c.m;
  FD_TRY(dalloc_t(c, &c.rhs, (size_t)m * c.ntot));
  FD_TRY(dalloc_t(c, &c.rhs_p_cells, (size_t)m * c.N * c.np));
  FD_CUDA(cudaMemsetAsync(c.rhs, 0, sizeof(double) * (size_t)m * c.ntot, c.stream));
  FD_CUDA(cudaMemsetAsync(c.rhs_p_cells, 0, sizeof(double) * (size_t)m * c.N * c.np, c.stream));
  for (size_t b = 0; b < c.lat.size(); ++b) {
    const fetidp_problem& p = probs[b];
    const LatticeSpan& ls = c.lat[b];
    std::vector<int> body(m);
    bool any_body = false;
    for (int l = 0; l < m; ++l) {
      body[l] = p.load_kind[l] == 1 ? 1 : 0;
      any_body = any_body || body[l];
      if (body[l]) continue;
      const int ax = p.load_axis[l];
      if (ax < 0 || ax > 2) { set_error("bad load axis"); return FETIDP_EINVAL; }
      if (ax >= d && p.load_side[l]) continue;   // 2D: every cell lies on side 0 of the third axis, none on side 1
      long long work = 1;
      for (int k = 0; k < d; ++k)
        if (k < d && k != ax) work *= (long long)ls.geo.nc[k] * (c.e + 1);
      const double* dir = p.load_dir + (size_t)l * d;
      traction_kernel<<<grid_of(work, 128), 128, 0, c.stream>>>(
          ls.geo, c.nr, c.np, c.perm + c.n, ax, p.load_side[l] ? 1 : 0, dir[0], dir[1], d == 3 ? dir[2] : 0.0, ls.cell0,
          c.rhs + (size_t)l * c.ntot, c.rhs_p_cells + (size_t)l * c.N * c.np);
      FD_CHECK_LAUNCH();
    }
    if (any_body) {
      int* body_d = nullptr;
      double* dirs_d = nullptr;
      FD_TRY(tmp_alloc(c, reinterpret_cast<void**>(&body_d), sizeof(int) * m));
      FD_TRY(tmp_alloc(c, reinterpret_cast<void**>(&dirs_d), sizeof(double) * (size_t)m * d));
      FD_CUDA(cudaMemcpyAsync(body_d, body.data(), sizeof(int) * m, cudaMemcpyHostToDevice, c.stream));
      FD_CUDA(cudaMemcpyAsync(dirs_d, p.load_dir, sizeof(double) * (size_t)m * d, cudaMemcpyHostToDevice, c.stream));
      FD_TRY(k_body_loads(c, ls, c.perm, dirs_d, body_d, c.rhs, c.ntot, c.rhs_p_cells));
      FD_CUDA(cudaStreamSynchronize(c.stream));   // host vectors go out of scope
      tmp_free(c, body_d);
      tmp_free(c, dirs_d);
    }
  }
  // f_P from every cell's corner loads (Eq. 18)
  return k_primal_assemble(c, CCellVec{c.rhs_p_cells, c.N * c.np, c.np}, c.rhs + c.N * c.nr, c.ntot, 1.0, 0.0, m);
}

}  // namespace fetidp
