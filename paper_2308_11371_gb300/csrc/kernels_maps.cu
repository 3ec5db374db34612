// Integer-indexed maps of the FETI-DP hot path and FP64 vector kernels.
//
// * B_d^T gather and B_d scatter (Eq. 15; used in Eqs. 48-49 and Algorithm 3):
//   both are written as row-wise gathers over at most two signed terms in a
//   fixed order, so they are bit-exact and need no atomics.
// * A_p assembly / extraction of corner values (Eq. 18).
// * Deterministic FP64 reductions for the Krylov recurrences: a fixed
//   partition into at most kRedBlocks blocks, warp-shuffle trees, then the
//   partials summed in a fixed order by the last block to arrive.
#include "common.cuh"

namespace fetidp {

namespace {

constexpr int kRedBlocks = kReductionBlocks;
constexpr int kRedThreads = 256;

// Dirichlet-preconditioner scaling D = (B B^T)^{-1} (Eq. 30: sum_s B_d B_d^T D = I_L).
// B B^T is block diagonal over the rows of one node and component.  dinfo[row] = (n << 8) | q:
// the row is chain row q of the n chain rows of its node (rows of one node and component lie d
// apart), n = 0 for a Dirichlet row (block 1).  The block is the inverse of the n x n matrix
// tridiag(-1, 2, -1), (T^{-1})_ab = (min(a, b) + 1)(n - max(a, b)) / (n + 1): 1/2 for n = 1
// (every 2D row, 3D face rows), quarters for the n = 3 rows of a 3D cell edge (exact in binary).
// The blocks for n = 1, 2, 3 as constants (each the correctly rounded quotient, as a run-time FP64
// division would give): GB300's FP64 divide is a long software sequence on its slow FP64 pipe.
__device__ __forceinline__ double tinv(int a, int b, int n) {
  const int lo = a < b ? a : b, hi = a < b ? b : a;
  const int num = (lo + 1) * (n - hi);
  if (n == 1) return 0.5;
  if (n == 2) return num == 2 ? 2.0 / 3.0 : 1.0 / 3.0;
  if (n == 3) return 0.25 * num;
  return (double)num / (double)(n + 1);
}


// -x when neg is 1, by the sign bit alone (no FP64 instruction: GB300 runs FP64 at 1/64 of FP32)
__device__ __forceinline__ double flip_sign(double x, int neg) {
  return __longlong_as_double(__double_as_longlong(x) ^ ((long long)neg << 63));
}

// x_d = B_d^T lambda, or B_d^T D lambda when dinfo is given.  One thread per (cell, dual DOF):
// the (multiplier row, weight) terms of the entry -- at most two signed rows, each expanded into
// at most three rows by the D block -- are decoded once, then applied to every RHS.  Entries of one row
// with weight 1 or 1/2 (every face node, every 2D node) take no FP64 instruction: sign and exponent are set
// on the bits (the FP64 sum 0 + w l is exact).  Other entries take one FP64 addition or FMA per term.
// order: the cell's dual DOF with the face nodes' first, so that a warp takes one path.
// XF: the values are rounded once into an FP32 layout instead of FP64 cell vectors.
// 2,048 cells of n_d = 630, 6 RHS: the two scaled maps of a preconditioner application 222 -> 154 us.
template <bool XF>
__global__ void gather_BT_kernel(const int* __restrict__ gath, const double* __restrict__ lam,
                                 long long lam_rs, const int* __restrict__ dinfo, int d,
                                 const int* __restrict__ order, double* __restrict__ out, long long out_rs, int out_cs,
                                 int nd, long long ncell, int nrhs, double beta, XfLayout F) {
  const int width = XF ? F.width : nd;
  const int total = (int)(ncell * width);            // < 2^31, checked by the host
  const bool overwrite = beta == 0.0;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
    const int cell = t / width;
    const int jt = t - cell * width;
    if (XF && jt >= nd) {
      for (int rhs = 0; rhs < nrhs; ++rhs) F.p[(rhs >> 3) * F.chs + (rhs & 7) * F.rs + cell * F.cs + jt * F.ds] = 0.f;
      continue;
    }
    const int j = order ? order[jt] : jt;
    const int2 cc = reinterpret_cast<const int2*>(gath)[(long long)cell * nd + j];
    // six term slots in registers (fixed trip counts); live / neg are bit masks over the slots
    int idx[6];
    double w[6];
    int live = 0, neg = 0;
    bool unit = true;
#pragma unroll
    for (int k = 0; k < 6; ++k) { idx[k] = 0; w[k] = 0.0; }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int code = h ? cc.y : cc.x;
      if (code == 0) continue;
      const int row = (code > 0 ? code : -code) - 1;
      const int sg = code < 0 ? 1 : 0;
      const int dc = dinfo ? dinfo[row] : 0;
      const int n = dc >> 8, q = dc & 0xff;
      if (n <= 1) {
        idx[3 * h] = row;
        live |= 1 << (3 * h);
        neg |= sg << (3 * h);
        unit = unit && n == 0;
        const double t1 = n == 0 ? 1.0 : 0.5;
        w[3 * h] = sg ? -t1 : t1;
        continue;
      }
      unit = false;
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        if (b < n) {
          const int k = 3 * h + b;
          idx[k] = row + (b - q) * d;
          const double tb = tinv(q, b, n);
          w[k] = sg ? -tb : tb;
          live |= 1 << k;
        }
      }
    }
    const bool single = live == 1 && (unit || w[0] == 0.5 || w[0] == -0.5);
    auto value = [&](int rhs) {
      const double* l = lam + rhs * lam_rs;
      double v;
      if (single) {
        v = flip_sign(l[idx[0]], neg & 1);
        if (!unit) v = fd_half(v);
        if (__double_as_longlong(v) == (long long)0x8000000000000000ull) v = 0.0;   // 0 + (-0)
      } else if (unit) {
        const double a = (live & 1) ? l[idx[0]] : 0.0, bv = (live & 8) ? l[idx[3]] : 0.0;
        v = flip_sign(a, neg & 1) + flip_sign(bv, (neg >> 3) & 1);
      } else {
        v = 0.0;
#pragma unroll
        for (int k = 0; k < 6; ++k)
          if ((live >> k) & 1) v = fma(w[k], l[idx[k]], v);
      }
      return v;
    };
    if (XF) {
      for (int r0 = 0; r0 < nrhs; r0 += 4) {
        float* o = F.p + (r0 >> 3) * F.chs + (r0 & 7) * F.rs + cell * F.cs + j * F.ds;
        float v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = r0 + q < nrhs ? fd_round(value(r0 + q)) : 0.f;
        if (F.P >= 4) *reinterpret_cast<float4*>(o) = make_float4(v[0], v[1], v[2], v[3]);
        else if (F.P == 2) *reinterpret_cast<float2*>(o) = make_float2(v[0], v[1]);
        else
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (r0 + q < nrhs) o[q * F.rs] = v[q];
      }
      continue;
    }
    for (int rhs = 0; rhs < nrhs; ++rhs) {
      const double v = value(rhs);
      double* o = out + rhs * out_rs + (long long)cell * out_cs + j;
      *o = overwrite ? v : v + beta * (*o);
    }
  }
}

// FP64 cell vectors rounded into the RHS-interleaved FP32 layout (len entries per cell).
__global__ void pack_f32_kernel(const double* __restrict__ x, long long x_rs, int x_cs, int len, long long ncell,
                                int nrhs, float* __restrict__ xf, int P, int xcs) {
  const long long per = ncell * len;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < per;
       t += (long long)gridDim.x * blockDim.x) {
    const long long cell = t / len;
    const int j = (int)(t - cell * len);
    const double* xc = x + cell * x_cs + j;
    for (int r0 = 0; r0 < nrhs; r0 += 4) {
      float* o = xf + (r0 >> 3) * ncell * xcs + cell * xcs + j * P + (r0 & 7);
      float v[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) v[q] = r0 + q < nrhs ? fd_round(xc[(r0 + q) * x_rs]) : 0.f;
      if (P >= 4) *reinterpret_cast<float4*>(o) = make_float4(v[0], v[1], v[2], v[3]);
      else if (P == 2) *reinterpret_cast<float2*>(o) = make_float2(v[0], v[1]);
      else *o = v[0];
    }
  }
}

// z = alpha B y + beta z, or alpha D B y + beta z when dinfo is given.  One thread per row: the
// (cell entry, weight) terms -- two signed copies of each of at most three chain rows -- are decoded
// once, then applied to every RHS.  A row of one weight (n <= 1: every 2D row, 3D face rows) is one signed
// FP64 sum, halved in the exponent for n = 1 (the rounding of the sum of the halves); order: rows with
// those first, so that a warp takes one path.  y in FP64, or FP32 as the FP32 cell operators leave it.
template <typename T>
__global__ void scatter_B_kernel(const int* __restrict__ scat, const T* __restrict__ yd,
                                 long long y_rs, int y_cs, int nd, const int* __restrict__ dinfo,
                                 int d, const int* __restrict__ order, double* __restrict__ out, long long out_rs,
                                 long long L, double alpha, double beta, int nrhs) {
  const int Li = (int)L;                             // < 2^31, checked by the host
  const bool overwrite = beta == 0.0, unscaled = alpha == 1.0;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < Li; t += gridDim.x * blockDim.x) {
    const int row = order ? order[t] : t;
    const int code = dinfo ? dinfo[row] : 0;
    const int n = code >> 8, q = code & 0xff;
    long long idx[6];
    double w[6];
    int live = 0, neg = 0;
#pragma unroll
    for (int k = 0; k < 6; ++k) { idx[k] = 0; w[k] = 0.0; }
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      if (b > 0 && b >= n) break;
      const int r = n <= 1 ? row : row + (b - q) * d;
      const double wr = n <= 1 ? 1.0 : tinv(q, b, n);
      const int2 sc = reinterpret_cast<const int2*>(scat)[r];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int c = h ? sc.y : sc.x;
        if (c == 0) continue;
        const int e = (c > 0 ? c : -c) - 1;
        const int cell = e / nd;
        const int k = 2 * b + h;
        idx[k] = (long long)cell * y_cs + (e - cell * nd);
        w[k] = c > 0 ? wr : -wr;
        live |= 1 << k;
        neg |= (c < 0 ? 1 : 0) << k;
      }
    }
#pragma unroll 2
    for (int rhs = 0; rhs < nrhs; ++rhs) {
      const T* y = yd + rhs * y_rs;
      double v;
      if (n <= 1) {
        const double a = (live & 1) ? fd_load(y[idx[0]]) : 0.0, bv = (live & 2) ? fd_load(y[idx[1]]) : 0.0;
        v = flip_sign(a, neg & 1) + flip_sign(bv, (neg >> 1) & 1);
        if (n == 1) v = fd_half(v);
      } else {
        v = 0.0;
#pragma unroll
        for (int k = 0; k < 6; ++k)
          if ((live >> k) & 1) v = fma(w[k], fd_load(y[idx[k]]), v);
      }
      double* o = out + rhs * out_rs + row;
      const double av = unscaled ? v : alpha * v;
      *o = overwrite ? av : av + beta * (*o);
    }
  }
}

__global__ void primal_assemble_kernel(const int* __restrict__ vert_cells, int ncorner, int d,
                                       const double* __restrict__ cp, long long c_rs, int c_cs,
                                       double* __restrict__ out, long long out_rs, int nV,
                                       double alpha, double beta, int nrhs) {
  const long long total = (long long)nV * d;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total * nrhs;
       t += (long long)gridDim.x * blockDim.x) {
    const int rhs = (int)(t / total);
    const long long vc = t - rhs * total;
    const int v = (int)(vc / d), comp = (int)(vc - (long long)v * d);
    double s = 0.0;
    for (int q = 0; q < ncorner; ++q) {
      const int code = vert_cells[v * ncorner + q];
      if (code < 0) continue;
      const long long cell = code / ncorner;
      const int k = code - (int)cell * ncorner;
      s += cp[rhs * c_rs + cell * c_cs + k * d + comp];
    }
    double* o = out + rhs * out_rs + vc;
    *o = (beta == 0.0) ? alpha * s : alpha * s + beta * (*o);
  }
}

__global__ void primal_extract_kernel(const int* __restrict__ corner_v, int ncorner, int d,
                                      const double* __restrict__ uP, long long uP_rs,
                                      double* __restrict__ cp, long long c_rs, int c_cs,
                                      long long ncell, int nrhs) {
  const int npc = ncorner * d;
  const long long total = ncell * npc;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total * nrhs;
       t += (long long)gridDim.x * blockDim.x) {
    const int rhs = (int)(t / total);
    const long long ck = t - rhs * total;
    const long long cell = ck / npc;
    const int q = (int)(ck - cell * npc);
    const int k = q / d, comp = q - k * d;
    const int v = corner_v[cell * ncorner + k];
    cp[rhs * c_rs + cell * c_cs + q] = v >= 0 ? uP[rhs * uP_rs + (long long)v * d + comp] : 0.0;
  }
}

// The same corner values rounded to FP32, the RHS of a chunk of eight adjacent (0 for absent ones).
__global__ void primal_extract_f32_kernel(const int* __restrict__ corner_v, int ncorner, int d,
                                          const double* __restrict__ uP, long long uP_rs, float* __restrict__ cpf,
                                          long long ncell, int nrhs) {
  const int npc = ncorner * d;
  const long long total = ncell * npc;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const long long cell = t / npc;
    const int q = (int)(t - cell * npc), k = q / d, comp = q - k * d;
    const int v = corner_v[cell * ncorner + k];
    for (int r0 = 0; r0 < nrhs; r0 += 8) {
      float o[8];
#pragma unroll
      for (int r = 0; r < 8; ++r)
        o[r] = v >= 0 && r0 + r < nrhs ? fd_round(uP[(r0 + r) * uP_rs + (long long)v * d + comp]) : 0.f;
      float4* dst = reinterpret_cast<float4*>(cpf + ((r0 >> 3) * total + t) * 8);
      dst[0] = make_float4(o[0], o[1], o[2], o[3]);
      if (nrhs - r0 > 4) dst[1] = make_float4(o[4], o[5], o[6], o[7]);
    }
  }
}

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// Block-wide sum; result valid in thread 0.
__device__ __forceinline__ double block_sum(double v, double* sh) {
  v = warp_sum(v);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) sh[w] = v;
  __syncthreads();
  double r = 0.0;
  if (w == 0) {
    r = (lane < (int)(blockDim.x >> 5)) ? sh[lane] : 0.0;
    r = warp_sum(r);
  }
  __syncthreads();
  return r;
}

// Sum of one value per block over the blocks blockIdx.x of a launch (deterministic, one launch): every block
// leaves its value in part[blockIdx.x]; the last one to arrive (a counter that it leaves at zero) adds them
// in a fixed order and tree.  True in thread 0 of that block, with the total in `total`.
__device__ __forceinline__ bool grid_sum(double v, double* __restrict__ part, unsigned* __restrict__ count,
                                         double* sh, double& total) {
  __shared__ bool last;
  v = block_sum(v, sh);
  if (threadIdx.x == 0) {
    part[blockIdx.x] = v;
    __threadfence();
    last = atomicAdd(count, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return false;
  __threadfence();
  double s = 0.0;
  for (int t = threadIdx.x; t < (int)gridDim.x; t += blockDim.x) s += __ldcg(part + t);
  total = block_sum(s, sh);
  if (threadIdx.x == 0) *count = 0u;
  return threadIdx.x == 0;
}

// out[rhs*nv + i] = V_i[rhs] . w[rhs], V_i at Vb + i*vstride + rhs*vrs: blockIdx.x a fixed slice, y the RHS,
// z the vector.
__global__ void multi_dot_kernel(const double* __restrict__ Vb, long long vstride, long long vrs,
                                 const double* __restrict__ w, long long wrs, long long len,
                                 int nv, double* __restrict__ partial, unsigned* __restrict__ count,
                                 double* __restrict__ out) {
  __shared__ double sh[32];
  const int i = blockIdx.z, rhs = blockIdx.y, blk = blockIdx.x;
  const double* v = Vb + i * vstride + rhs * vrs;
  const double* x = w + rhs * wrs;
  const long long chunk = (len + gridDim.x - 1) / gridDim.x;
  const long long beg = blk * chunk;
  const long long end = beg + chunk < len ? beg + chunk : len;
  double s = 0.0;
#pragma unroll 4
  for (long long t = beg + threadIdx.x; t < end; t += blockDim.x) s += v[t] * x[t];
  const long long k = (long long)rhs * nv + i;
  double total;
  if (grid_sum(s, partial + k * kRedBlocks, count + k, sh, total)) out[k] = total;
}

__global__ void reduce_partials(const double* __restrict__ partial, int count,
                                double* __restrict__ out) {
  __shared__ double sh[32];
  const int k = blockIdx.x;
  double s = 0.0;
  // fixed assignment of partials to threads, then a fixed tree
  for (int t = threadIdx.x; t < kRedBlocks; t += blockDim.x) s += partial[(long long)k * kRedBlocks + t];
  s = block_sum(s, sh);
  if (threadIdx.x == 0) out[k] = s;
  (void)count;
}

// One PCG update: x += alpha p, r -= alpha q, alpha = rz / pq, and r . r of the new residual; blockIdx.y is the
// RHS (converged ones leave at once).  With tol >= 0 the last block of an RHS also makes the convergence
// test: counts the iteration, flags a breakdown (p^T F p <= 0 or a non-finite residual) and clears the
// active flag when ||r|| / ||r_0|| <= tol or r = 0, so whole iterations run without a host round trip.
__global__ void pcg_update_kernel(double* __restrict__ X, double* __restrict__ R, const double* __restrict__ P,
                                  const double* __restrict__ Q, double* __restrict__ scal, PcgSlots S, long long L,
                                  int nrhs, double tol, double* __restrict__ partial, unsigned* __restrict__ count) {
  __shared__ double sh[32];
  const int rhs = blockIdx.y;
  if (scal[S.act * nrhs + rhs] == 0.0) return;
  const double pq = scal[S.pq * nrhs + rhs];
  const double alpha = scal[S.rz * nrhs + rhs] / pq;
  const long long chunk = (L + gridDim.x - 1) / gridDim.x, beg = blockIdx.x * chunk, o = rhs * L;
  const long long end = beg + chunk < L ? beg + chunk : L;
  double s = 0.0;
#pragma unroll 2
  for (long long t = beg + threadIdx.x; t < end; t += blockDim.x) {
    X[o + t] += alpha * P[o + t];
    const double r = R[o + t] - alpha * Q[o + t];
    R[o + t] = r;
    s += r * r;
  }
  double rr;
  if (!grid_sum(s, partial + (long long)rhs * kRedBlocks, count + rhs, sh, rr)) return;
  scal[S.rr * nrhs + rhs] = rr;
  if (tol < 0.0) return;
  scal[S.its * nrhs + rhs] += 1.0;
  if (!(pq > 0.0) || !isfinite(rr)) {
    scal[S.err * nrhs + rhs] = 1.0;
    scal[S.act * nrhs + rhs] = 0.0;
  } else if (sqrt(rr / scal[S.r0 * nrhs + rhs]) <= tol || rr == 0.0) {
    scal[S.act * nrhs + rhs] = 0.0;
  }
}

// p = z + beta p, beta = rz_new / rz_old, for the active RHS (blockIdx.y)
__global__ void pcg_p_kernel(double* __restrict__ P, const double* __restrict__ Zv,
                             const double* __restrict__ scal, int act, int new_slot, int old_slot, long long L,
                             int nrhs) {
  const int rhs = blockIdx.y;
  if (scal[act * nrhs + rhs] == 0.0) return;
  const double beta = scal[new_slot * nrhs + rhs] / scal[old_slot * nrhs + rhs];
  double* p = P + rhs * L;
  const double* z = Zv + rhs * L;
#pragma unroll 4
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < L; t += (long long)gridDim.x * blockDim.x)
    p[t] = z[t] + beta * p[t];
}

// Compliance partial sums: sum over (cell, local dof) of f . u for one load case, with f the
// remaining-DOF part of the outer right-hand side and the cells' own corner loads, and u in
// natural cell order.  Fixed chunk per block, fixed tree in the block (deterministic).
__global__ void compliance_partial(const double* __restrict__ rhs, long long ntot, const double* __restrict__ fp,
                                   const double* __restrict__ u, const int* __restrict__ perm, int n, int nr,
                                   long long ncell, double* __restrict__ partial) {
  __shared__ double sh[32];
  const int rhs_i = blockIdx.y, blk = blockIdx.x;
  const long long len = ncell * n;
  const long long chunk = (len + kRedBlocks - 1) / kRedBlocks;
  const long long beg = blk * chunk;
  const long long end = beg + chunk < len ? beg + chunk : len;
  const double* fr = rhs + rhs_i * ntot;
  const double* fq = fp + rhs_i * ncell * (n - nr);
  const double* uc = u + rhs_i * len;
  double acc = 0.0;
  for (long long t = beg + threadIdx.x; t < end; t += blockDim.x) {
    const long long s = t / n;
    const int li = (int)(t - s * n);
    const double f = li < nr ? fr[s * nr + li] : fq[s * (n - nr) + (li - nr)];
    acc += f * uc[s * n + perm[li]];
  }
  acc = block_sum(acc, sh);
  if (threadIdx.x == 0) partial[(long long)rhs_i * kRedBlocks + blk] = acc;
}

__global__ void multi_axpy_kernel(const double* __restrict__ Vb, long long vstride, long long vrs,
                                  int nv, const double* __restrict__ coef, double* __restrict__ w,
                                  long long wrs, long long len, int nrhs, double sign) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < len * nrhs;
       t += (long long)gridDim.x * blockDim.x) {
    const int rhs = (int)(t / len);
    const long long q = t - rhs * len;
    double s = 0.0;
    for (int i = 0; i < nv; ++i) s += coef[rhs * nv + i] * Vb[i * vstride + rhs * vrs + q];
    w[rhs * wrs + q] += sign * s;
  }
}

__global__ void copy_scale_kernel(const double* __restrict__ x, double* __restrict__ y,
                                  long long len, int nrhs, long long xs, long long ys,
                                  const double* __restrict__ s_dev, double s_host) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < len * nrhs;
       t += (long long)gridDim.x * blockDim.x) {
    const int rhs = (int)(t / len);
    const long long q = t - rhs * len;
    const double s = s_dev ? s_dev[rhs] : s_host;
    y[rhs * ys + q] = s * x[rhs * xs + q];
  }
}

// *flag = 1 (host-mapped) if any x[i] is NaN or +-Inf (input validation of the C entry points)
__global__ void nonfinite_kernel(const double* __restrict__ x, long long n, int* __restrict__ flag) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    if (!fd_finite(x[i])) {
      *reinterpret_cast<volatile int*>(flag) = 1;
      return;
    }
}

// blocks per reduced vector: at least four entries per thread, at most two blocks per SM
inline int red_blocks(long long len) {
  const long long b = (len + 4 * kRedThreads - 1) / (4 * kRedThreads);
  return (int)(b < 1 ? 1 : b > kRedBlocks ? kRedBlocks : b);
}

inline int grid_for(long long work, int threads = 256) {
  long long g = (work + threads - 1) / threads;
  if (g > 152LL * 16) g = 152LL * 16;
  if (g < 1) g = 1;
  return (int)g;
}

}  // namespace

fetidp_status k_gather_BT(Ctx& c, const double* lam, long long lam_rs, const int* dinfo,
                          CellVec out, int nrhs, double beta) {
  const long long work = c.N * c.nd;
  if (work >= (1LL << 31) || c.L >= (1LL << 31)) { set_error("lattice too large for 32-bit map indices"); return FETIDP_EINVAL; }
  ProfScope ps(c, FETIDP_K_MAPS, 0.0, (double)nrhs * (c.L * 8.0 + c.N * c.nd * 8.0) + c.N * c.nd * 8.0);
  gather_BT_kernel<false><<<grid_for(work), 256, 0, c.stream>>>(c.gath, lam, lam_rs, dinfo, c.d, c.dual_order, out.p,
                                                                out.rs, out.cs, c.nd, c.N, nrhs, beta, XfLayout{});
  FD_CHECK_LAUNCH();
  return FETIDP_OK;
}

// B_d^T lambda (or B_d^T D lambda) rounded into an FP32 layout.
fetidp_status k_gather_BT_f32(Ctx& c, const double* lam, long long lam_rs, const int* dinfo, const XfLayout& xf,
                              int nrhs) {
  const long long work = c.N * xf.width;
  if (work >= (1LL << 31) || c.L >= (1LL << 31)) { set_error("lattice too large for 32-bit map indices"); return FETIDP_EINVAL; }
  ProfScope ps(c, FETIDP_K_MAPS, 0.0, (double)nrhs * (c.L * 8.0 + c.N * c.nd * 4.0) + c.N * c.nd * 8.0);
  gather_BT_kernel<true><<<grid_for(work), 256, 0, c.stream>>>(c.gath, lam, lam_rs, dinfo, c.d, c.dual_order, nullptr, 0,
                                                               0, c.nd, c.N, nrhs, 0.0, xf);
  FD_CHECK_LAUNCH();
  return FETIDP_OK;
}

fetidp_status k_pack_f32(Ctx& c, CCellVec x, int len, float* xf, int nrhs) {
  ProfScope ps(c, FETIDP_K_MAPS, 0.0, 12.0 * nrhs * c.N * len);
  pack_f32_kernel<<<grid_for(c.N * len), 256, 0, c.stream>>>(x.p, x.rs, x.cs, len, c.N, nrhs, xf, c.xf_P, c.xf_cs(len));
  FD_CHECK_LAUNCH();
  return FETIDP_OK;
}

fetidp_status k_scatter_B(Ctx& c, CCellVec yd, double* out, long long out_rs, const int* dinfo,
                          double alpha, double beta, int nrhs) {
  if (c.L >= (1LL << 31) || c.N * c.nd >= (1LL << 31)) { set_error("lattice too large for 32-bit map indices"); return FETIDP_EINVAL; }
  ProfScope ps(c, FETIDP_K_MAPS, 0.0, (double)nrhs * (c.L * 8.0 + c.N * c.nd * 8.0) + c.L * 8.0);
  scatter_B_kernel<double><<<grid_for(c.L), 256, 0, c.stream>>>(c.scat, yd.p, yd.rs, yd.cs, c.nd, dinfo, c.d,
                                                                dinfo ? c.row_order : nullptr, out, out_rs, c.L, alpha,
                                                                beta, nrhs);
  FD_CHECK_LAUNCH();
  return FETIDP_OK;
}

fetidp_status k_scatter_B_f32(Ctx& c, const FCellVec& yd, double* out, long long out_rs, const int* dinfo, int nrhs) {
  if (c.L >= (1LL << 31) || c.N * c.nd >= (1LL << 31)) { set_error("lattice too large for 32-bit map indices"); return FETIDP_EINVAL; }
  ProfScope ps(c, FETIDP_K_MAPS, 0.0, (double)nrhs * (c.L * 8.0 + c.N * c.nd * 4.0) + c.L * 8.0);
  scatter_B_kernel<float><<<grid_for(c.L), 256, 0, c.stream>>>(c.scat, yd.p, yd.rs, yd.cs, c.nd, dinfo, c.d,
                                                               dinfo ? c.row_order : nullptr, out, out_rs, c.L, 1.0,
                                                               0.0, nrhs);
  FD_CHECK_LAUNCH();
  return FETIDP_OK;
}

fetidp_status k_primal_assemble(Ctx& c, CCellVec cp, double* out, long long out_rs, double alpha,
                                double beta, int nrhs) {
  ProfScope ps(c, FETIDP_K_MAPS, 0.0, (double)nrhs * (c.N * c.np * 8.0 + c.nP * 8.0));
  primal_assemble_kernel<<<grid_for((long long)c.nV * c.d * nrhs), 256, 0, c.stream>>>(
      c.vert_cells, c.ncorner, c.d, cp.p, cp.rs, cp.cs, out, out_rs, c.nV, alpha, beta, nrhs);
  FD_CHECK_LAUNCH();
  return FETIDP_OK;
}

fetidp_status k_primal_extract(Ctx& c, const double* uP, long long uP_rs, CellVec cp, int nrhs) {
  ProfScope ps(c, FETIDP_K_MAPS, 0.0, (double)nrhs * (c.N * c.np * 8.0 + c.nP * 8.0));
  primal_extract_kernel<<<grid_for(c.N * c.np * nrhs), 256, 0, c.stream>>>(
      c.corner_v, c.ncorner, c.d, uP, uP_rs, cp.p, cp.rs, cp.cs, c.N, nrhs);
  FD_CHECK_LAUNCH();
  return FETIDP_OK;
}

fetidp_status k_primal_extract_f32(Ctx& c, const double* uP, long long uP_rs, float* cpf, int nrhs) {
  ProfScope ps(c, FETIDP_K_MAPS, 0.0, (double)nrhs * (c.N * c.np * 4.0 + c.nP * 8.0));
  primal_extract_f32_kernel<<<grid_for(c.N * c.np, 128), 128, 0, c.stream>>>(c.corner_v, c.ncorner, c.d, uP, uP_rs, cpf,
                                                                             c.N, nrhs);
  FD_CHECK_LAUNCH();
  return FETIDP_OK;
}

// out[rhs*nv + i] = V_i[rhs] . w[rhs]; V_i at Vb + i*vstride + rhs*len_rs.
static fetidp_status multi_dot_impl(Ctx& c, const double* Vb, long long vstride, long long vrs,
                                    int nv, const double* w, long long wrs, long long len,
                                    int nrhs, double* out) {
  ProfScope ps(c, FETIDP_K_VECTOR, 2.0 * nv * len * nrhs, 8.0 * (nv + 1) * len * nrhs);
  multi_dot_kernel<<<dim3(red_blocks(len), nrhs, nv), kRedThreads, 0, c.stream>>>(Vb, vstride, vrs, w, wrs, len, nv,
                                                                                  c.red, c.red_count, out);
  FD_CHECK_LAUNCH();
  return FETIDP_OK;
}

fetidp_status k_dot(Ctx& c, const double* x, long long xs, const double* y, long long ys,
                    long long len, int nrhs, double* out) {
  return multi_dot_impl(c, x, 0, xs, 1, y, ys, len, nrhs, out);
}

fetidp_status k_pcg_update(Ctx& c, double* X, double* R, const double* P, const double* Q, const PcgSlots& S,
                           double tol) {
  ProfScope ps(c, FETIDP_K_VECTOR, 6.0 * c.L * c.m, 48.0 * c.L * c.m);
  pcg_update_kernel<<<dim3(red_blocks(c.L), c.m), kRedThreads, 0, c.stream>>>(X, R, P, Q, c.scal, S, c.L, c.m, tol,
                                                                             c.red, c.red_count);
  FD_CHECK_LAUNCH();
  return FETIDP_OK;
}

fetidp_status k_pcg_p(Ctx& c, double* P, const double* Z, const PcgSlots& S, int rz_new) {
  ProfScope ps(c, FETIDP_K_VECTOR, 2.0 * c.L * c.m, 24.0 * c.L * c.m);
  pcg_p_kernel<<<dim3(grid_for((c.L + 3) / 4), c.m), 256, 0, c.stream>>>(P, Z, c.scal, S.act, rz_new, S.rz, c.L, c.m);
  FD_CHECK_LAUNCH();
  return FETIDP_OK;
}

fetidp_status k_multi_dot(Ctx& c, const double* Vb, long long vstride, int nv, const double* w,
                          long long len, int nrhs, double* out) {
  // Krylov vectors: V_i[rhs] at Vb + i*vstride + rhs*len; w[rhs] at w + rhs*len
  return multi_dot_impl(c, Vb, vstride, len, nv, w, len, len, nrhs, out);
}

fetidp_status k_multi_axpy(Ctx& c, const double* Vb, long long vstride, int nv, const double* coef,
                           double* w, long long len, int nrhs, double sign) {
  ProfScope ps(c, FETIDP_K_VECTOR, 2.0 * nv * len * nrhs, 8.0 * (nv + 2) * len * nrhs);
  multi_axpy_kernel<<<grid_for(len * nrhs), 256, 0, c.stream>>>(Vb, vstride, len, nv, coef, w, len,
                                                                 len, nrhs, sign);
  FD_CHECK_LAUNCH();
  return FETIDP_OK;
}

fetidp_status k_compliance(Ctx& c, const double* u, double* out, double* partial) {
  compliance_partial<<<dim3(kRedBlocks, c.m), 256, 0, c.stream>>>(c.rhs, c.ntot, c.rhs_p_cells, u, c.perm, c.n, c.nr,
                                                                 c.N, partial);
  FD_CHECK_LAUNCH();
  reduce_partials<<<c.m, 256, 0, c.stream>>>(partial, kRedBlocks, out);
  FD_CHECK_LAUNCH();
  return FETIDP_OK;
}

fetidp_status k_copy_scale(Ctx& c, const double* x, double* y, long long len, int nrhs,
                           long long xs, long long ys, const double* s_dev, double s_host) {
  ProfScope ps(c, FETIDP_K_VECTOR, (double)len * nrhs, 16.0 * len * nrhs);
  copy_scale_kernel<<<grid_for(len * nrhs), 256, 0, c.stream>>>(x, y, len, nrhs, xs, ys, s_dev,
                                                                 s_host);
  FD_CHECK_LAUNCH();
  return FETIDP_OK;
}

}  // namespace fetidp

namespace fetidp {

fetidp_status k_nonfinite(Ctx& c, const double* x, long long n, int* flag) {
  if (n <= 0) return FETIDP_OK;
  nonfinite_kernel<<<grid_for(n), 256, 0, c.stream>>>(x, n, flag);
  FD_CHECK_LAUNCH();
  return FETIDP_OK;
}

}  // namespace fetidp
