// K6/K7 -- CLR linear combination (the T_n polynomial of Section 4.2 is
// (15 I - 10 X_n + 3 X_n^2) / 8), distance to the identity (NS convergence test), CLR
// matrix-vector products (alpha estimate) and transposes (adjoint products).
#include <cooperative_groups.h>

#include "clr_internal.h"

namespace clr {

constexpr int kT = 256;

__device__ __forceinline__ double wsum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ double bsum(double v, double* sh) {
  v = wsum(v);
  const int w = threadIdx.x / 32, l = threadIdx.x % 32;
  __syncthreads();
  if (l == 0) sh[w] = v;
  __syncthreads();
  double s = 0.0;
  for (int i = 0; i < (int)(blockDim.x / 32); ++i) s += sh[i];
  __syncthreads();
  return s;
}

// Route of each output block of out = a X + b Y + diag I (rules of Section 4.1 low-rank
// addition; see clr.h).
__global__ void lincomb_route_kernel(double a, MatView X, double b, MatView Y, double diag,
                                     Plan p) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= p.nI * p.nJ) return;
  const int I = t / p.nJ, J = t % p.nJ;
  const int m = X.row_off[I + 1] - X.row_off[I];
  const int n = X.col_off[J + 1] - X.col_off[J];
  int kx = X.kind[t], ky = Y.kind[t];
  if (a == 0.0) kx = CLR_KIND_ZERO;
  if (b == 0.0) ky = CLR_KIND_ZERO;
  const bool shift = I == J && diag != 0.0;
  int route = ROUTE_ZERO, rs = 0;
  if (kx == CLR_KIND_ZERO && ky == CLR_KIND_ZERO && !shift) {
    route = ROUTE_ZERO;
  } else if (!shift && (kx == CLR_KIND_ZERO || ky == CLR_KIND_ZERO)) {
    route = -1;  // exact scaled copy
  } else if (shift || kx == CLR_KIND_DENSE || ky == CLR_KIND_DENSE) {
    route = ROUTE_DENSE;
  } else {
    const int R = X.rank[t] + Y.rank[t];
    const int lim = (m < n ? m : n) / 2;
    if (R <= lim) { route = ROUTE_QR; rs = R; } else { route = ROUTE_DACC; }
  }
  p.t_count[t] = 0;
  p.t_route[t] = route < 0 ? ROUTE_ZERO : route;
  p.t_rsum[t] = rs;
  // the copy case is re-derived by the apply kernel from the operand kinds
}

// A cluster of CS CTAs per block, its elements in turn (a dense sum of low-rank blocks takes m n r
// FMAs on the FP64 pipe, and with one CTA per block the largest block was the kernel's time: 4.9 ms
// for the 3D lattice's iterates at N = 2048, now 1.2); the norm's parts are added in a fixed order.
template <int CS>
__global__ void __cluster_dims__(CS, 1, 1) __launch_bounds__(kT)
    lincomb_apply_kernel(double a, MatView X, double b, MatView Y, double diag, MatView O, Plan p,
                         double* ws) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  __shared__ double red[kT / 32];
  __shared__ double part_sq;
  const int t = blockIdx.x / CS, rank = (int)cluster.block_rank();
  const int tid = threadIdx.x + kT * rank;
  constexpr int kAll = kT * CS;
  const int I = t / p.nJ, J = t % p.nJ;
  const int m = X.row_off[I + 1] - X.row_off[I];
  const int n = X.col_off[J + 1] - X.col_off[J];
  int kx = X.kind[t], ky = Y.kind[t];
  if (a == 0.0) kx = CLR_KIND_ZERO;
  if (b == 0.0) ky = CLR_KIND_ZERO;
  const bool shift = I == J && diag != 0.0;
  const int64_t sl = slot_of(O, I, J, m);
  const double* xs = X.pool + sl;
  const double* ys = Y.pool + sl;
  double* os = O.pool + sl;
  const int route = p.t_route[t];
  const int rx = X.rank[t], ry = Y.rank[t];
  if (kx == CLR_KIND_ZERO && ky == CLR_KIND_ZERO && !shift) {
    if (tid == 0) { O.kind[t] = CLR_KIND_ZERO; O.rank[t] = 0; O.norm[t] = 0.0; }
    return;
  }
  if (!shift && (kx == CLR_KIND_ZERO || ky == CLR_KIND_ZERO)) {
    const bool fromx = ky == CLR_KIND_ZERO;
    const MatView& S = fromx ? X : Y;
    const double c = fromx ? a : b;
    const double* ss = fromx ? xs : ys;
    const int kind = S.kind[t], r = S.rank[t];
    if (kind == CLR_KIND_DENSE) {
      for (int e = tid; e < m * n; e += kAll) os[e] = c * ss[e];
    } else {
      for (int e = tid; e < m * r; e += kAll) os[e] = c * ss[e];
      for (int e = tid; e < n * r; e += kAll) os[m * r + e] = ss[m * r + e];
    }
    if (tid == 0) { O.kind[t] = kind; O.rank[t] = r; O.norm[t] = fabs(c) * S.norm[t]; }
    return;
  }
  if (route == ROUTE_QR) {
    const int R = rx + ry;
    double* Xc = ws + 2 * sl;
    double* Wc = Xc + (int64_t)m * R;
    for (int e = tid; e < m * rx; e += kAll) Xc[e] = a * xs[e];
    for (int e = tid; e < m * ry; e += kAll) Xc[m * rx + e] = b * ys[e];
    for (int e = tid; e < n * rx; e += kAll) Wc[e] = xs[m * rx + e];
    for (int e = tid; e < n * ry; e += kAll) Wc[n * rx + e] = ys[m * ry + e];
    return;
  }
  // dense sum (ROUTE_DENSE or ROUTE_DACC)
  double part = 0.0;
  for (int e = tid; e < m * n; e += kAll) {
    const int i = e % m, j = e / m;
    double v = 0.0;
    if (kx == CLR_KIND_DENSE) {
      v = a * xs[e];
    } else if (kx == CLR_KIND_LR) {
      double s = 0.0;
      for (int c = 0; c < rx; ++c) s = fma(xs[i + c * m], xs[m * rx + j + c * n], s);
      v = a * s;
    }
    if (ky == CLR_KIND_DENSE) {
      v = fma(b, ys[e], v);
    } else if (ky == CLR_KIND_LR) {
      double s = 0.0;
      for (int c = 0; c < ry; ++c) s = fma(ys[i + c * m], ys[m * ry + j + c * n], s);
      v = fma(b, s, v);
    }
    if (shift && i == j) v += diag;
    os[e] = v;
    part = fma(v, v, part);
  }
  const double own = bsum(part, red);
  if (threadIdx.x == 0) part_sq = own;
  cluster.sync();
  if (tid == 0) {
    double nsq = 0.0;
    for (int c = 0; c < CS; ++c) nsq += *cluster.map_shared_rank(&part_sq, c);
    O.kind[t] = CLR_KIND_DENSE;
    O.rank[t] = m < n ? m : n;
    O.norm[t] = sqrt(nsq);
  }
  cluster.sync();   // no CTA's part goes before it has been read
}

void launch_plan_scan(const Plan& p, int recompress_dense, cudaStream_t st);

void launch_lincomb_plan(double a, const MatView& X, double b, const MatView& Y, double diag,
                         const MatView& O, const Plan& p, double* ws, int recompress_dense,
                         cudaStream_t st) {
  const int n = p.nI * p.nJ;
  cudaMemsetAsync(p.counters, 0, kPlanCountersClear, st);
  lincomb_route_kernel<<<(n + 127) / 128, 128, 0, st>>>(a, X, b, Y, diag, p);
  launch_plan_scan(p, recompress_dense, st);
  // CTAs per block, fewer the more blocks there are: starting CTAs for blocks without work is then
  // what the launch takes (a sum of 141376 blocks, 1126 of them not zero: 2840 us with recompression
  // by eights, 1360 by ones; 8281 blocks, 3D lattice: 95.3 and 97.9 ms, by twos 95.9; 2116: equal
  // with 8 and 4).  A scaled copy has no FMAs to share: by ones from 3072 on (8100 blocks, chain:
  // 214, 134 and 123 us by eights, twos and ones).
  const int many = a == 0.0 || b == 0.0 ? 3072 : 16384;
  if (n <= 1024) lincomb_apply_kernel<8><<<n * 8, kT, 0, st>>>(a, X, b, Y, diag, O, p, ws);
  else if (n <= 3072) lincomb_apply_kernel<4><<<n * 4, kT, 0, st>>>(a, X, b, Y, diag, O, p, ws);
  else if (n <= many) lincomb_apply_kernel<2><<<n * 2, kT, 0, st>>>(a, X, b, Y, diag, O, p, ws);
  else lincomb_apply_kernel<1><<<n, kT, 0, st>>>(a, X, b, Y, diag, O, p, ws);
}

// Per block: ||M_IJ - delta_IJ I||_F^2, then a deterministic single-CTA sum.
__global__ void __launch_bounds__(kT) identity_distance_block_kernel(MatView M, double* part) {
  __shared__ double red[kT / 32];
  const int t = blockIdx.x;
  const int I = t / M.nc, J = t % M.nc;
  const int m = M.row_off[I + 1] - M.row_off[I];
  const int n = M.col_off[J + 1] - M.col_off[J];
  const int kind = M.kind[t];
  if (I != J) {
    if (threadIdx.x == 0) part[t] = M.norm[t] * M.norm[t];
    return;
  }
  const double* s = M.pool + slot_of(M, I, J, m);
  double acc = 0.0;
  if (kind == CLR_KIND_DENSE) {
    for (int e = threadIdx.x; e < m * n; e += kT) {
      const double v = s[e] - ((e % m) == (e / m) ? 1.0 : 0.0);
      acc = fma(v, v, acc);
    }
  } else if (kind == CLR_KIND_LR) {
    // ||X W^T||^2 - 2 tr(X W^T) + m
    const int r = M.rank[t];
    for (int e = threadIdx.x; e < m * r; e += kT) {
      const int i = e % m, c = e / m;
      acc -= 2.0 * s[e] * s[m * r + i + c * n];
    }
  }
  const double tot = bsum(acc, red);
  if (threadIdx.x == 0) {
    if (kind == CLR_KIND_DENSE) part[t] = tot;
    else if (kind == CLR_KIND_LR) part[t] = M.norm[t] * M.norm[t] + tot + (double)m;
    else part[t] = (double)m;
  }
}

__global__ void __launch_bounds__(1024) sum_kernel(const double* part, int n, double* out) {
  __shared__ double red[32];
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) s += part[i];
  s = wsum(s);
  if (threadIdx.x % 32 == 0) red[threadIdx.x / 32] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double tot = 0.0;
    for (int i = 0; i < (int)(blockDim.x / 32); ++i) tot += red[i];
    *out = tot;
  }
}

void launch_identity_distance(const MatView& X, double* out_sq, cudaStream_t st) {
  // out_sq[0] receives the sum; out_sq[1 ...] holds the per-block parts
  const int nb = X.nr * X.nc;
  identity_distance_block_kernel<<<nb, kT, 0, st>>>(X, out_sq + 1);
  sum_kernel<<<1, 1024, 0, st>>>(out_sq + 1, nb, out_sq);
}

// y_I = sum_J M_IJ x_J.  Bound by reading the blocks once (70 MB for the 3D lattice at N = 4096)
// and by the FP64 pipe (an FMA per double read), 15 us each there, so the block-row is spread
// over a cluster of CS CTAs (blocks J in turn) whose partial sums are added, in a fixed order,
// through distributed shared memory: no workspace, so calls on different streams do not meet.
// (One CTA per block-row, walking its blocks one after the other, took 690 us; eight take 60.)
// Inside a CTA a warp takes four columns of W at a time for W^T x and sums them together; for X t
// (and dense blocks) it owns a group of 32 rows and a share of the columns, its row sums in
// registers until the end.  The kinds, ranks and places of 32 of the CTA's blocks are read at once: in
// a chain matrix nearly all are zero, and read one after the other they were most of the time.
constexpr int kMvThreads = 512;
constexpr int kMvWarps = kMvThreads / 32;

template <int CS>
__global__ void __cluster_dims__(CS, 1, 1) __launch_bounds__(kMvThreads)
    matvec_kernel(MatView M, const double* x, double* y) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  __shared__ double part[kMvWarps][CLR_MAX_CLUSTER];   // [0] ends as this CTA's sum
  __shared__ double tw[2][CLR_MAX_CLUSTER / 2];
  const int I = blockIdx.x / CS, rank = (int)cluster.block_rank();
  const int m = M.row_off[I + 1] - M.row_off[I];
  const int w = threadIdx.x / 32, l = threadIdx.x % 32;
  const int groups = (m + 31) / 32, slices = kMvWarps / groups;
  const int i = (w % groups) * 32 + l, slice = w / groups;
  const bool mine = slice < slices && i < m;
  double acc = 0.0;
  int buf = 0;
  for (int J0 = rank; J0 < M.nc; J0 += 32 * CS) {
    const int Jl = J0 + l * CS;
    const bool in = Jl < M.nc;
    const int kind = in ? M.kind[I * M.nc + Jl] : CLR_KIND_ZERO;
    const int rank_l = in ? M.rank[I * M.nc + Jl] : 0;
    const int off_l = in ? M.col_off[Jl] : 0, end_l = in ? M.col_off[Jl + 1] : 0;
    const unsigned lr = __ballot_sync(0xffffffffu, kind == CLR_KIND_LR);
    for (unsigned todo = __ballot_sync(0xffffffffu, kind != CLR_KIND_ZERO); todo; todo &= todo - 1) {
      const int bit = __ffs(todo) - 1;
      const int off = __shfl_sync(0xffffffffu, off_l, bit);
      const int n = __shfl_sync(0xffffffffu, end_l, bit) - off;
      const double* s = M.pool + (int64_t)M.row_off[I] * M.n_cols + (int64_t)m * off;
      const double* xj = x + off;
      const double* v = xj;
      int cols = n;
      if (lr >> bit & 1u) {
        const int r = __shfl_sync(0xffffffffu, rank_l, bit);
        const double* W = s + (int64_t)m * r;
        for (int c0 = 4 * w; c0 < r; c0 += 4 * kMvWarps) {
          double d[4] = {0.0, 0.0, 0.0, 0.0};
          const double* wc[4];
#pragma unroll
          for (int c = 0; c < 4; ++c) wc[c] = W + (int64_t)(c0 + c < r ? c0 + c : c0) * n;
#pragma unroll 4
          for (int j = l; j < n; j += 32) {
            const double xv = xj[j];
#pragma unroll
            for (int c = 0; c < 4; ++c) d[c] = fma(wc[c][j], xv, d[c]);
          }
          // lane l: the sum of column c0 + l / 8
          const bool h16 = (l & 16) != 0, h8 = (l & 8) != 0;
          double a0 = h16 ? d[2] : d[0], a1 = h16 ? d[3] : d[1];
          a0 += __shfl_xor_sync(0xffffffffu, h16 ? d[0] : d[2], 16);
          a1 += __shfl_xor_sync(0xffffffffu, h16 ? d[1] : d[3], 16);
          double a = h8 ? a1 : a0;
          a += __shfl_xor_sync(0xffffffffu, h8 ? a0 : a1, 8);
          a += __shfl_xor_sync(0xffffffffu, a, 4);
          a += __shfl_xor_sync(0xffffffffu, a, 2);
          a += __shfl_xor_sync(0xffffffffu, a, 1);
          if (l % 8 == 0 && c0 + l / 8 < r) tw[buf][c0 + l / 8] = a;
        }
        // (the other buffer is written only past the next barrier: one barrier per block)
        __syncthreads();
        v = tw[buf];
        cols = r;
        buf ^= 1;
      }
      if (mine) {
        const double* si = s + i;
#pragma unroll 8
        for (int c = slice; c < cols; c += slices) acc = fma(si[(int64_t)c * m], v[c], acc);
      }
    }
  }
  if (mine) part[slice][i] = acc;
  __syncthreads();
  for (int r = threadIdx.x; r < m; r += kMvThreads) {
    double sum = part[0][r];
    for (int q = 1; q < slices; ++q) sum += part[q][r];
    part[0][r] = sum;
  }
  cluster.sync();
  for (int r = rank + CS * threadIdx.x; r < m; r += CS * kMvThreads) {
    double sum = 0.0;
    for (int q = 0; q < CS; ++q) sum += cluster.map_shared_rank(&part[0][0], q)[r];
    y[M.row_off[I] + r] = sum;
  }
  cluster.sync();   // no CTA's shared memory goes before the others have read it
}

void launch_matvec(const MatView& M, const double* x, double* y, cudaStream_t st) {
  // Eight CTAs a block-row while that makes at most six rounds of the two an SM holds; beyond, two
  // (chain matrices, 259 and 376 block-rows: 79 and 65 us by eights, 40 and 33 by twos; full ones at
  // 91 and 220 block-rows: 359 and 486 us by eights, 496 and 563 by twos).
  if (M.nr <= 228) matvec_kernel<8><<<M.nr * 8, kMvThreads, 0, st>>>(M, x, y);
  else matvec_kernel<2><<<M.nr * 2, kMvThreads, 0, st>>>(M, x, y);
}

// T = S^T: block (J,I) of T is block (I,J) of S transposed (dense, 32 x 32 tiles through shared
// memory so that both sides are accessed along their columns) or with X and W swapped.  Bound by
// HBM; several parts per block where blocks alone are too few or too large to spread evenly.  A CTA
// looks at 32 of its (block, part) items at once, as in a chain matrix nearly all are zero (67081
// blocks, 775 not zero: 129 us with the allocation, 208 with a CTA per block).
constexpr unsigned kTransposeCtas = 9728;   // eight rounds of what 152 SMs hold

__global__ void __launch_bounds__(256) transpose_kernel(MatView S, MatView T, unsigned parts) {
  __shared__ double tile[32][33];
  const int l = threadIdx.x % 32, w = threadIdx.x / 32;
  const unsigned items = (unsigned)(S.nr * S.nc) * parts;
  for (unsigned it0 = blockIdx.x; it0 < items; it0 += 32 * gridDim.x) {
    const unsigned own = it0 + l * gridDim.x;
    int kind = CLR_KIND_ZERO;
    if (own < items) {
      const int t = (int)(own / parts);
      kind = S.kind[t];
      if (w == 0 && own % parts == 0) {
        const int tt = t % S.nc * T.nc + t / S.nc;
        T.kind[tt] = kind;
        T.rank[tt] = S.rank[t];
        T.norm[tt] = S.norm[t];
      }
    }
    const unsigned dense = __ballot_sync(0xffffffffu, kind == CLR_KIND_DENSE);
    for (unsigned todo = __ballot_sync(0xffffffffu, kind != CLR_KIND_ZERO); todo; todo &= todo - 1) {
      const unsigned bit = __ffs(todo) - 1, it = it0 + bit * gridDim.x;
      const int t = (int)(it / parts), part = (int)(it % parts), np = (int)parts;
      const int I = t / S.nc, J = t % S.nc;
      const int m = S.row_off[I + 1] - S.row_off[I];
      const int n = S.col_off[J + 1] - S.col_off[J];
      const double* s = S.pool + slot_of(S, I, J, m);
      double* d = T.pool + slot_of(T, J, I, n);
      if (dense >> bit & 1u) {
        const int ti = (m + 31) / 32, tj = (n + 31) / 32;
        for (int q = part; q < ti * tj; q += np) {
          const int i0 = (q % ti) * 32, j0 = (q / ti) * 32;
          for (int c = w; c < 32; c += 8)
            if (i0 + l < m && j0 + c < n) tile[c][l] = s[i0 + l + (int64_t)(j0 + c) * m];
          __syncthreads();
          for (int c = w; c < 32; c += 8)
            if (j0 + l < n && i0 + c < m) d[j0 + l + (int64_t)(i0 + c) * n] = tile[l][c];
          __syncthreads();
        }
      } else {
        const int r = S.rank[t], e0 = threadIdx.x + 256 * part, step = 256 * np;
        for (int e = e0; e < n * r; e += step) d[e] = s[(int64_t)m * r + e];
        for (int e = e0; e < m * r; e += step) d[(int64_t)n * r + e] = s[e];
      }
    }
  }
}

void launch_transpose(const MatView& S, const MatView& T, cudaStream_t st) {
  const int64_t nb = (int64_t)S.nr * S.nc, area = S.n_rows * S.n_cols / nb;
  // (3D lattice, 4624 and 8281 blocks of 180^2: 337 and 430 us with one part, 249 and 327 with four,
  // as fast as with eight; 48400 blocks of 37^2: 229 with one, 337 with four)
  const unsigned parts = nb <= 1024 ? 8 : area >= 8192 ? 4 : area >= 4096 ? 2 : 1;
  const unsigned items = (unsigned)nb * parts;
  transpose_kernel<<<items < kTransposeCtas ? items : kTransposeCtas, 256, 0, st>>>(S, T, parts);
}

}  // namespace clr
