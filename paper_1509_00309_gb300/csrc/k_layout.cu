// Layout conversions between a row-major dense matrix and the block-slot pool, through
// 32 x 32 shared-memory tiles so that both sides are accessed coalesced.  In the pool, the
// block-row panel of block-row R is an m_R x n_cols column-major matrix, so element (r, c)
// of a dense block lives at row_off[R] * n_cols + (r - row_off[R]) + c * m_R.
#include "clr_internal.h"

namespace clr {

__device__ __forceinline__ int64_t panel_index(const MatView& M, int R, int64_t r, int64_t c,
                                               int mR) {
  return (int64_t)M.row_off[R] * M.n_cols + (r - M.row_off[R]) + c * mR;
}

// pool <- row-major src for every block (used when every kept block is dense).
__global__ void __launch_bounds__(256) rowmajor_to_pool_kernel(MatView M, const int* row_idx,
                                                               const double* src, int64_t lds) {
  __shared__ double tile[32][33];
  const int64_t tiles_r = (M.n_rows + 31) / 32;
  const int64_t r0 = (int64_t)(blockIdx.x % tiles_r) * 32;
  const int64_t c0 = (int64_t)(blockIdx.x / tiles_r) * 32;
  const int tx = threadIdx.x % 32, ty = threadIdx.x / 32;
  for (int rr = ty; rr < 32; rr += 8) {  // coalesced along columns
    const int64_t r = r0 + rr, c = c0 + tx;
    tile[rr][tx] = (r < M.n_rows && c < M.n_cols) ? src[r * lds + c] : 0.0;
  }
  __syncthreads();
  const int64_t r = r0 + tx;
  if (r >= M.n_rows) return;
  const int R = row_idx[r];
  const int mR = M.row_off[R + 1] - M.row_off[R];
  for (int cc = ty; cc < 32; cc += 8) {  // coalesced along rows of a block-row panel
    const int64_t c = c0 + cc;
    if (c < M.n_cols) M.pool[panel_index(M, R, r, c, mR)] = tile[tx][cc];
  }
}

void launch_rowmajor_to_pool(const MatView& M, const int* row_idx, const double* src,
                             int64_t lds, cudaStream_t st) {
  const int64_t n = ((M.n_rows + 31) / 32) * ((M.n_cols + 31) / 32);
  rowmajor_to_pool_kernel<<<(unsigned)n, 256, 0, st>>>(M, row_idx, src, lds);
}

// After rowmajor_to_pool and block norms: keep every block dense unless its norm is below
// drop_norm (or zero); non-finite norms raise the error flag.
__global__ void dense_kinds_kernel(MatView M, double drop_norm, int* err) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= M.nr * M.nc) return;
  const int I = t / M.nc, J = t % M.nc;
  const int m = M.row_off[I + 1] - M.row_off[I];
  const int n = M.col_off[J + 1] - M.col_off[J];
  const double nrm = M.norm[t];
  if (!isfinite(nrm)) atomicCAS(err, 0, 3);  // an earlier error keeps precedence
  if (!(nrm >= drop_norm) || nrm == 0.0) {
    M.kind[t] = CLR_KIND_ZERO;
    M.rank[t] = 0;
    M.norm[t] = 0.0;
  } else {
    M.kind[t] = CLR_KIND_DENSE;
    M.rank[t] = m < n ? m : n;
  }
}

void launch_dense_kinds(const MatView& M, double drop_norm, int* err, cudaStream_t st) {
  const int n = M.nr * M.nc;
  dense_kinds_kernel<<<(n + 127) / 128, 128, 0, st>>>(M, drop_norm, err);
}

// row-major out <- reconstruction of every block.  Dense blocks are bound by HBM (16 bytes an
// element), low-rank ones by the FP64 pipe (rank FMAs an element).  A CTA takes a T x T tile and a
// lane T / 32 of its rows in T / 8 adjacent columns, all of whose kinds and then dense values are
// loaded before the first is used: with 32 x 32 tiles and a chain of index, kind and value loads per
// element the dense N = 16384 result took 1.74 ms, with T = 64 0.77 (4.3 GB: 0.63 at the copy
// rate).  Where the lane's columns lie in one block their low-rank sums run side by side: one load
// of X a step for all of them, and no FMA waits for the one before (3D lattice, N = 8192: 4.22 ms, an
// element at a time 4.74; its FMAs alone take 4.0).
template <int T>
__global__ void __launch_bounds__(256) pool_to_rowmajor_kernel(MatView M, const int* row_idx,
                                                               const int* col_idx, double* out,
                                                               int64_t ldo) {
  __shared__ double tile[T][T + 1];
  constexpr int kRows = T / 32, kCols = T / 8;
  const int64_t tiles_r = (M.n_rows + T - 1) / T;
  const int64_t r0 = (int64_t)(blockIdx.x % tiles_r) * T;
  const int64_t c0 = (int64_t)(blockIdx.x / tiles_r) * T;
  const int l = threadIdx.x % 32, w = threadIdx.x / 32;
  int R[kRows], mR[kRows], rloc[kRows];
  int64_t base[kRows];
#pragma unroll
  for (int h = 0; h < kRows; ++h) {
    const int64_t r = r0 + l + 32 * h;
    R[h] = r < M.n_rows ? row_idx[r] : -1;
    const int off = R[h] >= 0 ? M.row_off[R[h]] : 0;
    mR[h] = R[h] >= 0 ? M.row_off[R[h] + 1] - off : 0;
    rloc[h] = (int)(r - off);
    base[h] = (int64_t)off * M.n_cols + rloc[h];
  }
  const int64_t cw = c0 + kCols * w;   // the warp's first column
  unsigned dense = 0, lr = 0;          // by element: bit kRows q + h
  bool one;                            // the warp's columns lie in one cluster
  {
    int Cc[kCols], kind[kCols][kRows];
#pragma unroll
    for (int q = 0; q < kCols; ++q) Cc[q] = cw + q < M.n_cols ? col_idx[cw + q] : -1;
#pragma unroll
    for (int q = 0; q < kCols; ++q)
#pragma unroll
      for (int h = 0; h < kRows; ++h)
        kind[q][h] = R[h] >= 0 && Cc[q] >= 0 ? M.kind[(int64_t)R[h] * M.nc + Cc[q]] : CLR_KIND_ZERO;
#pragma unroll
    for (int q = 0; q < kCols; ++q)
#pragma unroll
      for (int h = 0; h < kRows; ++h) {
        dense |= (unsigned)(kind[q][h] == CLR_KIND_DENSE) << (kRows * q + h);
        lr |= (unsigned)(kind[q][h] == CLR_KIND_LR) << (kRows * q + h);
      }
    one = Cc[0] >= 0 && Cc[0] == Cc[kCols - 1];
  }
  {
    double v[kCols][kRows];
#pragma unroll
    for (int q = 0; q < kCols; ++q)
#pragma unroll
      for (int h = 0; h < kRows; ++h)
        v[q][h] = dense >> (kRows * q + h) & 1u ? M.pool[base[h] + (cw + q) * mR[h]] : 0.0;
#pragma unroll
    for (int q = 0; q < kCols; ++q)
#pragma unroll
      for (int h = 0; h < kRows; ++h) tile[l + 32 * h][kCols * w + q] = v[q][h];
  }
  // (the factors of the block of row h's cluster and column c)
  auto factors = [&](int h, int64_t c, const double** X, const double** W, int* n) {
    const int C = col_idx[c], coff = M.col_off[C];
    const int rk = M.rank[(int64_t)R[h] * M.nc + C];
    *n = M.col_off[C + 1] - coff;
    *X = M.pool + base[h] + (int64_t)mR[h] * coff;
    *W = *X - rloc[h] + (int64_t)mR[h] * rk + (c - coff);
    return rk;
  };
#pragma unroll
  for (int h = 0; h < kRows; ++h) {
    const double *X, *W;
    int n;
    double* to = &tile[l + 32 * h][kCols * w];
    if (one) {
      if (!(lr >> h & 1u)) continue;
      const int rk = factors(h, cw, &X, &W, &n);
      double s[kCols];
#pragma unroll
      for (int q = 0; q < kCols; ++q) s[q] = 0.0;
#pragma unroll 2
      for (int k = 0; k < rk; ++k) {
        const double x = *X;
        X += mR[h];
#pragma unroll
        for (int q = 0; q < kCols; ++q) s[q] = fma(x, W[q], s[q]);
        W += n;
      }
#pragma unroll
      for (int q = 0; q < kCols; ++q) to[q] = s[q];
    } else {
      for (int q = 0; q < kCols; ++q) {
        if (!(lr >> (kRows * q + h) & 1u)) continue;
        const int rk = factors(h, cw + q, &X, &W, &n);
        double s = 0.0;
        for (int k = 0; k < rk; ++k) s = fma(X[(int64_t)k * mR[h]], W[(int64_t)k * n], s);
        to[q] = s;
      }
    }
  }
  __syncthreads();
  for (int rr = w; rr < T; rr += 8) {
    const int64_t r = r0 + rr;
    if (r >= M.n_rows) break;
#pragma unroll
    for (int h = 0; h < kRows; ++h) {
      const int64_t c = c0 + l + 32 * h;
      if (c < M.n_cols) out[r * ldo + c] = tile[rr][l + 32 * h];
    }
  }
}

void launch_pool_to_rowmajor(const MatView& M, const int* row_idx, const int* col_idx,
                             double* out, int64_t ldo, cudaStream_t st) {
  // T = 64 once such tiles are enough (N = 512 to 4096 with low rank blocks: 77 to 1190 us with 64,
  // 44 to 1127 with 32; dense N = 4096 66 and 80, N = 16384 0.77 and 1.0 ms)
  auto tiles = [&](int64_t t) { return ((M.n_rows + t - 1) / t) * ((M.n_cols + t - 1) / t); };
  if (tiles(64) > 4096)
    pool_to_rowmajor_kernel<64><<<(unsigned)tiles(64), 256, 0, st>>>(M, row_idx, col_idx, out, ldo);
  else
    pool_to_rowmajor_kernel<32><<<(unsigned)tiles(32), 256, 0, st>>>(M, row_idx, col_idx, out, ldo);
}

}  // namespace clr
