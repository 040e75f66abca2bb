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
// element), low-rank ones by the FP64 pipe (rank FMAs an element).  A CTA takes a 64 x 64 tile and a
// lane 16 of its elements, all of whose kinds and then values are loaded before the first is used:
// with 32 x 32 tiles and a chain of index, kind and value loads per element the dense N = 16384
// result took 1.73 ms, now 0.80 (4.3 GB: 0.63 at the copy rate).
constexpr int kOutTile = 64;
__global__ void __launch_bounds__(256) pool_to_rowmajor_kernel(MatView M, const int* row_idx,
                                                               const int* col_idx, double* out,
                                                               int64_t ldo) {
  __shared__ double tile[kOutTile][kOutTile + 1];
  const int64_t tiles_r = (M.n_rows + kOutTile - 1) / kOutTile;
  const int64_t r0 = (int64_t)(blockIdx.x % tiles_r) * kOutTile;
  const int64_t c0 = (int64_t)(blockIdx.x / tiles_r) * kOutTile;
  const int l = threadIdx.x % 32, w = threadIdx.x / 32;
  int R[2], mR[2], rloc[2];
  int64_t base[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int64_t r = r0 + l + 32 * h;
    R[h] = r < M.n_rows ? row_idx[r] : -1;
    const int off = R[h] >= 0 ? M.row_off[R[h]] : 0;
    mR[h] = R[h] >= 0 ? M.row_off[R[h] + 1] - off : 0;
    rloc[h] = (int)(r - off);
    base[h] = (int64_t)off * M.n_cols + rloc[h];
  }
  constexpr int kCols = kOutTile / 8;
  int Cc[kCols], kind[kCols][2];
  double v[kCols][2];
#pragma unroll
  for (int q = 0; q < kCols; ++q) {
    const int64_t c = c0 + w + 8 * q;
    Cc[q] = c < M.n_cols ? col_idx[c] : -1;
  }
#pragma unroll
  for (int q = 0; q < kCols; ++q)
#pragma unroll
    for (int h = 0; h < 2; ++h)
      kind[q][h] = R[h] >= 0 && Cc[q] >= 0 ? M.kind[(int64_t)R[h] * M.nc + Cc[q]] : CLR_KIND_ZERO;
  bool lr = false;
#pragma unroll
  for (int q = 0; q < kCols; ++q)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      v[q][h] = kind[q][h] == CLR_KIND_DENSE ? M.pool[base[h] + (c0 + w + 8 * q) * mR[h]] : 0.0;
      lr = lr || kind[q][h] == CLR_KIND_LR;
    }
  if (lr) {
#pragma unroll
    for (int q = 0; q < kCols; ++q)
#pragma unroll
      for (int h = 0; h < 2; ++h)
        if (kind[q][h] == CLR_KIND_LR) {
          const int coff = M.col_off[Cc[q]];
          const int n = M.col_off[Cc[q] + 1] - coff;
          const int rk = M.rank[(int64_t)R[h] * M.nc + Cc[q]];
          const double* X = M.pool + base[h] - rloc[h] + (int64_t)mR[h] * coff;
          const double* W = X + (int64_t)mR[h] * rk + (c0 + w + 8 * q - coff);
          X += rloc[h];
          double s = 0.0;
          for (int k = 0; k < rk; ++k) s = fma(X[(int64_t)k * mR[h]], W[(int64_t)k * n], s);
          v[q][h] = s;
        }
  }
#pragma unroll
  for (int q = 0; q < kCols; ++q)
#pragma unroll
    for (int h = 0; h < 2; ++h) tile[l + 32 * h][w + 8 * q] = v[q][h];
  __syncthreads();
  for (int rr = w; rr < kOutTile; rr += 8) {
    const int64_t r = r0 + rr;
    if (r >= M.n_rows) break;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int64_t c = c0 + l + 32 * h;
      if (c < M.n_cols) out[r * ldo + c] = tile[rr][l + 32 * h];
    }
  }
}

void launch_pool_to_rowmajor(const MatView& M, const int* row_idx, const int* col_idx,
                             double* out, int64_t ldo, cudaStream_t st) {
  const int64_t n =
      ((M.n_rows + kOutTile - 1) / kOutTile) * ((M.n_cols + kOutTile - 1) / kOutTile);
  pool_to_rowmajor_kernel<<<(unsigned)n, 256, 0, st>>>(M, row_idx, col_idx, out, ldo);
}

}  // namespace clr
