// FP64 dense tile kernels: dense x dense tile products (the plain-precision form of the
// block GEMM task of Section 3.2, C_ij += A_ik B_kj), reconstruction, and per-tile kind
// bookkeeping.
//
// On GB300 FP64 runs on the CUDA cores at a small fraction of the tensor rate (~2 FMAs per clock
// per SM: a warp's FMA holds its sub-partition's pipe for 64 cycles), so these kernels are
// FP64-pipe-bound and the work is cut to waste no FMAs and to reach every SM: a C tile (m x n, up
// to 256 x 256) is cut into sub-tiles of 64, 32 or 16 rows and columns and a ragged last one; one
// CTA computes a sub-tile in registers (16 x 16 threads, up to 4 x 4 entries each, rows and
// columns beyond the next multiple of 16 skipped), walking that tile's dense x dense products in
// k order (deterministic, no atomics).  Sub-tiles are taken from a launch-wide counter over the
// tiles in decreasing cost order (longest-processing-time scheduling).
#include <cooperative_groups.h>

#include "clr_internal.h"

namespace clr {

constexpr int kSub = 64;                     // largest sub-tile edge
constexpr int kStage = 64 * 17;              // doubles of an operand's staged k chunk
constexpr int kSubPerTile = (CLR_MAX_CLUSTER / kSub) * (CLR_MAX_CLUSTER / kSub);
constexpr int kDdThreads = 256;
constexpr int kPrefixTiles = 1024;           // tiles whose sub-tiles are numbered exactly
constexpr int kItemsPerSm = 6;

// The sub-tile of edge 16 NA at (i0, j0) of C tile t.  Chunks of 64 / NA k are staged.
template <int NA>
__device__ __forceinline__ void dd_sub_tile(const MatView& A, const MatView& B, const MatView& C,
                                            const Plan& p, int t, int i0, int j0, double* As,
                                            double* Bs) {
  constexpr int E = 16 * NA, LD = E + 1, KC = 64 / NA;
  const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
  const int I = t / p.nJ, J = t % p.nJ;
  const int m = C.row_off[I + 1] - C.row_off[I];
  const int n = C.col_off[J + 1] - C.col_off[J];
  const int h = min(E, m - i0), g = min(E, n - j0);
  const int na = (h + 15) / 16, nb = (g + 15) / 16;
  double acc[NA][NA];
#pragma unroll
  for (int a = 0; a < NA; ++a)
#pragma unroll
    for (int b = 0; b < NA; ++b) acc[a][b] = 0.0;
  const int start = p.t_start[t], count = p.t_count[t];
  for (int q = 0; q < count; ++q) {
    const Triple tr = p.triples[start + q];
    if (tr.kind != T_DD) continue;
    const int K = tr.k;
    const int k = A.col_off[K + 1] - A.col_off[K];
    const double* Ab = A.pool + slot_of(A, I, K, m) + i0;                // m x k, column-major
    const double* Bb = B.pool + slot_of(B, K, J, k) + (int64_t)j0 * k;   // k x n, column-major
    for (int k0 = 0; k0 < k; k0 += KC) {
      const int kc = min(KC, k - k0);
      for (int e = tid; e < KC * E; e += kDdThreads) {
        const int r = e % E, kk = e / E;
        As[kk * LD + r] = (r < h && kk < kc) ? Ab[r + (int64_t)(k0 + kk) * m] : 0.0;
        const int kk2 = e % KC, c = e / KC;
        Bs[kk2 * LD + c] = (c < g && kk2 < kc) ? Bb[(k0 + kk2) + (int64_t)c * k] : 0.0;
      }
      __syncthreads();
#pragma unroll 4
      for (int kk = 0; kk < kc; ++kk) {
        double av[NA], bv[NA];
#pragma unroll
        for (int a = 0; a < NA; ++a) av[a] = As[kk * LD + ty + 16 * a];
#pragma unroll
        for (int b = 0; b < NA; ++b) bv[b] = Bs[kk * LD + tx + 16 * b];
#pragma unroll
        for (int a = 0; a < NA; ++a)
          if (a < na) {
#pragma unroll
            for (int b = 0; b < NA; ++b)
              if (b < nb) acc[a][b] = fma(av[a], bv[b], acc[a][b]);
          }
      }
      __syncthreads();
    }
  }
  double* D = C.pool + slot_of(C, I, J, m);
#pragma unroll
  for (int a = 0; a < NA; ++a)
#pragma unroll
    for (int b = 0; b < NA; ++b) {
      const int r = ty + 16 * a, c = tx + 16 * b;
      if (r < h && c < g) D[i0 + r + (int64_t)(j0 + c) * m] = acc[a][b];
    }
}

// The sub-tile edge: the largest of 64, 32, 16 that still gives every SM kItemsPerSm sub-tiles
// (16 x 128^2 tiles, the 1D chain at N = 2048: 64 sub-tiles of 64 on 152 SMs took 525 us, 1024 of 16 take 98), with
// the tiles' sub-tiles numbered by a prefix sum; with more than kPrefixTiles tiles, 64 with 16
// numbers per tile, of which those past the tile's end are empty.
__global__ void __launch_bounds__(kDdThreads) dd_fp64_kernel(MatView A, MatView B, MatView C,
                                                             Plan p, int n_sm) {
  __shared__ double As[kStage], Bs[kStage];
  __shared__ int prefix[kPrefixTiles];   // inclusive, of the chosen edge
  __shared__ int warp_tot[3][kDdThreads / 32];
  __shared__ int sh_next;
  const int tid = threadIdx.x, w = tid / 32, l = tid % 32;
  const int n_dense = p.counters->n_dense;
  int* sched = &p.counters->sched[3];
  auto subs = [&](int it, int edge, int* nsi) {
    const int t = p.l_dense_s[it];
    const int I = t / p.nJ, J = t % p.nJ;
    *nsi = (C.row_off[I + 1] - C.row_off[I] + edge - 1) / edge;
    return *nsi * ((C.col_off[J + 1] - C.col_off[J] + edge - 1) / edge);
  };
  int edge = kSub, n_items = n_dense * kSubPerTile;
  const bool exact = n_dense <= kPrefixTiles;
  if (exact) {
    constexpr int kPer = kPrefixTiles / kDdThreads;
    int tot[3] = {0, 0, 0}, nsi;
    for (int x = 0; x < kPer; ++x) {
      const int it = tid * kPer + x;
      if (it < n_dense)
        for (int e = 0; e < 3; ++e) tot[e] += subs(it, kSub >> e, &nsi);
    }
    for (int e = 0; e < 3; ++e) {
      const int s = __reduce_add_sync(0xffffffffu, tot[e]);
      if (l == 0) warp_tot[e][w] = s;
    }
    __syncthreads();
    int sel = 2;
    for (int e = 1; e >= 0; --e) {
      int s = 0;
      for (int q = 0; q < kDdThreads / 32; ++q) s += warp_tot[e][q];
      if (s >= kItemsPerSm * n_sm) sel = e;
    }
    edge = kSub >> sel;
    int own = tot[0];
    if (sel == 1) own = tot[1];
    if (sel == 2) own = tot[2];
    int incl = own;
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (l >= o) incl += v;
    }
    int base = incl - own;
    n_items = 0;
    for (int q = 0; q < kDdThreads / 32; ++q) {
      if (q < w) base += warp_tot[sel][q];
      n_items += warp_tot[sel][q];
    }
    for (int x = 0; x < kPer; ++x) {
      const int it = tid * kPer + x;
      if (it < n_dense) prefix[it] = base += subs(it, edge, &nsi);
    }
    __syncthreads();
  }
  for (int item = next_item(sched, &sh_next); item < n_items;
       item = next_item(sched, &sh_next)) {
    int it, si, sj, nsi;
    if (exact) {
      int lo = 0, hi = n_dense - 1;   // the first tile whose inclusive count exceeds item
      while (lo < hi) {
        const int mid = (lo + hi) / 2;
        if (prefix[mid] > item) hi = mid; else lo = mid + 1;
      }
      it = lo;
      const int s = item - (it > 0 ? prefix[it - 1] : 0);
      subs(it, edge, &nsi);
      si = s % nsi;
      sj = s / nsi;
    } else {
      it = item / kSubPerTile;
      const int s = item % kSubPerTile;
      si = s / (CLR_MAX_CLUSTER / kSub);
      sj = s % (CLR_MAX_CLUSTER / kSub);
      const int total = subs(it, edge, &nsi);
      if (si >= nsi || sj >= total / nsi) continue;
    }
    const int t = p.l_dense_s[it];
    if (edge == 64) dd_sub_tile<4>(A, B, C, p, t, si * 64, sj * 64, As, Bs);
    else if (edge == 32) dd_sub_tile<2>(A, B, C, p, t, si * 32, sj * 32, As, Bs);
    else dd_sub_tile<1>(A, B, C, p, t, si * 16, sj * 16, As, Bs);
  }
}

void launch_dd_fp64(const MatView& A, const MatView& B, const MatView& C, const Plan& p,
                    int n_sm, cudaStream_t st) {
  dd_fp64_kernel<<<4 * n_sm, kDdThreads, 0, st>>>(A, B, C, p, n_sm);
}

// After planning: kinds of tiles that get no contribution (zero) or a dense accumulation.
__global__ void set_route_kinds_kernel(MatView C, Plan p) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= p.nI * p.nJ) return;
  const int route = p.t_route[t];
  const int I = t / p.nJ, J = t % p.nJ;
  const int m = C.row_off[I + 1] - C.row_off[I];
  const int n = C.col_off[J + 1] - C.col_off[J];
  if (route == ROUTE_ZERO) {
    C.kind[t] = CLR_KIND_ZERO;
    C.rank[t] = 0;
    C.norm[t] = 0.0;
  } else if (route == ROUTE_DENSE) {
    C.kind[t] = CLR_KIND_DENSE;
    C.rank[t] = m < n ? m : n;
    C.norm[t] = 0.0;  // a sum of squares when the dense kernel's epilogue forms the norms
  }
}

void launch_set_route_kinds(const MatView& C, const Plan& p, cudaStream_t st) {
  const int n = p.nI * p.nJ;
  set_route_kinds_kernel<<<(n + 127) / 128, 128, 0, st>>>(C, p);
}

// Frobenius norms of the dense-accumulated tiles (those not recompressed afterwards): a cluster of
// CTAs per tile, its parts added in a fixed order (with one CTA a tile's loads took 20 us), while
// the tiles are few (kNormFew a cluster: 512); beyond, CTAs fill the SMs with a tile each and a
// cluster would only wait at its barriers (48400 tiles of at most 48^2: 2350 us by clusters, 330 by
// CTAs).  Nor has a small tile (kNormSmall on average) loads to share: 169 tiles of 39^2 16 and 8 us.
constexpr int kNormCtas = 8;
constexpr int kNormGrid = 1024;
constexpr int kNormFew = 4;
constexpr int kNormSmall = 4096;
__global__ void __cluster_dims__(kNormCtas, 1, 1) __launch_bounds__(256)
    dense_tile_norms_kernel(MatView C, Plan p) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  __shared__ double red[8];
  __shared__ double part;
  const int n_items = p.counters->n_dense;
  const bool alone = n_items > kNormFew * (int)(gridDim.x / kNormCtas) ||
                     C.n_rows * C.n_cols <= (int64_t)kNormSmall * p.nI * p.nJ;
  const int rank = alone ? 0 : (int)cluster.block_rank(), ctas = alone ? 1 : kNormCtas;
  for (int it = blockIdx.x / ctas; it < n_items; it += gridDim.x / ctas) {
    const int t = p.l_dense[it];
    const int I = t / p.nJ, J = t % p.nJ;
    const int m = C.row_off[I + 1] - C.row_off[I];
    const int n = C.col_off[J + 1] - C.col_off[J];
    const double* D = C.pool + slot_of(C, I, J, m);
    double s = 0.0;
#pragma unroll 4
    for (int e = threadIdx.x + 256 * rank; e < m * n; e += 256 * ctas) s = fma(D[e], D[e], s);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (threadIdx.x % 32 == 0) red[threadIdx.x / 32] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
      double tot = 0.0;
      for (int i = 0; i < 8; ++i) tot += red[i];
      part = tot;
    }
    if (alone) {
      if (threadIdx.x == 0) C.norm[t] = sqrt(part);
      __syncthreads();
      continue;
    }
    cluster.sync();
    if (rank == 0 && threadIdx.x == 0) {
      double tot = 0.0;
      for (int c = 0; c < kNormCtas; ++c) tot += *cluster.map_shared_rank(&part, c);
      C.norm[t] = sqrt(tot);
    }
    cluster.sync();   // the parts have been read
  }
}

void launch_dense_tile_norms(const MatView& C, const Plan& p, cudaStream_t st) {
  dense_tile_norms_kernel<<<kNormGrid, 256, 0, st>>>(C, p);
}

__global__ void sqrt_dense_norms_kernel(MatView C, Plan p) {
  const int n_items = p.counters->n_dense;
  for (int it = blockIdx.x * blockDim.x + threadIdx.x; it < n_items; it += gridDim.x * blockDim.x) {
    const int t = p.l_dense[it];
    C.norm[t] = sqrt(C.norm[t]);
  }
}

void launch_sqrt_dense_norms(const MatView& C, const Plan& p, cudaStream_t st) {
  sqrt_dense_norms_kernel<<<64, 256, 0, st>>>(C, p);
}

}  // namespace clr
