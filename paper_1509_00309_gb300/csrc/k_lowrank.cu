// K2/K3/K4 -- low-rank tile products and their accumulation into C tiles (FP64).
//
// Section 4.1: products are kept in low-rank form whenever an operand is low rank.
//   dense x LR  (DL):  A_IK (X_B W_B^T)          -> (A_IK X_B) W_B^T        rank r_B
//   LR x dense  (LD):  (X_A W_A^T) B_KJ          -> X_A (B_KJ^T W_A)^T      rank r_A
//   LR x LR     (LL):  Z = W_A^T X_B (r_A x r_B), then X_A Z with W_B (rank r_B) or X_A with
//                      W_B Z^T (rank r_A), whichever output rank is smaller (Eq. 1; tie: X_A Z)
// Low-rank sums are concatenations of factors (Eq. lr_addition).  One cluster of CTAs owns one C
// tile and walks its products in k order:
//   ROUTE_QR     the factor pairs are written side by side into the tile's concatenation
//                workspace (X_cat m x R, W_cat n x R) for recompression by K5;
//   ROUTE_DENSE  the tile already holds the dense x dense sum; every low-rank product is
//                added as X_t W_t^T;
//   ROUTE_DACC   the concatenated rank exceeds floor(min(m,n)/2), so the sum is accumulated
//                densely (from zero) and K5 takes a dense truncated SVD.
// With a tensor-core GEMM (split precision or exact slices: Plan::dense_by_gemm) the GEMM sums all
// contributions of DENSE and DACC_G tiles, which are not in the list then; this kernel builds the
// ROUTE_QR concatenations and the FP64 DACC sums.
//
// The work is FP64-pipe-bound (~2 FMAs per clock and SM).  While the tiles with low-rank work are
// few, or differ by an order of magnitude, a tile is spread over the CTAs of a cluster: CTA c owns
// the rows [m c / CS, m (c + 1) / CS) of the tile, of X_cat and of every X_t, and that share of the
// rows of W_cat.  What every CTA needs whole (Z, and a computed W_t of a dense accumulation) is
// formed in shares into the cluster's scratch and exchanged by one cluster barrier; two buffers in
// turn make that barrier the only one.  Measured (one tile per CTA before): Coulomb-like lattice at
// N = 2048 (144 tiles, 1452 LL products of rank ~40) 25.3 -> 7.7 ms (1 of it by taking the most
// expensive tiles first); 1D chain at N = 2048 257 -> 70 us.  With more than kTilesPerCta tiles a
// CTA they fill the SMs one to a CTA, and shares only cost barriers and ragged micro-tiles (CS = 1;
// ms with CS = 4 / 1: 3D lattice, 529 tiles 48 / 49, 1156 tiles (Coulomb-like) 133 / 117, 2116
// 306 / 263; clusters of at most 48 points, 48400 tiles, 1106 / 581).
#include <cooperative_groups.h>

#include "clr_internal.h"

namespace clr {

namespace cg = cooperative_groups;

constexpr int kLrThreads = 256;
// Tiles with work, a CTA of the grid, from which each CTA takes its own (608 at two CTAs an SM:
// between the 529 and the 784 tiles measured).
constexpr int kTilesPerCta = 2;

// out(i,j) (= or +=) sum_l a(i,l) b(l,j) for a P x Q output with arbitrary element strides, the
// micro-tile by the size of the output (clr_internal.h).
__device__ __forceinline__ void cta_gemm(int P, int Q, int L, const double* a, int64_t a_r,
                                         int64_t a_c, const double* b, int64_t b_r, int64_t b_c,
                                         double* out, int64_t ldo, bool accumulate) {
  cta_gemm_auto((int)threadIdx.x, kLrThreads, P, Q, L, a, a_r, a_c, b, b_r, b_c, out, ldo, accumulate);
}

__device__ void cta_copy_cols(int rows, int cols, const double* src, int64_t lds, double* dst,
                              int64_t ldd) {
  for (int e = threadIdx.x; e < rows * cols; e += kLrThreads) {
    const int i = e % rows, j = e / rows;
    dst[i + (int64_t)j * ldd] = src[i + (int64_t)j * lds];
  }
}

constexpr int64_t kZElems = (int64_t)(CLR_MAX_CLUSTER / 2) * (CLR_MAX_CLUSTER / 2);
constexpr int64_t kFElems = (int64_t)CLR_MAX_CLUSTER * (CLR_MAX_CLUSTER / 2);
// scratch: per cluster (in its first CTA's part) two buffers of Z and of a shared W_t, then per
// CTA its rows of X_t
static_assert(2 * (kZElems + kFElems) + kFElems <= kSvdScratchPerCta, "low-rank scratch");

template <int CS>
__global__ void __cluster_dims__(CS, 1, 1) __launch_bounds__(kLrThreads)
    lr_products_kernel(MatView A, MatView B, MatView C, Plan p, double* ws, double* scratch,
                       int64_t scratch_per_cta, int few) {
  cg::cluster_group cluster = cg::this_cluster();
  __shared__ int sh_next[2];
  const int n_lr = p.counters->n_lr;
  if (few != 0 && (n_lr > few) != (CS == 1)) return;   // the other launch's work
  const int rank = CS > 1 ? (int)cluster.block_rank() : 0;
  auto tile_sync = [&]() {
    if constexpr (CS == 1) __syncthreads(); else cluster.sync();
  };
  double* shared_scr = scratch + (int64_t)(blockIdx.x - rank) * scratch_per_cta;
  double* scrX = scratch + (int64_t)blockIdx.x * scratch_per_cta + 2 * (kZElems + kFElems);
  int* sched = &p.counters->sched[0];
  int slot = 0, par = 0;
  // a CTA's shared memory may be written by another only once it is known to have started
  if (CS > 1) cluster.sync();
  while (true) {
    // the cluster's next tile (two slots: one is read while the other is written)
    if (rank == 0 && threadIdx.x == 0) {
      const int v = atomicAdd(sched, 1);
      if (CS == 1) sh_next[slot] = v;
      else
        for (int c = 0; c < CS; ++c) *cluster.map_shared_rank(&sh_next[slot], c) = v;
    }
    tile_sync();
    const int li = sh_next[slot];
    slot ^= 1;
    if (li >= n_lr) break;
    const int t = p.l_lr_s[li];
    const int I = t / p.nJ, J = t % p.nJ;
    const int m = C.row_off[I + 1] - C.row_off[I];
    const int n = C.col_off[J + 1] - C.col_off[J];
    const int route = p.t_route[t];
    const int R = p.t_rsum[t];
    const int64_t sC = slot_of(C, I, J, m);
    double* D = C.pool + sC;
    double* Xcat = ws + 2 * sC;
    double* Wcat = Xcat + (int64_t)m * R;
    const bool concat = route == ROUTE_QR;
    // this CTA's rows of the tile (and of X_t), and of W_t
    const int x0 = m * rank / CS, xr = m * (rank + 1) / CS - x0;
    const int w0 = n * rank / CS, wr = n * (rank + 1) / CS - w0;
    bool first = route == ROUTE_DACC;   // a DACC sum starts from zero
    const int start = p.t_start[t], count = p.t_count[t];
    for (int q = 0; q < count; ++q) {
      const Triple tr = p.triples[start + q];
      if (tr.kind == T_DD) continue;
      const int K = tr.k;
      const int k = A.col_off[K + 1] - A.col_off[K];
      const int ra = A.rank[I * A.nc + K], rb = B.rank[K * B.nc + J];
      const double* Ab = A.pool + slot_of(A, I, K, m);
      const double* Bb = B.pool + slot_of(B, K, J, k);
      const double* XA = Ab;                        // low-rank A: m x ra, then k x ra
      const double* WA = Ab + (int64_t)m * ra;
      const double* XB = Bb;                        // low-rank B: k x rb, then n x rb
      const double* WB = Bb + (int64_t)k * rb;
      const bool x_side = tr.kind == T_DL || (tr.kind == T_LL && rb <= ra);
      double* scrZ = shared_scr + par * (kZElems + kFElems);
      double* scrF = scrZ + kZElems;
      if (tr.kind == T_LL) {
        // Z = W_A^T X_B (ra x rb, column-major), its columns in shares
        const int z0 = rb * rank / CS, zc = rb * (rank + 1) / CS - z0;
        cta_gemm(ra, zc, k, WA, k, 1, XB + (int64_t)z0 * k, 1, k, scrZ + (int64_t)z0 * ra, ra,
                 false);
        tile_sync();
        par ^= 1;
      }
      const int rt = x_side ? rb : ra;
      if (x_side) {
        // X_t = A_IK X_B or X_A Z, this CTA's rows; W_t = W_B
        double* dst = concat ? Xcat + (int64_t)m * tr.col + x0 : scrX;
        const int64_t ldd = concat ? m : xr;
        if (tr.kind == T_DL)
          cta_gemm(xr, rb, k, Ab + x0, 1, m, XB, 1, k, dst, ldd, false);
        else
          cta_gemm(xr, rb, ra, XA + x0, 1, m, scrZ, 1, ra, dst, ldd, false);
        if (concat) cta_copy_cols(wr, rb, WB + w0, n, Wcat + (int64_t)n * tr.col + w0, n);
      } else {
        // X_t = X_A; W_t = B_KJ^T W_A or W_B Z^T, this CTA's rows
        double* dst = (concat ? Wcat + (int64_t)n * tr.col : scrF) + w0;
        if (tr.kind == T_LD)
          cta_gemm(wr, ra, k, Bb + (int64_t)w0 * k, k, 1, WA, 1, k, dst, n, false);
        else
          cta_gemm(wr, ra, rb, WB + w0, 1, n, scrZ, ra, 1, dst, n, false);
        if (concat) cta_copy_cols(xr, ra, XA + x0, m, Xcat + (int64_t)m * tr.col + x0, m);
      }
      if (!concat) {
        // D += X_t W_t^T, this CTA's rows (the whole of W_t)
        const double* Xt = x_side ? scrX : XA + x0;
        const int64_t ldx = x_side ? xr : m;
        if (x_side) {
          __syncthreads();
        } else {
          tile_sync();
          if (tr.kind == T_LD) par ^= 1;   // (an LL product has switched buffers already)
        }
        cta_gemm(xr, n, rt, Xt, 1, ldx, x_side ? WB : scrF, n, 1, D + x0, m, !first);
        first = false;
        __syncthreads();
      }
    }
    __syncthreads();
  }
}

int launch_lr_products(const MatView& A, const MatView& B, const MatView& C, const Plan& p,
                       double* ws, double* scratch, int64_t scratch_per_cta, int grid,
                       cudaStream_t st) {
  // Eight CTAs a tile while the tiles are few (the 1D chain at N = 512: 16 tiles on 152 SMs), else
  // four (from about 64 tiles on four already fill the SMs, with fewer exchanges) or one.  How many
  // tiles have work is the device's to know: of two launches the one whose case it is not returns.
  const int tiles = p.nI * p.nJ, few = kTilesPerCta * grid;
  auto launch = [&](auto kernel, int cs) {
    const int g = grid / cs > 0 ? grid / cs * cs : cs;
    kernel<<<g, kLrThreads, 0, st>>>(A, B, C, p, ws, scratch, scratch_per_cta,
                                     tiles > few ? few : 0);
  };
  if (tiles <= 64) launch(lr_products_kernel<8>, 8); else launch(lr_products_kernel<4>, 4);
  if (tiles <= few) return 1;
  launch(lr_products_kernel<1>, 1);
  return 2;
}

}  // namespace clr
