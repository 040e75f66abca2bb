// K0 -- the product's work list.
//
// The paper's task-based SUMMA (Section 3.2) issues one multiply task per (i,k,j) block
// triple and reduces the partial products into C_ij; on one GPU that task graph becomes a
// triple list built on the device, sorted by C tile (then by k) so that one CTA can own each
// C tile and accumulate its products without atomics (the GEMM-update case of Section 3.2).
// Tiles are screened with the Frobenius-norm estimate of Section 4.1.
#include "clr_internal.h"

namespace clr {

__device__ __forceinline__ int out_rank(int kind, int ra, int rb) {
  // Section 4.1, Eq. 1: Z = W_A^T X_B is contracted on the side of smaller output rank.
  if (kind == T_DL) return rb;
  if (kind == T_LD) return ra;
  if (kind == T_LL) return rb <= ra ? rb : ra;
  return 0;
}

__device__ __forceinline__ unsigned long long triple_flops(int kind, long long m, long long k,
                                                           long long n, long long ra,
                                                           long long rb) {
  if (kind == T_DD) return 2ull * m * k * n;
  if (kind == T_DL) return 2ull * m * k * rb;
  if (kind == T_LD) return 2ull * k * n * ra;
  return 2ull * k * ra * rb + (rb <= ra ? 2ull * m * ra * rb : 2ull * n * ra * rb);
}

// One warp per C tile (I, J), its lanes over the inner clusters K.
// gemm_dacc_bound > 0 (split precision): a tile that would be accumulated densely in FP64
// (ROUTE_DACC) is summed by the tensor-core GEMM instead (ROUTE_DACC_G) when its norm estimate
// sum_K ||A_IK|| ||B_KJ|| is at most gemm_dacc_bound = eps / (16 u_split).
// oz.sa non-null (exact slices): the same when the estimate of the sliced sum's error,
// from the exponents of the tile's rows and columns per K segment, sum over segments
// s of sa[I][s] sb[J][s] (sa[I][s] = sum over rows i of I of 4^e_is), is at most oz.bound2.
__global__ void plan_count_kernel(MatView A, MatView B, Plan p, double eps_sp,
                                  double gemm_dacc_bound, OzDaccRule oz) {
  const int t = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 32);
  const int lane = threadIdx.x % 32;
  if (t >= p.nI * p.nJ) return;  // the whole warp
  const int I = t / p.nJ, J = t % p.nJ;
  const int m = A.row_off[I + 1] - A.row_off[I];
  const int n = B.col_off[J + 1] - B.col_off[J];
  bool pass = true;
  double est = 0.0;
  if (eps_sp > 0.0 || gemm_dacc_bound > 0.0) {
    for (int K = lane; K < p.nK; K += 32) {
      const int ka = A.kind[I * A.nc + K], kb = B.kind[K * B.nc + J];
      if (ka != CLR_KIND_ZERO && kb != CLR_KIND_ZERO)
        est += A.norm[I * A.nc + K] * B.norm[K * B.nc + J];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) est += __shfl_xor_sync(0xffffffffu, est, o);
    if (eps_sp > 0.0) pass = est > eps_sp * (double)m * (double)n;
  }
  int count = 0, has_dd = 0, rsum = 0;
  unsigned long long fl = 0;
  int byk[4] = {0, 0, 0, 0};
  if (pass) {
    for (int K = lane; K < p.nK; K += 32) {
      const int ka = A.kind[I * A.nc + K], kb = B.kind[K * B.nc + J];
      if (ka == CLR_KIND_ZERO || kb == CLR_KIND_ZERO) continue;
      const int kind = (ka == CLR_KIND_DENSE ? 0 : 2) + (kb == CLR_KIND_DENSE ? 0 : 1);
      const int ra = A.rank[I * A.nc + K], rb = B.rank[K * B.nc + J];
      const int k = A.col_off[K + 1] - A.col_off[K];
      ++count;
      byk[kind]++;
      fl += triple_flops(kind, m, k, n, ra, rb);
      if (kind == T_DD) has_dd = 1; else rsum += out_rank(kind, ra, rb);
    }
  }
  count = __reduce_add_sync(0xffffffffu, (unsigned)count);
  rsum = __reduce_add_sync(0xffffffffu, (unsigned)rsum);
  has_dd = __any_sync(0xffffffffu, has_dd);
#pragma unroll
  for (int q = 0; q < 4; ++q) byk[q] = __reduce_add_sync(0xffffffffu, (unsigned)byk[q]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) fl += __shfl_xor_sync(0xffffffffu, fl, o);
  if (lane != 0) return;
  int route = ROUTE_ZERO;
  if (count > 0) {
    int lim = (m < n ? m : n) / 2;
    route = has_dd ? ROUTE_DENSE : (rsum <= lim ? ROUTE_QR : ROUTE_DACC);
    if (route == ROUTE_DACC && gemm_dacc_bound > 0.0 && est <= gemm_dacc_bound) {
      route = ROUTE_DACC_G;
      atomicAdd(&p.counters->n_gemm_dacc, 1ull);
    }
    if (route == ROUTE_DACC && oz.sa) {
      double e2 = 0.0;
      for (int sg = 0; sg < oz.n_seg; ++sg)
        e2 += oz.sa[(int64_t)I * oz.n_seg + sg] * oz.sb[(int64_t)J * oz.n_seg + sg];
      if (e2 <= oz.bound2) {
        route = ROUTE_DACC_G;
        atomicAdd(&p.counters->n_gemm_dacc, 1ull);
      }
    }
  }
  p.t_count[t] = count;
  p.t_route[t] = route;
  p.t_rsum[t] = rsum;
  if (count > 0) {
    atomicAdd(&p.counters->n_triples, (unsigned long long)count);
    for (int q = 0; q < 4; ++q)
      if (byk[q]) atomicAdd(&p.counters->by_kind[q], (unsigned long long)byk[q]);
    atomicAdd(&p.counters->flops, fl);
    atomicAdd(&p.counters->by_mode[has_dd ? 1 : 2], 1ull);
    if (!has_dd) atomicMax(&p.counters->max_rsum, (unsigned long long)rsum);
  } else {
    atomicAdd(&p.counters->by_mode[0], 1ull);
  }
}

// Single-CTA scan: t_start = exclusive prefix sum of t_count, plus the tile lists in tile
// order.  Tile counts are at most a few hundred thousand, so one CTA of 1024 threads walking
// contiguous chunks is enough.
constexpr int kScanThreads = 1024;
constexpr int kScanQ = 5;
constexpr int kCostBuckets = 128;   // four an octave

// Bucket (4 log2, rounded down) of a tile's cost (which = 0: QR route recompression, 1: dense SVD, 2: dense x
// dense products, m n times the tile's number of products, 3: low-rank products: an X_t or W_t of
// ~32 (m + n) FMAs a column of the concatenation and, unless it is concatenated, m n for the sum).  A dense recompression's cost
// depends on the path the tile takes (dense certificate ~0.4, pivoted QR and the SVD of R
// ~1.1 when stored low rank and ~2 when stored dense, SM cycles per m n min(m, n) on the
// lattice iterates), known only once it ran: the cycles
// measured the last time a tile of this matrix was recompressed (Newton-Schulz reuses its
// matrices for the same products every iteration) replace the size estimate (2 m n min(m, n)
// cycles) when present.
__device__ __forceinline__ int cost_bucket(const Plan& p, int t, int which) {
  const int I = t / p.nJ, J = t % p.nJ;
  const long long m = p.row_off[I + 1] - p.row_off[I];
  const long long n = p.col_off[J + 1] - p.col_off[J];
  long long c;
  if (which == 0) {
    const long long R = p.t_rsum[t];
    c = (m + n) * R * R + R * R * R;
  } else if (which == 1) {
    const unsigned kc = p.c_cost ? p.c_cost[t] : 0u;
    c = kc ? (long long)kc << 10 : 2 * m * n * (m < n ? m : n);
  } else if (which == 2) {
    c = m * n * (long long)p.t_count[t];
  } else {
    c = (p.t_route[t] == ROUTE_QR ? 32 * (m + n) : m * n + 32 * (m + n)) * (long long)p.t_rsum[t];
  }
  if (c < 4) return 0;
  const int b = 63 - __clzll(c);
  const int q = 4 * b + (int)(c >> (b - 2) & 3);
  return q < kCostBuckets ? q : kCostBuckets - 1;
}

// How many of the most expensive recompressions take a team of kTeamCtas CTAs each instead of one
// CTA (compress_dense_team_kernel): with few tiles the launch takes what its largest tile takes
// while most SMs idle.  A team halves a tile's time and so doubles what it costs, hence the
// estimate max((E + E_K) / CTAs, e_0 / 2, e_K) of the launch's time for the K leading tiles, e_K
// the cost of the next one; the cut lies at the end of a bucket, within one tile a team, and is
// taken only for a tenth of the time or more.  By one warp; lane l holds the counts of the
// buckets kCostBuckets - 1 - 4 l and the three below.
__device__ __forceinline__ int team_tiles(const int (&cnt)[4], int n_ctas) {
  constexpr unsigned kAll = 0xffffffffu;
  const int l = threadIdx.x % 32;
  float e[4], own = 0.f, first = 0.f;
  int own_n = 0;
#pragma unroll
  for (int x = 3; x >= 0; --x) {
    const int b = kCostBuckets - 1 - 4 * l - x;
    e[x] = ldexpf(4.5f + (float)(b & 3), (b >> 2) - 2);   // the middle of the bucket
    own += (float)cnt[x] * e[x];
    own_n += cnt[x];
    if (cnt[x]) first = e[x];
  }
  float sum = own;
  int num = own_n;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const float v = __shfl_up_sync(kAll, sum, o);
    const int u = __shfl_up_sync(kAll, num, o);
    if (l >= o) {
      sum += v;
      num += u;
    }
  }
  const float all = __shfl_sync(kAll, sum, 31);
  const unsigned busy = __ballot_sync(kAll, own_n > 0);
  if (!busy) return 0;
  const float top = __shfl_sync(kAll, first, __ffs(busy) - 1);
  const unsigned later = l < 31 ? busy >> (l + 1) : 0u;
  float below = __shfl_sync(kAll, first, later ? l + __ffs(later) : l);
  if (!later) below = 0.f;   // nothing below this lane's buckets
  const float none = fmaxf(all / (float)n_ctas, top);
  float best = none;
  int cut = 0;
  float next[4];
#pragma unroll
  for (int x = 3; x >= 0; --x) {
    next[x] = below;
    if (cnt[x]) below = e[x];
  }
  sum -= own;
  num -= own_n;
#pragma unroll
  for (int x = 0; x < 4; ++x) {
    sum += (float)cnt[x] * e[x];
    num += cnt[x];
    const float t = fmaxf(fmaxf((all + sum) / (float)n_ctas, 0.5f * top), next[x]);
    if (cnt[x] && num <= n_ctas / kTeamCtas && t < best) {
      best = t;
      cut = num;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float t = __shfl_xor_sync(kAll, best, o);
    const int c = __shfl_xor_sync(kAll, cut, o);
    if (t < best || (t == best && c < cut)) {
      best = t;
      cut = c;
    }
  }
  return best < 0.9f * none ? cut : 0;
}

__global__ void __launch_bounds__(kScanThreads) plan_scan_kernel(Plan p, int recompress_dense) {
  __shared__ int sh[kScanQ][kScanThreads];
  const int n = p.nI * p.nJ;
  const int tid = threadIdx.x;
  const int chunk = (n + kScanThreads - 1) / kScanThreads;
  const int lo = min(n, tid * chunk), hi = min(n, lo + chunk);
  int s[kScanQ] = {0, 0, 0, 0, 0};
  // with a tensor-core GEMM the dense tiles and the DACC_G tiles take every contribution there
  // (low-rank operand blocks staged as X W^T)
  auto takes_lr = [&](int i, int route) {
    return p.t_rsum[i] > 0 && route != ROUTE_DACC_G && !(p.dense_by_gemm && route == ROUTE_DENSE);
  };
  for (int i = lo; i < hi; ++i) {
    int route = p.t_route[i];
    s[0] += p.t_count[i];
    s[1] += route == ROUTE_DENSE;
    s[2] += takes_lr(i, route);
    s[3] += route == ROUTE_QR;
    s[4] += route == ROUTE_DACC || route == ROUTE_DACC_G ||
            (route == ROUTE_DENSE && recompress_dense);
  }
  for (int q = 0; q < kScanQ; ++q) sh[q][tid] = s[q];
  __syncthreads();
  // Hillis-Steele inclusive scan over the 1024 partial sums.
  for (int off = 1; off < kScanThreads; off <<= 1) {
    int v[kScanQ];
    for (int q = 0; q < kScanQ; ++q) v[q] = tid >= off ? sh[q][tid - off] : 0;
    __syncthreads();
    for (int q = 0; q < kScanQ; ++q) sh[q][tid] += v[q];
    __syncthreads();
  }
  int base[kScanQ];
  for (int q = 0; q < kScanQ; ++q) base[q] = sh[q][tid] - s[q];
  for (int i = lo; i < hi; ++i) {
    int route = p.t_route[i];
    p.t_start[i] = base[0];
    base[0] += p.t_count[i];
    if (route == ROUTE_DENSE) p.l_dense[base[1]++] = i;
    if (takes_lr(i, route)) p.l_lr[base[2]++] = i;
    if (route == ROUTE_QR) p.l_qr[base[3]++] = i;
    if (route == ROUTE_DACC || route == ROUTE_DACC_G ||
        (route == ROUTE_DENSE && recompress_dense))
      p.l_dcomp[base[4]++] = i;
  }
  if (tid == kScanThreads - 1) {
    p.counters->n_dense = sh[1][tid];
    p.counters->n_lr = sh[2][tid];
    p.counters->n_qr = sh[3][tid];
    p.counters->n_dcomp = sh[4][tid];
    p.counters->n_dacc = 0;
  }
  // The recompression lists and those of dense and low-rank products again, largest cost first
  // (longest-processing-time order for the dynamically distributed kernels): a counting sort on
  // a quarter of an octave of the cost, m n min(m, n) for a dense SVD, (m + n) R^2 for a QR route, m n times the
  // number of products for dense x dense products.  The order within a bucket is immaterial:
  // every tile is processed independently.
  __syncthreads();
  const int n_qr = sh[3][kScanThreads - 1], n_dc = sh[4][kScanThreads - 1];
  const int n_de = sh[1][kScanThreads - 1], n_lr = sh[2][kScanThreads - 1];
  __shared__ int bcount[4][kCostBuckets], boff[4][kCostBuckets];
  static_assert(4 * kCostBuckets <= kScanThreads && kCostBuckets == 4 * 32, "buckets");
  if (tid < 4 * kCostBuckets) (&bcount[0][0])[tid] = 0;
  __syncthreads();
  auto item = [&](int i, int* which) {
    *which = i < n_qr ? 0 : i < n_qr + n_dc ? 1 : i < n_qr + n_dc + n_de ? 2 : 3;
    return *which == 0   ? p.l_qr[i]
           : *which == 1 ? p.l_dcomp[i - n_qr]
           : *which == 2 ? p.l_dense[i - n_qr - n_dc]
                         : p.l_lr[i - n_qr - n_dc - n_de];
  };
  const int n_all = n_qr + n_dc + n_de + n_lr;
  for (int i = tid; i < n_all; i += kScanThreads) {
    int which;
    const int t = item(i, &which);
    atomicAdd(&bcount[which][cost_bucket(p, t, which)], 1);
  }
  __syncthreads();
  if (tid < 4 * 32) {
    const int which = tid / 32, l = tid % 32;
    int cnt[4], own = 0;
#pragma unroll
    for (int x = 0; x < 4; ++x) own += cnt[x] = bcount[which][kCostBuckets - 1 - 4 * l - x];
    int incl = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (l >= o) incl += v;
    }
    int acc = incl - own;
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      boff[which][kCostBuckets - 1 - 4 * l - x] = acc;
      acc += cnt[x];
    }
    if (which == 1) {
      const int k = n_dc > 0 ? team_tiles(cnt, p.n_sm / kTeamCtas * kTeamCtas) : 0;
      if (l == 0) p.counters->n_team = k;
    }
  }
  __syncthreads();
  for (int i = tid; i < n_all; i += kScanThreads) {
    int which;
    const int t = item(i, &which);
    const int pos = atomicAdd(&boff[which][cost_bucket(p, t, which)], 1);
    (which == 0 ? p.l_qr_s : which == 1 ? p.l_dcomp_s : which == 2 ? p.l_dense_s : p.l_lr_s)[pos] = t;
  }
}

// One warp per C tile: its lanes take 32 inner clusters at a time; a ballot gives each
// nonzero triple its place (K order) and a warp scan of the output ranks its first factor
// column in the tile's concatenation.
__global__ void plan_fill_kernel(MatView A, MatView B, Plan p) {
  const int t = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 32);
  const int lane = threadIdx.x % 32;
  if (t >= p.nI * p.nJ) return;  // the whole warp
  if (p.t_count[t] == 0) return;
  const int I = t / p.nJ, J = t % p.nJ;
  int64_t pos = p.t_start[t];
  int col = 0;
  for (int K0 = 0; K0 < p.nK; K0 += 32) {
    const int K = K0 + lane;
    int ka = CLR_KIND_ZERO, kb = CLR_KIND_ZERO;
    if (K < p.nK) {
      ka = A.kind[I * A.nc + K];
      kb = B.kind[K * B.nc + J];
    }
    const bool on = ka != CLR_KIND_ZERO && kb != CLR_KIND_ZERO;
    const unsigned mask = __ballot_sync(0xffffffffu, on);
    const int kind = (ka == CLR_KIND_DENSE ? 0 : 2) + (kb == CLR_KIND_DENSE ? 0 : 1);
    const int r = on ? out_rank(kind, A.rank[I * A.nc + K], B.rank[K * B.nc + J]) : 0;
    int incl = r;  // inclusive prefix sum of the output ranks over the lanes
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    if (on) {
      Triple tr;
      tr.tile = t;
      tr.k = K;
      tr.kind = kind;
      tr.col = col + incl - r;
      const int64_t at = pos + __popc(mask & ((1u << lane) - 1u));
      if (at < p.max_triples) p.triples[at] = tr; else atomicCAS(&p.counters->err, 0, 2);
    }
    pos += __popc(mask);
    col += __shfl_sync(0xffffffffu, incl, 31);
  }
}

void launch_plan_scan(const Plan& p, int recompress_dense, cudaStream_t st) {
  plan_scan_kernel<<<1, kScanThreads, 0, st>>>(p, recompress_dense);
}

void launch_plan(const MatView& A, const MatView& B, const Plan& p, double eps_sp,
                 int recompress_dense, double gemm_dacc_bound, const OzDaccRule& oz,
                 cudaStream_t st) {
  const int n = p.nI * p.nJ;
  const int threads = 128;  // 4 tiles per block: one warp each
  const int blocks = (int)(((int64_t)n * 32 + threads - 1) / threads);
  cudaMemsetAsync(p.counters, 0, kPlanCountersClear, st);
  plan_count_kernel<<<blocks, threads, 0, st>>>(A, B, p, eps_sp, gemm_dacc_bound, oz);
  plan_scan_kernel<<<1, kScanThreads, 0, st>>>(p, recompress_dense);
  plan_fill_kernel<<<blocks, threads, 0, st>>>(A, B, p);
}

}  // namespace clr
