// K5 -- recompression of C tiles (FP64), and the truncated SVD used to build CLR matrices.
//
// Section 4.1 recompresses a low-rank sum X W^T by QR of both factors, X = Q_X R_X and
// W = Q_W R_W, a low-rank decomposition of the small core M = R_X R_W^T, and re-expansion
// X' = Q_X X_M, W' = Q_W W_M.  The decomposition of M is taken to be its SVD (the paper does
// not name it); truncation keeps the smallest rank whose Frobenius error is <= eps, with the
// singular values on the left factor (X' = Q_X U_r S_r, W' = Q_W V_r).  A block whose rank
// exceeds floor(min(m,n)/2) is stored dense.
//
// A CTA (16 warps), or a team of CTAs (compress_dense_body, compress_qr_kernel's pairs), handles one
// tile at a time, taking tiles from a launch-wide counter:
//   Householder QR         LAPACK-style reflectors H = I - tau v v^T, v_0 = 1;
//   one-sided Jacobi SVD   Hestenes rotations on column pairs, round-robin ordering so a
//                          round's pairs are disjoint (one warp per pair), until no pair has
//                          |g_a.g_b| > tol ||g_a|| ||g_b|| or the sweep limit is reached
//                          (mixed FP32/FP64 stages, svd_mixed);
//   rank-revealing QR      the paper's construction for building from dense (option).
// FP64 working arrays live in the tile's workspace slot (2 m n doubles per tile, enough for
// either route); the FP32 copies of the mixed-precision SVD in shared memory, or in a per-CTA
// scratch where they do not fit.
#include <cooperative_groups.h>

#include <cfloat>
#include <mutex>
#include <type_traits>

#include "clr_internal.h"

namespace clr {

constexpr int kThreads = 512;
// index of the per-path cycle counters in the profiling counters (third block of 8)
constexpr int kPathCounters = 16;
// compress_dense_kernel's full-SVD stages while profiling (block 3 of the counters): cycles of
// the pivoted QR attempt, the five stages of svd_mixed (the fifth: FP64 sweeps, near the noise
// floor only), truncation and stores; then the count
constexpr int kFullStageCounters = 24;
// the same for the pre-reduced path (block 4): the QR, the five stages of svd_mixed on R^T,
// truncation, recovery and the factors' stores; then the count
constexpr int kPreStageCounters = 32;
// tiles taken by a team of CTAs (block 5)
constexpr int kTeamTileCounter = 40;
constexpr int kWarps = kThreads / 32;

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sum over the CTA, returned to every thread.  The 16 warps' partial sums are added by one warp:
// an FP64 instruction holds its sub-partition's FP64 pipe for 64 cycles whatever its lanes do, so
// the same 16 additions made by every warp took 4.9k cycles a call, these four take 0.4k.
__device__ double block_sum(double v, double* sh) {
  v = warp_sum(v);
  const int w = threadIdx.x / 32, l = threadIdx.x % 32;
  __syncthreads();
  if (l == 0) sh[w] = v;
  __syncthreads();
  if (w == 0) {
    double s = l < kWarps ? sh[l] : 0.0;
#pragma unroll
    for (int o = kWarps / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (l == 0) sh[0] = s;
  }
  __syncthreads();
  const double s = sh[0];
  __syncthreads();
  return s;
}

// The CTAs that work on one tile: one, or a whole cluster (compress_dense_kernel while tiles are
// few).  Data in global memory is shared out by tid / nt and w / nw; what every CTA needs in
// shared memory each keeps a copy of, computed alike from the same data or written to every copy
// by put().
// (One is the team of a single CTA, known when the kernel is compiled.)
struct Team {
  int rank, size;   // this CTA and the number of CTAs
  int tid, nt;      // this thread and the threads of the team
  int w, nw;        // this warp (warps are dealt over the CTAs) and the warps of the team
  __device__ __forceinline__ Team(int r, int n)
      : rank(r), size(n), tid(r * kThreads + threadIdx.x), nt(n * kThreads),
        w(r + n * (int)(threadIdx.x / 32)), nw(n * kWarps) {}
  __device__ __forceinline__ void sync() const {
    if (size == 1) __syncthreads(); else cooperative_groups::this_cluster().sync();
  }
  template <class T>
  __device__ __forceinline__ void put(T* local, T v) const {
    if (size == 1) {
      *local = v;
    } else {
      cooperative_groups::cluster_group c = cooperative_groups::this_cluster();
      for (int r = 0; r < size; ++r) *c.map_shared_rank(local, r) = v;
    }
  }
};
struct One {
  static constexpr int rank = 0, size = 1, nt = kThreads, nw = kWarps;
  int tid, w;
  __device__ __forceinline__ One() : tid(threadIdx.x), w(threadIdx.x / 32) {}
  __device__ __forceinline__ void sync() const { __syncthreads(); }
  template <class T>
  __device__ __forceinline__ void put(T* local, T v) const {
    *local = v;
  }
};

// ---------------------------------------------------------------------------------------------
// Householder steps.  What bounds them is the FP64 pipe: one warp-instruction per 19 cycles and
// SM, an addition in a reduction as dear as a fused multiply-add, and a scalar square root or
// division (9 such instructions) repeated by 16 warps dearer than the column work of a small
// step.  So:
//  - a warp takes eight columns at a time, eight lanes to a column and two columns to a lane: the
//    inner products need 3 additions for the eight columns (with a warp per column 5 each), no
//    more than 7 rows' lanes idle in a column's last instruction, and the scalars that follow
//    (the multiplier, the new entry of R, the downdated norm) are formed for the eight columns
//    by one instruction each, in the lanes that hold their sums;
//  - the reflector is not scaled: v = (v_0, x_{j+1}, ...) with x the column as it is, and
//    H y = y - v (v.y) rn rv with rn = 1 / ||x_j..||, rv = 1 / |v_0| (v.v / 2 = ||x|| |v_0|; two
//    factors, so that neither over- nor underflows before ||x||^2 does).  One warp forms these
//    while the others already take their columns' inner products with x, which need no scalar.
// Measured: the two 16-column QRs of a 164 x 132 tile took 580k SM cycles with a warp per column
// and the scalars by every warp; 96k now (in registers, a CTA each, below).
// ---------------------------------------------------------------------------------------------
constexpr int kRowsPerLane = CLR_MAX_CLUSTER / 32;
constexpr int kGroup = 8;   // columns a warp takes together in a step
constexpr int kQuad = 4;    // and where it holds whole columns (warp_sum4)

// The warp's sums of s[0..3]: lane l receives the sum of s[l / 8].
__device__ __forceinline__ double warp_sum4(const double (&s)[kQuad]) {
  const int l = threadIdx.x % 32;
  const bool h16 = (l & 16) != 0, h8 = (l & 8) != 0;
  double a0 = h16 ? s[2] : s[0], a1 = h16 ? s[3] : s[1];
  a0 += __shfl_xor_sync(0xffffffffu, h16 ? s[0] : s[2], 16);
  a1 += __shfl_xor_sync(0xffffffffu, h16 ? s[1] : s[3], 16);
  double a = h8 ? a1 : a0;
  a += __shfl_xor_sync(0xffffffffu, h8 ? a0 : a1, 8);
  a += __shfl_xor_sync(0xffffffffu, a, 4);
  a += __shfl_xor_sync(0xffffffffu, a, 2);
  a += __shfl_xor_sync(0xffffffffu, a, 1);
  return a;
}

__device__ __forceinline__ void group_sync(int bar, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(threads) : "memory");
}

// One group of a step: columns c0 .. c0 + 7 of ncol (col(c): the column's n rows), lane l works on
// columns c0 + l / 8 and c0 + 4 + l / 8, rows l % 8, l % 8 + 8, ...; the sums arrive in the lanes
// of group_column.
__device__ __forceinline__ int group_column(int c0) {
  const int l = threadIdx.x % 32;
  return c0 + l / 8 + (l & 4);
}
__device__ __forceinline__ double group_sum(double s0, double s1) {
  const bool hi = (threadIdx.x & 4) != 0;
  double a = hi ? s1 : s0;
  a += __shfl_xor_sync(0xffffffffu, hi ? s0 : s1, 4);
  a += __shfl_xor_sync(0xffffffffu, a, 2);
  a += __shfl_xor_sync(0xffffffffu, a, 1);
  return a;
}
template <class Col>
__device__ __forceinline__ double group_dot(const double* x, int n, int c0, int ncol, Col col) {
  const int l = threadIdx.x % 32, a = c0 + l / 8, b = a + 4;
  const double* ya = col(a < ncol ? a : c0);
  const double* yb = col(b < ncol ? b : c0);
  double s0 = 0.0, s1 = 0.0;
  if (c0 + 4 < ncol) {
#pragma unroll 4
    for (int i = l % 8; i < n; i += 8) {
      const double xv = x[i];
      s0 = fma(xv, ya[i], s0);
      s1 = fma(xv, yb[i], s1);
    }
  } else {
#pragma unroll 4
    for (int i = l % 8; i < n; i += 8) s0 = fma(x[i], ya[i], s0);
  }
  return group_sum(s0, s1);
}
// y_c -= f_c x, f_c in the lanes of group_column
template <class Col>
__device__ __forceinline__ void group_update(const double* x, double f, int n, int c0, int ncol,
                                             Col col) {
  const int l = threadIdx.x % 32, a = c0 + l / 8, b = a + 4;
  const double fa = -__shfl_sync(0xffffffffu, f, l & 24);
  const double fb = -__shfl_sync(0xffffffffu, f, (l & 24) + 4);
  double* ya = col(a < ncol ? a : c0);
  double* yb = col(b < ncol ? b : c0);
  if (b < ncol) {
#pragma unroll 4
    for (int i = l % 8; i < n; i += 8) {
      const double xv = x[i];
      const double u = fma(fa, xv, ya[i]), v = fma(fb, xv, yb[i]);
      ya[i] = u;
      yb[i] = v;
    }
  } else if (a < ncol) {
#pragma unroll 4
    for (int i = l % 8; i < n; i += 8) ya[i] = fma(fa, x[i], ya[i]);
  }
  __syncwarp();
}
template <class Col>
__device__ __forceinline__ double group_squares(int n, int c0, int ncol, Col col) {
  const int l = threadIdx.x % 32, a = c0 + l / 8, b = a + 4;
  const double* ya = col(a < ncol ? a : c0);
  const double* yb = col(b < ncol ? b : c0);
  double s0 = 0.0, s1 = 0.0;
#pragma unroll 4
  for (int i = l % 8; i < n; i += 8) {
    s0 = fma(ya[i], ya[i], s0);
    s1 = fma(yb[i], yb[i], s1);
  }
  return group_sum(s0, s1);
}

// The reflector of a column (x0 above the n rows x), by one warp: *v0, *rn, *rv as above (rn =
// 0 and H = I when the rows below are zero) and the new diagonal entry (returned).
__device__ __forceinline__ double make_reflector(const double* x, int n, double x0, double* v0,
                                                 double* rn, double* rv) {
  double s = 0.0;
  for (int i = threadIdx.x % 32; i < n; i += 32) s = fma(x[i], x[i], s);
  s = warp_sum(s);
  double beta = x0, a = 0.0, b = 0.0, c = 0.0;
  if (s > 0.0) {
    const double t2 = fma(x0, x0, s);
    b = rsqrt(t2);
    const double nrm = t2 * b;
    a = x0 + copysign(nrm, x0);
    c = 1.0 / fabs(a);
    beta = -copysign(nrm, x0);
  }
  *v0 = a;
  *rn = b;
  *rv = c;
  return beta;
}

// The reflectors of one QR in shared memory: H_j = I - v v^T rn[j] rv[j], v = (v0[j], rows
// below the diagonal of column j).
struct Reflectors {
  double v0[CLR_MAX_CLUSTER], rn[CLR_MAX_CLUSTER], rv[CLR_MAX_CLUSTER];
  double x0, beta;   // of the current step (householder_qr_regs)
};

// In-place Householder QR of the p x q column-major matrix a (ld p), p >= q, by the nw warps of
// a group (warp w of it; bar: the group's named barrier).  R is left in the upper triangle, the
// reflector rows below it.
__device__ __noinline__ void householder_qr(double* a, int p, int q, Reflectors& h, int w, int nw,
                                            int bar) {
  const int l = threadIdx.x % 32;
  for (int j = 0; j < q; ++j) {
    double* cj = a + (int64_t)j * p;
    const int n = p - j - 1, ncol = q - j - 1;
    auto col = [&](int c) { return a + (int64_t)(j + 1 + c) * p + j + 1; };
    const double* x = cj + j + 1;
    double d = 0.0;
    if (w == 0) {
      double v0, rn, rv;
      const double beta = make_reflector(x, n, cj[j], &v0, &rn, &rv);
      __syncwarp();
      if (l == 0) {
        cj[j] = beta;
        h.v0[j] = v0;
        h.rn[j] = rn;
        h.rv[j] = rv;
      }
    } else if (kGroup * (w - 1) < ncol) {
      d = group_dot(x, n, kGroup * (w - 1), ncol, col);
    }
    group_sync(bar, 32 * nw);
    const double v0 = h.v0[j], rn = h.rn[j], rv = h.rv[j];
    // the groups taken above, then the rest over all warps
    for (int gi = w > 0 ? w - 1 : nw - 1; kGroup * gi < ncol; gi = (gi < nw - 1 ? nw - 1 + w : gi + nw)) {
      const int c0 = kGroup * gi, c = group_column(c0);
      if (gi >= nw - 1) d = group_dot(x, n, c0, ncol, col);
      const double yj = c < ncol ? col(c)[-1] : 0.0;
      const double f = fma(v0, yj, d) * rn * rv;
      group_update(x, f, n, c0, ncol, col);
      if (c < ncol && l % 4 == 0) col(c)[-1] = fma(-f, v0, yj);
    }
    group_sync(bar, 32 * nw);
  }
}

// The same QR where a lane can keep its share of a column: each of the group's nw warps holds four
// columns (q <= 4 nw) in registers from the first step to the last, eight lanes a column, rows
// l % 8, l % 8 + 8, ... of them (kRows >= ceil(p / 8)); only the step's reflector goes through
// shared memory (xs: 512 doubles of the group, two buffers in turn).  A step of a small factor is
// bound by latency, its loads above all: with the columns in global memory a step took 16k SM
// cycles at 16 columns.  The last warp forms the scalars.
template <int kRows>
__device__ __noinline__ void householder_qr_regs(double* a, int p, int q, Reflectors& h,
                                                 double* xs, int w, int nw, int bar) {
  const int l = threadIdx.x % 32, r8 = l % 8;
  const int c = kQuad * w + l / 8;   // this lane's column
  double y[kRows];
#pragma unroll
  for (int t = 0; t < kRows; ++t)
    y[t] = c < q && r8 + 8 * t < p ? a[r8 + 8 * t + (int64_t)c * p] : 0.0;
  const int nt = (p + 7) / 8;
  for (int j = 0; j < q; ++j) {
    double* x = xs + (j & 1) * CLR_MAX_CLUSTER;
    const int t0 = j / 8;
    const bool mine = kQuad * w < q && kQuad * w + kQuad - 1 >= j;   // a column from j on (warp)
    double yj = 0.0;   // row j of this lane's column
    if (mine) {
#pragma unroll
      for (int t = 0; t < kRows; ++t)
        if (t == t0) yj = y[t];
      yj = __shfl_sync(0xffffffffu, yj, (l & 24) + j % 8);
      if (c == j) {
#pragma unroll
        for (int t = 0; t < kRows; ++t)
          if (t <= nt) x[r8 + 8 * t] = r8 + 8 * t > j ? y[t] : 0.0;
        if (r8 == 0) h.x0 = yj;
      }
    }
    group_sync(bar, 32 * nw);
    const double x0 = h.x0;
    if (w == nw - 1) {
      double v0, rn, rv;
      const double beta = make_reflector(x + j + 1, p - j - 1, x0, &v0, &rn, &rv);
      if (l == 0) {
        h.beta = beta;
        h.v0[j] = v0;
        h.rn[j] = rn;
        h.rv[j] = rv;
      }
    }
    double d = 0.0;
    if (mine) {
#pragma unroll
      for (int t = 0; t < kRows; t += 2)   // (two rows' loads together)
        if (t + 1 >= t0 && t < nt) {
          const double xa = x[r8 + 8 * t], xb = x[r8 + 8 * t + 8];
          d = fma(xa, y[t], d);
          d = fma(xb, y[t + 1], d);
        }
      d += __shfl_xor_sync(0xffffffffu, d, 4);
      d += __shfl_xor_sync(0xffffffffu, d, 2);
      d += __shfl_xor_sync(0xffffffffu, d, 1);
    }
    group_sync(bar, 32 * nw);
    if (mine) {
      const double v0 = h.v0[j];
      const double f = c > j ? fma(v0, yj, d) * h.rn[j] * h.rv[j] : 0.0;
#pragma unroll
      for (int t = 0; t < kRows; t += 2)
        if (t + 1 >= t0 && t < nt) {
          const double xa = x[r8 + 8 * t], xb = x[r8 + 8 * t + 8];
          y[t] = fma(-f, xa, y[t]);
          y[t + 1] = fma(-f, xb, y[t + 1]);
        }
      const double yn = c == j ? h.beta : fma(-f, v0, yj);
      const bool row_j = r8 == j % 8 && c >= j;
#pragma unroll
      for (int t = 0; t < kRows; ++t)
        if (t == t0 && row_j) y[t] = yn;
    }
  }
#pragma unroll
  for (int t = 0; t < kRows; ++t)
    if (c < q && r8 + 8 * t < p) a[r8 + 8 * t + (int64_t)c * p] = y[t];
}

// The QR of a factor by a warp group, in registers where it fits.
__device__ __forceinline__ void factor_qr(double* a, int p, int q, Reflectors& h, double* xs,
                                          int w, int nw, int bar) {
  if (q > kQuad * nw) householder_qr(a, p, q, h, w, nw, bar);
  else if (p <= 128) householder_qr_regs<16>(a, p, q, h, xs, w, nw, bar);
  else if (p <= 192) householder_qr_regs<24>(a, p, q, h, xs, w, nw, bar);
  else householder_qr_regs<32>(a, p, q, h, xs, w, nw, bar);
}

// y (p x r, ld ldy) <- Q y with Q = H_0 H_1 ... H_{k-1}; the rows of reflector j are in column
// perm[j] (j when perm is null) of v (ld p).  Each warp carries four columns of y at a time through
// all reflectors in registers (eight lanes a column): no step waits for another warp.
template <int kRows>
__device__ __noinline__ void apply_q_regs(const double* v, int p, int k, const Reflectors& h,
                                          const int* perm, double* y, int r, int64_t ldy, int w,
                                          int nw) {
  const int l = threadIdx.x % 32, r8 = l % 8;
  const int nt = (p + 7) / 8;
  for (int g0 = kQuad * w; g0 < r; g0 += kQuad * nw) {
    const int c = g0 + l / 8;
    double* yc = y + (int64_t)c * ldy;
    double yr[kRows];
#pragma unroll
    for (int t = 0; t < kRows; ++t) yr[t] = c < r && r8 + 8 * t < p ? yc[r8 + 8 * t] : 0.0;
    for (int j = k - 1; j >= 0; --j) {
      const double* vj = v + (int64_t)(perm ? perm[j] : j) * p;
      const double v0 = h.v0[j];
      // rows two at a time, so that their loads go out together
      auto xv = [&](int i) { return i > j && i < p ? vj[i] : (i == j ? v0 : 0.0); };
      double s = 0.0;
#pragma unroll
      for (int t = 0; t < kRows; t += 2)
        if (8 * (t + 2) > j && t < nt) {
          const double xa = xv(r8 + 8 * t), xb = xv(r8 + 8 * t + 8);
          s = fma(xa, yr[t], s);
          s = fma(xb, yr[t + 1], s);
        }
      s += __shfl_xor_sync(0xffffffffu, s, 4);
      s += __shfl_xor_sync(0xffffffffu, s, 2);
      s += __shfl_xor_sync(0xffffffffu, s, 1);
      const double f = -s * h.rn[j] * h.rv[j];
#pragma unroll
      for (int t = 0; t < kRows; t += 2)
        if (8 * (t + 2) > j && t < nt) {
          const double xa = xv(r8 + 8 * t), xb = xv(r8 + 8 * t + 8);
          yr[t] = fma(f, xa, yr[t]);
          yr[t + 1] = fma(f, xb, yr[t + 1]);
        }
    }
#pragma unroll
    for (int t = 0; t < kRows; ++t)
      if (c < r && r8 + 8 * t < p) yc[r8 + 8 * t] = yr[t];
  }
}

__device__ __forceinline__ void apply_q(const double* v, int p, int k, const Reflectors& h,
                                        const int* perm, double* y, int r, int64_t ldy, int w,
                                        int nw) {
  if (p <= 128) apply_q_regs<16>(v, p, k, h, perm, y, r, ldy, w, nw);
  else if (p <= 192) apply_q_regs<24>(v, p, k, h, perm, y, r, ldy, w, nw);
  else apply_q_regs<32>(v, p, k, h, perm, y, r, ldy, w, nw);
}

// ---------------------------------------------------------------------------------------------
// One-sided Jacobi.  The columns' pairs of a round are disjoint (cyclic round-robin order).  A
// pair found converged (or below the floor) is checked again only once one of its columns has
// been rotated: each pair meets at the same round of every sweep, so when neither column has been
// rotated since the pair's check one sweep earlier, its inner product is the one that check
// computed and the pair is skipped.  Late sweeps, and the refinement of columns that are already
// orthogonal to each other, then touch only the pairs of recently rotated columns.
//
// The rotation (Rutishauser): zeta = (b - a) / 2g, t = sign(zeta) / (|zeta| + sqrt(1 + zeta^2)),
// c = 1 / sqrt(1 + t^2), s = c t, with a, b the squared norms and g the inner product.
// ---------------------------------------------------------------------------------------------
// columns (a, b) of pair k in a round over qq slots
__device__ __forceinline__ void round_pair(int round, int k, int qq, int* a, int* b) {
  int x = round, y = qq - 1;
  if (k > 0) {
    x = round + k;
    if (x >= qq - 1) x -= qq - 1;
    y = round - k;
    if (y < 0) y += qq - 1;
  }
  *a = x;
  *b = y;
}

// FP64 (the allocation-free entry point, and svd_mixed near the noise floor): the tests compare
// squares, the rotation's tangent t is found in FP32 from zeta where the angle is small (its
// accuracy only sets how far one rotation reduces the pair's inner product) and c is refined in
// FP64 by two Newton steps from the FP32 seed, so that c^2 + s^2 = 1 to FP64 rounding and the
// rotation is orthogonal.
__device__ __forceinline__ void rotation(double al, double be, double g, double& c, double& s,
                                         double& t) {
  // zeta in FP64 (the operands may lie far outside the FP32 range).  For a large angle
  // (|cos| > 1e-3: the first sweeps of a fresh start, nearly parallel columns) the tangent in
  // FP64, since a rotation that is off by u32 there leaves a leak that is large relative to the
  // smaller column; for the small angles of a refinement in FP32 where |zeta| < 2^100 (from 2^40 on,
  // where its square may overflow, by the asymptote 1 / (2 zeta)), else the asymptote in FP64.
  const double zeta = (be - al) / (2.0 * g);
  if (g * g > 1e-6 * (al * be)) {
    t = copysign(1.0 / (fabs(zeta) + sqrt(fma(zeta, zeta, 1.0))), zeta);
  } else if (fabs(zeta) < 0x1p100) {
    const float z = (float)zeta, az = fabsf(z), w = fmaf(z, z, 1.f);
    t = (double)(az > 0x1p40f ? __fdividef(0.5f, z)
                              : copysignf(__fdividef(1.f, az + w * rsqrtf(w)), z));
  } else {
    t = 0.5 / zeta;
  }
  const double u = fma(t, t, 1.0);
  double r = (double)rsqrtf((float)u);
  r = r * fma(-0.5 * u, r * r, 1.5);
  r = r * fma(-0.5 * u, r * r, 1.5);
  c = r;
  s = r * t;
}

struct JacobiShared {
  float2 nrm[CLR_MAX_CLUSTER];     // column norms: squared, and the root
  int last_rot[CLR_MAX_CLUSTER];   // the step of the column's last rotation, -1 if none
  int rotated, sweeps;
};

// One-sided Jacobi in FP64 on the q columns of g (p x q, ld p); v (q x q) accumulates the rotations:
// kOnto: onto its contents, row-major, else from I, column-major.  On return g = U S and the
// input equals g v^T (times the initial v^T where v is not reset).  Pairs whose
// inner product is below floor2, or below the FP64 epsilon times sqrt(p) relative to the norms,
// are left alone.  Returns the number of sweeps.  jac: its norms' place holds the column norms
// squared, recomputed exactly at every sweep start and refreshed (fused into the rotation pass) for
// the two columns of every rotated pair, so a pair costs one inner product unless it is rotated.
template <bool kOnto>
__device__ __noinline__ int jacobi_svd(double* g, int p, int q, double* v, int max_sweeps,
                                       int* sh_flag, double floor2, JacobiShared& jac) {
  double* nrm2 = reinterpret_cast<double*>(jac.nrm);
  int* last_rot = jac.last_rot;   // the step (sweep * (qq - 1) + round) of its last rotation, -1
  const int w = threadIdx.x / 32, l = threadIdx.x % 32;
  if (!kOnto)
    for (int e = threadIdx.x; e < q * q; e += kThreads) v[e] = (e % q == e / q) ? 1.0 : 0.0;
  const int qq = q + (q & 1);  // even number of slots; slot q is a dummy when q is odd
  const double tol = DBL_EPSILON * sqrt((double)p);
  for (int c = threadIdx.x; c < q; c += kThreads) last_rot[c] = -1;
  __syncthreads();
  int sweep = 0;
  for (; sweep < max_sweeps; ++sweep) {
    for (int c = w; c < q; c += kWarps) {
      const double* gc = g + (int64_t)c * p;
      double s2 = 0;
      for (int i = l; i < p; i += 32) s2 = fma(gc[i], gc[i], s2);
      s2 = warp_sum(s2);
      if (l == 0) nrm2[c] = s2;
    }
    if (threadIdx.x == 0) *sh_flag = 0;
    __syncthreads();
    for (int round = 0; round < qq - 1; ++round) {
      for (int k = w; k < qq / 2; k += kWarps) {
        int a, b;
        round_pair(round, k, qq, &a, &b);
        if (a >= q || b >= q) continue;
        const int step = sweep * (qq - 1) + round;
        if (sweep > 0 && last_rot[a] < step - (qq - 1) && last_rot[b] < step - (qq - 1))
          continue;
        const double al = nrm2[a], be = nrm2[b], ab = al * be;
        // both columns at the noise floor: |g_a . g_b| <= |g_a| |g_b| <= floor2, nothing to do
        if (ab == 0.0 || ab <= floor2 * floor2) continue;
        double* ga = g + (int64_t)a * p;
        double* gb = g + (int64_t)b * p;
        // kOnto: the two columns are read again for the rotation (in a kernel with all its registers
        // in use the callee's are spilled by every caller: compress_qr_kernel 210 -> 216 us where no
        // such sweep runs); else they stay in registers in between
        constexpr int kHold = kOnto ? 1 : kRowsPerLane;
        double xa[kHold], xb[kHold], d = 0;
        if constexpr (kOnto) {
#pragma unroll 2
          for (int i = l; i < p; i += 32) d = fma(ga[i], gb[i], d);
        } else {
#pragma unroll
          for (int j = 0; j < kHold; ++j) {
            if (32 * j >= p) break;
            const int i = l + 32 * j;
            xa[j] = i < p ? ga[i] : 0.0;
            xb[j] = i < p ? gb[i] : 0.0;
            d = fma(xa[j], xb[j], d);
          }
        }
        d = warp_sum(d);
        if (d * d <= tol * tol * ab || d * d <= floor2 * floor2) continue;
        double c, sn, t;
        rotation(al, be, d, c, sn, t);
        if constexpr (kOnto) {
#pragma unroll 2
          for (int i = l; i < p; i += 32) {
            const double x = ga[i], y = gb[i];
            ga[i] = c * x - sn * y;
            gb[i] = sn * x + c * y;
          }
        } else {
#pragma unroll
          for (int j = 0; j < kHold; ++j) {
            if (32 * j >= p) break;
            const int i = l + 32 * j;
            if (i < p) {
              ga[i] = c * xa[j] - sn * xb[j];
              gb[i] = sn * xa[j] + c * xb[j];
            }
          }
        }
        // new squared norms: a - t g and b + t g exactly; recomputed from the rotated columns
        // when the update cancels (a column losing more than 63/64 of its square)
        double na = al - t * d, nb = be + t * d;
        if (!(na > al * 0.015625) || !(nb > be * 0.015625)) {
          __syncwarp();
          double sa = 0, sb = 0;
          for (int i = l; i < p; i += 32) {
            sa = fma(ga[i], ga[i], sa);
            sb = fma(gb[i], gb[i], sb);
          }
          na = warp_sum(sa);
          nb = warp_sum(sb);
        }
        double* va = v + (kOnto ? a : a * q);
        double* vb = v + (kOnto ? b : b * q);
        const int v_r = kOnto ? q : 1;
        for (int i = l; i < q; i += 32) {
          const double x = va[i * v_r], y = vb[i * v_r];
          va[i * v_r] = c * x - sn * y;
          vb[i * v_r] = sn * x + c * y;
        }
        if (l == 0) {
          nrm2[a] = na;
          nrm2[b] = nb;
          last_rot[a] = step;
          last_rot[b] = step;
          *sh_flag = 1;
        }
      }
      __syncthreads();
    }
    const int rotated = *sh_flag;
    __syncthreads();
    if (!rotated) break;
  }
  return sweep;
}

// FP32 building blocks: the approximate units (a few ulp) serve throughout, as the FP32 stages
// only find rotations that FP64 products apply; two rows at a time by the packed FP32 pipe.
__device__ __forceinline__ float fast_rsqrt(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float fast_rcp(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float fast_sqrt(float x) {
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float x, float y) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ float sum2(f32x2 a) {
  float x, y;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a));
  return x + y;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

// One-sided Jacobi in FP32 with the working copies in shared memory (or, where they do not fit,
// in the per-CTA scratch), for the FP32 stages of svd_mixed.  What bounds it is the latency of a
// round (a column pair's inner product, its rotation, and a barrier), so a round is kept short:
//  - LP lanes per pair and 2 kVec rows a lane (as packed pairs), so that a round's pairs fill the
//    CTA once where they can: a warp alone issues an instruction every ~5 cycles, so a round
//    costs what one of its warps has to issue;
//  - the norms' roots are kept beside their squares, so that the tests need no square root (and
//    the squares so that the rotation angles see no more than the rounding of their updates:
//    squared approximate roots drift, and clustered columns then stop converging);
//  - only the warps that have pairs take part, with their own barrier (none for a single warp).
// g: p x q, ld ldg (even, the row p of an odd p zero); v: q x q, ld ldv (even), reset to I.
// tol, floor2: a pair is converged when its inner product is at most tol times the norms, or
// floor2.  Measured (core of 16 columns, both FP32 stages): 259k SM cycles with the copies in the
// global scratch, a warp per pair and 8 masked rows a lane.
// kShared: both copies in shared memory, g and v given as offsets into it (addressed as such: a
// generic pointer's loads are slower).
// Copies that do not fit there (more than ~156 columns) make a sweep bound by what one SM can move
// to and from L2 (8 KB a pair: 23k SM cycles a round of 119 pairs), so a team takes such a sweep
// together: the pairs dealt over its warps, the norms and marks in every CTA's copy, a cluster
// barrier a round.  The rotations are the same ones in the same order.
template <int LP, int kVec, bool kShared, class TM>
__device__ __noinline__ int jacobi32(const TM& tm, float* g_ptr, int q, int ldg, float* v_ptr,
                                     int ldv, int max_sweeps, float tol, float floor2,
                                     JacobiShared& sh) {
  extern __shared__ __align__(16) float svd_smem[];
  float* const g = kShared ? svd_smem + (int)(g_ptr - svd_smem) : g_ptr;
  float* const v = kShared ? svd_smem + (int)(v_ptr - svd_smem) : v_ptr;
  float2* nrm = sh.nrm;
  int* last_rot = sh.last_rot;
  constexpr unsigned kAll = 0xffffffffu;
  const int w = threadIdx.x / 32, li = threadIdx.x % LP;
  const int qq = q + (q & 1), half = qq / 2;   // slot q is a dummy when q is odd
  const int n_act = min(kWarps, (half * LP + 31) / 32);   // warps with pairs
  const int grp = tm.w * (32 / LP) + (threadIdx.x % 32) / LP;
  const int ngrp = n_act * (32 / LP) * tm.size;
  const int p2 = ldg / 2, q2 = ldv / 2;        // packed rows
  for (int e = tm.tid; e < ldv * q; e += tm.nt) v[e] = e % ldv == e / ldv ? 1.f : 0.f;
  for (int c = threadIdx.x; c < q; c += kThreads) last_rot[c] = -1;
  tm.sync();
  if (w < n_act) {
    auto act_sync = [&]() {
      if (tm.size > 1) tm.sync();   // (all warps have pairs then)
      else if (n_act == 1) __syncwarp();
      else group_sync(3, 32 * n_act);
    };
    auto sum_lp = [&](float x) {
#pragma unroll
      for (int o = LP / 2; o > 0; o >>= 1) x += __shfl_xor_sync(kAll, x, o);
      return x;
    };
    int sweep = 0;
    for (; sweep < max_sweeps; ++sweep) {
      for (int c0 = 0; c0 < q; c0 += ngrp) {
        const int c = c0 + grp;
        f32x2 s2 = 0;
        if (c < q) {
          const f32x2* gc = reinterpret_cast<const f32x2*>(g + c * ldg);
#pragma unroll
          for (int j = 0; j < kVec; ++j) {
            const f32x2 x = li + LP * j < p2 ? gc[li + LP * j] : 0;
            s2 = fma2(x, x, s2);
          }
        }
        const float s = sum_lp(sum2(s2));
        if (li == 0 && c < q) tm.put(&nrm[c], make_float2(s, fast_sqrt(s)));
      }
      if (threadIdx.x == 0) sh.rotated = 0;
      act_sync();
      for (int round = 0; round < qq - 1; ++round) {
        const int step = sweep * (qq - 1) + round;
        for (int k0 = 0; k0 < half; k0 += ngrp) {
          const int k = k0 + grp;
          int a, b;
          round_pair(round, k, qq, &a, &b);
          bool on = k < half && a < q && b < q;
          float2 na = make_float2(0.f, 0.f), nb = na;
          if (on) {
            // neither column rotated since this pair's check one sweep ago
            on = !(sweep > 0 && last_rot[a] < step - (qq - 1) && last_rot[b] < step - (qq - 1));
            na = nrm[a];
            nb = nrm[b];
          }
          const float ab = na.y * nb.y;
          on = on && ab > floor2;
          if (!__any_sync(kAll, on)) continue;
          f32x2* ga = reinterpret_cast<f32x2*>(g + a * ldg);
          f32x2* gb = reinterpret_cast<f32x2*>(g + b * ldg);
          f32x2 xa[kVec], xb[kVec], d2 = 0;
#pragma unroll
          for (int j = 0; j < kVec; ++j) {
            const int i = li + LP * j;
            const bool in = on && i < p2;
            xa[j] = in ? ga[i] : 0;
            xb[j] = in ? gb[i] : 0;
            d2 = fma2(xa[j], xb[j], d2);
          }
          const float d = sum_lp(sum2(d2)), ad = fabsf(d);
          // (inner products at the end of the FP32 range are left alone)
          on = on && ad > tol * ab && ad > floor2 && ad > 1e-37f;
          if (!__any_sync(kAll, on)) continue;
          float a2 = na.x, b2 = nb.x;
          bool again = false;
          if (on) {
            f32x2* va = reinterpret_cast<f32x2*>(v + a * ldv);
            f32x2* vb = reinterpret_cast<f32x2*>(v + b * ldv);
            f32x2 ya[kVec], yb[kVec];
#pragma unroll
            for (int j = 0; j < kVec; ++j) {
              const int i = li + LP * j;
              ya[j] = i < q2 ? va[i] : 0;
              yb[j] = i < q2 ? vb[i] : 0;
            }
            const float z = (b2 - a2) * (0.5f * fast_rcp(d)), az = fabsf(z);
            // (for |zeta| > 2^40, where its square may overflow, the asymptote 1 / (2 zeta))
            const float t =
                copysignf(fast_rcp(az + (az > 0x1p40f ? az : fast_sqrt(fmaf(az, az, 1.f)))), z);
            // one Newton step on the approximate root: c^2 + s^2 drifts less from 1 over many
            // rotations
            const float u = fmaf(t, t, 1.f);
            float c = fast_rsqrt(u);
            c = c * fmaf(-0.5f * u, c * c, 1.5f);
            const float sn = c * t;
            const f32x2 cc = pack2(c, c), ss = pack2(sn, sn), ns = pack2(-sn, -sn);
#pragma unroll
            for (int j = 0; j < kVec; ++j) {
              const int i = li + LP * j;
              const f32x2 x = fma2(ns, xb[j], mul2(cc, xa[j]));
              xb[j] = fma2(cc, xb[j], mul2(ss, xa[j]));
              xa[j] = x;
              if (i < p2) {
                ga[i] = xa[j];
                gb[i] = xb[j];
              }
              if (i < q2) {
                va[i] = fma2(ns, yb[j], mul2(cc, ya[j]));
                vb[i] = fma2(cc, yb[j], mul2(ss, ya[j]));
              }
            }
            // a - t g and b + t g, recomputed from the rotated columns when that cancels
            const float ra = fmaf(-t, d, a2), rb = fmaf(t, d, b2);
            again = !(ra > a2 * 0.015625f) || !(rb > b2 * 0.015625f);
            a2 = ra;
            b2 = rb;
          }
          if (__any_sync(kAll, again)) {
            f32x2 sa = 0, sb = 0;
#pragma unroll
            for (int j = 0; j < kVec; ++j) {
              sa = fma2(xa[j], xa[j], sa);
              sb = fma2(xb[j], xb[j], sb);
            }
            const float fa = sum_lp(sum2(sa)), fb = sum_lp(sum2(sb));
            if (again) {
              a2 = fa;
              b2 = fb;
            }
          }
          if (on && li == 0) {
            tm.put(&nrm[a], make_float2(a2, fast_sqrt(a2)));
            tm.put(&nrm[b], make_float2(b2, fast_sqrt(b2)));
            tm.put(&last_rot[a], step);
            tm.put(&last_rot[b], step);
            tm.put(&sh.rotated, 1);
          }
        }
        act_sync();
      }
      const int rotated = sh.rotated;
      act_sync();
      if (!rotated) break;
    }
    if (threadIdx.x == 0) sh.sweeps = sweep;
  }
  __syncthreads();
  return sh.sweeps;
}

// The FP32 working copies of svd_mixed (G: p x q, V: q x q): lanes per pair and packed rows per
// lane, leading dimensions and place.
struct Work32 {
  float *g, *v;
  int ldg, ldv, lp, vec;
};
// Dynamic shared memory of the recompression kernels: with their static part (34 KB) nearly all
// that a CTA can have, enough for a 256 x 133 pair of copies or a 156 x 156 one.
constexpr int kSvdSmemBytes = 192 * 1024;
// Of this launch: none where L1 is to cache the copies in the scratch (launch_compress_dense).
__device__ __forceinline__ int svd_smem_bytes() {
  int b;
  asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(b));
  return b;
}

// Lanes and packed rows per lane for columns of p rows: 16 lanes a pair put up to 32 pairs into one
// pass over the CTA's 16 warps, 32 lanes up to 16; one packed row a lane while the rows are few.
__device__ __forceinline__ void split32(Work32& k, int p, int q) {
  k.ldg = (p + 1) & ~1;
  k.ldv = (q + 1) & ~1;
  k.lp = p <= 32 || (q > 32 && p <= 128) ? 16 : 32;
  k.vec = (k.ldg / 2 + k.lp - 1) / k.lp;
}

__device__ __forceinline__ Work32 work32(int p, int q, double* sc) {
  extern __shared__ __align__(16) float svd_smem[];
  Work32 k;
  split32(k, p, q);
  const bool fits = (int64_t)(k.ldg + k.ldv) * q * (int)sizeof(float) <= svd_smem_bytes();
  k.g = fits ? svd_smem : reinterpret_cast<float*>(sc);
  k.v = k.g + k.ldg * q;
  return k;
}

// Whether the sweeps on a graded p x q matrix run on its FP32 triangular factor instead: rotations
// of A = Q R from the right are those of R, whose columns are q long, and Householder QR keeps
// each column's error relative to its own norm, as the grading needs.  The QR works in shared
// memory (p q floats).
__device__ __forceinline__ bool use_qr32(int p, int q) {
  return 8 * p >= 9 * q && (int64_t)((p + 1) & ~1) * q * (int)sizeof(float) <= svd_smem_bytes();
}

// k.g (p x q, ld k.ldg, in shared memory) <- its triangular factor (q x q, zero below the diagonal),
// k set up for it: V beside it in shared memory, or in the scratch.  One barrier a step: every
// warp forms the reflector itself and takes its columns.  Measured (256 x 100): 4.0 M SM cycles of
// sweeps on A, 2.4 M with this.
__device__ __noinline__ void qr32(Work32& k, int p, int q, double* sc) {
  extern __shared__ __align__(16) float svd_smem[];
  const int w = threadIdx.x / 32, l = threadIdx.x % 32;
  constexpr int kPer = CLR_MAX_CLUSTER / 32;
  float beta = 0.f;
  for (int j = 0; j < q; ++j) {
    const float* x = k.g + j * k.ldg;
    float xr[kPer], s = 0.f;
#pragma unroll
    for (int t = 0; t < kPer; ++t) {
      const int i = l + 32 * t;
      xr[t] = i > j && i < p ? x[i] : 0.f;
      s = fmaf(xr[t], xr[t], s);
    }
    const float x0 = x[j];
    s = warp_sum(s);
    // v = (v0, x below the diagonal), H = I - v v^T / (||x|| |v0|)
    const float nrm = sqrtf(fmaf(x0, x0, s)), v0 = x0 + copysignf(nrm, x0);
    const float tau = s > 0.f ? __fdividef(1.f, nrm) * __fdividef(1.f, fabsf(v0)) : 0.f;
    beta = s > 0.f ? -copysignf(nrm, x0) : x0;
    if (l == j % 32) {
#pragma unroll
      for (int t = 0; t < kPer; ++t)
        if (t == j / 32) xr[t] = v0;
    }
    for (int c = j + 1 + w; c < q; c += kWarps) {
      float* y = k.g + c * k.ldg;
      float yr[kPer], d = 0.f;
#pragma unroll
      for (int t = 0; t < kPer; ++t) {
        const int i = l + 32 * t;
        yr[t] = i >= j && i < p ? y[i] : 0.f;
        d = fmaf(xr[t], yr[t], d);
      }
      const float f = tau * warp_sum(d);
#pragma unroll
      for (int t = 0; t < kPer; ++t) {
        const int i = l + 32 * t;
        if (i >= j && i < p) y[i] = fmaf(-f, xr[t], yr[t]);
      }
    }
    __syncthreads();
    if (threadIdx.x == 0) k.g[j * k.ldg + j] = beta;   // (read no more by the steps to come)
  }
  __syncthreads();
  // columns moved together, to the even leading dimension of q rows: a column's new place ends
  // before the next one's old place starts
  const int ldp = k.ldg;
  Work32 n = k;
  split32(n, q, q);
  for (int c = 0; c < q; ++c) {
    const int i = threadIdx.x;
    const float v = i <= c ? k.g[c * ldp + i] : 0.f;
    __syncthreads();
    if (i < n.ldg) n.g[c * n.ldg + i] = v;
  }
  const bool fits = (int64_t)2 * n.ldg * q * (int)sizeof(float) <= svd_smem_bytes();
  n.v = fits ? n.g + n.ldg * q : reinterpret_cast<float*>(sc);
  k = n;
  __syncthreads();
}

// (tm: one CTA, or the team with both copies in global memory)
template <class TM>
__device__ __forceinline__ int run_jacobi32(const TM& tm, const Work32& k, int q, int max_sweeps,
                                            float tol, float floor2, JacobiShared& sh) {
  extern __shared__ __align__(16) float svd_smem[];
#define CLR_JACOBI32(LP, VEC, SH) \
  return jacobi32<LP, VEC, SH>(tm, k.g, q, k.ldg, k.v, k.ldv, max_sweeps, tol, floor2, sh)
  const float* end = svd_smem + svd_smem_bytes() / (int)sizeof(float);
  if (!(k.g >= svd_smem && k.g < end && k.v >= svd_smem && k.v < end)) {
    if (k.vec <= 3) CLR_JACOBI32(32, 3, false);   // (columns of more than 128 rows only)
    CLR_JACOBI32(32, 4, false);
  }
  if constexpr (std::is_same<TM, One>::value) {
    if (k.lp == 16) {
      switch (k.vec) {
        case 1: CLR_JACOBI32(16, 1, true);
        case 2: CLR_JACOBI32(16, 2, true);
        case 3: CLR_JACOBI32(16, 3, true);
        default: CLR_JACOBI32(16, 4, true);
      }
    }
    switch (k.vec) {
      case 1:
      case 2: CLR_JACOBI32(32, 2, true);
      case 3: CLR_JACOBI32(32, 3, true);
      default: CLR_JACOBI32(32, 4, true);
    }
  }
  return 0;   // (not reached: a team's copies are in global memory)
#undef CLR_JACOBI32
}

// Where small_series keeps its 2 q^2 floats: the place of the FP32 copies, which the
// orthonormalisation has read by then.
__device__ __forceinline__ float* series_f32(int q, double* sc) {
  extern __shared__ __align__(16) float svd_smem[];
  return (int64_t)2 * q * q * (int)sizeof(float) <= svd_smem_bytes() ? svd_smem
                                                                 : reinterpret_cast<float*>(sc);
}

struct SvdShared {
  double red[kWarps];
  double sigma[CLR_MAX_CLUSTER];    // by column
  double sorted[CLR_MAX_CLUSTER];   // descending
  double sigma_inv[CLR_MAX_CLUSTER];   // tail_lower_bound_sq: 1 / R_ii
  int perm[CLR_MAX_CLUSTER];        // sorted position -> column
  int flag;
  int v_tracked;  // svd_mixed: 1 when v holds the right singular vectors (else recover_right)
  int ls_recover; // svd_mixed: 1 when G's kept columns are orthogonal to the FP32 stages' tolerance
                  // only: the right factor needs the least-squares form (ls_solve)
  int rank;
  double kept_sq;
  // reflectors of the pivoted QR, of rrqr_block, or of the QR route's X factor; and of its W
  Reflectors refl, refl_w;
  int qr_perm[CLR_MAX_CLUSTER];   // pivoted QR: column order (columns are not moved)
  double qr_diag[CLR_MAX_CLUSTER];   // and R's diagonal (the columns keep their x_j there)
  int sweeps;      // of the second FP32 stage (every CTA's copy)
  JacobiShared jac;
  double cert;    // tail_lower_bound_sq's result
  // compress_by_pivoted_qr, by parity of the step: each column's trailing norm^2, downdated, and
  // its value when it was last summed exactly (the downdated norms are recomputed once they fall
  // below kDowndateFloor of it); and the FMAs of those recomputations
  double qr_nu[2][CLR_MAX_CLUSTER];
  double qr_nref[2][CLR_MAX_CLUSTER];
  unsigned long long qr_recomputed;
};
// Downdated column norms^2 are summed again exactly once they fall below this fraction of the
// last exact value: a downdate nu'^2 = nu^2 - r^2 carries an absolute error of a few u nu_ref^2,
// so the relative error stays below ~1e-9 between recomputations.
constexpr double kDowndateFloor = 1e-6;

// Column norms of g, their descending order, and the truncation rank at eps.  (Norms >= 0 are
// ordered by their bit patterns: integer comparisons instead of q^2 on the FP64 pipe, and the
// rank from one warp's suffix sums instead of a serial chain with a square root per step.)
__device__ void sort_and_truncate(const double* g, int p, int q, int64_t ldg, double eps,
                                  SvdShared& sh) {
  const int w = threadIdx.x / 32, l = threadIdx.x % 32;
  for (int c0 = kQuad * w; c0 < q; c0 += kQuad * kWarps) {
    double s[kQuad];
#pragma unroll
    for (int c = 0; c < kQuad; ++c) {
      s[c] = 0.0;
      if (c0 + c < q) {
        const double* gc = g + (int64_t)(c0 + c) * ldg;
        for (int i = l; i < p; i += 32) s[c] = fma(gc[i], gc[i], s[c]);
      }
    }
    const double d = warp_sum4(s);
    if (l % 8 == 0 && c0 + l / 8 < q) sh.sigma[c0 + l / 8] = d;
  }
  __syncthreads();
  for (int c = threadIdx.x; c < q; c += kThreads) sh.sigma[c] = sqrt(sh.sigma[c]);
  __syncthreads();
  for (int j = threadIdx.x; j < q; j += kThreads) {
    const unsigned long long sj = (unsigned long long)__double_as_longlong(sh.sigma[j]);
    int pos = 0;
    for (int i = 0; i < q; ++i) {
      const unsigned long long si = (unsigned long long)__double_as_longlong(sh.sigma[i]);
      pos += (si > sj) || (si == sj && i < j);
    }
    sh.perm[pos] = j;
    sh.sorted[pos] = sh.sigma[j];
  }
  __syncthreads();
  if (w == 0) {
    // smallest r with sum_{i >= r} s_i^2 <= eps^2: lane l sums chunk l from the small end
    const int ch = (q + 31) / 32;
    const int hi = q - l * ch, lo = hi - ch > 0 ? hi - ch : 0;   // indices [lo, hi)
    double own = 0.0;
    for (int i = hi - 1; i >= lo; --i) own = fma(sh.sorted[i], sh.sorted[i], own);
    double incl = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double v = __shfl_up_sync(0xffffffffu, incl, o);
      if (l >= o) incl += v;
    }
    double tail = __shfl_up_sync(0xffffffffu, incl, 1);
    if (l == 0) tail = 0.0;
    const double eps2 = eps * eps;
    int dropped = 0;
    double kept = 0.0;
    for (int i = hi - 1; i >= lo; --i) {
      const double s2 = sh.sorted[i] * sh.sorted[i];
      tail += s2;
      if (tail <= eps2) ++dropped; else kept += s2;
    }
    dropped = __reduce_add_sync(0xffffffffu, dropped);
    kept = warp_sum(kept);
    if (l == 0) {
      sh.rank = q - dropped;
      sh.kept_sq = kept;
    }
  }
  __syncthreads();
}

// Read-only view of the p x q working matrix: element (i, j) = src[i * s_r + j * s_c], or of its
// transpose when tr is set.
struct SrcView {
  const double* src;
  int64_t s_r, s_c;
  bool tr;
  __device__ __forceinline__ double at(int i, int j) const {
    return tr ? src[(int64_t)j * s_r + (int64_t)i * s_c] : src[(int64_t)i * s_r + (int64_t)j * s_c];
  }
};

// How the FP32 matrices at f (series_f32) are written: in its own shared memory by every CTA of the
// team for itself, in the team's one global scratch (more than ~156 columns) dealt over the team
// (3D lattice iterates, N = 2048: orthonormalisation and projection 1870 -> 1750 M SM cycles).
struct FloatShare {
  bool own;
  int t0, step;
  template <class TM>
  __device__ __forceinline__ FloatShare(const TM& tm, const float* f) {
    extern __shared__ __align__(16) float svd_smem[];
    own = tm.size == 1 || f == svd_smem;
    t0 = own ? (int)threadIdx.x : tm.tid;
    step = own ? kThreads : tm.nt;
  }
};

// The matrix function of a small symmetric E (q x q) that both uses below need, in place:
//   e <- c1 E + c2 E^2 + c3 E^3.
// The powers are taken in FP32 (f: 2 q^2 floats): their error is 6e-8 c2 ||E||_F^2, 1e-15 at the
// ||E||_F = 2e-4 (kSeriesFro) that its callers take for the last time; not at all where E^2 is below
// 1e-18 (kTinyFro).  Returns ||E||_F^2.
constexpr double kTinyFro = 1e-9;

template <class TM>
__device__ __noinline__ double small_series(const TM& tm, double* e, int q, double c1, float c2,
                                            float c3, float* f, SvdShared& sh) {
  const FloatShare fs(tm, f);
  float* t = f + q * q;
  float part = 0.f;
  for (int x = threadIdx.x; x < q * q; x += kThreads) {
    const float v = (float)e[x];
    if (fs.own) f[x] = v;
    part = fmaf(v, v, part);
  }
  const double fro2 = block_sum((double)part, sh.red);
  if (fro2 <= kTinyFro * kTinyFro) {
    tm.sync();   // (every CTA has read E)
    for (int x = tm.tid; x < q * q; x += tm.nt) e[x] *= c1;
    tm.sync();
    return fro2;
  }
  if (!fs.own) {
    for (int x = fs.t0; x < q * q; x += fs.step) f[x] = (float)e[x];
    tm.sync();
  }
  cta_gemm_auto(fs.t0, fs.step, q, q, q, f, 1, q, f, 1, q, t, q);
  tm.sync();
  // E^3 = F T an output at a time, added to the rest of the series
  for (int x = tm.tid; x < q * q; x += tm.nt) {
    const int i = x % q, j = x / q;
    float s = 0.f;
    for (int l = 0; l < q; ++l) s = fmaf(f[i + l * q], t[l + j * q], s);
    e[x] = fma(c1, e[x], (double)fmaf(c2, t[x], c3 * s));
  }
  tm.sync();
  return fro2;
}

// e (q x q) <- G^T G scaled by d on both sides (d null: unscaled) minus I, for G (n x q) given
// row-major (element (l, i) at a[l q + i]): the lower triangle in 2 x 2 blocks, mirrored.
template <class TM>
__device__ void gram_minus_identity(const TM& tm, const double* a, int n, int q,
                                    const double* d, double* e) {
  const int nb = (q + 1) / 2;
  for (int t = tm.tid; t < nb * (nb + 1) / 2; t += tm.nt) {
    int bi = (int)((sqrtf(8.f * (float)t + 1.f) - 1.f) * 0.5f);
    while (bi * (bi + 1) / 2 > t) --bi;
    while ((bi + 1) * (bi + 2) / 2 <= t) ++bi;
    const int i0 = 2 * bi, j0 = 2 * (t - bi * (bi + 1) / 2);
    const int i1 = i0 + 1 < q ? i0 + 1 : i0, j1 = j0 + 1 < q ? j0 + 1 : j0;
    double s00 = 0.0, s01 = 0.0, s10 = 0.0, s11 = 0.0;
    const double* r = a;
    for (int l = 0; l < n; ++l, r += q) {
      const double x0 = r[i0], x1 = r[i1], y0 = r[j0], y1 = r[j1];
      s00 = fma(x0, y0, s00);
      s01 = fma(x0, y1, s01);
      s10 = fma(x1, y0, s10);
      s11 = fma(x1, y1, s11);
    }
    auto put = [&](int i, int j, double s) {
      if (d) s *= d[i] * d[j];
      if (i == j) s -= 1.0;
      e[i + (int64_t)j * q] = s;
      e[j + (int64_t)i * q] = s;
    };
    put(i0, j0, s00);
    if (j0 + 1 < q) put(i0, j1, s01);
    if (i0 + 1 < q) put(i1, j0, s10);
    if (i0 + 1 < q && j0 + 1 < q) put(i1, j1, s11);
  }
  tm.sync();
}

// m (rows x q, row-major) <- m (I + w) (add_identity) or m w in FP64, w q x q row-major, row by
// row in place: one warp per row, the row held in registers (8 entries per lane) and broadcast
// by shuffles, 8 output columns per lane.  m's element (i, k) is at m[i m_r + k m_c].
template <class TM>
__device__ void right_multiply_fp64(const TM& tm, double* m, int rows, int64_t m_r, int64_t m_c,
                                    int q, const double* wt, bool add_identity) {
  constexpr int kPer = CLR_MAX_CLUSTER / 32;
  const int l = threadIdx.x % 32;
  for (int i = tm.w; i < rows; i += tm.nw) {
    double r[kPer], acc[kPer];
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
      const int k = l + 32 * j;
      r[j] = k < q ? m[i * m_r + k * m_c] : 0.0;
      acc[j] = add_identity ? r[j] : 0.0;
    }
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
      if (32 * j >= q) break;
      for (int kk = 0; kk < 32; ++kk) {
        const int k = 32 * j + kk;
        const double rk = __shfl_sync(0xffffffffu, r[j], kk);
        if (k >= q) break;
#pragma unroll
        for (int o = 0; o < kPer; ++o) {
          if (32 * o < q) {
            const int c = l + 32 * o;
            acc[o] = fma(rk, c < q ? wt[(int64_t)k * q + c] : 0.0, acc[o]);
          }
        }
      }
    }
    __syncwarp();
#pragma unroll
    for (int o = 0; o < kPer; ++o) {
      const int c = l + 32 * o;
      if (c < q) m[i * m_r + c * m_c] = acc[o];
    }
  }
  tm.sync();
}

// Above this ||E||_F the series in small_series, cut after E^3 and with FP32 powers, is not FP64
// accurate (at it the first term left out, 35/128 E^4, is 4e-16 and the powers' error 1e-15).
// ||V^T V - I||_F afterwards, against extended precision, and that of Gram-Schmidt: 16 columns 1.2e-15
// and 7e-16 at this limit (6e-16 at the usual ||E||_F of 1e-5), 100 columns 3.3e-15 and 3.4e-15, 240
// columns 8.0e-15 and 7.4e-15, after two passes 7.4e-15.
constexpr double kSeriesFro = 2e-4;
constexpr double kRefineFro = 0.05;   // up to this, by refinement (ls_solve)

// v (q x q, row-major) <- the orthogonal polar factor of the FP32 matrix v32 (ld ldv) in FP64:
// V (V^T V)^-1/2 by its series in E = V^T V - I, which rotations accumulated in FP32 keep at
// about 1e-5; repeated until ||E||_F has been below kSeriesFro.  Two products of q^3 FMAs (one of
// them symmetric) that fill the CTA, against Gram-Schmidt's q^3 FMAs in q dependent steps of
// reductions.  Measured (q = 16, with the product that follows): 218k -> 25k SM cycles; 3D lattice
// product at N = 4096, both stages over all blocks: 3.1 -> 2.1 G cycles.  From ~200 columns on a
// second pass is needed; its E is below kTinyFro (a few 1e-13), so that V E / 2 taken in FP32 is
// exact to 1e-19 (with FP64 products that pass made whole blocks of 256 columns slower than
// Gram-Schmidt).  v32 is the team's first CTA's; e: q^2 doubles, f: 2 q^2 floats, not overlapping
// v32's matrix until it has been read.
template <class TM>
__device__ __noinline__ void orthonormalise_fp64(const TM& tm, const float* v32, int ldv,
                                                 double* v, int q, double* e, float* f,
                                                 SvdShared& sh) {
  if (tm.rank == 0)
    for (int x = threadIdx.x; x < q * q; x += kThreads) {
      const int i = x / q, j = x - i * q;
      v[x] = (double)v32[i + j * ldv];
    }
  tm.sync();
  for (int pass = 0; pass < 4; ++pass) {
    gram_minus_identity(tm, v, q, q, nullptr, e);
    const double fro2 = small_series(tm, e, q, -0.5, 0.375f, -0.3125f, f, sh);
    if (fro2 <= kTinyFro * kTinyFro) {
      float* w = f + q * q;
      float* d = reinterpret_cast<float*>(e);   // V (-E / 2), in E's place
      const FloatShare fs(tm, f);
      for (int x = fs.t0; x < q * q; x += fs.step) {
        f[x] = (float)v[x];
        w[x] = (float)e[x];
      }
      tm.sync();
      cta_gemm_auto(tm.tid, tm.nt, q, q, q, w, 1, q, f, 1, q, d, q);
      tm.sync();
      for (int x = tm.tid; x < q * q; x += tm.nt) v[x] += (double)d[x];
      tm.sync();
      break;
    }
    right_multiply_fp64(tm, v, q, q, 1, q, e, true);
    if (!(fro2 > kSeriesFro * kSeriesFro)) break;
  }
}

// g (p x q, ld p) = A v in FP64, v row-major.  lower: A(i, l) = 0 for l > i (the transposed
// triangular factor), half of its first q rows.
template <class TM>
__device__ void project_fp64(const TM& tm, const SrcView& a, int p, int q, const double* v,
                             double* g, bool lower) {
  const int64_t a_i = a.tr ? a.s_c : a.s_r, a_k = a.tr ? a.s_r : a.s_c;
  if (lower)
    cta_gemm_auto<1>(tm.tid, tm.nt, p, q, q, a.src, a_i, a_k, v, q, 1, g, p);
  else
    cta_gemm_auto(tm.tid, tm.nt, p, q, q, a.src, a_i, a_k, v, q, 1, g, p);
  tm.sync();
}

// y (q x r, row-major) = A^T G_r in FP64, G_r the r kept columns of g (p x q, ld p) in the order
// perm; with G_r = U_r S_r this is V_r S_r^2.  G_r is first gathered row-major into `gather`
// (p r doubles, not overlapping g or y).  lower: A(i, j) = 0 for i < j.
template <class TM>
__device__ void recover_right(const TM& tm, const SrcView& a, int p, int q, const double* g,
                              const int* perm, int r, double* y, double* gather, bool lower) {
  for (int e = tm.tid; e < p * r; e += tm.nt) {
    const int k = e / r, c = e - k * r;
    gather[e] = g[k + (int64_t)perm[c] * p];
  }
  tm.sync();
  // y^T(c, j) = sum_k G_r(k, c) A(k, j)
  const int64_t a_j = a.tr ? a.s_r : a.s_c, a_k = a.tr ? a.s_c : a.s_r;
  if (lower)
    cta_gemm_auto<2>(tm.tid, tm.nt, r, q, p, gather, 1, r, a.src, a_k, a_j, y, r);
  else
    cta_gemm_auto(tm.tid, tm.nt, r, q, p, gather, 1, r, a.src, a_k, a_j, y, r);
  tm.sync();
}

// y (q x r, row-major) <- y (G_r^T G_r)^-1 in FP64, G_r the kept columns gathered row-major in
// `gr` (p x r), with norms d: the least-squares right factor when G_r is not orthogonal to FP64
// precision.  The Gram matrix of the normalised columns is I + E, E at the FP32 stages' tolerance
// (~1e-5), and its inverse N = I - E + E^2 - E^3; above kSeriesFro the result is refined,
// x += (y - x (I + E)) N, until the series' relative error to the power of the steps is below
// 1e-16; above kRefineFro a Cholesky factorisation in mw (a chain of one row's steps per thread:
// 10-40 M SM cycles at r ~ 110, which the relaxed test of a graded A made common before the
// refinement).  mw, e: r^2 doubles, f: 2 r^2 floats, z: q r doubles; gr is used again (q r).
// Returns false, with y unchanged, when the Cholesky factorisation meets a pivot that is not positive (kept columns at
// the rounding level of a block whose norm is near eps); the caller then uses the
// orthogonal-columns formula y S^-2.
template <class TM>
__device__ __noinline__ bool ls_solve(const TM& tm, double* y, int q, int r, double* gr, int p,
                                      const double* d, double* e, double* mw, double* z,
                                      float* f, SvdShared& sh) {
  double* rd = sh.sigma_inv;
  for (int c = threadIdx.x; c < r; c += kThreads) rd[c] = 1.0 / d[c];
  __syncthreads();
  gram_minus_identity(tm, gr, p, r, rd, e);
  for (int x = tm.tid; x < r * r; x += tm.nt) mw[x] = e[x];
  tm.sync();
  const double fro2 = small_series(tm, e, r, -1.0, 1.0f, -1.0f, f, sh);
  if (fro2 <= kRefineFro * kRefineFro) {
    // the series' relative error: its first omitted term and the FP32 powers'
    const double err = fro2 * fro2 + 1e-7 * fro2;
    int steps = 0;
    if (fro2 > kSeriesFro * kSeriesFro)
      for (double x = err; x > 1e-16; x *= err) ++steps;
    for (int x = tm.tid; x < q * r; x += tm.nt) {
      const double v = y[x] * rd[x % r];
      y[x] = v;
      gr[x] = v;
    }
    tm.sync();
    right_multiply_fp64(tm, y, q, r, 1, r, e, true);
    for (; steps > 0; --steps) {
      for (int x = tm.tid; x < q * r; x += tm.nt) z[x] = y[x];
      tm.sync();
      right_multiply_fp64(tm, z, q, r, 1, r, mw, true);
      for (int x = tm.tid; x < q * r; x += tm.nt) z[x] = gr[x] - z[x];
      tm.sync();
      right_multiply_fp64(tm, z, q, r, 1, r, e, true);
      for (int x = tm.tid; x < q * r; x += tm.nt) y[x] += z[x];
      tm.sync();
    }
    for (int x = tm.tid; x < q * r; x += tm.nt) y[x] *= rd[x % r];
    tm.sync();
    return true;
  }
  if (tm.rank == 0) {   // (by the first CTA alone)
    if (threadIdx.x == 0) sh.flag = 1;
    for (int x = threadIdx.x; x < r; x += kThreads) mw[x + (int64_t)x * r] += 1.0;
    __syncthreads();
    for (int j = 0; j < r; ++j) {  // lower Cholesky, column by column
      if (threadIdx.x == 0) {
        double a = mw[j + (int64_t)j * r];
        for (int k = 0; k < j; ++k) a -= mw[j + (int64_t)k * r] * mw[j + (int64_t)k * r];
        if (!(a > 0.0) || !isfinite(a)) {
          sh.flag = 0;
          a = 1.0;
        }
        mw[j + (int64_t)j * r] = sqrt(a);
      }
      __syncthreads();
      const double ljj = mw[j + (int64_t)j * r];
      for (int i = j + 1 + threadIdx.x; i < r; i += kThreads) {
        double a = mw[i + (int64_t)j * r];
        for (int k = 0; k < j; ++k) a -= mw[i + (int64_t)k * r] * mw[j + (int64_t)k * r];
        mw[i + (int64_t)j * r] = a / ljj;
      }
      __syncthreads();
    }
    // each row t: x = (y_t D^-1) (L L^T)^-1 D^-1 (no row when a pivot failed)
    for (int t = sh.flag ? threadIdx.x : q; t < q; t += kThreads) {
      double* yt = y + (int64_t)t * r;
      for (int i = 0; i < r; ++i) {  // forward: L u = (y_t D^-1)^T
        double a = yt[i] / d[i];
        for (int k = 0; k < i; ++k) a -= mw[i + (int64_t)k * r] * yt[k];
        yt[i] = a / mw[i + (int64_t)i * r];
      }
      for (int i = r - 1; i >= 0; --i) {  // back: L^T x = u
        double a = yt[i];
        for (int k = i + 1; k < r; ++k) a -= mw[k + (int64_t)i * r] * yt[k];
        yt[i] = a / mw[i + (int64_t)i * r];
      }
      for (int i = 0; i < r; ++i) yt[i] /= d[i];
    }
    if (threadIdx.x == 0) tm.put(&sh.flag, sh.flag);
  }
  tm.sync();
  return sh.flag != 0;
}

// x 2^k by integer arithmetic on the exponent (an FP64 multiplication holds the pipe for 64 cycles a
// warp): zero where the exponent leaves the range below; the caller keeps it in range above.
__device__ __forceinline__ int double_exponent(double x) {
  return __double2hiint(x) >> 20 & 0x7ff;
}
__device__ __forceinline__ double scaled(double x, int k) {
  const int e = double_exponent(x);
  return e > 0 && e + k > 0 ? __hiloint2double(__double2hiint(x) + (k << 20), __double2loint(x))
                            : 0.0;
}

// Mixed-precision one-sided Jacobi SVD of the p x q (p >= q) matrix A given by `a`.  FP64 runs
// at a small fraction of the FP32 rate on this part, so the rotations are found in FP32 and only
// applied, once per stage, in FP64:
//  1. FP32 sweeps on a copy of A until converged at FP32 accuracy, accumulating V1;
//  2. V = V1 orthonormalised in FP64 (its polar factor) and G = A V in FP64.  G's columns
//     are orthogonal to FP32 accuracy relative to ||A||; the part of the spectrum below
//     u32 ||A|| is still unresolved (it was rounding noise in the FP32 copy of A);
//  3. FP32 sweeps on a copy of G, whose columns are rounded relative to their own norms, so
//     the small columns are resolved against each other and against the large ones; V2
//     orthonormalised in FP64 and G <- G V2.
//  For the transposed triangular factor of the pivoted QR (`lower`) stage 1 resolves the small
//     columns too: that matrix is graded, row i of R at most |r_ii|, so its columns are rounded
//     relative to their own norms already and one-sided Jacobi is relatively accurate on them
//     (Drmac and Veselic).  Stage 1 then sweeps down to stage 3's floor, and stage 3 only runs
//     where a pair of G's columns is further than 16 times the stages' tolerance (cosine ~1e-4)
//     from orthogonal.  At that angle well separated columns' norms are within 1e-8 relative of the
//     singular values; of a cluster only the sum of squares is (two equal columns at a cosine c have
//     singular values c / 2 to either side), so a truncation inside a cluster may keep or drop a
//     column whose singular value is within 1e-4 of its norm; the error is the dropped columns' norm
//     either way, and what a kept column can carry of a dropped one is 1e-4 eps.  Measured on the
//     3D lattice product at N = 4096 (376 blocks): stages 1, 3 and 4 took 0.26 + 1.34 + 1.38 G
//     SM cycles, now 1.49 + 0.13 + 0.02.
//  The right factor: for kept columns G_r = U_r S_r it is V_r = A^T G_r S_r^-2 (recover_right),
//     and G_r (A^T G_r S_r^-2)^T = P A with P the orthogonal projector onto span(G_r), so
//     rounding in V_r is scaled back by S_r; near the noise floor V is accumulated instead.
// Pairs whose inner product is below the noise floor are not rotated: p u ||A||_F in FP32 on A,
// and max(p u ||A||_F, 1e-3 eps) on G and on a graded A (columns that small cannot move a
// truncation at eps).
// On return g = U S in FP64, and v the right factor when sh.v_tracked (else workspace).  sc:
// kSvdScratchPerCta doubles.
//
// Certified dense exit (dense_h >= 0): the block is stored dense when its eps-rank exceeds
// dense_h, i.e. when the singular-value tail sqrt(sum_{i >= dense_h} s_i^2) exceeds eps.  After
// stage 1 every sorted column norm c_i of G32 is within delta of s_i(A), with
//   delta = 2 u32 ||A||_F (4 q sqrt(p) + p sqrt(q) + 2 s32 q + 1)
// (backward error of s32 FP32 sweeps of rotations, the rounding of A to FP32, and the residual
// non-orthogonality of G32's columns: pairs within 4 u32 sqrt(p) of orthogonal or below the FP32
// noise floor).  So tail(A) >= tail(c) - sqrt(q - dense_h) delta, and when that exceeds eps the
// later stages could only confirm "dense": they are skipped and the function returns 1.
template <class TM>
__device__ __noinline__ int svd_mixed(const TM& tm, const SrcView& a, int p, int q, double* g, double* v,
                                      double* sc, int max_sweeps, double eps, int dense_h,
                                      double fro, bool lower, SvdShared& sh,
                                      unsigned long long* jstats,
                                      unsigned long long* stage_clk = nullptr) {
  extern __shared__ __align__(16) float svd_smem[];
  // while profiling the full-SVD path: SM cycles per stage (1..5 of kFullStageCounters)
  long long ck = stage_clk ? clock64() : 0;
  auto mark = [&](int stage) {
    if (stage_clk && tm.tid == 0) {
      const long long now = clock64();
      atomicAdd(&stage_clk[stage], (unsigned long long)(now - ck));
      ck = now;
    }
  };
  Work32 wk = work32(p, q, sc);
  const bool tri32 = lower && use_qr32(p, q);
  if (tri32) wk.g = svd_smem;
  // the team's sweeps where the copies (of A, or of its triangular factor) do not fit one CTA's
  // shared memory
  const int q_even = (q + 1) & ~1;
  const bool spread1 =
      tm.size > 1 && (tri32 ? 2 * q_even * q : (wk.ldg + wk.ldv) * q) * (int)sizeof(float) >
                         svd_smem_bytes();
  constexpr int64_t kSq = (int64_t)CLR_MAX_CLUSTER * CLR_MAX_CLUSTER;
  double* v2 = sc + kSq;       // after p q + q^2 floats
  double* e = sc + 4 * kSq;    // the orthonormalisations' E, and their FP32 powers
  float* f = series_f32(q, sc);
  const int w = threadIdx.x / 32, l = threadIdx.x % 32;
  // The FP64 noise floor, raised to 1e-3 eps: columns below it hold less than 1e-6 eps^2 each, so
  // their mutual (non-)orthogonality cannot move a truncation decision at eps except within a
  // hair of the threshold, while orthogonalising them costs most of the sweeps
  const double floor64 = fmax((double)p * DBL_EPSILON * fro, 1e-3 * eps);
  // The FP32 copies (and the floors beside them) are scaled by the power of two that brings
  // ||A||_F to 1..2: their squares and inner products then stay inside the FP32 range whatever
  // the block's norm is, and V does not depend on the scale.  (Unscaled, no pair of columns was
  // rotated in blocks of norm below ~1e-18 or above 1.8e19, and their ranks were those of the
  // columns as they came.)
  const int fro_exp = double_exponent(fro), shift = fro_exp < 0x7ff ? 0x3ff - fro_exp : 0;
  const float floor_g = (float)scaled(floor64, shift);
  const float tol32 = 4.f * FLT_EPSILON * sqrtf((float)p);
  const float floor32 = lower ? floor_g : (float)((double)p * FLT_EPSILON * scaled(fro, shift));
  // (else the FP32 stages are the first CTA's)
  int sw32 = 0;
  const One solo;
  if (spread1 && !tri32) {
    for (int e = tm.tid; e < wk.ldg * q; e += tm.nt) {
      const int i = e % wk.ldg;
      wk.g[e] = i < p ? (float)scaled(a.at(i, e / wk.ldg), shift) : 0.f;
    }
    tm.sync();
    sw32 = run_jacobi32(tm, wk, q, max_sweeps, tol32, floor32 * floor32, sh.jac);
  } else if (tm.rank == 0) {
    for (int e = threadIdx.x; e < wk.ldg * q; e += kThreads) {
      const int i = e % wk.ldg;
      wk.g[e] = i < p ? (float)scaled(a.at(i, e / wk.ldg), shift) : 0.f;
    }
    __syncthreads();
    if (tri32) qr32(wk, p, q, sc);
    if (!spread1) sw32 = run_jacobi32(solo, wk, q, max_sweeps, tol32, floor32 * floor32, sh.jac);
  }
  if (spread1 && tri32) {
    // the triangular factor from the first CTA's shared memory to where the team reads it
    float* g32 = reinterpret_cast<float*>(sc);
    split32(wk, q, q);
    if (tm.rank == 0)
      for (int e = threadIdx.x; e < wk.ldg * q; e += kThreads) g32[e] = wk.g[e];
    wk.g = g32;
    wk.v = g32 + wk.ldg * q;
    tm.sync();
    sw32 = run_jacobi32(tm, wk, q, max_sweeps, tol32, floor32 * floor32, sh.jac);
  }
  mark(1);
  if (dense_h >= 0 && dense_h < q) {   // (full SVDs: a team of one)
    for (int c = w; c < q; c += kWarps) {
      const float* gc = wk.g + c * wk.ldg;
      double s2 = 0.0;
      for (int i = l; i < p; i += 32) s2 = fma((double)gc[i], (double)gc[i], s2);
      s2 = warp_sum(s2);
      if (l == 0) sh.sigma[c] = scaled(sqrt(s2), -shift);
    }
    __syncthreads();
    double part = 0.0;
    for (int j = threadIdx.x; j < q; j += kThreads) {
      const double sj = sh.sigma[j];
      int pos = 0;
      for (int i = 0; i < q; ++i) {
        const double si = sh.sigma[i];
        pos += (si > sj) || (si == sj && i < j);
      }
      if (pos >= dense_h) part = fma(sj, sj, part);
    }
    const double tail = sqrt(block_sum(part, sh.red));
    const double delta = 2.0 * FLT_EPSILON * fro *
                         (4.0 * q * sqrt((double)p) + p * sqrt((double)q) + 2.0 * sw32 * q + 1.0);
    if (tail - sqrt((double)(q - dense_h)) * delta > eps) {
      if (jstats && tm.tid == 0) {
        atomicAdd(&jstats[0], 1ull);
        atomicAdd(&jstats[1], (unsigned long long)sw32);
        atomicAdd(&jstats[3], 1ull);
        atomicAdd(&jstats[5], 4ull * p * q * q * sw32);
      }
      return 1;
    }
  }
  orthonormalise_fp64(tm, wk.v, wk.ldv, v, q, e, f, sh);
  project_fp64(tm, a, p, q, v, g, lower);
  mark(2);
  wk = work32(p, q, sc);
  const float tol_g = lower ? 16.f * tol32 : tol32;
  int sw32b = 0;
  if (tm.size > 1 && (wk.ldg + wk.ldv) * q * (int)sizeof(float) > svd_smem_bytes()) {
    for (int e = tm.tid; e < wk.ldg * q; e += tm.nt) {
      const int i = e % wk.ldg;
      wk.g[e] = i < p ? (float)scaled(g[i + (int64_t)(e / wk.ldg) * p], shift) : 0.f;
    }
    tm.sync();
    sw32b = run_jacobi32(tm, wk, q, max_sweeps, tol_g, floor_g * floor_g, sh.jac);
  } else {
    if (tm.rank == 0) {
      for (int e = threadIdx.x; e < wk.ldg * q; e += kThreads) {
        const int i = e % wk.ldg;
        wk.g[e] = i < p ? (float)scaled(g[i + (int64_t)(e / wk.ldg) * p], shift) : 0.f;
      }
      __syncthreads();
      const int sw = run_jacobi32(solo, wk, q, max_sweeps, tol_g, floor_g * floor_g, sh.jac);
      if (threadIdx.x == 0) tm.put(&sh.sweeps, sw);
    }
    tm.sync();
    sw32b = sh.sweeps;
  }
  mark(3);
  // When eps is well above the noise floor the right factor of the kept columns is recovered
  // from A and G afterwards (recover_right).  Near the floor (eps < 1e3 p u ||A||_F) kept
  // columns may lie below it, unorthogonalised, where that recovery is not a projection: V is
  // accumulated instead.
  const bool track_v = floor64 > 1e-3 * eps;
  if (sw32b > 0) {
    orthonormalise_fp64(tm, wk.v, wk.ldv, v2, q, e, f, sh);
    right_multiply_fp64(tm, g, p, 1, p, q, v2, false);
    if (track_v) right_multiply_fp64(tm, v, q, q, 1, q, v2, false);
  }
  if (threadIdx.x == 0) sh.v_tracked = track_v ? 1 : 0;
  mark(4);
  // Near the noise floor a matrix that is not graded needs FP64 sweeps too: V2 is FP32, so the small
  // columns of G V2 keep ~u32^2 ||A||_F sqrt(p q) of the large ones, which can exceed eps (a sum of
  // two low-rank blocks of a common column space, eps = 1e-13: rank 48 where it is 24).
  // Elsewhere no FP64 sweep follows: the columns of G are orthogonal to the FP32 stages' tolerance
  // (cosines ~1e-5, for a graded A up to ~1e-4, relative to their own norms), and the truncation
  // error does not depend on their being orthogonal: with V accumulated A = G V^T and dropping
  // columns leaves ||G_tail V_tail^T||_F = ||G_tail||_F (V is orthogonal to FP64 rounding); without
  // it, the least-squares right factor (ls_solve) makes X W^T the orthogonal projection of A onto
  // span(G_r), with error ||(I - P) G_tail|| <= ||G_tail||_F <= eps for any G = A V_eff.
  // (FP64 sweeps to convergence wherever V is accumulated, the earlier choice, took 3.6 of 12.5 G
  // cycles of the lattice product's recompression at N = 4096, of graded factors.)
  int sw64 = 0;
  if (track_v && !lower)   // (one CTA: teams have graded factors)
    sw64 = jacobi_svd<true>(g, p, q, v, max_sweeps, &sh.flag, floor64 * floor64, sh.jac);
  mark(5);
  if (threadIdx.x == 0) sh.ls_recover = track_v ? 0 : 1;
  if (jstats && tm.tid == 0) {
    // algorithmic flops: Jacobi 4 p q^2 per sweep, orthonormalisation 3 q^3, products 2 p q^2
    const unsigned long long pq2 = (unsigned long long)p * q * q, q3 = (unsigned long long)q * q * q;
    unsigned long long f64 = 2 * q3 + 2 * pq2;
    if (sw32b > 0) f64 += 2 * q3 + 2 * pq2 + (track_v ? 2 * q3 : 0);
    f64 += 4 * pq2 * (unsigned long long)sw64;
    atomicAdd(&jstats[0], 1ull);
    atomicAdd(&jstats[1], (unsigned long long)(sw32 + sw32b));
    atomicAdd(&jstats[2], (unsigned long long)sw64);
    atomicAdd(&jstats[4], f64);
    atomicAdd(&jstats[5], 4 * pq2 * (unsigned long long)(sw32 + sw32b));
  }
  return 0;
}

// ---------------------------------------------------------------------------------------------
// ROUTE_QR tiles: X_cat (m x R) and W_cat (n x R) in the workspace slot.
//
// Small factors (the 1D chain's have 16 columns) make this a chain of latencies on a few SMs, so
// the CTAs come in clusters of two: while the tiles are at most half the CTAs a pair takes one
// tile, one CTA the QR of X_cat and the final Q_X product, the other W_cat's; the core and its SVD
// both compute (the same bits: nothing needs to be exchanged but the triangular factors, which
// are read after one cluster barrier).  With more tiles each CTA takes its own, eight warps a
// factor.  Measured, a 164 x 132 tile with R = 16 (SM cycles): QRs 262k -> 96k, application of Q
// 149k -> 70k; compress_qr_kernel of the 1D chain at N = 512 374 -> 260 us.
// ---------------------------------------------------------------------------------------------
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
    compress_qr_kernel(MatView C, const int* list, const int* count, const int* rsum, double* ws,
                       double* svd_scratch, double eps, int max_sweeps, int* sched,
                       unsigned long long* jstats) {
  extern __shared__ __align__(16) float svd_smem[];
  __shared__ SvdShared sh;
  __shared__ int sh_next;
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  constexpr int64_t kSq = (int64_t)CLR_MAX_CLUSTER * CLR_MAX_CLUSTER;
  double* sc = svd_scratch + (int64_t)blockIdx.x * kSvdScratchPerCta;
  const int n_items = *count;
  const bool pair = 2 * n_items <= (int)gridDim.x;
  const int rank = (int)cluster.block_rank();
  const One solo;   // the core is each CTA's own
  const bool lead = !pair || rank == 0;   // writes what a tile has once
  int it = pair ? (int)(blockIdx.x / 2) : next_item(sched, &sh_next);
  while (it < n_items) {
    const int t = list[it];
    const int I = t / C.nc, J = t % C.nc;
    const int m = C.row_off[I + 1] - C.row_off[I];
    const int n = C.col_off[J + 1] - C.col_off[J];
    const int R = rsum[t];
    const int64_t sC = slot_of(C, I, J, m);
    double* Xc = ws + 2 * sC;
    double* Wc = Xc + (int64_t)m * R;
    // R <= 128: the core and its SVD's factors in the third part of the CTA's scratch
    double* M = sc + 2 * kSq;
    double* V = M + (int64_t)R * R;
    double* G = V + (int64_t)R * R;
    // this warp's factor (X_cat or W_cat), its group of warps and the group's barrier
    const int wg = threadIdx.x / 32, half = pair ? rank : wg / (kWarps / 2);
    const int nw = pair ? kWarps : kWarps / 2;
    // (alone, W's first warps sit on other sub-partitions than X's)
    const int hw = pair ? wg : half ? (wg + 6) % (kWarps / 2) : wg;
    double* F = half ? Wc : Xc;
    const int f_rows = half ? n : m;
    Reflectors& refl = half ? sh.refl_w : sh.refl;
    factor_qr(F, f_rows, R, refl, reinterpret_cast<double*>(svd_smem) + half * 2 * CLR_MAX_CLUSTER,
              hw, nw, 1 + half);
    if (pair) cluster.sync(); else __syncthreads();
    // M = R_X R_W^T (both upper triangular R x R)
    for (int e = threadIdx.x; e < R * R; e += kThreads) {
      const int a = e % R, b = e / R;
      double s = 0.0;
      for (int c = (a > b ? a : b); c < R; ++c)
        s = fma(Xc[a + (int64_t)c * m], Wc[b + (int64_t)c * n], s);
      M[e] = s;
    }
    __syncthreads();
    unsigned long long* js = lead ? jstats : nullptr;
    {
      double part = 0.0;
      for (int e = threadIdx.x; e < R * R; e += kThreads) part = fma(M[e], M[e], part);
      const double mfro = sqrt(block_sum(part, sh.red));
      SrcView mv{M, 1, R, false};
      svd_mixed(solo, mv, R, R, G, V, sc, max_sweeps, eps, -1, mfro, false, sh, js);
    }
    sort_and_truncate(G, R, R, R, eps, sh);
    const int r = sh.rank;
    const bool tracked = sh.v_tracked;
    bool ls = !tracked && sh.ls_recover;
    if (!tracked) {
      // V_r S_r^2 = M^T G_r into V (M is still intact), or the least-squares V_r
      SrcView mv{M, 1, R, false};
      recover_right(solo, mv, R, R, G, sh.perm, r, V, sc, false);
      if (ls)
        ls = ls_solve(solo, V, R, r, sc, R, sh.sorted, sc + 4 * kSq, sc + kSq, sc + 3 * kSq,
                      series_f32(r, sc), sh);
    }
    double* Xo = C.pool + sC;
    double* Wo = Xo + (int64_t)m * r;
    if (!pair || rank == 0)
      for (int e = threadIdx.x; e < m * r; e += kThreads) {
        const int i = e % m, c = e / m;
        Xo[e] = i < R ? G[i + (int64_t)sh.perm[c] * R] : 0.0;
      }
    if (!pair || rank == 1)
      for (int e = threadIdx.x; e < n * r; e += kThreads) {
        const int j = e % n, c = e / n;
        Wo[e] = j >= R ? 0.0
                : tracked ? V[(int64_t)j * R + sh.perm[c]]
                : ls      ? V[(int64_t)j * r + c]
                          : V[(int64_t)j * r + c] / (sh.sorted[c] * sh.sorted[c]);
      }
    // the reflectors in shared memory where they fit (the FP32 copies there are dead): a lone
    // warp's step would wait for each reflector from L2
    const double* Fs = F;
    const int64_t room = (pair ? 1 : 2) * (int64_t)f_rows * R * (int64_t)sizeof(double);
    if (room <= kSvdSmemBytes) {
      double* st = reinterpret_cast<double*>(svd_smem) +
                   (pair || !half ? 0 : kSvdSmemBytes / (int64_t)sizeof(double) / 2);
      for (int e = hw * 32 + threadIdx.x % 32; e < f_rows * R; e += nw * 32) st[e] = F[e];
      Fs = st;
    }
    __syncthreads();
    apply_q(Fs, f_rows, R, refl, nullptr, half ? Wo : Xo, r, f_rows, hw, nw);
    if (js && threadIdx.x == 0) {
      // Householder QRs 2(m+n)R^2, core R_X R_W^T (2/3)R^3, recovery 2R^2 r (when not
      // accumulated), re-expansion 4(m+n)R r
      const unsigned long long mn = (unsigned long long)(m + n), RR = (unsigned long long)R * R;
      atomicAdd(&js[4], 2 * mn * RR + 2 * RR * R / 3 + (tracked ? 0 : 2 * RR * r) +
                            4 * mn * R * r);
    }
    if (lead && threadIdx.x == 0) {
      C.kind[t] = r > 0 ? CLR_KIND_LR : CLR_KIND_ZERO;
      C.rank[t] = r;
      C.norm[t] = sqrt(sh.kept_sq);
    }
    __syncthreads();
    if (pair) break;   // at most one tile a pair
    it = next_item(sched, &sh_next);
  }
}

// Launch shape of a recompression kernel: one CTA per SM (512 threads x 128 registers fill the
// register file) within the caller's grid (the scratch is sized for it), with all the shared
// memory a CTA can have for the FP32 working copies.
template <typename K>
int svd_launch_grid(K kernel, int grid_max, bool* attr_done) {
  int dev = 0;
  cudaGetDevice(&dev);
  int n_sm = 1;
  cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
  // set once per device (outside any stream capture the first time a product runs)
  if (dev >= 0 && dev < 64 && !attr_done[dev]) {
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSvdSmemBytes);
    // (as much L1 as a launch's shared memory leaves)
    cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 0);
    attr_done[dev] = true;
  }
  int grid = n_sm;
  if (grid > grid_max) grid = grid_max;
  return grid < 1 ? 1 : grid;
}

void launch_compress_qr(const MatView& C, const int* list, const int* count, const int* rsum,
                        double* ws, double* svd_scratch, double eps, int max_sweeps, int grid,
                        int* err, int* sched,
                        unsigned long long* jstats, cudaStream_t st) {
  (void)err;
  static bool attr_done[64] = {false};
  int g = svd_launch_grid(compress_qr_kernel, grid, attr_done);
  g = g < 2 ? 2 : g & ~1;   // pairs of CTAs
  compress_qr_kernel<<<g, kThreads, kSvdSmemBytes, st>>>(C, list, count, rsum, ws, svd_scratch, eps,
                                             max_sweeps, sched, jstats);
}

// ---------------------------------------------------------------------------------------------
// Rank-revealing QR of one block (the paper's construction of X and W, Section 4.1): Householder
// QR with greedy column pivoting (at step j the remaining column of largest norm over rows
// j..m-1, first maximum; the norms are recomputed exactly every step), stopped at the first j
// whose trailing block has ||R_22||_F <= eps.  g: m x n work copy (ld m); on return its upper
// trapezoid holds R, the reflector rows lie below the diagonal (sh.refl), the column order is in
// sh.perm.  Returns the rank r.
// ---------------------------------------------------------------------------------------------
__device__ int rrqr_block(const double* S, int64_t s_r, int64_t s_c, int m, int n, double eps,
                          double* g, SvdShared& sh) {
  const int w = threadIdx.x / 32, l = threadIdx.x % 32;
  for (int e = threadIdx.x; e < m * n; e += kThreads) {
    const int i = e % m, j = e / m;
    g[e] = S[i * s_r + j * s_c];
  }
  for (int c = threadIdx.x; c < n; c += kThreads) sh.perm[c] = c;
  __syncthreads();
  const int k = m < n ? m : n;
  int r = k;
  for (int j = 0; j < k; ++j) {
    for (int c = j + w; c < n; c += kWarps) {
      const double* gc = g + (int64_t)c * m;
      double s2 = 0.0;
      for (int i = j + l; i < m; i += 32) s2 = fma(gc[i], gc[i], s2);
      s2 = warp_sum(s2);
      if (l == 0) sh.sigma[c] = s2;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      double tot = 0.0, best = -1.0;
      int arg = j;
      for (int c = j; c < n; ++c) {
        tot += sh.sigma[c];
        if (sh.sigma[c] > best) { best = sh.sigma[c]; arg = c; }
      }
      sh.kept_sq = tot;
      sh.flag = arg;
    }
    __syncthreads();
    if (sqrt(sh.kept_sq) <= eps) {
      r = j;
      break;
    }
    const int piv = sh.flag;
    if (piv != j) {
      double* a = g + (int64_t)j * m;
      double* b = g + (int64_t)piv * m;
      for (int i = threadIdx.x; i < m; i += kThreads) {
        const double t = a[i];
        a[i] = b[i];
        b[i] = t;
      }
      if (threadIdx.x == 0) {
        const int t = sh.perm[j];
        sh.perm[j] = sh.perm[piv];
        sh.perm[piv] = t;
      }
    }
    __syncthreads();
    // Householder reflector of column j and its application (as householder_qr)
    double* cj = g + (int64_t)j * m;
    const int nr = m - j - 1, ncol = n - j - 1;
    auto col = [&](int c) { return g + (int64_t)(j + 1 + c) * m + j + 1; };
    const double* x = cj + j + 1;
    if (w == 0) {
      double v0, rn, rv;
      const double beta = make_reflector(x, nr, cj[j], &v0, &rn, &rv);
      __syncwarp();
      if (l == 0) {
        cj[j] = beta;
        sh.refl.v0[j] = v0;
        sh.refl.rn[j] = rn;
        sh.refl.rv[j] = rv;
      }
    }
    __syncthreads();
    const double v0 = sh.refl.v0[j], rn = sh.refl.rn[j], rv = sh.refl.rv[j];
    for (int c0 = kGroup * w; c0 < ncol; c0 += kGroup * kWarps) {
      const double d = group_dot(x, nr, c0, ncol, col);
      const int c = group_column(c0);
      const double yj = c < ncol ? col(c)[-1] : 0.0;
      const double f = fma(v0, yj, d) * rn * rv;
      group_update(x, f, nr, c0, ncol, col);
      if (c < ncol && l % 4 == 0) col(c)[-1] = fma(-f, v0, yj);
    }
    __syncthreads();
  }
  return r;
}

// ---------------------------------------------------------------------------------------------
// Truncated SVD of a block of low numerical rank through a column-pivoted QR (pre-reduction).
//
// A (p x q, the block or its transpose, p >= q) is reduced by Householder QR with column
// pivoting (at step j the remaining column of largest norm over rows j..p-1, first maximum on
// ties; the norms are downdated and summed again exactly once they have fallen by 1e6, and the
// stop is always decided on exact sums), stopped at the first step k whose trailing block has
// ||R_22||_F <= tau = eps/16:
//   A P = Q [R_11 R_12; 0 R_22].
// R_22 is dropped and the k x q factor R = [R_11 R_12] gets the mixed-precision SVD, truncated
// at the remaining budget sqrt(eps^2 - ||R_22||_F^2).  The two errors are orthogonal (rows
// 0..k-1 and k..p-1 of Q^T A P), so ||A - X W^T||_F <= eps, with X = Q_k X_R and W = P W_R.
// Cost: about 3 p q k FP64 FMAs for the QR and O(q k^2) for the SVD of R, instead of the
// O(p q^2)-per-sweep Jacobi on all q columns.  Ranks can exceed the minimal eps-rank where the
// singular-value tail crosses eps within the budget split (the rank reading allows one).
// Blocks of numerical rank above q/2 (stored dense): the QR stops after J = floor(q/2) + 1
// steps, and the block is certified dense when sigma_min(R_11) > eps for the leading J x J
// triangle: R_11 is a submatrix of Q^T A P, so sigma_J(A) >= sigma_min(R_11), and the eps-rank
// exceeds q/2 as soon as sigma_{q/2+1}(A) > eps.  sigma_min(R_11) is bounded below by
// 1 / ||R_11^-1||_F (a triangular inverse, J^3/6 FMAs).
// A block that meets neither goes on to its QR rank k at eps/16 (at most q).  Past 3q/5 steps
// it is first certified dense when a leading triangle R_K' bounds the tail
// sum_{i > q/2} sigma_i(A)^2 above eps^2: sigma_min alone certifies only blocks whose
// (q/2 + 1)-th singular value exceeds eps, while the tail of a block with many singular
// values just below eps also exceeds it (tail_lower_bound_sq).  Otherwise the SVD of its R
// decides, at any k: rank <= q/2 is stored low rank, else the block is stored dense (the
// untouched source).  One-sided Jacobi on R^T after a pivoted QR
// converges in fewer sweeps than on A itself (R is graded by the pivoting: the
// preconditioning of Drmac and Veselic, "New fast and accurate Jacobi SVD algorithm", SIAM
// J. Matrix Anal. Appl. 29, 2008), so even k near q costs less than the full SVD of A.
// Returns 1 when the block is done (low rank or zero, written to slot and the outputs), 2 when
// it is certified dense, 3 when the SVD of R found it dense (for 2 and 3 the source is
// untouched: the caller stores the kind and copies an external source into the slot), 0 only
// when a trailing norm is not finite; the caller then takes the full SVD on the source.
// g: p x q copy (ld p); wv: the tile's second workspace half (p q doubles); slot: the block's
// m n output slot (also the source of product tiles, overwritten only by a low-rank result);
// sc: the CTA's SVD scratch (kSvdScratchPerCta doubles: svd_mixed's working copies in the
// first two CLR_MAX_CLUSTER^2, the k x k right factor of R^T in the third, R in the fourth).
// ---------------------------------------------------------------------------------------------
// A lower bound on sum_{i > h} sigma_i(A)^2 from the leading K x K upper triangle R_K of the
// pivoted QR in g (ld p).  For every K' in (h, K], R_K' is the upper part of the first K'
// columns of Q^T A P, so sigma_i(A) >= sigma_i(R_K') (removing columns does not raise singular
// values), and the Cauchy-Schwarz inequality over the K' - h smallest singular values of R_K'
// gives  sum_{i > h} sigma_i(R_K')^2 >= (K' - h)^2 / sum_{i > h} sigma_i(R_K')^-2
// >= (K' - h)^2 / ||R_K'^-1||_F^2.  The columns of R_K^-1 come by back substitution of the unit
// vectors, one warp per column; column c depends only on the leading
// (c + 1) x (c + 1) triangle, so R_K'^-1 is the leading block of R_K^-1 and its squared
// Frobenius norm a prefix sum of column norms.  Returns the largest of the K - h bounds
// (h = K - 1: 1 / ||R_K^-1||_F^2 <= sigma_min(R_K)^2).
template <class TM>
__device__ __noinline__ double tail_lower_bound_sq(const TM& tm, const double* g, int p, int h,
                                                   int K, SvdShared& sh) {
  const int w = threadIdx.x / 32, l = threadIdx.x % 32;
  for (int i = threadIdx.x; i < K; i += kThreads) sh.sigma_inv[i] = 1.0 / sh.qr_diag[i];
  __syncthreads();
  // column c by columns of R from the last: x_i is final when its turn comes and is subtracted
  // from the rows above it, so no step needs a reduction (with an inner product and a division
  // per entry this test took half of a certified tile's time)
  for (int c = tm.w; c < K; c += tm.nw) {
    double x[kRowsPerLane];
#pragma unroll
    for (int t = 0; t < kRowsPerLane; ++t) x[t] = l + 32 * t == c ? 1.0 : 0.0;
#pragma unroll
    for (int b = kRowsPerLane - 1; b >= 0; --b) {
      if (32 * b > c) continue;
      for (int i = min(c, 32 * b + 31); i >= 32 * b; --i) {
        const double* ri = g + (int64_t)sh.qr_perm[i] * p;
        const double xi = __shfl_sync(0xffffffffu, x[b], i - 32 * b) * sh.sigma_inv[i];
#pragma unroll
        for (int t = 0; t < kRowsPerLane; ++t)
          if (t <= b) {
            const double u = l + 32 * t < i ? ri[l + 32 * t] : 0.0;
            x[t] = fma(-u, xi, x[t]);
          }
        if (l == i - 32 * b) x[b] = xi;
      }
    }
    double s2 = 0.0;
#pragma unroll
    for (int t = 0; t < kRowsPerLane; ++t)
      if (32 * t <= c) s2 = fma(x[t], x[t], s2);
    s2 = warp_sum(s2);
    if (l == 0) tm.put(&sh.sorted[c], s2);
  }
  tm.sync();
  if (w == 0) {
    // the prefix sums f_c, until a zero pivot makes them useless, and the best bound
    const int ch = (K + 31) / 32, lo = l * ch, hi = min(K, lo + ch);
    double own = 0.0;
    for (int c = lo; c < hi; ++c) own += sh.sorted[c];
    double incl = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double v = __shfl_up_sync(0xffffffffu, incl, o);
      if (l >= o) incl += v;
    }
    double f = __shfl_up_sync(0xffffffffu, incl, 1);
    if (l == 0) f = 0.0;
    double best = 0.0;
    for (int c = lo; c < hi; ++c) {
      f += sh.sorted[c];
      if (!(f > 0.0) || !isfinite(f)) break;   // a zero pivot: no larger K' bounds anything
      const int kk = c + 1;
      if (kk > h) best = fmax(best, (double)(kk - h) * (double)(kk - h) / f);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) best = fmax(best, __shfl_xor_sync(0xffffffffu, best, o));
    if (l == 0) sh.cert = best;
  }
  __syncthreads();
  return sh.cert;
}

// (not inlined: the kernel's register allocation stays with its own paths)
template <class TM>
__device__ __noinline__ int compress_by_pivoted_qr(const TM& tm, const SrcView& a, int p, int q,
                                                   bool tr, int m, int n, double eps, int max_sweeps,
                                                   double* g, double* wv, double* sc,
                                                   double* slot, int* kind_out, int* rank_out,
                                                   double* norm_out, SvdShared& sh,
                                                   unsigned long long* jstats) {
  const int w = threadIdx.x / 32, l = threadIdx.x % 32;
  const long long c_entry = clock64();
  // Once the QR has met the threshold, R (k x q) goes to the fourth part of sc, the left SVD
  // factor of R^T (q x k <= p q doubles) to wv and the right one (k x k) to the third part of
  // sc; the source stays untouched until a low-rank result overwrites it.  Ranks up to q/2
  // are stored low rank.
  const int kmax = q / 2;
  // steps after which a block still above the threshold is tested for the sigma_min
  // certificate, and the QR rank above which the tail certificate is tried before the SVD
  // (the steps past jtail cost a few percent of the first ones: their trailing blocks are
  // small)
  const int jcert = q / 2 + 1 <= q ? q / 2 + 1 : q;
  const int jtail = (3 * q) / 5 > jcert ? (3 * q) / 5 : jcert;
  const double tau2 = (eps / 16.0) * (eps / 16.0);
  // copy with the column norms
  for (int c = tm.w; c < q; c += tm.nw) {
    double* gc = g + (int64_t)c * p;
    double s2 = 0.0;
    for (int i = l; i < p; i += 32) {
      const double x = a.at(i, c);
      gc[i] = x;
      s2 = fma(x, x, s2);
    }
    s2 = warp_sum(s2);
    if (l == 0) {
      tm.put(&sh.qr_nu[0][c], s2);
      tm.put(&sh.qr_nref[0][c], s2);
    }
  }
  for (int c = threadIdx.x; c < q; c += kThreads) sh.qr_perm[c] = c;
  if (threadIdx.x == 0) sh.qr_recomputed = 0;
  tm.sync();
  unsigned long long fma_count = 0;
  bool exact = true;   // the trailing norms were all summed exactly at this step
  int k = -1;
  for (int j = 0; j <= q; ++j) {
    // pivot (warp 0): the largest trailing norm, first maximum (norms >= 0: compared as
    // integers); their sum only when the largest could let it meet the threshold.  Columns are
    // exchanged in the order qr_perm, not moved.
    // (two buffers of the norms, by step: a CTA of the team that is ahead writes the next step's
    // into every copy while another still chooses its pivot)
    double* nu = sh.qr_nu[j & 1];
    double* nref = sh.qr_nref[j & 1];
    if (w == 0) {
      unsigned long long best = 0;
      int arg = j;
      for (int c = j + l; c < q; c += 32) {
        const unsigned long long v = (unsigned long long)__double_as_longlong(nu[c]);
        if (v > best) { best = v; arg = c; }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long ob = __shfl_xor_sync(0xffffffffu, best, o);
        const int oa = __shfl_xor_sync(0xffffffffu, arg, o);
        if (ob > best || (ob == best && oa < arg)) { best = ob; arg = oa; }
      }
      double tot = __longlong_as_double((long long)best);
      if (tot <= tau2) {
        tot = 0.0;
        for (int c = j + l; c < q; c += 32) tot += nu[c];
        tot = warp_sum(tot);
      }
      if (l == 0) {
        sh.kept_sq = tot;
        if (!(tot <= tau2) && arg != j) {
          const double t = nu[j];
          nu[j] = nu[arg];
          nu[arg] = t;
          const double tr = nref[j];
          nref[j] = nref[arg];
          nref[arg] = tr;
          const int ti = sh.qr_perm[j];
          sh.qr_perm[j] = sh.qr_perm[arg];
          sh.qr_perm[arg] = ti;
        }
      }
    }
    __syncthreads();
    if (sh.kept_sq <= tau2 && !exact) {
      tm.sync();   // (every CTA has chosen)
      // the downdated norms meet the threshold: sum the trailing norms exactly and decide (and
      // pivot) on those
      for (int c0 = j + kQuad * tm.w; c0 < q; c0 += kQuad * tm.nw) {
        double s2[kQuad];
#pragma unroll
        for (int c = 0; c < kQuad; ++c) {
          s2[c] = 0.0;
          if (c0 + c < q) {
            const double* y = g + (int64_t)sh.qr_perm[c0 + c] * p;
            for (int i = j + l; i < p; i += 32) s2[c] = fma(y[i], y[i], s2[c]);
          }
        }
        const double d = warp_sum4(s2);
        if (l % 8 == 0 && c0 + l / 8 < q) {
          tm.put(&nu[c0 + l / 8], d);
          tm.put(&nref[c0 + l / 8], d);
        }
      }
      fma_count += (unsigned long long)(p - j) * (unsigned long long)(q - j);
      exact = true;
      tm.sync();
      --j;   // the same step again
      continue;
    }
    if (sh.kept_sq <= tau2) {
      k = j;
      break;
    }
    if (j == jcert) {
      // still above the threshold after floor(q/2) + 1 steps: dense if sigma_min(R_11) > eps
      const double b2 = tail_lower_bound_sq(tm, g, p, jcert - 1, jcert, sh);
      if (jstats && tm.tid == 0)
        atomicAdd(&jstats[4], 2ull * fma_count + (unsigned long long)jcert * jcert * jcert / 3);
      fma_count = 0;
      if (b2 > eps * eps) return 2;
    }
    // (the trailing block after q steps is empty: only a non-finite norm gets here)
    if (j == q) break;
    // Householder reflector of the pivot column and its application to the remaining columns
    // (as householder_qr).  The reflector keeps the norm of each column's rows j..p-1 and moves
    // its row j into R, so the trailing norm^2 over rows j+1..p-1 is the old one minus the new
    // row-j entry squared (downdate), summed again exactly when it has fallen below
    // kDowndateFloor of its last exact value (or is not positive).
    double* cj = g + (int64_t)sh.qr_perm[j] * p;
    const int n = p - j - 1, ncol = q - j - 1;
    auto col = [&](int c) { return g + (int64_t)sh.qr_perm[j + 1 + c] * p + j + 1; };
    const double* x = cj + j + 1;
    // Groups of eight columns, or in a team of four where that still leaves no warp more than one
    // (shorter, though more of the pipe in all); each CTA's first warp forms the reflector (all alike), so the first groups go to the others.
    const int gc = tm.size > 1 && ncol <= 4 * (kWarps - 1) * tm.size ? 4 : kGroup;
    const int first = (kWarps - 1) * tm.size;   // groups taken before the scalars are known
    auto end = [&](int c0) { return c0 + gc < ncol ? c0 + gc : ncol; };
    double d = 0.0;
    if (w == 0) {
      double v0, rn, rv;
      const double beta = make_reflector(x, n, cj[j], &v0, &rn, &rv);
      __syncwarp();
      if (l == 0) {
        sh.qr_diag[j] = beta;
        sh.refl.v0[j] = v0;
        sh.refl.rn[j] = rn;
        sh.refl.rv[j] = rv;
      }
    } else if (gc * (tm.w - tm.size) < ncol) {
      const int c0 = gc * (tm.w - tm.size);
      d = group_dot(x, n, c0, end(c0), col);
    }
    __syncthreads();
    const double v0 = sh.refl.v0[j], rn = sh.refl.rn[j], rv = sh.refl.rv[j];
    for (int gi = w > 0 ? tm.w - tm.size : first + tm.w; gc * gi < ncol;
         gi = gi < first ? first + tm.w : gi + tm.nw) {
      const int c0 = gc * gi, c1 = end(c0);
      const int cg = group_column(c0), c = cg < c1 ? cg : ncol;   // (ncol: no column)
      if (gi >= first) d = group_dot(x, n, c0, c1, col);
      const double yj = c < ncol ? col(c)[-1] : 0.0;
      const double f = fma(v0, yj, d) * rn * rv;
      group_update(x, f, n, c0, c1, col);
      const double yn = fma(-f, v0, yj);
      double nu2 = 0.0, ref = 0.0;
      bool again = false;
      if (c < ncol) {
        ref = nref[j + 1 + c];
        nu2 = fma(-yn, yn, nu[j + 1 + c]);
        again = !(nu2 > kDowndateFloor * ref);
      }
      if (__any_sync(0xffffffffu, again)) {
        const double s2 = group_squares(n, c0, c1, col);
        if (again) {
          ref = nu2 = s2;
          if (l % 4 == 0) atomicAdd(&sh.qr_recomputed, (unsigned long long)n);
        }
      }
      __syncwarp();
      if (c < ncol && l % 4 == 0) {
        col(c)[-1] = yn;
        tm.put(&sh.qr_nu[(j + 1) & 1][j + 1 + c], nu2);
        tm.put(&sh.qr_nref[(j + 1) & 1][j + 1 + c], ref);
      }
    }
    fma_count += 2ull * (unsigned long long)(p - j) * (unsigned long long)(q - j - 1) + (p - j);
    exact = false;
    tm.sync();
  }
  if (jstats && threadIdx.x == 0)   // (the QR's flops after the certificate test)
    atomicAdd(&jstats[4], 2ull * ((tm.rank == 0 ? fma_count : 0) + sh.qr_recomputed));
  if (k < 0) return 0;
  if (k > jtail) {
    // dense when sum_{i > q/2} sigma_i^2 > eps^2 is certified by some leading triangle of the
    // k completed steps, else the SVD of R decides
    const double b2 = tail_lower_bound_sq(tm, g, p, kmax, k, sh);
    if (jstats && tm.tid == 0)
      atomicAdd(&jstats[4], (unsigned long long)k * k * k / 3);
    if (b2 > eps * eps) return 2;
  }
  const double trail2 = sh.kept_sq;
  __syncthreads();
  if (k == 0) {
    if (tm.tid == 0) { *kind_out = CLR_KIND_ZERO; *rank_out = 0; *norm_out = 0.0; }
    __syncthreads();
    return 1;
  }
  // M = R^T (q x k, ld q, zero above the diagonal: consecutive threads of its products read
  // consecutive rows) and its SVD
  constexpr int64_t kSq = (int64_t)CLR_MAX_CLUSTER * CLR_MAX_CLUSTER;
  double* rb = sc + 3 * kSq;   // q x k
  double* gs = wv;             // q x k
  double* vs = sc + 2 * kSq;   // k x k
  double part = 0.0;
  for (int e = tm.tid; e < k * q; e += tm.nt) {
    const int i = e % k, c = e / k;
    rb[c + (int64_t)i * q] = i < c    ? g[i + (int64_t)sh.qr_perm[c] * p]
                             : i == c ? sh.qr_diag[i]
                                      : 0.0;
  }
  tm.sync();
  for (int e = threadIdx.x; e < k * q; e += kThreads) part = fma(rb[e], rb[e], part);
  const double rfro = sqrt(block_sum(part, sh.red));
  const double budget = sqrt(fmax(eps * eps - trail2, 0.0));
  const SrcView mv{rb, 1, q, false};
  unsigned long long* stage_clk = jstats ? jstats + kPreStageCounters : nullptr;
  if (stage_clk && tm.tid == 0)
    atomicAdd(&stage_clk[0], (unsigned long long)(clock64() - c_entry));
  svd_mixed(tm, mv, q, k, gs, vs, sc, max_sweeps, budget, -1, rfro, true, sh, jstats, stage_clk);
  const long long c_after = clock64();
  sort_and_truncate(gs, q, k, q, budget, sh);
  const int r = sh.rank;
  if (r == 0) {
    if (tm.tid == 0) { *kind_out = CLR_KIND_ZERO; *rank_out = 0; *norm_out = 0.0; }
    __syncthreads();
    return 1;
  }
  if (r > kmax) {
    // stored dense: the source is untouched (R lives in the scratch), so the block is kept
    // exactly (the caller copies an external source into the slot)
    if (jstats && tm.tid == 0) {
      atomicAdd(&stage_clk[6], (unsigned long long)(clock64() - c_after));
      atomicAdd(&stage_clk[7], 1ull);
    }
    __syncthreads();
    return 3;
  }
  const bool tracked = sh.v_tracked;
  bool ls = !tracked && sh.ls_recover;
  if (!tracked) recover_right(tm, mv, q, k, gs, sh.perm, r, vs, sc, true);   // Y = R G_r (k x r)
  // (R is no longer needed: its place is work space)
  if (ls)
    ls = ls_solve(tm, vs, k, r, sc, q, sh.sorted, sc + 4 * kSq, sc + kSq, rb, series_f32(r, sc), sh);
  // R = V_M S U_M^T:  X_R = (V_M S)_r (k x r), W_R = (U_M)_r (q x r); A ~ (Q_k X_R) (P W_R)^T
  // (the source in the slot is no longer read: the factors overwrite it)
  tm.sync();
  double* xa = tr ? slot + (int64_t)m * r : slot;   // Q_k X_R: p x r, ld p
  double* wa = tr ? slot : slot + (int64_t)m * r;   // P W_R: q x r, ld q
  for (int e = tm.tid; e < p * r; e += tm.nt) {
    const int i = e % p, c = e / p;
    double v = 0.0;
    if (i < k)
      v = tracked ? vs[(int64_t)i * k + sh.perm[c]] * sh.sorted[c]
          : ls    ? vs[(int64_t)i * r + c]
                  : vs[(int64_t)i * r + c] / sh.sorted[c];
    xa[e] = v;
  }
  for (int e = tm.tid; e < q * r; e += tm.nt) {
    const int j = e % q, c = e / q;
    const double v = gs[j + (int64_t)sh.perm[c] * q];
    wa[sh.qr_perm[j] + (int64_t)c * q] = ls ? v : v / sh.sorted[c];
  }
  __syncthreads();
  // the reflectors in shared memory where they fit
  if ((int64_t)p * k * (int64_t)sizeof(double) <= svd_smem_bytes()) {
    extern __shared__ __align__(16) float svd_smem[];
    double* st = reinterpret_cast<double*>(svd_smem);
    for (int c = w; c < k; c += kWarps)
      for (int i = c + 1 + l; i < p; i += 32) st[i + c * p] = g[i + (int64_t)sh.qr_perm[c] * p];
    tm.sync();   // (and the factors' entries)
    apply_q(st, p, k, sh.refl, nullptr, xa, r, p, tm.w, tm.nw);
  } else {
    tm.sync();
    apply_q(g, p, k, sh.refl, sh.qr_perm, xa, r, p, tm.w, tm.nw);
  }
  if (tm.tid == 0) {
    *kind_out = CLR_KIND_LR;
    *rank_out = r;
    *norm_out = sqrt(sh.kept_sq);
    if (jstats) {
      atomicAdd(&jstats[4], 4ull * (unsigned long long)p * k * r);
      atomicAdd(&jstats[6], 1ull);
      atomicAdd(&stage_clk[6], (unsigned long long)(clock64() - c_after));
      atomicAdd(&stage_clk[7], 1ull);
    }
  }
  __syncthreads();
  return 1;
}

// ---------------------------------------------------------------------------------------------
// Dense truncated SVD of whole blocks (ROUTE_DACC tiles, recompressed dense tiles, building a
// CLR matrix from a dense one).
//
// A tile is FP64-pipe-bound for 5 to 20 ms of one SM at 256 x 256 (and bound by its FP32 sweeps for
// up to 45 where its QR rank is ~240), so with few tiles the launch takes what its largest tile takes
// while most SMs idle.  With few tiles the CTAs come in clusters of four, and a cluster can work on
// one tile as a team (the columns of the QR, the rows and blocks of the products, the pairs of
// FP32 sweeps that leave shared memory).  A team takes a 256 x 240 tile of QR rank ~235 in 45 M SM
// cycles, one CTA in 100 (of QR rank ~60 in 5.1 and 9.3), so that about half of its SMs' time is
// lost.  Teams take all tiles while these are at most half
// the CTAs (64 tiles, gradient of the 1D chain at N = 1024: 3.6 ms against 5.1), else the leading
// n_team ones of the list (team_tiles, by their costs), after which each CTA takes its own: with
// 144 tiles on 152 SMs all by teams were no faster than none (Coulomb-like lattice at N = 2048,
// 6.2 ms against 5.8), the largest few are (3D lattice iterates at N = 2048, 29 launches: 247 ->
// 192 ms, the longest 43 -> 18).  Either way a tile's arithmetic is the same to the bit.
// ---------------------------------------------------------------------------------------------
template <bool kTeams>
__device__ __forceinline__ void compress_dense_body(
    MatView C, const int* list, const int* count, const int* order, const double* src,
    int64_t lds, double* ws, double* svd_scratch, double eps, double drop_norm,
    int dense_only, int rrqr, int prereduce, int max_sweeps, int* err, int* sched,
    const int* n_team, unsigned long long* jstats) {
  __shared__ SvdShared sh;
  __shared__ int sh_next[2];
  const int n_items = list ? *count : C.nr * C.nc;
  const int cta = kTeams ? (int)cooperative_groups::this_cluster().block_rank() : 0;
  // the leading tiles of the list that teams take
  const int lead = !kTeams ? 0 : 2 * n_items <= (int)gridDim.x ? n_items : n_team ? *n_team : 0;
  bool team = lead > 0;
  auto make = [&]() {
    if constexpr (kTeams) return Team(team ? cta : 0, team ? kTeamCtas : 1);
    else return One();
  };
  auto tm = make();
  double* sc = svd_scratch + (int64_t)(blockIdx.x - tm.rank) * kSvdScratchPerCta;
  // a CTA's shared memory may be written by another (put) only once it is known to have started
  // (lead is the same in all of a cluster's CTAs)
  if (team) tm.sync();
  int next_slot = 0;
  auto next = [&]() {
    if constexpr (kTeams)
      if (team) {
        // (two slots: one is read while the other is written)
        if (tm.tid == 0) tm.put(&sh_next[next_slot], atomicAdd(sched, 1));
        tm.sync();
        next_slot ^= 1;
        const int it = sh_next[next_slot ^ 1];
        if (it < lead) return it;
        // from here on each CTA takes its own tiles, the first one this one
        __syncthreads();
        team = false;
        tm = make();
        sc = svd_scratch + (int64_t)blockIdx.x * kSvdScratchPerCta;
        if (cta == 0) return it;
      }
    return next_item(sched, &sh_next[0]);
  };
  // each tile's SM kilocycles go to C.cost (the next plan's scheduling cost), written when the
  // CTA takes its next tile (every path of the loop body ends there) and after the last one
  // (a team's time twice over: about what one CTA takes)
  int prev_t = -1, prev_x = 1;
  long long prev_c = 0;
  auto record_cost = [&](long long now) {
    if (C.cost && prev_t >= 0 && threadIdx.x == 0) {
      const long long kc = (now - prev_c) * prev_x >> 10;
      C.cost[prev_t] = (unsigned int)(kc < 1 ? 1 : kc > 0xFFFFFFFFll ? 0xFFFFFFFFll : kc);
    }
  };
  for (int it = next(); it < n_items; it = next()) {
    const int t = list ? list[it] : (order ? order[it] : it);
    const long long now = clock64();
    record_cost(now);
    prev_t = tm.rank == 0 ? t : -1;
    prev_c = now;
    prev_x = tm.size > 1 ? 2 : 1;
    if (jstats && tm.size > 1 && tm.tid == 0) atomicAdd(&jstats[kTeamTileCounter], 1ull);
    const int I = t / C.nc, J = t % C.nc;
    const int m = C.row_off[I + 1] - C.row_off[I];
    const int n = C.col_off[J + 1] - C.col_off[J];
    const int64_t sC = slot_of(C, I, J, m);
    double* slot = C.pool + sC;
    const double* S = src ? src + (int64_t)C.row_off[I] * lds + C.col_off[J] : slot;
    const int64_t s_r = src ? lds : 1;   // element (i,j) at S[i * s_r + j * s_c]
    const int64_t s_c = src ? 1 : m;
    const bool tr = m < n;
    const int p = tr ? n : m, q = tr ? m : n;
    double* G = ws + 2 * sC;             // p x q, ld p
    double* V = G + (int64_t)m * n;      // q x q, ld q
    double part = 0.0;
    for (int e = threadIdx.x; e < m * n; e += kThreads) {
      int i, j;
      if (src) { i = e / n; j = e % n; } else { i = e % m; j = e / m; }
      const double x = S[i * s_r + j * s_c];
      part = fma(x, x, part);
    }
    const double nsq = block_sum(part, sh.red);
    if (!isfinite(nsq)) {
      if (tm.tid == 0) atomicCAS(err, 0, 3);  // a timeout (1) keeps precedence
    }
    const double nrm = sqrt(nsq);
    int kind;
    if (!(nrm >= drop_norm) || nsq == 0.0 || !isfinite(nsq)) {
      kind = CLR_KIND_ZERO;
      if (tm.tid == 0) { C.kind[t] = kind; C.rank[t] = 0; C.norm[t] = 0.0; }
      __syncthreads();
      continue;
    }
    const One solo;
    int r = q;
    bool alone = false;      // a full SVD in a team: the rest is the first CTA's
    long long c_full = -1;   // while profiling: start of a full-SVD block's truncation
    if (rrqr && !dense_only) {
      r = rrqr_block(S, s_r, s_c, m, n, eps, G, sh);
      if (r > 0 && r <= q / 2) {
        // X = Q_r (the first r columns of H_0 ... H_{r-1}), W = P R_r^T
        double* Xo = slot;
        double* Wo = slot + (int64_t)m * r;
        for (int e = threadIdx.x; e < m * r; e += kThreads) Xo[e] = (e % m == e / m) ? 1.0 : 0.0;
        __syncthreads();
        apply_q(G, m, r, sh.refl, nullptr, Xo, r, m, threadIdx.x / 32, kWarps);
        __syncthreads();
        double part = 0.0;
        for (int e = threadIdx.x; e < n * r; e += kThreads) {
          const int c = e % n, i = e / n;
          const double v = c >= i ? G[i + (int64_t)c * m] : 0.0;
          Wo[sh.perm[c] + (int64_t)i * n] = v;
          part = fma(v, v, part);
        }
        const double kept = block_sum(part, sh.red);
        if (threadIdx.x == 0) {
          C.kind[t] = CLR_KIND_LR;
          C.rank[t] = r;
          C.norm[t] = sqrt(kept);
        }
        __syncthreads();
        continue;
      }
    } else if (!dense_only) {
      const SrcView view{S, s_r, s_c, tr};
      const long long c0 = clock64();
      // pivoted QR first: blocks of low numerical rank are truncated through the SVD of
      // the k x q factor, blocks of rank above q/2 certified dense
      const int pre = prereduce ? compress_by_pivoted_qr(tm, view, p, q, tr, m, n, eps, max_sweeps,
                                                         G, V, sc, slot, &C.kind[t], &C.rank[t],
                                                         &C.norm[t], sh, jstats)
                                : 0;
      // (the full SVD is one CTA's)
      if (pre == 0 && tm.rank != 0) continue;
      alone = pre == 0;
      if (pre == 0) {
        unsigned long long* stage_clk = jstats ? jstats + kFullStageCounters : nullptr;
        if (stage_clk && threadIdx.x == 0)
          atomicAdd(&stage_clk[0], (unsigned long long)(clock64() - c0));
        const int early_dense = svd_mixed(solo, view, p, q, G, V, sc, max_sweeps, eps, q / 2, nrm,
                                          false, sh, jstats, stage_clk);
        if (!early_dense) {
          c_full = clock64();
          sort_and_truncate(G, p, q, p, eps, sh);
          r = sh.rank;
        }
      } else if (pre >= 2 && jstats && tm.tid == 0) {
        atomicAdd(&jstats[3], 1ull);   // stored dense without a full SVD
      }
      // SM cycles per path while profiling (block 2 of the counters): QR and the SVD of R
      // stored low rank, certified dense by the QR's triangles, full SVD (prereduce off, or a
      // non-finite QR norm), QR and the SVD of R stored dense
      if (jstats && tm.tid == 0) {
        const int path = pre == 1 ? 0 : pre == 2 ? 1 : pre == 3 ? 3 : 2;
        atomicAdd(&jstats[kPathCounters + 2 * path], (unsigned long long)(clock64() - c0));
        atomicAdd(&jstats[kPathCounters + 2 * path + 1], 1ull);
      }
      if (pre == 1) continue;
    }
    const int lim = q / 2;
    if (r == 0) {
      if (tm.tid == 0) { C.kind[t] = CLR_KIND_ZERO; C.rank[t] = 0; C.norm[t] = 0.0; }
    } else if (dense_only || r > lim) {
      if (src) {
        for (int e = alone ? threadIdx.x : tm.tid; e < m * n; e += alone ? kThreads : tm.nt) {
          const int i = e % m, j = e / m;
          slot[e] = S[i * s_r + j * s_c];
        }
      }
      if (tm.tid == 0) { C.kind[t] = CLR_KIND_DENSE; C.rank[t] = q; C.norm[t] = nrm; }
    } else {
      // Y = A^T G_r (q x r) into V before the slot (possibly the source) is overwritten, or
      // Y = V_r S_r^2 from the accumulated V
      const SrcView view{S, s_r, s_c, tr};
      const bool tracked = sh.v_tracked;
      bool ls = !tracked && sh.ls_recover;
      constexpr int64_t kSq = (int64_t)CLR_MAX_CLUSTER * CLR_MAX_CLUSTER;
      if (!tracked) recover_right(solo, view, p, q, G, sh.perm, r, V, sc, false);
      if (ls)
        ls = ls_solve(solo, V, q, r, sc, p, sh.sorted, sc + 4 * kSq, sc + kSq, sc + 3 * kSq,
                      series_f32(r, sc), sh);
      if (jstats && threadIdx.x == 0 && !tracked)
        atomicAdd(&jstats[4], 2ull * p * q * r);
      double* Xo = slot;
      double* Wo = slot + (int64_t)m * r;
      if (!tr) {
        // G = U S (m x n), Y = V S^2:  X = (U S)_r, W = V_r
        for (int e = threadIdx.x; e < m * r; e += kThreads) {
          const int i = e % m, c = e / m;
          Xo[e] = G[i + (int64_t)sh.perm[c] * p];
        }
        for (int e = threadIdx.x; e < n * r; e += kThreads) {
          const int j = e % n, c = e / n;
          Wo[e] = tracked ? V[(int64_t)j * q + sh.perm[c]]
                  : ls    ? V[(int64_t)j * r + c]
                          : V[(int64_t)j * r + c] / (sh.sorted[c] * sh.sorted[c]);
        }
      } else {
        // G = U' S (n x m) of the transposed block, Y = V' S^2 (m x r): block = V' S U'^T ->
        // X = V'_r S_r = Y S^-1, W = U'_r = G_r S^-1
        for (int e = threadIdx.x; e < m * r; e += kThreads) {
          const int i = e % m, c = e / m;
          Xo[e] = tracked ? V[(int64_t)i * q + sh.perm[c]] * sh.sorted[c]
                  : ls    ? V[(int64_t)i * r + c]
                          : V[(int64_t)i * r + c] / sh.sorted[c];
        }
        for (int e = threadIdx.x; e < n * r; e += kThreads) {
          const int j = e % n, c = e / n;
          Wo[e] = ls ? G[j + (int64_t)sh.perm[c] * p] : G[j + (int64_t)sh.perm[c] * p] / sh.sorted[c];
        }
      }
      if (threadIdx.x == 0) {
        C.kind[t] = CLR_KIND_LR;
        C.rank[t] = r;
        C.norm[t] = sqrt(sh.kept_sq);
      }
    }
    __syncthreads();
    if (jstats && c_full >= 0 && threadIdx.x == 0) {
      atomicAdd(&jstats[kFullStageCounters + 6], (unsigned long long)(clock64() - c_full));
      atomicAdd(&jstats[kFullStageCounters + 7], 1ull);
      if (r > q / 2) atomicAdd(&jstats[7], 1ull);   // full SVD, stored dense
    }
  }
  record_cost(clock64());
}

// The kernel with CTAs in clusters, which leave a few SMs of a GPC unused, and the one without for
// launches that could not use a team.
__global__ void __cluster_dims__(kTeamCtas, 1, 1) __launch_bounds__(kThreads, 1)
    compress_dense_team_kernel(MatView C, const int* list, const int* count, const int* order,
                               const double* src, int64_t lds, double* ws, double* svd_scratch,
                               double eps, double drop_norm, int dense_only, int rrqr,
                               int prereduce, int max_sweeps, int* err, int* sched,
                               const int* n_team, unsigned long long* jstats) {
  compress_dense_body<true>(C, list, count, order, src, lds, ws, svd_scratch, eps, drop_norm, dense_only,
                      rrqr, prereduce, max_sweeps, err, sched, n_team, jstats);
}

__global__ void __launch_bounds__(kThreads, 1)
    compress_dense_kernel(MatView C, const int* list, const int* count, const int* order,
                          const double* src, int64_t lds, double* ws, double* svd_scratch,
                          double eps, double drop_norm, int dense_only, int rrqr, int prereduce,
                          int max_sweeps, int* err, int* sched, unsigned long long* jstats) {
  compress_dense_body<false>(C, list, count, order, src, lds, ws, svd_scratch, eps, drop_norm, dense_only,
                      rrqr, prereduce, max_sweeps, err, sched, nullptr, jstats);
}

void launch_compress_dense(const MatView& C, const int* list, const int* count,
                           const int* order, const double* src, int64_t lds, double* ws,
                           double* svd_scratch, double eps, double drop_norm,
                           int dense_only, int rrqr, int prereduce, int max_side, int max_sweeps,
                           int grid, int* err, int* sched, const int* n_team,
                           unsigned long long* jstats, cudaStream_t st) {
  static bool attr_done[64] = {false}, attr_done_team[64] = {false};
  const int g = svd_launch_grid(compress_dense_kernel, grid, attr_done);
  const int gt =
      svd_launch_grid(compress_dense_team_kernel, grid, attr_done_team) / kTeamCtas * kTeamCtas;
  // (how many tiles a product has is the device's to know; launches with more blocks than this are
  // rarely left with few enough for teams)
  if (gt > 0 && prereduce && !rrqr && !dense_only && C.nr * C.nc <= 2 * gt)
    compress_dense_team_kernel<<<gt, kThreads, kSvdSmemBytes, st>>>(
        C, list, count, order, src, lds, ws, svd_scratch, eps, drop_norm, dense_only, rrqr,
        prereduce, max_sweeps, err, sched, n_team, jstats);
  else
    // Without the pivoted QR a 256 x 256 block's sweeps run on 512 KB in the scratch; they are bound
    // by what L1 holds of it, and shared memory would take that (build of the 3D lattice, N = 1024
    // and 2048, clusters of up to 256: 87 and 76 ms, now 84 and 72).
    compress_dense_kernel<<<g, kThreads, !prereduce && 8 * max_side * max_side > kSvdSmemBytes
                                             ? 0 : kSvdSmemBytes, st>>>(
        C, list, count, order, src, lds, ws, svd_scratch, eps, drop_norm, dense_only, rrqr,
        prereduce, max_sweeps, err, sched, jstats);
}

// ---------------------------------------------------------------------------------------------
// Block Frobenius norms: dense directly, low rank as sqrt(sum_ab (X^T X)_ab (W^T W)_ab).
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kThreads) block_norms_kernel(MatView M) {
  __shared__ double red[kWarps];
  const int t = blockIdx.x;
  const int I = t / M.nc, J = t % M.nc;
  const int m = M.row_off[I + 1] - M.row_off[I];
  const int n = M.col_off[J + 1] - M.col_off[J];
  const int kind = M.kind[t];
  const double* s = M.pool + slot_of(M, I, J, m);
  double part = 0.0;
  if (kind == CLR_KIND_DENSE) {
    for (int e = threadIdx.x; e < m * n; e += kThreads) part = fma(s[e], s[e], part);
  } else if (kind == CLR_KIND_LR) {
    const int r = M.rank[t];
    const double* X = s;
    const double* W = s + (int64_t)m * r;
    for (int e = threadIdx.x; e < r * r; e += kThreads) {
      const int a = e % r, b = e / r;
      double gx = 0.0, gw = 0.0;
      for (int i = 0; i < m; ++i) gx = fma(X[i + (int64_t)a * m], X[i + (int64_t)b * m], gx);
      for (int j = 0; j < n; ++j) gw = fma(W[j + (int64_t)a * n], W[j + (int64_t)b * n], gw);
      part = fma(gx, gw, part);
    }
  }
  const double tot = block_sum(part, red);
  if (threadIdx.x == 0) M.norm[t] = kind == CLR_KIND_ZERO ? 0.0 : sqrt(fmax(tot, 0.0));
}

// Frobenius norm of every block's slot read as a dense block (kinds not yet known).
__global__ void __launch_bounds__(kThreads) block_norms_dense_kernel(MatView M) {
  __shared__ double red[kWarps];
  const int t = blockIdx.x;
  const int I = t / M.nc, J = t % M.nc;
  const int m = M.row_off[I + 1] - M.row_off[I];
  const int n = M.col_off[J + 1] - M.col_off[J];
  const double* s = M.pool + slot_of(M, I, J, m);
  double part = 0.0;
  for (int e = threadIdx.x; e < m * n; e += kThreads) part = fma(s[e], s[e], part);
  const double tot = block_sum(part, red);
  if (threadIdx.x == 0) M.norm[t] = sqrt(tot);
}

void launch_block_norms_dense(const MatView& M, cudaStream_t st) {
  block_norms_dense_kernel<<<M.nr * M.nc, kThreads, 0, st>>>(M);
}

void launch_block_norms(const MatView& M, cudaStream_t st) {
  block_norms_kernel<<<M.nr * M.nc, kThreads, 0, st>>>(M);
}

// alpha * M in place: dense values or the X factor, and the norms; several CTAs per block
// (lr_parts).
__global__ void scale_blocks_kernel(MatView M, double alpha) {
  const int t = blockIdx.x;
  const int I = t / M.nc, J = t % M.nc;
  const int m = M.row_off[I + 1] - M.row_off[I];
  const int n = M.col_off[J + 1] - M.col_off[J];
  const int kind = M.kind[t];
  double* s = M.pool + slot_of(M, I, J, m);
  int64_t len = kind == CLR_KIND_DENSE ? (int64_t)m * n
              : kind == CLR_KIND_LR ? (int64_t)m * M.rank[t] : 0;
  const int64_t step = (int64_t)blockDim.x * gridDim.y;
  for (int64_t e = threadIdx.x + (int64_t)blockDim.x * blockIdx.y; e < len; e += step)
    s[e] *= alpha;
  if (threadIdx.x == 0 && blockIdx.y == 0) M.norm[t] *= fabs(alpha);
}

void launch_scale_blocks(const MatView& M, double alpha, cudaStream_t st) {
  scale_blocks_kernel<<<dim3((unsigned)(M.nr * M.nc), (unsigned)lr_parts(M)), 256, 0,
                        st>>>(M, alpha);
}

}  // namespace clr

// =============================================================================================
// Allocation-free truncated SVD of one block (clr_block_compress_noalloc).
//
// Same computation as compress_dense_kernel for a single block, but its working memory (the
// block copy G and the rotation matrix V) lives in a fixed file-scope device array instead of a
// caller- or context-allocated workspace, so the entry point never allocates.  The array holds
// CLR_MAX_CLUSTER^2 doubles for G and as many for V (1 MiB), is loaded with every GPU that
// loads this library, and is shared by every call: G is fully rewritten and V reset to the
// identity by each call, so no stale contents are read, but calls that overlap on the GPU
// (different streams, concurrent host threads) race on it.
// =============================================================================================
namespace clr {
namespace {

constexpr int64_t kNoAllocScratchDoubles = 2LL * CLR_MAX_CLUSTER * CLR_MAX_CLUSTER;
__device__ __align__(256) double g_noalloc_scratch[kNoAllocScratchDoubles];

constexpr int kNoAllocMaxDevices = 64;
double* g_noalloc_ptr[kNoAllocMaxDevices] = {nullptr};
std::mutex g_noalloc_mutex;

// status[0] = kind, status[1] = rank, status[2] = error flag (3: non-finite input, 4: sweep
// limit reached before convergence)
__global__ void __launch_bounds__(kThreads) compress_block_noalloc_kernel(
    const double* src, int64_t lds, int m, int n, double eps, int max_sweeps, double* scratch,
    double* x_out, double* w_out, double* sigma_out, int* status) {
  __shared__ SvdShared sh;
  const bool tr = m < n;
  const int p = tr ? n : m, q = tr ? m : n;
  double* G = scratch;                                   // p x q, ld p
  double* V = scratch + (int64_t)CLR_MAX_CLUSTER * CLR_MAX_CLUSTER;  // q x q, ld q
  double part = 0.0;
  for (int e = threadIdx.x; e < m * n; e += kThreads) {
    const int i = e % m, j = e / m;
    const double x = src[i + (int64_t)j * lds];
    part = fma(x, x, part);
    if (tr) G[j + (int64_t)i * p] = x; else G[i + (int64_t)j * p] = x;
  }
  const double nsq = block_sum(part, sh.red);
  if (threadIdx.x == 0) status[2] = isfinite(nsq) ? 0 : 3;
  if (!isfinite(nsq) || nsq == 0.0) {
    if (threadIdx.x == 0) { status[0] = CLR_KIND_ZERO; status[1] = 0; }
    return;
  }
  // pairs of columns at the FP64 rounding level of the block (p u ||A||_F) are left alone:
  // rotating them changes nothing that a truncation can see, and they would keep the sweeps
  // from ever converging
  const double floor64 = (double)p * DBL_EPSILON * sqrt(nsq);
  const int sweeps =
      jacobi_svd<false>(G, p, q, V, max_sweeps, &sh.flag, floor64 * floor64, sh.jac);
  // every sweep still rotated a pair: the column norms the truncation uses may be inexact
  if (sweeps >= max_sweeps && threadIdx.x == 0) status[2] = 4;
  sort_and_truncate(G, p, q, p, eps, sh);
  const int r = sh.rank;
  if (sigma_out)
    for (int c = threadIdx.x; c < q; c += kThreads) sigma_out[c] = sh.sorted[c];
  if (r == 0) {
    if (threadIdx.x == 0) { status[0] = CLR_KIND_ZERO; status[1] = 0; }
    return;
  }
  if (r > q / 2) {
    if (threadIdx.x == 0) { status[0] = CLR_KIND_DENSE; status[1] = q; }
    return;
  }
  if (!tr) {
    for (int e = threadIdx.x; e < m * r; e += kThreads)
      x_out[e] = G[(e % m) + (int64_t)sh.perm[e / m] * p];
    for (int e = threadIdx.x; e < n * r; e += kThreads)
      w_out[e] = V[(e % n) + (int64_t)sh.perm[e / n] * q];
  } else {
    for (int e = threadIdx.x; e < m * r; e += kThreads)
      x_out[e] = V[(e % m) + (int64_t)sh.perm[e / m] * q] * sh.sorted[e / m];
    for (int e = threadIdx.x; e < n * r; e += kThreads)
      w_out[e] = G[(e % n) + (int64_t)sh.perm[e / n] * p] / sh.sorted[e / n];
  }
  if (threadIdx.x == 0) { status[0] = CLR_KIND_LR; status[1] = r; }
}

}  // namespace
}  // namespace clr

extern "C" int clr_block_compress_noalloc(int device, const double* block, int64_t ld, int m,
                                          int n, double eps, int max_sweeps, double* x_out,
                                          double* w_out, double* sigma_out, int32_t* status,
                                          void* stream) {
  using namespace clr;
  if (!block || !x_out || !w_out || !status) return CLR_EINVAL;
  if (m < 1 || n < 1 || m > CLR_MAX_CLUSTER || n > CLR_MAX_CLUSTER) return CLR_EINVAL;
  if (ld < m || !(eps >= 0.0) || max_sweeps < 1) return CLR_EINVAL;
  if (device < 0 || device >= kNoAllocMaxDevices) return CLR_EINVAL;
  int prev = 0;
  if (cudaGetDevice(&prev) != cudaSuccess) return CLR_ECUDA;
  if (prev != device && cudaSetDevice(device) != cudaSuccess) return CLR_ECUDA;
  double* scratch = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_ptr[device]) {
      void* ptr = nullptr;
      if (cudaGetSymbolAddress(&ptr, g_noalloc_scratch) != cudaSuccess || !ptr) {
        if (prev != device) cudaSetDevice(prev);
        return CLR_ECUDA;
      }
      g_noalloc_ptr[device] = (double*)ptr;
    }
    scratch = g_noalloc_ptr[device];
  }
  compress_block_noalloc_kernel<<<1, kThreads, 0, (cudaStream_t)stream>>>(
      block, ld, m, n, eps, max_sweeps, scratch, x_out, w_out, sigma_out, (int*)status);
  const cudaError_t e = cudaGetLastError();
  if (prev != device) cudaSetDevice(prev);
  return e == cudaSuccess ? CLR_OK : CLR_ECUDA;
}
