// stb_quantize: the paper's quantizer on the GPU -- Standardized Importance (Eq. 3), N of 8 per group (Section 3.3),
// the salient-column search and the break-point search of Algorithm 2, residual binarization (Eq. 4) and
// trisection -- i.e. the block loop of Algorithm 1 without its Hessian update, from a dense fp16 layer and the column
// norms of the calibration activations to the logical arrays stb_pack takes.  The paper runs this step in
// PyTorch for hours per model (Section 4.1); here every stage is a kernel.
//
// The definition is float64 and some of its sums round (the error of a candidate is added up row by row), so that a
// decision that hangs on the last bits depends on the order of the additions.  The output must be the definition's, bit
// for bit, yet walking the rows of a block one after the other, for each of its 32 + 70 candidates, leaves the chip
// idle (15.7 ms for 4096 x 4096, every warp waiting on its own chain).  So every decision is FILTERED:
//   * the quantity behind it is first computed in parallel, in float64, by a formula that is equal in exact arithmetic,
//     with a bound on how far the definition's rounded value can be from it;
//   * where the bound leaves one outcome, that is the outcome;
//   * where it leaves several (ties, or differences near 2^-53 of the value: rare, or blocks of few weights), the
//     definition's own sequence of roundings is carried out for the candidates that are left.
// Sums of |w| of fp16 values, and sums of w^2 over a row's 128 columns of ordinary range, are exact in float64 and may be
// taken in any order; products and differences whose rounding the definition fixes are never fused into multiply-adds.
// The layer-wide mean and deviation of Eq. 3 are the exception: their rounding moves every
// score by the same relative 1e-16, which can change a decision only where two scores tie to that precision (a layer whose
// |w| are all one value is such a tie everywhere: its deviation is rounding noise, and so is the definition's choice).
//
// 4096 x 4096 at 6:8: 15.7 ms with one warp per (block, candidate) walking the rows, now 0.28 ms: sums 22 us, spread 18,
// selection 42, salient search 33, break points 102, emit 63.
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "../../include/stb.h"

namespace stb {
namespace quant {

constexpr int kBeta = 128, kM = 8, kMaxSal = 32, kGrid = 160;
constexpr int kPoints = 70;            // grid points with p2 <= 0.9 max (the grid's fraction passes 0.45 between 69 and 70)
constexpr double kUlp = 1.1102230246251565e-16;   // 2^-53
constexpr int kPartials = 592;         // CTAs of spread_kernel: four per SM

struct Ws {
  double* rowsum;      // [n]            -- zeroed from here ...
  double* colsum;      // [m]
  double* colsq;       // [m]
  double* sgain;       // [nblk][32]     sum over rows of the salient candidates' a^2 / k terms
  double* bgain;       // [nblk][70]     the same for the grid points
  uint32_t* colmax;    // [m]            largest kept |w| of a column, as fp16 bits
  uint32_t* count;     // [2 + 2 nblk]   CTAs done: sums, spread, salient and break per block
  uint32_t* zero_end;  //                -- ... to here
  double* rinv;        // [n]            1 / row sum, 0 for a zero row
  double* cinv;        // [m]
  double* atot;        // [n][nblk]      kept |w| of a row and block
  double* partial;     // [kPartials][2]
  double* scalars;     // [0] mean, [1] sd, [2] lambda
  uint8_t* salflag;    // [nblk][128]
  double* bp;          // [nblk][2]
};

// |w| of fp16 bits (sign cleared) in float64: the bits are put in place as a (tiny) double, one exact product moves the exponent
__device__ __forceinline__ double abs_of(uint32_t bits15) { return __hiloint2double((int)(bits15 << 10), 0) * 0x1p1008; }
__device__ __forceinline__ double w_at(const __half* W, size_t ldw, int i, int j) { return (double)__half2float(W[(size_t)i * ldw + j]); }
__device__ __forceinline__ uint32_t bits_at(const __half* W, size_t ldw, int i, int j) { return __half_as_ushort(W[(size_t)i * ldw + j]); }
__device__ __forceinline__ bool kept_at(const uint8_t* keep, int ngrp, int i, int j) { return (keep[(size_t)i * ngrp + (j >> 3)] >> (j & 7)) & 1u; }
// error of binarizing a set with sum of squares q, l1 sum a, count k: q - k alpha^2, alpha = a / k (no fused operations)
__device__ __forceinline__ double binary_error(double q, double a, int k) {
  if (k == 0) return 0.0;
  const double alpha = __ddiv_rn(a, (double)k);
  return __dsub_rn(q, __dmul_rn(__dmul_rn((double)k, alpha), alpha));
}
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, d);
  return v;
}
// eight consecutive weights of a row as raw bits, two per word; kVec: rows are 16-byte aligned
template <bool kVec>
__device__ __forceinline__ uint4 load8(const __half* p) {
  if constexpr (kVec) {
    return __ldg(reinterpret_cast<const uint4*>(p));
  } else {
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) w[i] = (uint32_t)__half_as_ushort(p[2 * i]) | ((uint32_t)__half_as_ushort(p[2 * i + 1]) << 16);
    return make_uint4(w[0], w[1], w[2], w[3]);
  }
}
__device__ __forceinline__ uint32_t half_bits(const uint4& v, int c) {      // c: compile-time after unrolling
  const uint32_t w = c < 2 ? v.x : (c < 4 ? v.y : (c < 6 ? v.z : v.w));
  return (c & 1) ? (w >> 16) : (w & 0xFFFFu);
}
// One arrival on a counter per CTA; true for all threads of the CTA that arrives last (`flag`: a shared word).
// What the CTA wrote before is visible to that last one.
__device__ __forceinline__ bool last_arrival(uint32_t* counter, uint32_t arrivals, uint32_t* flag) {
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) *flag = atomicAdd(counter, 1u) == arrivals - 1u ? 1u : 0u;
  __syncthreads();
  const bool last = *flag != 0u;
  if (last) __threadfence();
  return last;
}

// ---- Eq. 3: sums of |W| per row and per column, sums of W^2 per column -----------------------------------------------
// CTA: 256 columns (8 per lane) x kRowsPerCta rows, one row per warp at a time.  The sums of |w| are exact (40 bits and
// the row count's): atomics may add them in any order.  Those of w^2 are not (80 bits; an outlier column of 4096 rows
// needs 55 of them): salient_kernel, which orders columns by them, looks again where that matters.
constexpr int kRowsPerCta = 64, kInFlight = 4;    // (rows of a warp whose loads are in flight together: the passes are bound by latency)
// abs_of reads the codes of infinities and NaN as numbers.  Where a lane's weights may have such a code, the sums they belong to are
// made infinite or NaN here, as the definition's are: with an infinite one mean and deviation are then NaN, so that every group is
// selected by select_exact; and the sums of squares of their blocks are not finite, so that no candidate of a search is filtered out.
__device__ __noinline__ void add_non_finite(const __half* W, size_t ldw, int r0, int r1, int j0, double* rowsum, double* colsum, double* colsq) {
  for (int r = r0; r < r1; r += 8)
    for (int c = 0; c < 8; ++c) {
      const double x = fabs(w_at(W, ldw, r, j0 + c));
      if (!(x < INFINITY)) { atomicAdd(rowsum + r, x); atomicAdd(colsum + j0 + c, x); atomicAdd(colsq + j0 + c, x); }
    }
}
constexpr double kInfiniteCode = 65536.0;         // what abs_of makes of an infinity (of NaN, more): no smaller sum holds one
template <bool kVec>
__global__ void __launch_bounds__(256) sums_kernel(const __half* __restrict__ W, size_t ldw, int n, int m, double* __restrict__ rowsum,
                                                   double* __restrict__ colsum, double* __restrict__ colsq) {
  __shared__ double red[8][256];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int j0 = blockIdx.x * 256 + 8 * lane;
  const bool live = j0 < m;
  const int r1 = min(n, (int)(blockIdx.y + 1) * kRowsPerCta);
  double a[8], q[8];
  bool large = false;
#pragma unroll
  for (int c = 0; c < 8; ++c) a[c] = q[c] = 0.0;
  for (int r = blockIdx.y * kRowsPerCta + warp; r < r1; r += 8 * kInFlight) {
    uint4 v[kInFlight];
#pragma unroll
    for (int k = 0; k < kInFlight; ++k) v[k] = live && r + 8 * k < r1 ? load8<kVec>(W + (size_t)(r + 8 * k) * ldw + j0) : make_uint4(0, 0, 0, 0);
    double s[kInFlight];
#pragma unroll
    for (int k = 0; k < kInFlight; ++k) {
      s[k] = 0.0;
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const double w = abs_of(half_bits(v[k], c) & 0x7FFFu);
        a[c] += w; q[c] += w * w; s[k] += w;
      }
      large = large || s[k] >= kInfiniteCode;
    }
#pragma unroll
    for (int k = 0; k < kInFlight; ++k) {
      s[k] = warp_sum(s[k]);
      if (lane == 0 && r + 8 * k < r1) atomicAdd(rowsum + r + 8 * k, s[k]);
    }
  }
  if (large) add_non_finite(W, ldw, blockIdx.y * kRowsPerCta + warp, r1, j0, rowsum, colsum, colsq);
#pragma unroll
  for (int pass = 0; pass < 2; ++pass) {
#pragma unroll
    for (int c = 0; c < 8; ++c) red[warp][32 * c + lane] = pass == 0 ? a[c] : q[c];
    __syncthreads();
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < 8; ++w) s += red[w][threadIdx.x];
    const int j = blockIdx.x * 256 + 8 * (threadIdx.x & 31) + (threadIdx.x >> 5);
    if (j < m) atomicAdd((pass == 0 ? colsum : colsq) + j, s);
    __syncthreads();
  }
}

// Reciprocals of the sums, and by the last CTA the mean of mu = |w| / rowsum + |w| / colsum over the layer -- every row with
// a sum contributes 1, every column too -- and lambda: the caller's, or 0.01 mean_j h_jj with h_jj = 2 ||X_:,j||^2.
__global__ void __launch_bounds__(256) scalars_kernel(int n, int m, const double* __restrict__ xnorm, double lambda_in, Ws w) {
  __shared__ double sh[8][2];
  __shared__ uint32_t flag;
  double cnt = 0.0, h = 0.0;
  for (int i = blockIdx.x * 256 + threadIdx.x; i < n + m; i += gridDim.x * 256) {
    const double v = i < n ? w.rowsum[i] : w.colsum[i - n];
    const double inv = v > 0.0 ? 1.0 / v : 0.0;
    if (v > 0.0) cnt += 1.0;
    if (v == INFINITY) cnt = NAN;              // (an infinite weight over its own sum; a NaN sum counts as none)
    if (i < n) w.rinv[i] = inv;
    else { w.cinv[i - n] = inv; h += 2.0 * xnorm[i - n] * xnorm[i - n]; }
  }
  auto cta_sum = [&]() {                 // the CTA's sums to thread 0
    cnt = warp_sum(cnt); h = warp_sum(h);
    if ((threadIdx.x & 31) == 0) { sh[threadIdx.x >> 5][0] = cnt; sh[threadIdx.x >> 5][1] = h; }
    __syncthreads();
    cnt = h = 0.0;
    for (int k = 0; k < 8; ++k) { cnt += sh[k][0]; h += sh[k][1]; }
    __syncthreads();
  };
  cta_sum();
  if (threadIdx.x == 0) { w.partial[2 * blockIdx.x] = cnt; w.partial[2 * blockIdx.x + 1] = h; }
  if (!last_arrival(w.count, gridDim.x, &flag)) return;
  cnt = h = 0.0;
  for (int k = threadIdx.x; k < (int)gridDim.x; k += 256) { cnt += __ldcg(w.partial + 2 * k); h += __ldcg(w.partial + 2 * k + 1); }
  cta_sum();
  if (threadIdx.x == 0) {
    w.scalars[0] = cnt / ((double)n * (double)m);
    w.scalars[2] = lambda_in < 0.0 ? 0.01 * h / (double)m : lambda_in;
  }
}

// Deviation of mu: sum of (mu - mean)^2 per CTA, finished by the last one.
template <bool kVec>
__global__ void __launch_bounds__(256) spread_kernel(const __half* __restrict__ W, size_t ldw, int n, int m, Ws w) {
  __shared__ double sh[8];
  __shared__ uint32_t flag;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const double mean = w.scalars[0];
  const double* __restrict__ rinv = w.rinv;
  const double* __restrict__ cinv = w.cinv;
  const int cols = (m + 255) / 256;
  const long long units = (long long)cols * ((n + 15) / 16);           // 256 columns x 16 rows, one unit per warp at a time
  double acc = 0.0;
  for (long long u = (long long)blockIdx.x * 8 + warp; u < units; u += (long long)gridDim.x * 8) {
    const int j0 = (int)(u % cols) * 256 + 8 * lane, r0 = (int)(u / cols) * 16, r1 = min(n, r0 + 16);
    if (j0 >= m) continue;
    double ci[8], a2[2] = {0.0, 0.0};
#pragma unroll
    for (int c = 0; c < 8; ++c) ci[c] = cinv[j0 + c];
    for (int r = r0; r < r1; r += kInFlight) {
      uint4 v[kInFlight];
      double ri[kInFlight];
#pragma unroll
      for (int k = 0; k < kInFlight; ++k) {
        const int rr = min(r + k, r1 - 1);
        v[k] = load8<kVec>(W + (size_t)rr * ldw + j0);
        ri[k] = rinv[rr];
      }
#pragma unroll
      for (int k = 0; k < kInFlight; ++k)
        if (r + k < r1) {
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            const double d = abs_of(half_bits(v[k], c) & 0x7FFFu) * (ri[k] + ci[c]) - mean;
            a2[c & 1] += d * d;
          }
        }
    }
    acc += a2[0] + a2[1];
  }
  auto cta_sum = [&]() {
    acc = warp_sum(acc);
    if (lane == 0) sh[warp] = acc;
    __syncthreads();
    acc = 0.0;
    for (int k = 0; k < 8; ++k) acc += sh[k];
    __syncthreads();
  };
  cta_sum();
  if (threadIdx.x == 0) w.partial[blockIdx.x] = acc;
  if (!last_arrival(w.count + 1, gridDim.x, &flag)) return;
  acc = 0.0;
  for (int k = threadIdx.x; k < (int)gridDim.x; k += 256) acc += __ldcg(w.partial + k);
  cta_sum();
  if (threadIdx.x == 0) w.scalars[1] = sqrt(acc / ((double)n * (double)m));
}

// ---- Section 3.3: keep the N highest scores of every 8 columns (ties: lower column) ---------------------------------
// The definition's score of column c: s = ((mu - mean) / sd) xnorm with its own roundings.  Ties are the lower column's.
__device__ __noinline__ uint32_t select_exact(const __half* W, size_t ldw, int i, int j0, int N, const double* rowsum, const double* colsum,
                                              const double* xnorm, double mean, double sd) {
  double s[kM];
  for (int c = 0; c < kM; ++c) {
    const double a = fabs(w_at(W, ldw, i, j0 + c));
    double mu = 0.0;
    if (rowsum[i] > 0.0) mu = __dadd_rn(mu, __ddiv_rn(a, rowsum[i]));
    if (colsum[j0 + c] > 0.0) mu = __dadd_rn(mu, __ddiv_rn(a, colsum[j0 + c]));
    const double z = sd > 0.0 ? __ddiv_rn(__dsub_rn(mu, mean), sd) : 0.0;
    s[c] = __dmul_rn(z, xnorm[j0 + c]);
  }
  uint32_t bits = 0;
  for (int c = 0; c < kM; ++c) {
    int rank = 0;
    for (int a = 0; a < kM; ++a) rank += (s[a] > s[c] || (s[a] == s[c] && a < c)) ? 1 : 0;
    if (rank < N) bits |= 1u << c;
  }
  return bits;
}
// Filter: without the divisions, and without 1 / sd > 0, which changes no order, the score is a (1 / rowsum + 1 / colsum) - mean
// times xnorm: three operations, with a rounding error below 16 ulp of (mu + mean) xnorm.  The definition's score (times
// sd) is as close to the exact one, so a gap above 64 ulp between the last kept and the first dropped column decides.
// Same CTA shape as sums_kernel; a lane's eight columns are one group, 16 lanes one block of 128.
template <bool kVec>
__global__ void __launch_bounds__(256) select_kernel(const __half* __restrict__ W, size_t ldw, int n, int m, int N, const double* __restrict__ xnorm,
                                                     Ws w, uint8_t* __restrict__ keep) {
  __shared__ uint32_t cmax[8][4][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int j0 = blockIdx.x * 256 + 8 * lane, ngrp = m / kM, nblk = m / kBeta;
  const bool live = j0 < m;
  const double mean = w.scalars[0], sd = w.scalars[1];
  double ci[8], xn[8], xmax = 0.0;
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    ci[c] = live ? w.cinv[j0 + c] : 0.0; xn[c] = live ? xnorm[j0 + c] : 0.0;
    xmax = fmax(xmax, xn[c]);
  }
  const double* __restrict__ rinv = w.rinv;
  uint32_t cm[4] = {0, 0, 0, 0};
  const int r1 = min(n, (int)(blockIdx.y + 1) * kRowsPerCta);
  const int r0 = blockIdx.y * kRowsPerCta + warp;
  uint4 vn = make_uint4(0, 0, 0, 0);
  double rn = 0.0;
  if (r0 < r1) { if (live) vn = load8<kVec>(W + (size_t)r0 * ldw + j0); rn = rinv[r0]; }
  for (int r = r0; r < r1; r += 8) {
    const uint4 v = vn;
    const double ri = rn;
    if (r + 8 < r1) { if (live) vn = load8<kVec>(W + (size_t)(r + 8) * ldw + j0); rn = rinv[r + 8]; }
    double a[8], s[8];
    uint32_t rank = 0;                      // a nibble per column: how many columns come before it
    int big = 0;                            // high word of the largest |s|
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      a[c] = abs_of(half_bits(v, c) & 0x7FFFu);
      s[c] = (a[c] * (ri + ci[c]) - mean) * xn[c];
      big = max(big, __double2hiint(s[c]) & 0x7FFFFFFF);
#pragma unroll
      for (int b = 0; b < c; ++b) rank += s[c] > s[b] ? (1u << (4 * b)) : (1u << (4 * c));
    }
    uint32_t bits = 0xFFu;
    if (N < 8) {
      double low_kept = 0.0, high_dropped = 0.0;       // the scores with ranks N - 1 and N
      bits = 0;
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const int rk = (int)((rank >> (4 * c)) & 0xFu);
        if (rk < N) bits |= 1u << c;
        if (rk == N - 1) low_kept = s[c];
        if (rk == N) high_dropped = s[c];
      }
      // (a comparison with a NaN is false: such a group takes the definition's way too)
      const double smax = __hiloint2double(big + 1, 0);
      if (live && !(low_kept - high_dropped > 64.0 * kUlp * (smax + 2.0 * mean * xmax)))
        bits = select_exact(W, ldw, r, j0, N, w.rowsum, w.colsum, xnorm, mean, sd);
    }
    double at = 0.0;
#pragma unroll
    for (int c = 0; c < 8; ++c) at += (bits >> c) & 1u ? a[c] : 0.0;
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      const uint32_t vw = p == 0 ? v.x : (p == 1 ? v.y : (p == 2 ? v.z : v.w));
      const uint32_t msk = ((bits >> (2 * p)) & 1u) * 0x7FFFu + ((bits >> (2 * p + 1)) & 1u) * 0x7FFF0000u;
      cm[p] = __vmaxu2(cm[p], vw & msk);
    }
#pragma unroll
    for (int d = 8; d > 0; d >>= 1) at += __shfl_xor_sync(0xFFFFFFFFu, at, d);
    if (live) {
      keep[(size_t)r * ngrp + blockIdx.x * 32 + lane] = (uint8_t)bits;
      if ((lane & 15) == 0) w.atot[(size_t)r * nblk + blockIdx.x * 2 + (lane >> 4)] = at;
    }
  }
#pragma unroll
  for (int p = 0; p < 4; ++p) cmax[warp][p][lane] = cm[p];
  __syncthreads();
  if (warp < 4) {
    uint32_t x = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) x = __vmaxu2(x, cmax[k][warp][lane]);
    if (live) { atomicMax(w.colmax + j0 + 2 * warp, x & 0xFFFFu); atomicMax(w.colmax + j0 + 2 * warp + 1, x >> 16); }
  }
}

// How far the definition's error of a candidate (K rounded terms per row, added row by row) and its parallel counterpart
// Q - gain can be apart, both sides of a comparison together: below (16 n + 64) 2^-53 of the block's sum of squares.
__device__ __forceinline__ double filter_window(double q, int n) { return (16.0 * n + 64.0) * kUlp * q; }

// ---- Algorithm 2, Salient: how many of the 32 best columns of a block to take ----------------------------------------
// Error of taking the first i candidates: sum over rows of two binary errors q - a^2 / k.  The q of both sets add up to
// the row's whatever i is, so the filter compares the gains a1^2 / k1 + a0^2 / k0 (larger is better).  CTA: one block
// of columns x 128 rows, one row per thread; a row's sums grow by one column per candidate.
constexpr int kSalThreads = 128, kSalPitch = 65;     // words per staged row: odd, so that a column of rows is conflict-free
__device__ __noinline__ double salient_exact(const __half* W, size_t ldw, int n, int m, const uint8_t* keep, const int* order, int b, int i) {
  const int lane = threadIdx.x & 31, ngrp = m / kM;
  double err = 0.0;
  for (int r0 = 0; r0 < n; r0 += 32) {
    double e = 0.0;
    const int r = r0 + lane;
    if (r < n) {
      double q0 = 0, q1 = 0, a0 = 0, a1 = 0;
      int k0 = 0, k1 = 0;
      for (int c = 0; c < kBeta; ++c) {
        const int j = b * kBeta + c;
        if (!kept_at(keep, ngrp, r, j)) continue;
        bool sal = false;
        for (int t = 0; t < i; ++t) sal = sal || order[t] == c;
        const double aw = fabs(w_at(W, ldw, r, j));
        if (sal) { q1 += aw * aw; a1 += aw; ++k1; } else { q0 += aw * aw; a0 += aw; ++k0; }
      }
      e = __dadd_rn(binary_error(q1, a1, k1), binary_error(q0, a0, k0));
    }
    for (int l = 0; l < 32 && r0 + l < n; ++l) err = __dadd_rn(err, __shfl_sync(0xFFFFFFFFu, e, l));
  }
  return err;
}
// A NaN score comes after all others, so that the ranks are a permutation whatever the norms are: every place of the
// candidates' order is filled, with a column.
__device__ __forceinline__ double column_score(double xn, double lambda, double squares) {
  const double sc = __dmul_rn(__dadd_rn(__dmul_rn(__dmul_rn(2.0, xn), xn), lambda), squares);
  return sc == sc ? sc : -INFINITY;
}
// the definition's sum of squares of a column: row by row (a square is exact, the sum is not)
__device__ __noinline__ double column_squares(const __half* W, size_t ldw, int n, int j) {
  double q = 0.0;
  for (int i = 0; i < n; i += 8) {
    double v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = i + k < n ? w_at(W, ldw, i + k, j) : 0.0;
#pragma unroll
    for (int k = 0; k < 8; ++k) q = __dadd_rn(q, v[k] * v[k]);
  }
  return q;
}
// 0.01 mean_j h_jj, h_jj = 2 ||X_:,j||^2, summed in column order
__device__ __noinline__ double definition_lambda(const double* xnorm, int m) {
  double h = 0.0;
  for (int j = 0; j < m; j += 8) {          // (m is a multiple of 128)
    double v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = xnorm[j + k];
#pragma unroll
    for (int k = 0; k < 8; ++k) h = __dadd_rn(h, __dmul_rn(__dmul_rn(2.0, v[k]), v[k]));
  }
  return __ddiv_rn(__dmul_rn(0.01, h), (double)m);
}
__device__ __noinline__ int rank_among(const double* score, int c) {
  int rank = 0;
  for (int a = 0; a < kBeta; ++a) rank += (score[a] > score[c] || (score[a] == score[c] && a < c)) ? 1 : 0;
  return rank;
}
template <bool kVec>
__global__ void __launch_bounds__(kSalThreads) salient_kernel(const __half* __restrict__ W, size_t ldw, int n, int m, int N, const uint8_t* __restrict__ keep,
                                                              const double* __restrict__ xnorm, double lambda_in, Ws w, uint64_t* __restrict__ salient) {
  __shared__ __align__(16) uint32_t tile[kSalThreads * kSalPitch];   // per weight: |w| bits, bit 15 = kept; later the gains
  __shared__ double score[kBeta], ranked[kBeta], inv[kBeta + 1], exact[kMaxSal];
  __shared__ int order[kMaxSal];
  __shared__ uint32_t flag, maybe;
  const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ngrp = m / kM, nblk = m / kBeta;
  {
    // candidate order: column score (h_jj + lambda) sum_i W_ij^2, ties to the lower column
    const int j = b * kBeta + tid;
    double sc = column_score(xnorm[j], w.scalars[2], w.colsq[j]);
    score[tid] = sc;
    inv[tid + 1] = 1.0 / (double)(tid + 1);
    if (tid == 0) inv[0] = 0.0;
    __syncthreads();
    // The sums of squares are rounded, in the order in which sums_kernel's CTAs came by: within n ulp of the exact sum, as is
    // the definition's row by row; the sum behind a default lambda likewise within m ulp.  Two scores further apart than both
    // can move are in the definition's order; the columns of closer ones (duplicated columns, as a rule) are summed again,
    // row by row, and lambda column by column.  Two zeros are exact.
    const double window = (4.0 * ((double)n + m) + 64.0) * kUlp;
    int rank = 0;
    for (int a = 0; a < kBeta; ++a) rank += (score[a] > sc || (score[a] == sc && a < tid)) ? 1 : 0;
    ranked[rank] = sc;
    __syncthreads();
    // (of scores within rounding of one another, those next to each other in rank are)
    auto near = [&](double hi, double lo) { return hi != 0.0 && !(hi - lo > window * hi); };
    const bool close = (rank > 0 && near(ranked[rank - 1], sc)) || (rank < kBeta - 1 && near(sc, ranked[rank + 1]));
    if (__syncthreads_or(close)) {
      if (tid == 0) exact[0] = lambda_in < 0.0 ? definition_lambda(xnorm, m) : lambda_in;
      __syncthreads();
      if (close) score[tid] = column_score(xnorm[j], exact[0], column_squares(W, ldw, n, j));
      __syncthreads();
      rank = rank_among(score, tid);
    }
    if (rank < kMaxSal) order[rank] = tid;
  }
  double acc[kMaxSal];
#pragma unroll
  for (int i = 0; i < kMaxSal; ++i) acc[i] = 0.0;
  const uint16_t* row = reinterpret_cast<const uint16_t*>(tile) + tid * (2 * kSalPitch);
  for (int r0 = blockIdx.y * kSalThreads; r0 < n; r0 += gridDim.y * kSalThreads) {
    __syncthreads();
    // a warp stages its own 32 rows, two rows (16 lanes x 8 columns) at a time
#pragma unroll 4
    for (int k = 0; k < 16; ++k) {
      const int tr = 32 * warp + 2 * k + (lane >> 4), r = r0 + tr, piece = lane & 15;
      uint4 v = make_uint4(0, 0, 0, 0);
      uint32_t kb = 0;
      if (r < n) { v = load8<kVec>(W + (size_t)r * ldw + b * kBeta + 8 * piece); kb = keep[(size_t)r * ngrp + b * 16 + piece]; }
      uint32_t* d = tile + tr * kSalPitch + 4 * piece;
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        const uint32_t vw = p == 0 ? v.x : (p == 1 ? v.y : (p == 2 ? v.z : v.w));
        d[p] = (vw & 0x7FFF7FFFu) | (((kb >> (2 * p)) & 1u) << 15) | (((kb >> (2 * p + 1)) & 1u) << 31);
      }
    }
    __syncthreads();
    if (r0 + tid < n) {
      const double at = w.atot[(size_t)(r0 + tid) * nblk + b];
      double a1 = 0.0;
      int k1 = 0;
#pragma unroll
      for (int i = 0; i < kMaxSal; ++i) {
        const uint32_t h = row[order[i]];
        if (h & 0x8000u) { a1 += abs_of(h & 0x7FFFu); ++k1; }
        const double a0 = at - a1;
        acc[i] += a1 * a1 * inv[k1] + a0 * a0 * inv[max(16 * N - k1, 0)];      // (groups of NaN scores keep more than N)
      }
    }
  }
  __syncthreads();
  // the CTA's gains, summed over its threads: 32 x 128 doubles in the tile's place
  double* red = reinterpret_cast<double*>(tile);
#pragma unroll
  for (int i = 0; i < kMaxSal; ++i) red[i * kSalThreads + tid] = acc[i];
  __syncthreads();
  for (int i = warp; i < kMaxSal; i += kSalThreads / 32) {
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < kSalThreads / 32; ++k) s += red[i * kSalThreads + 32 * k + lane];
    s = warp_sum(s);
    if (lane == 0) atomicAdd(w.sgain + b * kMaxSal + i, s);
  }
  if (!last_arrival(w.count + 2 + b, gridDim.y, &flag)) return;
  // the last CTA of the block decides
  if (warp == 0) {
    double q = 0.0;
    for (int c = lane; c < kBeta; c += 32) q += w.colsq[b * kBeta + c];
    q = warp_sum(q);
    const double g = __ldcg(w.sgain + b * kMaxSal + lane);
    double best = g;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) best = fmax(best, __shfl_xor_sync(0xFFFFFFFFu, best, d));
    const uint32_t in = __ballot_sync(0xFFFFFFFFu, !(g < best - filter_window(q, n)));
    if (lane == 0) maybe = in;
  }
  __syncthreads();
  const uint32_t cand = maybe;
  if (__popc(cand) > 1) {
    for (int i = warp; i < kMaxSal; i += kSalThreads / 32)
      if ((cand >> i) & 1u) {
        const double e = salient_exact(W, ldw, n, m, keep, order, b, i + 1);
        if (lane == 0) exact[i] = e;
      }
    __syncthreads();
  }
  int ns = 0;
  if (__popc(cand) == 1) ns = __ffs(cand);
  else {
    double best = INFINITY;
    for (int i = 0; i < kMaxSal; ++i)
      if (((cand >> i) & 1u) && exact[i] < best) { best = exact[i]; ns = i + 1; }
  }
  bool sal = false;
  for (int t = 0; t < ns; ++t) sal = sal || order[t] == tid;
  w.salflag[b * kBeta + tid] = sal ? 1 : 0;
  const uint32_t bal = __ballot_sync(0xFFFFFFFFu, sal);
  if (lane == 0) reinterpret_cast<uint32_t*>(score)[warp] = bal;
  __syncthreads();
  if (tid < 2) salient[2 * b + tid] = (uint64_t)reinterpret_cast<uint32_t*>(score)[2 * tid] | ((uint64_t)reinterpret_cast<uint32_t*>(score)[2 * tid + 1] << 32);
}

// ---- Algorithm 2, NonSalientAwareQuant: break-point search ---------------------------------------------------------
// Grid point t: p1 = (0.1 + 0.8 t / 159) max, p2 = 2 p1, taken while p2 <= 0.9 max: t < kPoints (p2 = 0.894 max at t = 69 and
// 0.904 max at t = 70).  With max = 0 every error is 0 and the first point stands.
__device__ __forceinline__ void grid_point(int t, double mx, double& p1, double& p2) {
  const double frac = __dadd_rn(0.1, __ddiv_rn(__dmul_rn(0.9 - 0.1, (double)t), (double)(kGrid - 1)));
  p1 = __dmul_rn(frac, mx);
  p2 = __dmul_rn(2.0, p1);
}
// the largest fp16 value <= p (p >= 0), as bits: for fp16 |w|,  |w| > p  is  bits(|w|) > floor_bits(p)
__device__ __forceinline__ uint32_t floor_bits(double p) {
  const __half h = __double2half(p);
  uint32_t b = __half_as_ushort(h);
  if (b > 0u && (double)__half2float(h) > p) --b;
  return b;
}
// the definition's error of one grid point, all lanes of a warp together
__device__ __noinline__ double break_exact(const __half* W, size_t ldw, int n, int m, const uint8_t* keep, const uint8_t* sal, int b, double p1, double p2) {
  const int lane = threadIdx.x & 31, ngrp = m / kM;
  double err = 0.0;
  for (int r0 = 0; r0 < n; r0 += 32) {
    double e[3] = {0, 0, 0};
    const int r = r0 + lane;
    if (r < n) {
      double q[3] = {0, 0, 0}, a[3] = {0, 0, 0};
      int k[3] = {0, 0, 0};
      for (int c = 0; c < kBeta; ++c) {
        const int j = b * kBeta + c;
        if (sal[c] || !kept_at(keep, ngrp, r, j)) continue;
        const double aw = fabs(w_at(W, ldw, r, j));
        const int reg = aw > p2 ? 2 : (aw > p1 ? 1 : 0);
#pragma unroll
        for (int g = 0; g < 3; ++g)
          if (g == reg) { q[g] += aw * aw; a[g] += aw; ++k[g]; }
      }
#pragma unroll
      for (int g = 0; g < 3; ++g) e[g] = binary_error(q[g], a[g], k[g]);
    }
    for (int l = 0; l < 32 && r0 + l < n; ++l)
#pragma unroll
      for (int g = 0; g < 3; ++g) err = __dadd_rn(err, __shfl_sync(0xFFFFFFFFu, e[g], l));
  }
  return err;
}

// The filter again compares gains, here a^2 / k summed over the three regions.  A warp takes 32 rows, one per lane.  A
// weight's bin is the number of the 140 thresholds (p1 and p2 of every point) below it, one table look-up by its fp16 code, and
// the sums above a threshold are suffix sums over the bins.  A bin holds the sum and the count in ONE float64: every
// weight adds |w| + K, K a power of two at least 512 x the block's largest weight, so that the sum (below K / 4) and the
// count come apart again by rounding to a multiple of K; both stay exact while the largest weight is below 2^13 (beyond that,
// weights no layer has, the definition decides alone).  The bins of a warp are lane-minor, so that 32 lanes in 32 different
// bins never conflict; they fill the shared memory (35 KB per warp), which leaves six warps per SM: the loop is bound by
// issue and latency of its read-modify-writes, so it has no branches (a dropped weight adds 0) and runs two columns at a time.
constexpr int kBrkWarps = 6, kBrkThreads = 32 * kBrkWarps, kTabMax = 4096, kBins = 2 * kPoints + 1;
struct BreakSmem {
  static constexpr uint32_t hist = 0;                                             // per warp: [kBins][32] x 8 B
  static constexpr uint32_t hist_warp = (uint32_t)kBins * 32u * 8u;
  static constexpr uint32_t tab = hist + kBrkWarps * hist_warp;                   // bin by fp16 code
  static constexpr uint32_t inv = tab + 2u * kTabMax;                             // 1 / k
  static constexpr uint32_t misc = inv + 8u * (kBeta + 2);                        // thresholds, scan, flags
  static constexpr uint32_t sal = misc + 12u * kPoints + 64u;
  static constexpr uint32_t total = sal + kBeta;
};
static_assert(BreakSmem::total <= 232448 && BreakSmem::sal % 8 == 0, "one CTA per SM");

template <bool kVec>
__global__ void __launch_bounds__(kBrkThreads, 1) break_kernel(const __half* __restrict__ W, size_t ldw, int n, int m, const uint8_t* __restrict__ keep, Ws w) {
  extern __shared__ __align__(16) uint8_t smem[];
  const int b = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, ngrp = m / kM, nblk = m / kBeta;
  uint32_t* tab32 = reinterpret_cast<uint32_t*>(smem + BreakSmem::tab);
  const uint16_t* tab = reinterpret_cast<const uint16_t*>(smem + BreakSmem::tab);
  double* inv = reinterpret_cast<double*>(smem + BreakSmem::inv);
  uint32_t* thr = reinterpret_cast<uint32_t*>(smem + BreakSmem::misc);             // [2][kPoints]
  uint32_t* word = thr + 2 * kPoints;                                              // [0..7] scan, [8] flag, [9..11] candidates, [12] max
  uint32_t* pos = word + 16;                                                       // first bin above p1 | above p2 << 16, in bytes / 256
  uint8_t* sal = smem + BreakSmem::sal;
  __shared__ uint8_t nonsal[16];                                                   // a bit per column of the block that is not salient
  if (tid < 16) word[tid] = 0;
  __syncthreads();
  if (tid < kBeta) {
    const uint8_t f = w.salflag[b * kBeta + tid];
    sal[tid] = f;
    inv[tid + 1] = 1.0 / (double)(tid + 1);
    if (!f) atomicMax(word + 12, w.colmax[b * kBeta + tid]);
  }
  if (tid == 0) inv[0] = 0.0;
  if (tid < 16) {
    uint32_t x = 0;
    for (int c = 0; c < 8; ++c) x |= w.salflag[b * kBeta + 8 * tid + c] ? 0u : 1u << c;
    nonsal[tid] = (uint8_t)x;
  }
  for (int i = tid; i < kTabMax / 2; i += kBrkThreads) tab32[i] = 0;
  __syncthreads();
  const double mx = abs_of(word[12]);
  if (mx == 0.0) {                                     // the same for all CTAs of the block
    if (blockIdx.x == 0 && tid == 0) { w.bp[2 * b] = 0.0; w.bp[2 * b + 1] = 0.0; }
    return;
  }
  if (tid < kPoints) {
    double p1, p2;
    grid_point(tid, mx, p1, p2);
    thr[tid] = floor_bits(p1); thr[kPoints + tid] = floor_bits(p2);
  }
  __syncthreads();
  // Table over the fp16 codes from the first p1 threshold to just above the last p2 threshold (a range of 8.95 x: under 3400
  // codes): marks at the thresholds, then a running sum.
  const uint32_t code0 = thr[0];
  const uint32_t last = min(thr[2 * kPoints - 1] - code0 + 1u, (uint32_t)kTabMax - 1u);
  if (tid < 2 * kPoints) {
    const uint32_t idx = min(thr[tid] - code0 + 1u, last);
    atomicAdd(tab32 + (idx >> 1), 1u << (16 * (idx & 1)));
  }
  if (tid < kPoints) {
    uint32_t b1 = 0, b2 = 0;
    for (int i = 0; i < 2 * kPoints; ++i) { b1 += thr[i] <= thr[tid] ? 1u : 0u; b2 += thr[i] <= thr[kPoints + tid] ? 1u : 0u; }
    pos[tid] = b1 | (b2 << 16);
  }
  __syncthreads();
  {
    constexpr int kPer = (kTabMax / 2 + kBrkThreads - 1) / kBrkThreads;          // words (two entries) per thread
    uint32_t s = 0;
    for (int k = 0; k < kPer; ++k) {
      const int i = tid * kPer + k;
      if (i < kTabMax / 2) s += (tab32[i] & 0xFFFFu) + (tab32[i] >> 16);
    }
    uint32_t incl = s;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) { const uint32_t o = __shfl_up_sync(0xFFFFFFFFu, incl, d); if (lane >= d) incl += o; }
    if (lane == 31) word[warp] = incl;
    __syncthreads();
    uint32_t run = incl - s;
    for (int k = 0; k < warp; ++k) run += word[k];
    for (int k = 0; k < kPer; ++k) {
      const int i = tid * kPer + k;
      if (i < kTabMax / 2) {
        const uint32_t v = tab32[i], e0 = run + (v & 0xFFFFu), e1 = e0 + (v >> 16);
        tab32[i] = e0 | (e1 << 16);
        run = e1;
      }
    }
  }
  __syncthreads();

  // K and the constant that rounds a sum below 2^52 K to a multiple of K and leaves the count in the low word
  const double K = __hiloint2double((__double2hiint(mx) & 0x7FF00000) + (10 << 20), 0), magic = K * 0x1.8p52;
  double* h = reinterpret_cast<double*>(smem + BreakSmem::hist + warp * BreakSmem::hist_warp) + lane;
  double acc[kPoints];
#pragma unroll
  for (int t = 0; t < kPoints; ++t) acc[t] = 0.0;
  const int groups = (n + 31) / 32;
  for (int gr = blockIdx.x * kBrkWarps + warp; gr < groups; gr += gridDim.x * kBrkWarps) {
    const int r = gr * 32 + lane;
#pragma unroll 10
    for (int t = 0; t < kBins; ++t) h[32 * t] = 0.0;
    if (r < n) {
      const __half* wr = W + (size_t)r * ldw + b * kBeta;
      const uint8_t* kr = keep + (size_t)r * ngrp + b * 16;
      uint4 vn = load8<kVec>(wr);
      uint32_t kn = kr[0];
#pragma unroll 1
      for (int g = 0; g < 16; ++g) {
        const uint4 v = vn;
        const uint32_t kb = kn & nonsal[g];
        if (g < 15) { vn = load8<kVec>(wr + 8 * (g + 1)); kn = kr[g + 1]; }
#pragma unroll
        for (int c = 0; c < 8; c += 2) {
          double one[2];
          uint32_t bin[2];
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const uint32_t bits = half_bits(v, c + e) & 0x7FFFu;
            one[e] = (kb >> (c + e)) & 1u ? __fma_rn(__hiloint2double((int)(bits << 10), 0), 0x1p1008, K) : 0.0;
            bin[e] = 32u * tab[min(max(bits, code0) - code0, last)];
          }
          // both columns' bins are read before either is written; where they are the same bin the second sum has both
          const double x0 = h[bin[0]] + one[0], x1 = (bin[0] == bin[1] ? x0 : h[bin[1]]) + one[1];
          h[bin[0]] = x0;
          h[bin[1]] = x1;
        }
      }
    }
    double run = 0.0;                                  // suffix sums, in place
#pragma unroll 14
    for (int f = kBins - 1; f >= 0; --f) { run += h[32 * f]; h[32 * f] = run; }
    // (sum, count) of what lies above p1 and above p2, and of everything
    auto part = [&](double x, double& a, int& k) { const double m = x + magic; k = __double2loint(m); a = x - (m - magic); };
    double at, a12, a2;
    int kt, k12, k2;
    part(run, at, kt);
#pragma unroll
    for (int t = 0; t < kPoints; ++t) {
      const uint32_t ps = pos[t];
      part(h[32 * (ps & 0xFFFFu)], a12, k12);
      part(h[32 * (ps >> 16)], a2, k2);
      const double a0 = at - a12, a1 = a12 - a2;
      acc[t] += a0 * a0 * inv[kt - k12] + a1 * a1 * inv[k12 - k2] + a2 * a2 * inv[k2];
    }
  }
  // the warp's gains over its lanes, through its own bins
  __syncwarp();
  double* red = h - lane;
#pragma unroll
  for (int t = 0; t < kPoints; ++t) red[32 * t + lane] = acc[t];
  __syncwarp();
  for (int t = lane; t < kPoints; t += 32) {
    double s = 0.0;
    for (int l = 0; l < 32; ++l) s += red[32 * t + ((l + lane) & 31)];
    atomicAdd(w.bgain + b * kPoints + t, s);
  }
  if (!last_arrival(w.count + 2 + nblk + b, gridDim.x, word + 8)) return;
  double* gain = reinterpret_cast<double*>(smem);                                  // the bins are free now
  double* exact = gain + kPoints;
  if (warp == 0) {
    double q = 0.0, best = -INFINITY;
    for (int c = lane; c < kBeta; c += 32) q += w.colsq[b * kBeta + c];
    q = warp_sum(q);
    for (int t = lane; t < kPoints; t += 32) { gain[t] = __ldcg(w.bgain + b * kPoints + t); best = fmax(best, gain[t]); }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) best = fmax(best, __shfl_xor_sync(0xFFFFFFFFu, best, d));
    for (int k = 0; k < 3; ++k) {
      const int t = 32 * k + lane;
      const uint32_t in = __ballot_sync(0xFFFFFFFFu, t < kPoints && (mx >= 0x1p13 || !(gain[min(t, kPoints - 1)] < best - filter_window(q, n))));
      if (lane == 0) word[9 + k] = in;
    }
  }
  __syncthreads();
  const uint32_t c0 = word[9], c1 = word[10], c2 = word[11];
  const int many = __popc(c0) + __popc(c1) + __popc(c2);
  auto is_cand = [&](int t) { return (((t < 32 ? c0 : (t < 64 ? c1 : c2)) >> (t & 31)) & 1u) != 0u; };
  if (many > 1) {
    int k = 0;
    for (int t = 0; t < kPoints; ++t)
      if (is_cand(t) && (k++ % kBrkWarps) == warp) {
        double p1, p2;
        grid_point(t, mx, p1, p2);
        const double e = break_exact(W, ldw, n, m, keep, sal, b, p1, p2);
        if (lane == 0) exact[t] = e;
      }
    __syncthreads();
  }
  if (tid == 0) {
    double best = INFINITY, p1s = 0.0, p2s = 0.0;
    for (int t = 0; t < kPoints; ++t)
      if (is_cand(t) && (many == 1 || exact[t] < best)) { if (many > 1) best = exact[t]; grid_point(t, mx, p1s, p2s); }
    w.bp[2 * b] = p1s; w.bp[2 * b + 1] = p2s;
  }
}

// ---- Trisection, Res_Approx and the logical arrays: one thread per (row, block), loops in column order ----------------
// A row of a block that may keep an infinite or NaN weight: the definition's own comparisons and sums.
__device__ __noinline__ void emit_non_finite(const __half* wr, const uint8_t* kr, const uint8_t* sal, double p1, double p2, uint8_t* sign, uint16_t* region,
                                             uint32_t* sign2, uint16_t* scale) {
  double a[4] = {0, 0, 0, 0}, alpha[5], ar = 0.0;
  int k[4] = {0, 0, 0, 0}, ts = 0;
  uint32_t s2 = 0;
  auto region_of = [&](int c, double aw) { return sal[c] ? 3 : (aw > p2 ? 2 : (aw > p1 ? 1 : 0)); };
  for (int c = 0; c < kBeta; ++c)
    if ((kr[c >> 3] >> (c & 7)) & 1u) {
      const double aw = fabs((double)__half2float(wr[c]));
      const int reg = region_of(c, aw);
      for (int g = 0; g < 4; ++g)
        if (g == reg) { a[g] = __dadd_rn(a[g], aw); ++k[g]; }
    }
  for (int g = 0; g < 4; ++g) alpha[g] = k[g] ? __ddiv_rn(a[g], (double)k[g]) : 0.0;
  for (int c = 0; c < kBeta; ++c) {
    if (!sal[c]) continue;
    if ((kr[c >> 3] >> (c & 7)) & 1u) {
      const double w = (double)__half2float(wr[c]), d = __dsub_rn(w, __dmul_rn(alpha[3], w >= 0.0 ? 1.0 : -1.0));
      ar = __dadd_rn(ar, fabs(d));
      if (d >= 0.0) s2 |= 1u << ts;
    }
    ++ts;
  }
  alpha[4] = k[3] ? __ddiv_rn(ar, (double)k[3]) : 0.0;
  for (int q = 0; q < 5; ++q) scale[q] = __half_as_ushort(__double2half(alpha[q]));
  *sign2 = s2;
  for (int g = 0; g < 16; ++g) {
    uint32_t rank = 0, sv = 0, rv = 0;
    for (int c = 8 * g; c < 8 * g + 8; ++c)
      if ((kr[g] >> (c & 7)) & 1u) {
        const double w = (double)__half2float(wr[c]);
        sv |= (w >= 0.0 ? 1u : 0u) << rank;
        rv |= (uint32_t)region_of(c, fabs(w)) << (2u * rank);
        ++rank;
      }
    sign[g] = (uint8_t)sv; region[g] = (uint16_t)rv;
  }
}
template <bool kVec>
__global__ void __launch_bounds__(128) emit_kernel(const __half* __restrict__ W, size_t ldw, int n, int m, const uint8_t* __restrict__ keep, Ws w,
                                                   uint8_t* __restrict__ sign, uint16_t* __restrict__ region, uint32_t* __restrict__ sign2,
                                                   uint16_t* __restrict__ scale) {
  __shared__ uint32_t salw[4];                          // salient columns of the block, one bit each
  const int nblk = m / kBeta, ngrp = m / kM, b = blockIdx.x, r = blockIdx.y * 128 + threadIdx.x;
  {
    const uint32_t bal = __ballot_sync(0xFFFFFFFFu, w.salflag[b * kBeta + threadIdx.x] != 0);
    if ((threadIdx.x & 31) == 0) salw[threadIdx.x >> 5] = bal;
  }
  __syncthreads();
  if (r >= n) return;
  const uint32_t t1 = floor_bits(w.bp[2 * b]), t2 = floor_bits(w.bp[2 * b + 1]);
  const __half* wr = W + (size_t)r * ldw + b * kBeta;
  const uint8_t* kr = keep + (size_t)r * ngrp + b * 16;
  double above2 = 0.0, above1 = 0.0, all = 0.0, asal = 0.0;      // exact sums: above the second threshold, the first, all, salient
  int k2 = 0, k1 = 0, k0 = 0, ks = 0;
#pragma unroll 2
  for (int g = 0; g < 16; ++g) {
    const uint4 v = load8<kVec>(wr + 8 * g);
    const uint32_t sb = (salw[g >> 2] >> (8 * (g & 3))) & 0xFFu, kb = kr[g];
    uint32_t m1 = 0, m2 = 0;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const uint32_t bits = half_bits(v, c) & 0x7FFFu;
      const double aw = abs_of(bits);
      if ((sb >> c) & 1u) {                                      // (the same column for all lanes)
        if ((kb >> c) & 1u) asal += aw;
      } else {
        const bool kp = (kb >> c) & 1u, g1 = kp && bits > t1, g2 = kp && bits > t2;
        if (kp) all += aw;
        if (g1) { above1 += aw; m1 |= 1u << c; }
        if (g2) { above2 += aw; m2 |= 1u << c; }
      }
    }
    k2 += __popc(m2); k1 += __popc(m1); k0 += __popc(kb & ~sb); ks += __popc(kb & sb);
  }
  const size_t rb = (size_t)r * nblk + b;
  if (all + asal >= kInfiniteCode) {
    emit_non_finite(wr, kr, w.salflag + b * kBeta, w.bp[2 * b], w.bp[2 * b + 1], sign + (size_t)r * ngrp + b * 16, region + (size_t)r * ngrp + b * 16, sign2 + rb,
                    scale + rb * 5);
    return;
  }
  double alpha[5];
  const double set[4] = {all - above1, above1 - above2, above2, asal};
  const int cnt[4] = {k0 - k1, k1 - k2, k2, ks};
#pragma unroll
  for (int q = 0; q < 4; ++q) alpha[q] = cnt[q] ? __ddiv_rn(set[q], (double)cnt[q]) : 0.0;
  // residual of the salient weights, in column order: w - alpha sgn(w) is +-(|w| - alpha)
  double ar = 0.0;
  int ts = 0;
  uint32_t s2 = 0;
#pragma unroll 1
  for (int q = 0; q < 4; ++q)
    for (uint32_t rest = salw[q]; rest; rest &= rest - 1u, ++ts) {
      const int c = 32 * q + __ffs(rest) - 1;
      if (!((kr[c >> 3] >> (c & 7)) & 1u)) continue;
      const uint32_t h = __half_as_ushort(wr[c]);
      const double d = __dsub_rn(abs_of(h & 0x7FFFu), alpha[3]);
      ar = __dadd_rn(ar, fabs(d));
      const bool neg = h > 0x8000u;                     // -0 counts as positive
      if (neg ? d <= 0.0 : d >= 0.0) s2 |= 1u << ts;
    }
  alpha[4] = ks ? __ddiv_rn(ar, (double)ks) : 0.0;
#pragma unroll
  for (int q = 0; q < 5; ++q) scale[rb * 5 + q] = __half_as_ushort(__double2half(alpha[q]));
  sign2[rb] = s2;
#pragma unroll 1
  for (int g4 = 0; g4 < 4; ++g4) {
    uint32_t sg = 0, rgw[2] = {0, 0};
#pragma unroll
    for (int gi = 0; gi < 4; ++gi) {
      const int g = 4 * g4 + gi;
      const uint4 v = load8<kVec>(wr + 8 * g);
      const uint32_t kb = kr[g], sb = salw[g4] >> (8 * gi);
      uint32_t rank = 0, sv = 0, rv = 0;
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const uint32_t h = half_bits(v, c), bits = h & 0x7FFFu, kp = (kb >> c) & 1u;
        const uint32_t reg = (sb >> c) & 1u ? 3u : (bits > t2 ? 2u : (bits > t1 ? 1u : 0u));
        sv |= (h > 0x8000u ? 0u : kp) << rank;
        rv |= (kp ? reg : 0u) << (2u * rank);
        rank += kp;
      }
      if (kVec) { sg |= sv << (8 * gi); rgw[gi >> 1] |= rv << (16 * (gi & 1)); }
      else { sign[(size_t)r * ngrp + b * 16 + g] = (uint8_t)sv; region[(size_t)r * ngrp + b * 16 + g] = (uint16_t)rv; }
    }
    if (kVec) {
      *reinterpret_cast<uint32_t*>(sign + (size_t)r * ngrp + b * 16 + 4 * g4) = sg;
      *reinterpret_cast<uint2*>(region + (size_t)r * ngrp + b * 16 + 4 * g4) = make_uint2(rgw[0], rgw[1]);
    }
  }
}

static size_t a256(size_t v) { return (v + 255) & ~(size_t)255; }
static size_t carve(Ws& w, uint8_t* base, int n, int m) {
  const int nblk = m / kBeta;
  size_t o = 0;
  auto take = [&](size_t bytes) { uint8_t* p = base ? base + o : nullptr; o += a256(bytes); return p; };
  w.rowsum = (double*)take(sizeof(double) * n);
  w.colsum = (double*)take(sizeof(double) * m);
  w.colsq = (double*)take(sizeof(double) * m);
  w.sgain = (double*)take(sizeof(double) * nblk * kMaxSal);
  w.bgain = (double*)take(sizeof(double) * nblk * kPoints);
  w.colmax = (uint32_t*)take(sizeof(uint32_t) * m);
  w.count = (uint32_t*)take(sizeof(uint32_t) * (2 + 2 * (size_t)nblk));
  w.zero_end = (uint32_t*)take(0);
  w.rinv = (double*)take(sizeof(double) * n);
  w.cinv = (double*)take(sizeof(double) * m);
  w.atot = (double*)take(sizeof(double) * n * nblk);
  w.partial = (double*)take(sizeof(double) * 2 * kPartials);
  w.scalars = (double*)take(sizeof(double) * 8);
  w.salflag = (uint8_t*)take((size_t)nblk * kBeta);
  w.bp = (double*)take(sizeof(double) * nblk * 2);
  return o;
}

template <bool kVec>
static cudaError_t launch(const __half* W, size_t ldw, const double* xnorm, int n, int m, int N, double lambda, const stb_logical* out, const Ws& w,
                          cudaStream_t s) {
  const int nblk = m / kBeta;
  uint8_t* keep = const_cast<uint8_t*>(out->keep);
  // the shared-memory limit of a kernel is a per-device setting
  static bool attr_done[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64 || !attr_done[dev]) {
    e = cudaFuncSetAttribute(break_kernel<kVec>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)BreakSmem::total);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64) attr_done[dev] = true;
  }
  e = cudaMemsetAsync(w.rowsum, 0, (size_t)(reinterpret_cast<uint8_t*>(w.zero_end) - reinterpret_cast<uint8_t*>(w.rowsum)), s);
  if (e != cudaSuccess) return e;
  const dim3 strips((unsigned)((m + 255) / 256), (unsigned)((n + kRowsPerCta - 1) / kRowsPerCta));
  sums_kernel<kVec><<<strips, 256, 0, s>>>(W, ldw, n, m, w.rowsum, w.colsum, w.colsq);
  const int parts = (n + m + 255) / 256;
  scalars_kernel<<<parts < kPartials ? parts : kPartials, 256, 0, s>>>(n, m, xnorm, lambda, w);
  const long long units = (long long)((m + 255) / 256) * ((n + 15) / 16), wide = (units + 7) / 8;
  spread_kernel<kVec><<<(unsigned)(wide < kPartials ? wide : kPartials), 256, 0, s>>>(W, ldw, n, m, w);
  select_kernel<kVec><<<strips, 256, 0, s>>>(W, ldw, n, m, N, xnorm, w, keep);
  // four or so CTAs per SM in all, each with whole passes of 128 rows
  const int passes = (n + kSalThreads - 1) / kSalThreads;
  int per_block = (148 * 6 + nblk - 1) / nblk;
  if (per_block > passes) per_block = passes;
  salient_kernel<kVec><<<dim3((unsigned)nblk, (unsigned)per_block), kSalThreads, 0, s>>>(W, ldw, n, m, N, keep, xnorm, lambda, w, const_cast<uint64_t*>(out->salient));
  // break_kernel: one CTA per SM; the number of CTAs per block that makes waves x (rounds of 32 rows per warp + a CTA's
  // prologue, worth about half a round) smallest
  const int groups = (n + 31) / 32;
  int best = 1;
  double best_cost = 0.0;
  for (int c = 1; c <= 64 && (c == 1 || (c - 1) * kBrkWarps < groups); ++c) {
    const long long waves = ((long long)nblk * c + 147) / 148;
    const double cost = (double)waves * (0.5 + (double)((groups + c * kBrkWarps - 1) / (c * kBrkWarps)));
    if (c == 1 || cost < best_cost - 1e-9) { best_cost = cost; best = c; }
  }
  break_kernel<kVec><<<dim3((unsigned)best, (unsigned)nblk), kBrkThreads, BreakSmem::total, s>>>(W, ldw, n, m, keep, w);
  emit_kernel<kVec><<<dim3((unsigned)nblk, (unsigned)((n + 127) / 128)), 128, 0, s>>>(W, ldw, n, m, keep, w, const_cast<uint8_t*>(out->sign),
                                                                                      const_cast<uint16_t*>(out->region), const_cast<uint32_t*>(out->sign2),
                                                                                      const_cast<uint16_t*>(out->scale));
  return cudaGetLastError();
}

}  // namespace quant
}  // namespace stb

extern "C" int stb_quantize_workspace(int n, int m, size_t* bytes) {
  if (!bytes) return STB_ERR_ARG;
  if (n < 1 || m < 128 || m % 128 != 0) return STB_ERR_SHAPE;
  stb::quant::Ws w;
  *bytes = stb::quant::carve(w, nullptr, n, m);
  return STB_OK;
}

extern "C" int stb_quantize(const void* W, size_t ldw, const double* xnorm, int n, int m, int N, double lambda,
                            const stb_logical* out, void* ws, size_t ws_bytes, void* stream) {
  using namespace stb::quant;
  if (!W || !xnorm || !out || !ws) return STB_ERR_ARG;
  if (n < 1 || m < 128 || m % 128 != 0) return STB_ERR_SHAPE;
  if (N < 1 || N > 8) return STB_ERR_NM;
  if (ldw < (size_t)m || lambda != lambda) return STB_ERR_ARG;
  if (out->n != n || out->m != m || out->N != N) return STB_ERR_ARG;
  if (!out->keep || !out->sign || !out->region || !out->sign2 || !out->salient || !out->scale) return STB_ERR_ARG;
  Ws w;
  if (ws_bytes < carve(w, static_cast<uint8_t*>(ws), n, m)) return STB_ERR_SIZE;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const __half* Wh = static_cast<const __half*>(W);
  // 16-byte loads of W rows and 4- and 8-byte stores of signs and regions where the addresses allow them
  const bool vec = (reinterpret_cast<uintptr_t>(W) & 15u) == 0 && ldw % 8 == 0 && (reinterpret_cast<uintptr_t>(out->sign) & 3u) == 0 &&
                   (reinterpret_cast<uintptr_t>(out->region) & 7u) == 0;
  const cudaError_t e = vec ? launch<true>(Wh, ldw, xnorm, n, m, N, lambda, out, w, s) : launch<false>(Wh, ldw, xnorm, n, m, N, lambda, out, w, s);
  return e == cudaSuccess ? STB_OK : STB_ERR_CUDA;
}
