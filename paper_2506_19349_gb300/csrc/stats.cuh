// Step statistics of Section 3: highD (degree-weighted split), the
// dynamic-stepping gap of Eq. 1-3 and the traversal-optimisation profit of
// Eq. 4-6 with the clamping of Section 3.2.
#pragma once

#include "common.cuh"

namespace eic {

// highD over a degree multiset given per distinct degree: cnt[r] vertices of
// degree dvals[r] (ascending, >= 1). The threshold t splits the set into
// degrees < t and >= t with the smallest difference of total degree; t ranges
// over the degrees present, ties keep the smaller t, and an empty (zero total
// degree) set gives 0. The total degree is at most 2m < 2^32.
//
// The total degree below a rank, low, grows from present rank to present rank,
// so |total - 2 low| is smallest at the last present rank with 2 low <= total
// or at the next present one: one scan finds the thread whose ranks hold the
// former, and its warp walks that thread's ranks.
//
// In two parts with a block barrier between them and one behind (the caller's,
// so that other work can share them): highd_sums by all threads, at most 1024,
// then highd_cross by all threads; s.highd holds the result.
struct HighdScr {
  uint32_t wsum[32], wfirst[32];  // per warp: total degree, first present rank
  uint32_t highd;
};

struct HighdPart {
  uint32_t lo, hi;   // the thread's ranks
  uint32_t sum;      // their total degree
  uint32_t incl;     // inclusive sum in the warp
  uint32_t first;    // their first present rank
};

static __device__ __forceinline__ HighdPart highd_sums(const uint32_t* cnt, const uint32_t* dvals, uint32_t D,
                                                       HighdScr& s) {
  const uint32_t t = threadIdx.x, lane = t & 31u, per = (D + blockDim.x - 1) / blockDim.x;
  HighdPart p;
  p.lo = min(D, t * per);
  p.hi = min(D, p.lo + per);
  p.sum = 0;
  p.first = 0xFFFFFFFFu;
#pragma unroll 4
  for (uint32_t r = p.lo; r < p.hi; ++r) {
    const uint32_t c = __ldcg(&cnt[r]);
    if (c) p.first = min(p.first, r);
    p.sum += c * __ldg(&dvals[r]);
  }
  p.incl = warp_incl_scan(p.sum);
  const uint32_t f = __reduce_min_sync(EIC_FULL_MASK, p.first);
  if (lane == 31) {
    s.wsum[t >> 5] = p.incl;
    s.wfirst[t >> 5] = f;
  }
  if (t == 0) s.highd = 0;
  return p;
}

static __device__ __forceinline__ void highd_cross(const uint32_t* cnt, const uint32_t* dvals, uint32_t D,
                                                   const HighdPart& p, HighdScr& s) {
  const uint32_t t = threadIdx.x, lane = t & 31u, warp = t >> 5, nw = blockDim.x >> 5;
  const uint32_t all = warp_incl_scan(lane < nw ? s.wsum[lane] : 0u);
  const uint32_t total = __shfl_sync(EIC_FULL_MASK, all, 31);
  const uint32_t before = __shfl_sync(EIC_FULL_MASK, all, warp ? warp - 1 : 0);
  const uint32_t low0 = (warp ? before : 0u) + p.incl - p.sum;
  const bool cross = p.sum && 2ull * low0 <= total && 2ull * ((uint64_t)low0 + p.sum) > total;
  const uint32_t m = __ballot_sync(EIC_FULL_MASK, cross);
  if (!m) return;  // (one thread crosses when total > 0)
  const int src = __ffs(m) - 1;
  const uint32_t lo = __shfl_sync(EIC_FULL_MASK, p.lo, src), hi = __shfl_sync(EIC_FULL_MASK, p.hi, src);
  uint32_t run = __shfl_sync(EIC_FULL_MASK, low0, src);
  uint32_t r1 = 0, low1 = 0, low2 = 0, next = 0xFFFFFFFFu;  // the last rank with 2 low <= total, and the next present one
  for (uint32_t b = lo; b < hi; b += 32) {
    const uint32_t r = b + lane;
    const uint32_t c = r < hi ? __ldcg(&cnt[r]) : 0u;
    const uint32_t x = c ? c * __ldg(&dvals[r]) : 0u, incl = warp_incl_scan(x);
    const uint32_t here = __ballot_sync(EIC_FULL_MASK, c != 0);
    const uint32_t below = __ballot_sync(EIC_FULL_MASK, c != 0 && 2ull * (run + incl - x) <= total);
    uint32_t after = here;
    if (below) {
      const int j = 31 - __clz(below);
      r1 = b + j;
      low2 = run + __shfl_sync(EIC_FULL_MASK, incl, j);
      low1 = low2 - __shfl_sync(EIC_FULL_MASK, x, j);
      next = 0xFFFFFFFFu;
      after = j < 31 ? here & (0xFFFFFFFFu << (j + 1)) : 0u;
    }
    if (after && next == 0xFFFFFFFFu) next = b + __ffs(after) - 1;
    run += __shfl_sync(EIC_FULL_MASK, incl, 31);
  }
  if (next == 0xFFFFFFFFu) {  // in a later thread's ranks
    const uint32_t f = (int)lane > src ? p.first : 0xFFFFFFFFu;
    const uint32_t g = lane > warp && lane < nw ? s.wfirst[lane] : 0xFFFFFFFFu;
    next = __reduce_min_sync(EIC_FULL_MASK, min(f, g));
  }
  if (lane == 0)
    s.highd = dvals[low2 < total && 2ull * low2 - total < (uint64_t)total - 2ull * low1 ? next : r1];
}

// Eq. 1-3. maxW(G, ratio) is read from RtoW at index floor(ratio * (R - 1));
// Eq. 2 is evaluated as -expm1(log1p(-prob) / (prob * highD)). Every
// operation is an explicitly rounded IEEE double operation (no contraction).
__device__ __forceinline__ int64_t dev_gap(uint64_t sumd, uint64_t highd, uint64_t two_m, uint32_t alpha,
                                           double beta, const uint32_t* rtow) {
  const uint32_t R = EIC_RATIO_NUM;
  if (highd <= alpha || two_m == 0) return (int64_t)rtow[R - 1];
  uint64_t big = sumd > two_m - sumd ? sumd : two_m - sumd;
  double frac = __ddiv_rn((double)big, (double)two_m);
  double prob = frac < beta ? frac : beta;
  double ratio = -expm1(__ddiv_rn(log1p(-prob), __dmul_rn(prob, (double)highd)));
  double pos = __dmul_rn(ratio, (double)(R - 1));
  uint32_t idx = pos <= 0.0 ? 0u : (pos >= (double)(R - 1) ? R - 1 : (uint32_t)floor(pos));
  return (int64_t)rtow[idx];
}

// The same by a single-precision estimate of the RtoW position where that
// decides it, or -1. For prob <= 0.95 the estimate is off by less than 0.01:
// prob is off by 3 roundings of 2^-24, which log1p magnifies by at most
// prob / ((1 - prob) |log1p(-prob)|) < 6.4; with its own error, the
// quotient's and expm1's (which damps them) the ratio's relative error stays
// below 2.4e-6, times at most 4095.
__device__ __forceinline__ int64_t dev_gap_quick(uint64_t sumd, uint64_t highd, uint64_t two_m, uint32_t alpha,
                                                 double beta, const uint32_t* rtow) {
  const uint32_t R = EIC_RATIO_NUM;
  if (highd <= alpha || two_m == 0) return (int64_t)__ldg(&rtow[R - 1]);
  const uint64_t big = sumd > two_m - sumd ? sumd : two_m - sumd;
  const float prob = fminf((float)big / (float)two_m, (float)beta);
  if (!(prob <= 0.95f)) return -1;
  const float pos = -expm1f(log1pf(-prob) / (prob * (float)highd)) * (float)(R - 1), whole = floorf(pos);
  if (!(pos - whole > 0.02f && pos - whole < 0.98f)) return -1;
  return (int64_t)__ldg(&rtow[(uint32_t)whole]);
}

// Profit of candidate x for the next pair <lb, y> (Section 3.2):
//   x' = max(x, lb - maxW), ub0 = min(y, lb + maxW), ub1 = min(y, x' + maxW),
//   dsum = sumD(x') - sumD(lb),
//   pushed = (ub0 - lb) dsum / maxW, pulled = (ub1 - x') sumD(lb) / maxW,
//   long = pulled dsum / 2|E|,  profit = pushed - long - pulled.
__device__ __forceinline__ double dev_profit(int64_t x, int64_t lb, int64_t y, uint64_t dsum, uint64_t sumd_lb,
                                             uint32_t maxw, uint64_t two_m) {
  int64_t xc = x > lb - (int64_t)maxw ? x : lb - (int64_t)maxw;
  int64_t ub0 = y < lb + (int64_t)maxw ? y : lb + (int64_t)maxw;
  int64_t ub1 = y < xc + (int64_t)maxw ? y : xc + (int64_t)maxw;
  double pushed = __ddiv_rn(__dmul_rn((double)(ub0 - lb), (double)dsum), (double)maxw);
  double pulled = __ddiv_rn(__dmul_rn((double)(ub1 - xc), (double)sumd_lb), (double)maxw);
  double lng = __ddiv_rn(__dmul_rn(pulled, (double)dsum), (double)two_m);
  return __dsub_rn(__dsub_rn(pushed, lng), pulled);
}

}  // namespace eic
