// Window searches in a weight-sorted row [b, e) of the adjacency. The weight of
// entry i is read by a functor w(i), so that the index arithmetic compiles and
// can be checked without a GPU. Offsets are 32-bit and reach 2^32 - 2 (2m at
// the largest accepted graph): nothing is added to an offset that could wrap.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define EIC_HD __host__ __device__ __forceinline__
#else
#define EIC_HD inline
#endif

namespace eic {

// first index in [b, e) with weight >= t, or e
template <class W>
EIC_HD uint32_t lower_bound(const W& w, uint32_t b, uint32_t e, int64_t t) {
  if (t <= 1) return b;  // weights are >= 1
  while (b < e) {
    const uint32_t mid = b + ((e - b) >> 1);
    if ((int64_t)w(mid) < t)
      b = mid + 1;
    else
      e = mid;
  }
  return b;
}

// The same, given that the weight at lo is < t: exponential probes forward
// from lo, then a binary search in the last interval.
template <class W>
EIC_HD uint32_t gallop_past(const W& w, uint32_t lo, uint32_t e, int64_t t) {
  uint32_t hi;
  uint64_t step = 1;
  for (;;) {
    const uint64_t h = (uint64_t)lo + step;
    if (h >= e) {
      hi = e;
      break;
    }
    if ((int64_t)w((uint32_t)h) >= t) {
      hi = (uint32_t)h;
      break;
    }
    lo = (uint32_t)h;
    step <<= 1;
  }
  return lower_bound(w, lo + 1, hi, t);
}

// The same, given that every entry before p has weight < t. Costs O(log
// distance), and a short window costs one or two probes of one sector.
template <class W>
EIC_HD uint32_t gallop(const W& w, uint32_t p, uint32_t e, int64_t t) {
  if (t <= 1 || p >= e) return p;
  if ((int64_t)w(p) >= t) return p;
  return gallop_past(w, p, e, t);
}

// The same for windows that mostly end within four entries: the weights of the
// first four are read at once. (RMAT 2^25 2779 -> 2730 us, 15 M log-normal
// 1885 -> 1863 us; a window's average length there is 1.3 entries.)
template <class W>
EIC_HD uint32_t gallop4(const W& w, uint32_t p, uint32_t e, int64_t t) {
  if (t <= 1 || p >= e) return p;
  const uint32_t n = e - p;  // (p + k itself may wrap at the end of the largest adjacency)
  uint32_t x[4], c = 0;
#pragma unroll
  for (uint32_t k = 0; k < 4; ++k) x[k] = k < n ? w(p + k) : 0xFFFFFFFFu;
#pragma unroll
  for (uint32_t k = 0; k < 4; ++k) c += k < n && (int64_t)x[k] < t ? 1u : 0u;
  if (c < 4) return p + c;
  return gallop_past(w, p + 3, e, t);
}

}  // namespace eic
