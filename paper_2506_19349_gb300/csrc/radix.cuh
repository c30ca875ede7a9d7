// Device sort and scan primitives used by the CSR builder.
//
// LSD radix sort of 64-bit keys (optionally with 32-bit values) over a range of
// key bits, at most 9 bits per pass, in the reduce-then-scan form: a fixed grid
// of blocks each owns one contiguous slice of the input; pass = per-slice digit
// histogram -> exclusive scan of each digit's counts over the slices -> stable
// scatter of each slice in order. A pass is bound by memory (one read of the
// keys for the histogram, one read and one write for the scatter). The scatter
// therefore takes tiles of 4096 elements: it ranks them by digit (warps in
// order, 32-element rows of a warp in order, lanes in order, so it is stable),
// gathers them by digit in shared memory and writes runs of consecutive
// addresses, where a direct scatter writes 8 bytes here and there. Equal
// digits of a warp's row are found by a ballot per bit: match.any takes one
// instruction but 72% of its pipe's time.
// One pass over 32 M keys: scatter 225 us (2.3 TB/s, bound by instructions:
// 50% issue, most of it the ranking), histogram 45 us, scan 3 us; over 32 M
// pairs before (512-element rounds written directly, one block scanning all
// counts) 680, 50 and 426 us.
#pragma once

#include "common.cuh"

namespace eic {

constexpr int kSortThreads = 512;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kSortItems = 8;                           // elements per thread and tile
constexpr int kSortTile = kSortThreads * kSortItems;
constexpr int kSortBlocksMax = 152 * 2;                 // slices: the two blocks that every SM holds
constexpr int kRadixBits = 9;
constexpr int kRadixDigits = 1 << kRadixBits;

__device__ __forceinline__ uint32_t digit_of(uint64_t k, int shift, uint32_t mask) { return (uint32_t)(k >> shift) & mask; }

// Exclusive sum over a block of at most 1024 threads; s_w: 32 words. Every thread gets the block's total too.
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t x, uint32_t* s_w, uint32_t* total) {
  const uint32_t lane = threadIdx.x & 31u, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const uint32_t incl = warp_incl_scan(x);
  __syncthreads();
  if (lane == 31) s_w[w] = incl;
  __syncthreads();
  const uint32_t all = warp_incl_scan(lane < nw ? s_w[lane] : 0u);
  const uint32_t before = __shfl_sync(EIC_FULL_MASK, all, w ? w - 1 : 0);
  *total = __shfl_sync(EIC_FULL_MASK, all, 31);
  return (w ? before : 0u) + incl - x;
}

__global__ void __launch_bounds__(kSortThreads) k_radix_count(const uint64_t* __restrict__ keys, uint64_t n,
                                                              uint64_t per_block, int shift, uint32_t mask,
                                                              uint32_t* hist) {
  __shared__ uint32_t s_h[kSortWarps / 2][kRadixDigits];  // one table per two warps
  for (uint32_t i = threadIdx.x; i < kSortWarps / 2 * kRadixDigits; i += blockDim.x) (&s_h[0][0])[i] = 0;
  __syncthreads();
  const uint64_t lo = (uint64_t)blockIdx.x * per_block, hi = lo + per_block < n ? lo + per_block : n;
  uint32_t* h = s_h[threadIdx.x >> 6];
  uint64_t i = lo + threadIdx.x;
  for (; i + 3 * kSortThreads < hi; i += 4 * kSortThreads) {
    uint64_t k[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) k[j] = keys[i + j * kSortThreads];
#pragma unroll
    for (int j = 0; j < 4; ++j) atomicAdd(&h[digit_of(k[j], shift, mask)], 1u);
  }
  for (; i < hi; i += kSortThreads) atomicAdd(&h[digit_of(keys[i], shift, mask)], 1u);
  __syncthreads();
  for (uint32_t d = threadIdx.x; d <= mask; d += blockDim.x) {
    uint32_t s = 0;
    for (int j = 0; j < kSortWarps / 2; ++j) s += s_h[j][d];
    hist[(uint64_t)d * gridDim.x + blockIdx.x] = s;
  }
}

// One block per digit: its counts over the slices to exclusive sums, in place, and its total.
__global__ void __launch_bounds__(kSortThreads) k_radix_rows(uint32_t* hist, uint32_t slices, uint32_t* total) {
  __shared__ uint32_t s_w[32];
  static_assert(kSortBlocksMax <= kSortThreads, "one thread per slice");
  uint32_t* row = hist + (uint64_t)blockIdx.x * slices;
  const uint32_t x = threadIdx.x < slices ? row[threadIdx.x] : 0u;
  uint32_t sum;
  const uint32_t e = block_excl_scan(x, s_w, &sum);
  if (threadIdx.x < slices) row[threadIdx.x] = e;
  if (threadIdx.x == 0) total[blockIdx.x] = sum;
}

template <bool kHasVals>
__global__ void __launch_bounds__(kSortThreads, 2) k_radix_scatter(const uint64_t* __restrict__ keys,
                                                                   const uint32_t* __restrict__ vals, uint64_t n,
                                                                   uint64_t per_block, int shift, uint32_t mask,
                                                                   const uint32_t* __restrict__ hist,
                                                                   const uint32_t* __restrict__ total,
                                                                   uint64_t* __restrict__ keys_out,
                                                                   uint32_t* __restrict__ vals_out) {
  __shared__ uint64_t s_k[kSortTile];
  __shared__ uint32_t s_v[kHasVals ? kSortTile : 1];
  // per warp and digit: the tile's elements, then those of earlier warps (cleared two digits at a time)
  __shared__ __align__(4) uint16_t s_c[kSortWarps][kRadixDigits];
  __shared__ uint32_t s_start[kRadixDigits];          // a digit's first place in the tile
  __shared__ uint32_t s_out[kRadixDigits];            // ... and in the output, minus s_start
  __shared__ uint32_t s_w[32];
  static_assert(kRadixDigits <= kSortThreads, "one thread per digit");
  static_assert(kRadixDigits % 2 == 0, "a warp's row of s_c starts on a word");
  const uint32_t t = threadIdx.x, w = t >> 5, lane = t & 31u, lt = (1u << lane) - 1u;
  uint32_t sum;
  // the output place of the slice's next element of digit t
  uint32_t run = block_excl_scan(t <= mask ? total[t] : 0u, s_w, &sum);
  if (t <= mask) run += hist[(uint64_t)t * gridDim.x + blockIdx.x];
  const uint64_t lo = (uint64_t)blockIdx.x * per_block, hi = lo + per_block < n ? lo + per_block : n;
  for (uint64_t base = lo; base < hi; base += kSortTile) {
    const uint32_t cnt = hi - base < kSortTile ? (uint32_t)(hi - base) : (uint32_t)kSortTile;
    uint64_t k[kSortItems];
    uint32_t v[kHasVals ? kSortItems : 1], rank[kSortItems];
    const uint32_t i0 = w * 32 * kSortItems + lane;
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) {
      const uint32_t i = i0 + 32 * j;
      k[j] = i < cnt ? keys[base + i] : ~0ull;
      if (kHasVals) v[j] = i < cnt ? vals[base + i] : 0u;
    }
    for (uint32_t d = 2 * lane; d <= mask; d += 64) *(uint32_t*)&s_c[w][d] = 0u;
    __syncwarp();
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) {
      const bool in = i0 + 32 * j < cnt;
      const uint32_t d = digit_of(k[j], shift, mask);
      uint32_t peers = __ballot_sync(EIC_FULL_MASK, in);
#pragma unroll
      for (int b = 0; b < kRadixBits; ++b) {
        if (!((mask >> b) & 1u)) break;  // (the pass's digits are narrower)
        const uint32_t m = __ballot_sync(EIC_FULL_MASK, (d >> b) & 1u);
        peers &= (d >> b) & 1u ? m : ~m;
      }
      const uint32_t before = in ? s_c[w][d] : 0u;
      rank[j] = before + __popc(peers & lt);
      __syncwarp();
      if (in && !(peers & lt)) s_c[w][d] = (uint16_t)(before + __popc(peers));
      __syncwarp();
    }
    __syncthreads();
    uint32_t mine = 0;  // the tile's elements of digit t
    if (t <= mask)
      for (int j = 0; j < kSortWarps; ++j) {
        const uint32_t c = s_c[j][t];
        s_c[j][t] = (uint16_t)mine;
        mine += c;
      }
    const uint32_t start = block_excl_scan(mine, s_w, &sum);
    if (t <= mask) {
      s_start[t] = start;
      s_out[t] = run - start;
      run += mine;
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) {
      if (i0 + 32 * j >= cnt) continue;
      const uint32_t d = digit_of(k[j], shift, mask), p = s_start[d] + s_c[w][d] + rank[j];
      s_k[p] = k[j];
      if (kHasVals) s_v[p] = v[j];
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) {
      const uint32_t p = t + kSortThreads * j;
      if (p >= cnt) continue;
      const uint64_t x = s_k[p];
      const uint32_t o = s_out[digit_of(x, shift, mask)] + p;
      keys_out[o] = x;
      if (kHasVals) vals_out[o] = s_v[p];
    }
    __syncthreads();
  }
}

// Scratch of a sort, in uint32: the slices' digit counts and the digits' totals.
constexpr uint64_t kSortScratch = (uint64_t)kRadixDigits * kSortBlocksMax + kRadixDigits;

// Stably sort keys[0..n) (and vals when non-NULL) by the key bits [lo, lo +
// bits); n < 2^32. Ping-pongs between the two buffers; *in_alt tells which one
// holds the result. scratch holds kSortScratch uint32.
inline int radix_sort(uint64_t* keys, uint32_t* vals, uint64_t* keys_alt, uint32_t* vals_alt, uint64_t n, int lo,
                      int bits, uint32_t* scratch, cudaStream_t st, bool* in_alt) {
  *in_alt = false;
  if (n <= 1 || bits <= 0) return EIC_OK;
  const uint64_t tiles = (n + kSortTile - 1) / kSortTile;
  uint64_t slices = tiles < kSortBlocksMax ? tiles : kSortBlocksMax;
  const uint64_t per = (tiles + slices - 1) / slices * kSortTile;  // elements per slice, whole tiles
  slices = (n + per - 1) / per;
  uint32_t* total = scratch + (uint64_t)kRadixDigits * kSortBlocksMax;
  uint64_t *kin = keys, *kout = keys_alt;
  uint32_t *vin = vals, *vout = vals_alt;
  const int passes = (bits + kRadixBits - 1) / kRadixBits;
  for (int p = 0, shift = lo; p < passes; ++p) {
    const int width = (lo + bits - shift + passes - p - 1) / (passes - p);  // the bits left, spread evenly
    const uint32_t mask = (1u << width) - 1u;
    k_radix_count<<<(int)slices, kSortThreads, 0, st>>>(kin, n, per, shift, mask, scratch);
    k_radix_rows<<<(int)mask + 1, kSortThreads, 0, st>>>(scratch, (uint32_t)slices, total);
    if (vals)
      k_radix_scatter<true><<<(int)slices, kSortThreads, 0, st>>>(kin, vin, n, per, shift, mask, scratch, total, kout,
                                                                  vout);
    else
      k_radix_scatter<false><<<(int)slices, kSortThreads, 0, st>>>(kin, nullptr, n, per, shift, mask, scratch, total,
                                                                   kout, nullptr);
    EIC_CUDA_TRY(cudaGetLastError());
    uint64_t* tk = kin;
    kin = kout;
    kout = tk;
    uint32_t* tv = vin;
    vin = vout;
    vout = tv;
    *in_alt = !*in_alt;
    shift += width;
  }
  return EIC_OK;
}

// ------------------------------------------------------------------- scans

constexpr int kScanThreads = 1024;
constexpr int kScanBlocksMax = 1024;

template <typename TIn>
__global__ void __launch_bounds__(kScanThreads) k_block_sums(const TIn* __restrict__ in, uint64_t n, uint64_t per,
                                                             uint64_t* sums) {
  __shared__ uint64_t s_w[32];
  uint64_t lo = (uint64_t)blockIdx.x * per, hi = lo + per < n ? lo + per : n;
  uint64_t s = 0;
  for (uint64_t i = lo + threadIdx.x; i < hi; i += blockDim.x) s += (uint64_t)in[i];
  s = warp_sum_u64(s);
  if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    uint64_t t = threadIdx.x < blockDim.x / 32 ? s_w[threadIdx.x] : 0;
    t = warp_sum_u64(t);
    if (threadIdx.x == 0) sums[blockIdx.x] = t;
  }
}

// Exclusive sums of at most 1024 values in place, one thread each, and their total.
__global__ void __launch_bounds__(kScanBlocksMax) k_scan_sums(uint64_t* sums, int count, uint64_t* total) {
  __shared__ uint64_t s_w[32];
  const uint32_t t = threadIdx.x, lane = t & 31u, w = t >> 5;
  const uint64_t x = (int)t < count ? sums[t] : 0;
  uint64_t incl = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint64_t y = __shfl_up_sync(EIC_FULL_MASK, incl, o);
    if ((int)lane >= o) incl += y;
  }
  if (lane == 31) s_w[w] = incl;
  __syncthreads();
  uint64_t before = 0;
  for (uint32_t j = 0; j < w; ++j) before += s_w[j];
  if ((int)t < count) sums[t] = before + incl - x;
  if (t == blockDim.x - 1) *total = before + incl;
}

// out[i] = sum(in[0..i)) for i in [0, n], out[n] = total.
template <typename TIn>
__global__ void __launch_bounds__(kScanThreads) k_block_scan(const TIn* __restrict__ in, uint64_t n, uint64_t per,
                                                             const uint64_t* __restrict__ offs,
                                                             uint64_t* __restrict__ out) {
  __shared__ uint64_t s_w[32];
  __shared__ uint64_t s_carry;
  uint64_t lo = (uint64_t)blockIdx.x * per, hi = lo + per < n ? lo + per : n;
  if (threadIdx.x == 0) s_carry = offs[blockIdx.x];
  __syncthreads();
  for (uint64_t base = lo; base < hi; base += blockDim.x) {
    uint64_t i = base + threadIdx.x;
    uint64_t x = i < hi ? (uint64_t)in[i] : 0;
    uint64_t incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      uint64_t y = __shfl_up_sync(EIC_FULL_MASK, incl, o);
      if ((int)(threadIdx.x & 31) >= o) incl += y;
    }
    if ((threadIdx.x & 31) == 31) s_w[threadIdx.x >> 5] = incl;
    __syncthreads();
    if (threadIdx.x < 32) {
      uint64_t t = threadIdx.x < blockDim.x / 32 ? s_w[threadIdx.x] : 0;
      uint64_t ti = t;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        uint64_t y = __shfl_up_sync(EIC_FULL_MASK, ti, o);
        if ((int)threadIdx.x >= o) ti += y;
      }
      s_w[threadIdx.x] = ti - t;
    }
    __syncthreads();
    uint64_t carry = s_carry;
    if (i < hi) out[i] = carry + s_w[threadIdx.x >> 5] + incl - x;
    __syncthreads();
    if (threadIdx.x == blockDim.x - 1) s_carry = carry + s_w[threadIdx.x >> 5] + incl;
    __syncthreads();
  }
}

// out[0..n] exclusive prefix sums of in[0..n); out[n] = total. scratch holds
// kScanBlocksMax uint64.
template <typename TIn>
inline int exclusive_scan(const TIn* in, uint64_t n, uint64_t* out, uint64_t* scratch, cudaStream_t st) {
  int blocks = (int)((n + kScanThreads - 1) / kScanThreads);
  if (blocks > kScanBlocksMax) blocks = kScanBlocksMax;
  if (blocks < 1) blocks = 1;
  uint64_t per = (n + blocks - 1) / blocks;
  if (per == 0) per = 1;
  k_block_sums<TIn><<<blocks, kScanThreads, 0, st>>>(in, n, per, scratch);
  k_scan_sums<<<1, kScanBlocksMax, 0, st>>>(scratch, blocks, out + n);
  k_block_scan<TIn><<<blocks, kScanThreads, 0, st>>>(in, n, per, scratch, out);
  EIC_CUDA_TRY(cudaGetLastError());
  return EIC_OK;
}

}  // namespace eic
