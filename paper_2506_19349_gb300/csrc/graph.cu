// Device CSR builder and graph object (preprocessing of Section 4.1: every
// vertex's incident edges sorted in weight order, and the edge-weight
// distribution quantised into RtoW[RATIO_NUM]).
//
// Pipeline, all on the device:
//   1. validate the tuples; pack each pair as a (min, max) key with its weight
//      below it (as a 32-bit value beside it when that exceeds 64 bits),
//      self-loops dropped;
//   2. radix-sort by pair, keep the smallest weight of each distinct pair and
//      emit both directions of every pair in pair order (which lists each
//      row's neighbours in ascending order);
//   3. stably radix-sort by (row, weight): rows end up sorted by (weight,
//      neighbour), and their ends give the degrees;
//   4. relabel the vertices by degree and place the rows in the new order;
//   5. RtoW from the undirected weights; distinct-degree tables and highD(0)
//      for the step statistics; the list of non-isolated vertices.
// The work is passes over the tuples: 32 M tuples on 2 M vertices take five
// sorting passes over the pairs and four over the entries, each reading a key
// twice and writing it once, with the weight (and neighbour) inside the key. A
// build took 25.7 ms before (12-byte pairs in seven passes, one atomic per
// degree, a one-block scan per pass) and takes 6.4 ms, of which the sorts are
// 3.2 and allocation 1.9.
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <new>
#include <vector>

#include "graph.h"
#include "radix.cuh"
#include "stats.cuh"

using namespace eic;

namespace {

constexpr int kThreads = 256;

inline int grid_for(uint64_t n, int threads = kThreads) {
  uint64_t b = (n + threads - 1) / threads;
  if (b > 65535ull * 32) b = 65535ull * 32;
  return (int)(b ? b : 1);
}

// Blocks of a kernel that keeps per-block tables or ends in per-warp atomics: a few per SM.
inline int grid_few(uint64_t n, int threads = kThreads) {
  const uint64_t b = (n + threads - 1) / threads, most = 152 * 8;
  return (int)(b < most ? (b ? b : 1) : most);
}

inline int bits_for(uint64_t x) {  // bits needed to represent values 0..x
  int b = 0;
  while (b < 64 && (x >> b) != 0) ++b;
  return b;
}

// small: [0] pairs kept, [1] the largest weight among them; err: an endpoint or weight out of range
__global__ void k_validate(const uint32_t* __restrict__ src, const uint32_t* __restrict__ dst,
                           const uint32_t* __restrict__ w, uint64_t T, uint32_t n, uint32_t* small, int* err) {
  uint32_t kept = 0, wmax = 0;
  bool bad = false;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < T; i += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t a = src[i], b = dst[i], x = w[i];
    bad |= a >= n || b >= n || x == 0;
    if (a != b) {
      ++kept;
      wmax = max(wmax, x);
    }
  }
  kept = __reduce_add_sync(EIC_FULL_MASK, kept);
  wmax = __reduce_max_sync(EIC_FULL_MASK, wmax);
  if (bad) atomicExch(err, 1);
  if ((threadIdx.x & 31) == 0) {
    if (kept) atomicAdd(&small[0], kept);
    atomicMax(&small[1], wmax);
  }
}

// A tile of kTile elements is taken by one block, element base + j kThreads + t
// by thread t.
constexpr int kTileItems = 8;
constexpr uint32_t kTile = kThreads * kTileItems;

// The places, in element order, of the flagged ones of a tile (flag bit j: this
// thread's element j): rank[j] before it in the tile. s_c: kTileItems *
// kThreads / 32 words. Returns the tile's count.
__device__ __forceinline__ uint32_t tile_ranks(uint32_t flags, uint32_t (&rank)[kTileItems], uint32_t* s_c) {
  const uint32_t lane = threadIdx.x & 31u, w = threadIdx.x >> 5;
  constexpr uint32_t kW = kThreads / 32, kC = kTileItems * kW;
  static_assert(kC == 64, "two counts per lane of a warp");
  __syncthreads();
#pragma unroll
  for (int j = 0; j < kTileItems; ++j) {
    const uint32_t m = __ballot_sync(EIC_FULL_MASK, (flags >> j) & 1u);
    rank[j] = __popc(m & ((1u << lane) - 1u));
    if (lane == 0) s_c[j * kW + w] = __popc(m);
  }
  __syncthreads();
  const uint32_t a = s_c[2 * lane], b = s_c[2 * lane + 1], incl = warp_incl_scan(a + b);
  const uint32_t total = __shfl_sync(EIC_FULL_MASK, incl, 31);
  const uint32_t ea = incl - a - b, eb = incl - b;
#pragma unroll
  for (int j = 0; j < kTileItems; ++j) {
    const uint32_t q = j * kW + w;
    const uint32_t x = __shfl_sync(EIC_FULL_MASK, ea, q >> 1), y = __shfl_sync(EIC_FULL_MASK, eb, q >> 1);
    rank[j] += (q & 1u) ? y : x;
  }
  return total;
}

// Pair keys in any order: ((min << vbits) | max), above the weight's wb bits, or (kVals) with the weight beside it.
// One atomic per tile.
template <bool kVals>
__global__ void __launch_bounds__(kThreads) k_canon(const uint32_t* __restrict__ src, const uint32_t* __restrict__ dst,
                                                    const uint32_t* __restrict__ w, uint64_t T, int vbits, int wb,
                                                    uint64_t* keys, uint32_t* vals, uint32_t* count) {
  __shared__ uint32_t s_c[kTileItems * kThreads / 32], s_at;
  for (uint64_t base = (uint64_t)blockIdx.x * kTile; base < T; base += (uint64_t)gridDim.x * kTile) {
    uint32_t a[kTileItems], b[kTileItems], x[kTileItems], rank[kTileItems], flags = 0;
#pragma unroll
    for (int j = 0; j < kTileItems; ++j) {
      const uint64_t i = base + (uint64_t)j * kThreads + threadIdx.x;
      a[j] = i < T ? src[i] : 0u;
      b[j] = i < T ? dst[i] : 0u;
      x[j] = i < T ? w[i] : 0u;
      flags |= a[j] != b[j] ? 1u << j : 0u;
    }
    const uint32_t cnt = tile_ranks(flags, rank, s_c);
    if (threadIdx.x == 0) s_at = atomicAdd(count, cnt);
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kTileItems; ++j) {
      if (!((flags >> j) & 1u)) continue;
      const uint64_t pair = ((uint64_t)min(a[j], b[j]) << vbits) | max(a[j], b[j]);
      const uint32_t p = s_at + rank[j];
      keys[p] = kVals ? pair : (pair << wb) | x[j];
      if (kVals) vals[p] = x[j];
    }
  }
}

// Bit j: this thread's element j of the tile is the first of its pair (keys equal above bit lo).
__device__ __forceinline__ uint32_t tile_heads(const uint64_t* __restrict__ keys, uint64_t base, uint64_t K, int lo) {
  uint32_t flags = 0;
#pragma unroll
  for (int j = 0; j < kTileItems; ++j) {
    const uint64_t i = base + (uint64_t)j * kThreads + threadIdx.x;
    if (i < K && (i == 0 || (keys[i] >> lo) != (keys[i - 1] >> lo))) flags |= 1u << j;
  }
  return flags;
}

// Distinct pairs per tile of the sorted keys.
__global__ void __launch_bounds__(kThreads) k_heads(const uint64_t* __restrict__ keys, uint64_t K, int lo,
                                                    uint32_t* tile_cnt) {
  __shared__ uint32_t s_n;
  const uint64_t tiles = (K + kTile - 1) / kTile;
  for (uint64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    const uint32_t c = __reduce_add_sync(EIC_FULL_MASK, (uint32_t)__popc(tile_heads(keys, tile * kTile, K, lo)));
    if ((threadIdx.x & 31) == 0) atomicAdd(&s_n, c);
    __syncthreads();
    if (threadIdx.x == 0) tile_cnt[tile] = s_n;
    __syncthreads();
  }
}

constexpr uint32_t kWBins = 4096;      // weights counted in shared memory
constexpr uint32_t kWHist = 1u << 16;  // weights below this get RtoW from a histogram

// Every distinct pair with the smallest weight of its run, both directions, at
// 2 pos and 2 pos + 1: (row, weight, neighbour) in one key, or (kVals) (row,
// weight) with the neighbour beside it. small: [2] largest, [3] smallest
// weight; whist (or NULL): count of each weight.
template <bool kVals>
__global__ void __launch_bounds__(kThreads) k_emit(const uint64_t* __restrict__ keys, const uint32_t* __restrict__ vals,
                                                   uint64_t K, int vbits, int wb,
                                                   const uint64_t* __restrict__ tile_off, uint64_t* out, uint32_t* out_v,
                                                   uint32_t* whist, uint32_t* small) {
  __shared__ uint32_t s_c[kTileItems * kThreads / 32], s_h[kWBins];
  const int lo = kVals ? 0 : wb;
  const uint64_t vmask = (1ull << vbits) - 1, tiles = (K + kTile - 1) / kTile;
  for (uint32_t i = threadIdx.x; i < kWBins; i += kThreads) s_h[i] = 0;
  uint32_t lmax = 0, lmin = 0xFFFFFFFFu;
  for (uint64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const uint64_t base = tile * kTile;
    uint32_t rank[kTileItems];
    const uint32_t flags = tile_heads(keys, base, K, lo);
    tile_ranks(flags, rank, s_c);
    const uint64_t at = tile_off[tile];
#pragma unroll
    for (int j = 0; j < kTileItems; ++j) {
      if (!((flags >> j) & 1u)) continue;
      const uint64_t i = base + (uint64_t)j * kThreads + threadIdx.x, k = keys[i], pair = k >> lo;
      uint32_t w = kVals ? vals[i] : (uint32_t)(k & ((1ull << wb) - 1));
      for (uint64_t q = i + 1; q < K; ++q) {
        const uint64_t kq = keys[q];
        if ((kq >> lo) != pair) break;
        w = min(w, kVals ? vals[q] : (uint32_t)(kq & ((1ull << wb) - 1)));
      }
      const uint64_t a = pair >> vbits, b = pair & vmask, p = 2 * (at + rank[j]);
      if (kVals) {
        out[p] = (a << wb) | w;
        out[p + 1] = (b << wb) | w;
        *(uint2*)&out_v[p] = make_uint2((uint32_t)b, (uint32_t)a);
      } else {
        *(ulonglong2*)&out[p] = make_ulonglong2((((a << wb) | w) << vbits) | b, (((b << wb) | w) << vbits) | a);
      }
      lmax = max(lmax, w);
      lmin = min(lmin, w);
      if (whist) {
        if (w < kWBins)
          atomicAdd(&s_h[w], 1u);
        else
          atomicAdd(&whist[w], 1u);
      }
    }
  }
  lmax = __reduce_max_sync(EIC_FULL_MASK, lmax);
  lmin = __reduce_min_sync(EIC_FULL_MASK, lmin);
  if ((threadIdx.x & 31) == 0 && lmax) {
    atomicMax(&small[2], lmax);
    atomicMin(&small[3], lmin);
  }
  __syncthreads();
  if (whist)
    for (uint32_t i = threadIdx.x; i < kWBins; i += kThreads)
      if (s_h[i]) atomicAdd(&whist[i], s_h[i]);
}

// First entry and end of every row of the sorted entries (row = key >> lo; zero where a vertex has none).
__global__ void k_row_ends(const uint64_t* __restrict__ keys, uint64_t E, int lo, uint32_t* beg, uint32_t* end) {
  const uint32_t lane = threadIdx.x & 31u;  // (a lane's neighbours hold the entries beside its own)
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i - lane < E; i += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t none = ~0ull, r = i < E ? keys[i] >> lo : none;
    uint64_t before = __shfl_up_sync(EIC_FULL_MASK, r, 1), after = __shfl_down_sync(EIC_FULL_MASK, r, 1);
    if (lane == 0) before = i > 0 && i < E ? keys[i - 1] >> lo : none;
    if (lane == 31) after = i + 1 < E ? keys[i + 1] >> lo : none;
    if (i >= E) continue;
    if (before != r) beg[r] = (uint32_t)i;
    if (after != r) end[r] = (uint32_t)(i + 1);
  }
}

// deg[v] = end[v] - beg[v], in place of end; the largest to *maxdeg
__global__ void k_row_lengths(const uint32_t* __restrict__ beg, uint32_t* end, uint64_t n, uint32_t* maxdeg) {
  uint32_t lmax = 0;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t d = end[i] - beg[i];
    end[i] = d;
    lmax = max(lmax, d);
  }
  lmax = __reduce_max_sync(EIC_FULL_MASK, lmax);
  if ((threadIdx.x & 31) == 0 && lmax) atomicMax(maxdeg, lmax);
}

// beg[v] to what a row's entries move by (modulo 2^32): its place in internal order minus its first entry.
__global__ void k_row_shift(uint32_t* beg, uint64_t n, const uint32_t* __restrict__ orig2int,
                            const uint32_t* __restrict__ row) {
  for (uint64_t v = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; v < n; v += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t i = orig2int[v];
    if (i != 0xFFFFFFFFu) beg[v] = row[i] - beg[v];
  }
}

// The sorted entries to their places: rows in internal order, neighbours renamed.
template <bool kVals>
__global__ void k_place(const uint64_t* __restrict__ keys, const uint32_t* __restrict__ vals, uint64_t E, int vbits,
                        int wb, const uint32_t* __restrict__ shift, const uint32_t* __restrict__ orig2int, uint2* adj) {
  const uint64_t vmask = (1ull << vbits) - 1, wmask = (1ull << wb) - 1;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < E; i += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t k = keys[i], rw = kVals ? k : k >> vbits;
    const uint32_t v = kVals ? vals[i] : (uint32_t)(k & vmask), u = (uint32_t)(rw >> wb);
    adj[(uint32_t)i + shift[u]] = make_uint2(orig2int[v], (uint32_t)(rw & wmask));
  }
}

// key of non-isolated vertex v: (maxdeg - deg(v), v), at its compacted position
__global__ void k_relabel_keys(const uint32_t* __restrict__ deg, const uint32_t* __restrict__ flags,
                               const uint64_t* __restrict__ pos, uint32_t n, uint32_t maxdeg, int vbits,
                               uint64_t* keys) {
  for (uint64_t v = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; v < n; v += (uint64_t)gridDim.x * blockDim.x)
    if (flags[v]) keys[pos[v]] = ((uint64_t)(maxdeg - deg[v]) << vbits) | v;
}

__global__ void k_relabel_maps(const uint64_t* __restrict__ keys, uint32_t ni, int vbits, uint32_t* int2orig,
                               uint32_t* orig2int) {
  const uint64_t vmask = (1ull << vbits) - 1;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < ni; i += gridDim.x * blockDim.x) {
    const uint32_t v = (uint32_t)(keys[i] & vmask);
    int2orig[i] = v;
    orig2int[v] = i;
  }
}

__global__ void k_gather_u32(const uint32_t* __restrict__ src, const uint32_t* __restrict__ idx, uint32_t cnt,
                             uint32_t* out) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < cnt; i += gridDim.x * blockDim.x) out[i] = src[idx[i]];
}

// nz[i] = {i, smallest weight of row i, row begin, row end} for every internal vertex
__global__ void k_nz_fill(const uint32_t* __restrict__ row, const uint2* __restrict__ adj, uint32_t ni, uint4* nz) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < ni; i += gridDim.x * blockDim.x)
    nz[i] = make_uint4(i, adj[row[i]].y, row[i], row[i + 1]);
}

__global__ void k_weights_to_keys(const uint2* __restrict__ adj, uint64_t E, uint64_t* keys) {
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < E; i += (uint64_t)gridDim.x * blockDim.x)
    keys[i] = adj[i].y;
}

// RtoW[i] = the ceil(i m / (R-1))-th smallest weight (the smallest for i = 0),
// from the sorted weights of both directions (every weight twice).
__device__ __forceinline__ uint64_t rtow_rank(uint32_t i, uint64_t m) {
  const uint32_t R = EIC_RATIO_NUM;
  const uint64_t rank = ((uint64_t)i * m + (R - 2)) / (R - 1);
  return rank ? rank - 1 : 0;
}

__global__ void k_rtow(const uint64_t* __restrict__ sorted_w, uint64_t m, uint32_t* rtow) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < EIC_RATIO_NUM; i += gridDim.x * blockDim.x)
    rtow[i] = (uint32_t)sorted_w[2 * rtow_rank(i, m)];
}

// The same from the count of each weight (one block of 1024 threads, 64 bins each).
__global__ void __launch_bounds__(1024) k_rtow_hist(const uint32_t* __restrict__ whist, uint64_t m, uint32_t* rtow) {
  __shared__ uint32_t s_before[1024], s_w[32];
  constexpr uint32_t kPer = kWHist / 1024;
  const uint32_t t = threadIdx.x;
  uint32_t sum = 0, total;
  for (uint32_t j = 0; j < kPer; ++j) sum += whist[t * kPer + j];  // (m < 2^31)
  s_before[t] = block_excl_scan(sum, s_w, &total);
  __syncthreads();
  for (uint32_t i = t; i < EIC_RATIO_NUM; i += 1024) {
    const uint32_t r = (uint32_t)rtow_rank(i, m);
    uint32_t lo = 0, hi = 1023;  // the last thread's bins that start at or before r
    while (lo < hi) {
      const uint32_t mid = (lo + hi + 1) >> 1;
      if (s_before[mid] <= r)
        lo = mid;
      else
        hi = mid - 1;
    }
    uint32_t acc = s_before[lo], b = lo * kPer;
    while ((acc += whist[b]) <= r) ++b;
    rtow[i] = b;
  }
}

// Degree histogram; degrees below 1024 are counted in shared memory first.
__global__ void k_deg_hist(const uint32_t* __restrict__ deg, uint32_t n, uint32_t* hist) {
  __shared__ uint32_t s_h[1024];
  for (int i = threadIdx.x; i < 1024; i += blockDim.x) s_h[i] = 0;
  __syncthreads();
  for (uint64_t v = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; v < n; v += (uint64_t)gridDim.x * blockDim.x) {
    uint32_t d = deg[v];
    if (d < 1024)
      atomicAdd(&s_h[d], 1u);
    else
      atomicAdd(&hist[d], 1u);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < 1024; i += blockDim.x)
    if (s_h[i]) atomicAdd(&hist[i], s_h[i]);
}

__global__ void k_flag_present(const uint32_t* __restrict__ hist, uint32_t len, uint32_t* flags) {
  for (uint32_t d = blockIdx.x * blockDim.x + threadIdx.x; d < len; d += gridDim.x * blockDim.x)
    flags[d] = (d >= 1 && hist[d] > 0) ? 1u : 0u;
}

__global__ void k_degree_tables(const uint32_t* __restrict__ hist, const uint32_t* __restrict__ flags,
                                const uint64_t* __restrict__ pos, uint32_t len, uint32_t* dvals, uint32_t* dcnt0) {
  for (uint32_t d = blockIdx.x * blockDim.x + threadIdx.x; d < len; d += gridDim.x * blockDim.x) {
    if (flags[d]) {
      const uint32_t r = (uint32_t)pos[d];
      dvals[r] = d;
      dcnt0[r] = hist[d];
    }
  }
}

__global__ void k_highd0(const uint32_t* dcnt0, const uint32_t* dvals, uint32_t D, uint32_t* out) {
  __shared__ HighdScr s;
  const HighdPart p = highd_sums(dcnt0, dvals, D, s);
  __syncthreads();
  highd_cross(dcnt0, dvals, D, p, s);
  __syncthreads();
  if (threadIdx.x == 0) *out = s.highd;
}

__global__ void k_narrow(const uint64_t* __restrict__ in, uint64_t n, uint32_t* out) {
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x)
    out[i] = (uint32_t)in[i];
}

__global__ void k_nz_keys(const uint4* __restrict__ nz, uint32_t cnt, int vbits, uint64_t* keys) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < cnt; i += gridDim.x * blockDim.x)
    keys[i] = ((uint64_t)nz[i].y << vbits) | nz[i].x;
}

__global__ void k_nz_from_keys(const uint64_t* __restrict__ keys, uint32_t cnt, int vbits,
                               const uint32_t* __restrict__ row, uint4* nz) {
  const uint64_t vmask = (1ull << vbits) - 1;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < cnt; i += gridDim.x * blockDim.x) {
    const uint32_t v = (uint32_t)(keys[i] & vmask);
    nz[i] = make_uint4(v, (uint32_t)(keys[i] >> vbits), row[v], row[v + 1]);
  }
}

// lt[t] = number of entries of the weight-sorted nz with smallest weight < t, t < len
__global__ void k_nz_lt(const uint4* __restrict__ nz, uint32_t cnt, uint32_t len, uint32_t* lt) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i <= cnt; i += gridDim.x * blockDim.x) {
    const uint32_t lo = i == 0 ? 0 : nz[i - 1].y + 1;           // first t with entry i-1 counted
    const uint32_t hi = i == cnt ? len - 1 : nz[i].y;           // last t before entry i counts
    for (uint32_t t = lo; t <= hi && t < len; ++t) lt[t] = i;
  }
}

__global__ void k_flag_nonzero(const uint32_t* __restrict__ deg, uint32_t n, uint32_t* flags) {
  for (uint64_t v = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; v < n; v += (uint64_t)gridDim.x * blockDim.x)
    flags[v] = deg[v] ? 1u : 0u;
}

// Temporary device allocations released on every exit path.
struct Temps {
  void* p[24];
  int k = 0;
  ~Temps() {
    for (int i = 0; i < k; ++i) cudaFree(p[i]);
  }
  template <typename T>
  int alloc(T** out, uint64_t count) {
    *out = nullptr;
    if (count == 0) count = 1;
    if (cudaMalloc((void**)out, count * sizeof(T)) != cudaSuccess) {
      (void)cudaGetLastError();
      return EIC_ENOMEM;
    }
    p[k++] = *out;
    return EIC_OK;
  }
  void release(void* q) {
    for (int i = 0; i < k; ++i)
      if (p[i] == q) {
        cudaFree(q);
        p[i] = p[--k];
        return;
      }
  }
};

#define TRY(x)                   \
  do {                           \
    int rc_ = (x);               \
    if (rc_ != EIC_OK) return rc_; \
  } while (0)

template <typename T>
int galloc(eic_graph* g, T** out, uint64_t count) {
  *out = nullptr;
  if (count == 0) count = 1;
  if (cudaMalloc((void**)out, count * sizeof(T)) != cudaSuccess) {
    (void)cudaGetLastError();
    return EIC_ENOMEM;
  }
  g->bytes += count * sizeof(T);
  return EIC_OK;
}

void graph_free_arrays(eic_graph* g) {
  cudaFree(g->row);
  cudaFree(g->adj);
  cudaFree(g->dvals);
  cudaFree(g->dcnt0);
  cudaFree(g->dfirst);
  cudaFree(g->dhint);
  cudaFree(g->drow);
  cudaFree(g->rtow);
  cudaFree(g->nz);
  cudaFree(g->nz_lt);
  cudaFree(g->orig2int);
  cudaFree(g->int2orig);
}

int build(eic_graph* g, const uint32_t* src, const uint32_t* dst, const uint32_t* w, uint64_t T, uint32_t n,
          int on_device, cudaStream_t st) {
  Temps tmp;
  const uint32_t *dsrc = src, *ddst = dst, *dw = w;
  if (!on_device && T > 0) {
    uint32_t* up;
    TRY(tmp.alloc(&up, 3 * T));
    EIC_CUDA_TRY(cudaMemcpyAsync(up, src, T * 4, cudaMemcpyHostToDevice, st));
    EIC_CUDA_TRY(cudaMemcpyAsync(up + T, dst, T * 4, cudaMemcpyHostToDevice, st));
    EIC_CUDA_TRY(cudaMemcpyAsync(up + 2 * T, w, T * 4, cudaMemcpyHostToDevice, st));
    dsrc = up;
    ddst = up + T;
    dw = up + 2 * T;
  }
  const int vbits = bits_for(n > 1 ? n - 1 : 1);
  // [0] pairs kept, [1] their largest weight, [2] and [3] largest and smallest
  // weight of the distinct pairs, [4] largest degree, [5] highD(0), [6] error, [7] keys written
  uint32_t* small;
  uint64_t* scan_scratch;
  uint32_t* sort_scratch;
  TRY(tmp.alloc(&scan_scratch, kScanBlocksMax + kSortScratch / 2 + 8));
  sort_scratch = (uint32_t*)(scan_scratch + kScanBlocksMax);
  small = sort_scratch + kSortScratch;
  const uint32_t init_small[8] = {0, 0, 0, 0xFFFFFFFFu, 0, 0, 0, 0};
  EIC_CUDA_TRY(cudaMemcpyAsync(small, init_small, sizeof(init_small), cudaMemcpyHostToDevice, st));

  // 1. pair keys (min, max) with their weights, self-loops dropped
  if (T > 0) k_validate<<<grid_few(T), kThreads, 0, st>>>(dsrc, ddst, dw, T, n, small, (int*)(small + 6));
  EIC_CUDA_TRY(cudaGetLastError());
  uint32_t hs[8];
  EIC_CUDA_TRY(cudaMemcpyAsync(hs, small, sizeof(hs), cudaMemcpyDeviceToHost, st));
  EIC_CUDA_TRY(cudaStreamSynchronize(st));
  if (hs[6]) return EIC_EINVAL;
  const uint64_t K = hs[0];
  const int wb = bits_for(hs[1]);
  const bool packed = 2 * vbits + wb <= 64;  // pair and weight (row, weight and neighbour) in one key
  uint64_t *ka, *kb;                          // room for both directions of every pair
  uint32_t *va = nullptr, *vb = nullptr;
  TRY(tmp.alloc(&ka, 4 * K));
  kb = ka + 2 * K;
  if (!packed) {
    TRY(tmp.alloc(&va, 4 * K));
    vb = va + 2 * K;
  }
  uint64_t m = 0;
  uint32_t* whist = nullptr;  // count of each weight
  if (wb <= 16) {
    TRY(tmp.alloc(&whist, kWHist));
    EIC_CUDA_TRY(cudaMemsetAsync(whist, 0, kWHist * 4, st));
  }
  bool alt = false;
  if (K > 0) {
    const int lo = packed ? wb : 0;
    const uint64_t ktiles = (K + kTile - 1) / kTile;
    if (packed)
      k_canon<false><<<grid_for(T, kTile), kThreads, 0, st>>>(dsrc, ddst, dw, T, vbits, wb, ka, nullptr, small + 7);
    else
      k_canon<true><<<grid_for(T, kTile), kThreads, 0, st>>>(dsrc, ddst, dw, T, vbits, wb, ka, va, small + 7);
    EIC_CUDA_TRY(cudaGetLastError());
    // 2. sort by pair; each distinct pair keeps its smallest weight
    TRY(radix_sort(ka, va, kb, vb, K, lo, 2 * vbits, sort_scratch, st, &alt));
    if (alt) {
      std::swap(ka, kb);
      std::swap(va, vb);
    }
    uint64_t* toff;
    TRY(tmp.alloc(&toff, ktiles + 1 + (ktiles + 1) / 2));
    uint32_t* tcnt = (uint32_t*)(toff + ktiles + 1);
    k_heads<<<grid_few(ktiles, 1), kThreads, 0, st>>>(ka, K, lo, tcnt);
    TRY(exclusive_scan<uint32_t>(tcnt, ktiles, toff, scan_scratch, st));
    EIC_CUDA_TRY(cudaMemcpyAsync(&m, toff + ktiles, 8, cudaMemcpyDeviceToHost, st));
    if (packed)
      k_emit<false><<<grid_few(ktiles, 1), kThreads, 0, st>>>(ka, nullptr, K, vbits, wb, toff, kb, nullptr, whist, small);
    else
      k_emit<true><<<grid_few(ktiles, 1), kThreads, 0, st>>>(ka, va, K, vbits, wb, toff, kb, vb, whist, small);
    EIC_CUDA_TRY(cudaGetLastError());
    EIC_CUDA_TRY(cudaStreamSynchronize(st));
    // 3. both directions, stable sort by (row, weight)
    TRY(radix_sort(kb, vb, ka, va, 2 * m, packed ? vbits : 0, wb + vbits, sort_scratch, st, &alt));
    if (!alt) {
      std::swap(ka, kb);
      std::swap(va, vb);
    }
  }
  const uint64_t E = 2 * m;

  // the rows' places in the sorted entries, degrees in original ids
  uint32_t *beg, *deg;
  TRY(tmp.alloc(&beg, 2 * (uint64_t)n));
  deg = beg + n;
  EIC_CUDA_TRY(cudaMemsetAsync(beg, 0, 2 * (uint64_t)n * 4, st));
  if (E > 0) k_row_ends<<<grid_for(E), kThreads, 0, st>>>(ka, E, wb + (packed ? vbits : 0), beg, deg);
  k_row_lengths<<<grid_few(n), kThreads, 0, st>>>(beg, deg, n, small + 4);
  EIC_CUDA_TRY(cudaGetLastError());
  EIC_CUDA_TRY(cudaMemcpyAsync(hs, small, sizeof(hs), cudaMemcpyDeviceToHost, st));

  // 4. internal ids: the non-isolated vertices ordered by (degree descending,
  // original id), so that the most-touched vertices share cache lines
  uint32_t ni = 0, maxdeg = 0, maxw = 0, minw = 0;
  int wbits = 0;
  TRY(galloc(g, &g->orig2int, n));
  EIC_CUDA_TRY(cudaMemsetAsync(g->orig2int, 0xFF, (uint64_t)n * 4, st));
  {
    uint64_t* pos;
    TRY(tmp.alloc(&pos, (uint64_t)n + 1 + ((uint64_t)n + 1) / 2));
    uint32_t* flags = (uint32_t*)(pos + (uint64_t)n + 1);
    k_flag_nonzero<<<grid_for(n), kThreads, 0, st>>>(deg, n, flags);
    TRY(exclusive_scan<uint32_t>(flags, n, pos, scan_scratch, st));
    uint64_t c = 0;
    EIC_CUDA_TRY(cudaMemcpyAsync(&c, pos + n, 8, cudaMemcpyDeviceToHost, st));
    EIC_CUDA_TRY(cudaStreamSynchronize(st));
    ni = (uint32_t)c;
    maxdeg = hs[4];
    maxw = m ? hs[2] : 0;
    minw = m ? hs[3] : 0;
    wbits = bits_for(maxw);
    TRY(galloc(g, &g->int2orig, ni));
    uint64_t *rk0, *rk1;
    TRY(tmp.alloc(&rk0, 2 * (uint64_t)ni));
    rk1 = rk0 + ni;
    k_relabel_keys<<<grid_for(n), kThreads, 0, st>>>(deg, flags, pos, n, maxdeg, vbits, rk0);
    bool ralt = false;  // (the keys come in vertex order)
    TRY(radix_sort(rk0, nullptr, rk1, nullptr, ni, vbits, bits_for(maxdeg), sort_scratch, st, &ralt));
    k_relabel_maps<<<grid_for(ni), kThreads, 0, st>>>(ralt ? rk1 : rk0, ni, vbits, g->int2orig, g->orig2int);
    EIC_CUDA_TRY(cudaGetLastError());
    EIC_CUDA_TRY(cudaStreamSynchronize(st));
    tmp.release(rk0);
    tmp.release(pos);
  }
  const int ibits = bits_for(ni > 1 ? ni - 1 : 1);
  TRY(galloc(g, &g->row, (uint64_t)ni + 1));
  {
    uint64_t* row64;
    TRY(tmp.alloc(&row64, (uint64_t)ni + 1 + ((uint64_t)ni + 1) / 2));
    uint32_t* deg_int = (uint32_t*)(row64 + (uint64_t)ni + 1);
    k_gather_u32<<<grid_for(ni), kThreads, 0, st>>>(deg, g->int2orig, ni, deg_int);
    TRY(exclusive_scan<uint32_t>(deg_int, ni, row64, scan_scratch, st));
    k_narrow<<<grid_for((uint64_t)ni + 1), kThreads, 0, st>>>(row64, (uint64_t)ni + 1, g->row);
    EIC_CUDA_TRY(cudaGetLastError());
    EIC_CUDA_TRY(cudaStreamSynchronize(st));
    tmp.release(row64);
  }
  TRY(galloc(g, &g->adj, E + 2));  // two spare entries: a 16-byte pair load starting at the last entry stays inside
  if (E > 0) {
    k_row_shift<<<grid_for(n), kThreads, 0, st>>>(beg, n, g->orig2int, g->row);
    if (packed)
      k_place<false><<<grid_for(E), kThreads, 0, st>>>(ka, nullptr, E, vbits, wb, beg, g->orig2int, g->adj);
    else
      k_place<true><<<grid_for(E), kThreads, 0, st>>>(ka, va, E, vbits, wb, beg, g->orig2int, g->adj);
    EIC_CUDA_TRY(cudaGetLastError());
  }

  // 5a. RtoW from the undirected weights
  TRY(galloc(g, &g->rtow, EIC_RATIO_NUM));
  if (m > 0 && whist) {
    k_rtow_hist<<<1, 1024, 0, st>>>(whist, m, g->rtow);
    EIC_CUDA_TRY(cudaGetLastError());
  } else if (m > 0) {  // (the entries' keys have served)
    k_weights_to_keys<<<grid_for(E), kThreads, 0, st>>>(g->adj, E, ka);
    TRY(radix_sort(ka, nullptr, kb, nullptr, E, 0, wbits, sort_scratch, st, &alt));
    k_rtow<<<(EIC_RATIO_NUM + kThreads - 1) / kThreads, kThreads, 0, st>>>(alt ? kb : ka, m, g->rtow);
    EIC_CUDA_TRY(cudaGetLastError());
  } else {
    EIC_CUDA_TRY(cudaMemsetAsync(g->rtow, 0, EIC_RATIO_NUM * 4, st));
  }

  // 5b. distinct-degree tables and highD(0)
  const uint32_t hlen = maxdeg + 1;
  uint32_t D = 0, nlong = 0, nbig = 0, big_end = 0;
  {
    uint64_t* pos;
    TRY(tmp.alloc(&pos, 2 * ((uint64_t)hlen + 1)));
    uint32_t *dh = (uint32_t*)(pos + (uint64_t)hlen + 1), *flags = dh + hlen;
    EIC_CUDA_TRY(cudaMemsetAsync(dh, 0, (uint64_t)hlen * 4, st));
    k_deg_hist<<<grid_few(n), kThreads, 0, st>>>(deg, n, dh);
    k_flag_present<<<grid_for(hlen), kThreads, 0, st>>>(dh, hlen, flags);
    TRY(exclusive_scan<uint32_t>(flags, hlen, pos, scan_scratch, st));
    uint64_t dd = 0;
    EIC_CUDA_TRY(cudaMemcpyAsync(&dd, pos + hlen, 8, cudaMemcpyDeviceToHost, st));
    EIC_CUDA_TRY(cudaStreamSynchronize(st));
    D = (uint32_t)dd;
    TRY(galloc(g, &g->dvals, D));
    TRY(galloc(g, &g->dcnt0, D));
    k_degree_tables<<<grid_for(hlen), kThreads, 0, st>>>(dh, flags, pos, hlen, g->dvals, g->dcnt0);
    k_highd0<<<1, 1024, 0, st>>>(g->dcnt0, g->dvals, D, small + 5);
    EIC_CUDA_TRY(cudaGetLastError());
    // dfirst[r]: the first internal id of degree dvals[r] (ids by degree descending); drow[r]: the same with that
    // id's row offset and the degree
    TRY(galloc(g, &g->dfirst, D));
    TRY(galloc(g, &g->drow, D));
    if (D) {
      std::vector<uint32_t> cnt(D), first(D), vals(D);
      std::vector<uint4> rows(D);
      EIC_CUDA_TRY(cudaMemcpyAsync(cnt.data(), g->dcnt0, (uint64_t)D * 4, cudaMemcpyDeviceToHost, st));
      EIC_CUDA_TRY(cudaMemcpyAsync(vals.data(), g->dvals, (uint64_t)D * 4, cudaMemcpyDeviceToHost, st));
      EIC_CUDA_TRY(cudaStreamSynchronize(st));
      uint64_t acc = 0, off = 0;
      for (uint32_t r = D; r-- > 0;) {
        first[r] = (uint32_t)acc;
        rows[r] = make_uint4((uint32_t)acc, (uint32_t)off, vals[r], 0u);
        acc += cnt[r];
        off += (uint64_t)cnt[r] * vals[r];
        if (vals[r] > kCursorMin) nlong = (uint32_t)acc;  // ids [0, acc) have degree >= vals[r]
        if (vals[r] > kBigRow) {
          nbig = (uint32_t)acc;
          big_end = (uint32_t)off;
        }
      }
      EIC_CUDA_TRY(cudaMemcpyAsync(g->dfirst, first.data(), (uint64_t)D * 4, cudaMemcpyHostToDevice, st));
      EIC_CUDA_TRY(cudaMemcpyAsync(g->drow, rows.data(), (uint64_t)D * sizeof(uint4), cudaMemcpyHostToDevice, st));
      EIC_CUDA_TRY(cudaStreamSynchronize(st));
    }
    // dhint[b]: the ranks of ids 4096 b + 4095 and 4096 b (the range a rank search in block b needs)
    const uint64_t nblk = (uint64_t)ni / 4096 + 1;
    TRY(galloc(g, &g->dhint, nblk));
    if (D) {
      std::vector<uint32_t> first(D);
      EIC_CUDA_TRY(cudaMemcpyAsync(first.data(), g->dfirst, (uint64_t)D * 4, cudaMemcpyDeviceToHost, st));
      EIC_CUDA_TRY(cudaStreamSynchronize(st));
      auto rank_of = [&](uint64_t x) -> uint32_t {  // the smallest r with first[r] <= x
        uint32_t lo = 0, hi = D - 1;
        while (lo < hi) {
          const uint32_t mid = (lo + hi) / 2;
          if (first[mid] <= x)
            hi = mid;
          else
            lo = mid + 1;
        }
        return lo;
      };
      std::vector<uint2> hint(nblk);
      for (uint64_t b = 0; b < nblk; ++b) {
        const uint64_t x0 = b * 4096, x1 = std::min<uint64_t>(x0 + 4095, ni ? ni - 1 : 0);
        hint[b] = make_uint2(rank_of(x1), rank_of(std::min<uint64_t>(x0, x1)));
      }
      EIC_CUDA_TRY(cudaMemcpyAsync(g->dhint, hint.data(), nblk * sizeof(uint2), cudaMemcpyHostToDevice, st));
      EIC_CUDA_TRY(cudaStreamSynchronize(st));
    }
  }

  // 5c. every internal vertex with its smallest weight, ordered by (smallest
  // weight, id): the vertices a pull can touch (smallest weight below a bound)
  // form a prefix, located with nz_lt
  uint32_t nz_lt_len = 0;
  {
    TRY(galloc(g, &g->nz, ni));
    k_nz_fill<<<grid_for(ni), kThreads, 0, st>>>(g->row, g->adj, ni, g->nz);
    EIC_CUDA_TRY(cudaGetLastError());
    if (ni > 1) {
      uint64_t *kk0, *kk1;
      TRY(tmp.alloc(&kk0, 2 * (uint64_t)ni));
      kk1 = kk0 + ni;
      k_nz_keys<<<grid_for(ni), kThreads, 0, st>>>(g->nz, ni, ibits, kk0);
      bool alt = false;  // (the keys come in id order)
      TRY(radix_sort(kk0, nullptr, kk1, nullptr, ni, ibits, wbits, sort_scratch, st, &alt));
      k_nz_from_keys<<<grid_for(ni), kThreads, 0, st>>>(alt ? kk1 : kk0, ni, ibits, g->row, g->nz);
      EIC_CUDA_TRY(cudaGetLastError());
      EIC_CUDA_TRY(cudaStreamSynchronize(st));
      tmp.release(kk0);
    }
    nz_lt_len = (maxw < 65535u ? maxw + 1 : 65536u) + 1;
    TRY(galloc(g, &g->nz_lt, nz_lt_len));
    k_nz_lt<<<grid_for((uint64_t)ni + 1), kThreads, 0, st>>>(g->nz, ni, nz_lt_len, g->nz_lt);
    EIC_CUDA_TRY(cudaGetLastError());
  }
  EIC_CUDA_TRY(cudaMemcpyAsync(hs, small, sizeof(hs), cudaMemcpyDeviceToHost, st));
  EIC_CUDA_TRY(cudaStreamSynchronize(st));

  DevGraph& dg = g->dg;
  dg.n = n;
  dg.ni = ni;
  dg.orig2int = g->orig2int;
  dg.int2orig = g->int2orig;
  dg.two_m = E;
  dg.m = m;
  dg.row = g->row;
  dg.adj = g->adj;
  dg.dvals = g->dvals;
  dg.dcnt0 = g->dcnt0;
  dg.dfirst = g->dfirst;
  dg.dhint = g->dhint;
  dg.drow = g->drow;
  dg.nlong = nlong;
  dg.nbig = nbig;
  dg.big_end = big_end;
  dg.D = D;
  dg.rtow = g->rtow;
  dg.nz = g->nz;
  dg.nz_count = ni;
  dg.nz_lt = g->nz_lt;
  dg.nz_lt_len = nz_lt_len;
  dg.maxw = maxw;
  dg.minw = minw;
  dg.max_deg = maxdeg;
  dg.highd0 = hs[5];
  return EIC_OK;
}

}  // namespace

// ------------------------------------------------------------------ C ABI

extern "C" {

int eic_params_default(eic_params* p) {
  if (!p) return EIC_EINVAL;
  memset(p, 0, sizeof(*p));
  p->alpha = 3;
  p->beta = 0.9;
  p->st_num = 1024;
  return EIC_OK;
}

const char* eic_strerror(int status) {
  switch (status) {
    case EIC_OK: return "ok";
    case EIC_EINVAL: return "invalid argument";
    case EIC_ENOMEM: return "out of memory or capacity";
    case EIC_ECUDA: return "CUDA runtime error";
    case EIC_EOVERFLOW: return "distance overflow (max distance + max weight >= 2^32-1)";
    case EIC_ETIMEOUT: return "device wait timed out";
    case EIC_EBUSY: return "busy";
    case EIC_ESIZE: return "graph exceeds the limits of the allocation-free entry point";
    case EIC_EABORT: return "not run: every block group of the batch stopped at an earlier error";
    default: return "unknown status";
  }
}

int eic_version(void) { return 100; }

int eic_graph_create(const uint32_t* src, const uint32_t* dst, const uint32_t* w, uint64_t num_tuples,
                     uint32_t num_vertices, int ptrs_on_device, void* stream, eic_graph** out) {
  if (!out) return EIC_EINVAL;
  *out = nullptr;
  if (num_vertices == 0 || num_vertices >= 0xFFFFFFFFu) return EIC_EINVAL;
  if (num_tuples > 0 && (!src || !dst || !w)) return EIC_EINVAL;
  if (num_tuples >= (1ull << 31)) return EIC_EINVAL;
  eic_graph* g = new (std::nothrow) eic_graph();
  if (!g) return EIC_ENOMEM;
  if (cudaGetDevice(&g->device) != cudaSuccess) {
    (void)cudaGetLastError();
    delete g;
    return EIC_ECUDA;
  }
  int rc = build(g, src, dst, w, num_tuples, num_vertices, ptrs_on_device, (cudaStream_t)stream);
  if (rc != EIC_OK) {
    cudaStreamSynchronize((cudaStream_t)stream);
    (void)cudaGetLastError();
    graph_free_arrays(g);
    delete g;
    return rc;
  }
  *out = g;
  return EIC_OK;
}

int eic_graph_info(const eic_graph* g, uint32_t* n, uint64_t* m, uint32_t* max_deg, uint32_t* max_w,
                   uint32_t* min_w, uint32_t* highd0) {
  if (!g) return EIC_EINVAL;
  if (n) *n = g->dg.n;
  if (m) *m = g->dg.m;
  if (max_deg) *max_deg = g->dg.max_deg;
  if (max_w) *max_w = g->dg.maxw;
  if (min_w) *min_w = g->dg.minw;
  if (highd0) *highd0 = g->dg.highd0;
  return EIC_OK;
}

int eic_graph_export(const eic_graph* g, uint64_t* row_ptr, uint32_t* nbr, uint32_t* w, uint32_t* rtow) {
  if (!g) return EIC_EINVAL;
  int dev = 0;
  cudaGetDevice(&dev);
  cudaSetDevice(g->device);
  int rc = EIC_OK;
  const uint64_t n = g->dg.n, ni = g->dg.ni, E = g->dg.two_m;
  uint32_t* o2i = (uint32_t*)malloc((n ? n : 1) * 4);
  uint32_t* i2o = (uint32_t*)malloc((ni ? ni : 1) * 4);
  uint32_t* row = (uint32_t*)malloc((ni + 1) * 4);
  uint2* adj = (nbr || w) ? (uint2*)malloc((E ? E : 1) * sizeof(uint2)) : nullptr;
  if (!o2i || !i2o || !row || ((nbr || w) && !adj)) rc = EIC_ENOMEM;
  if (rc == EIC_OK && (cudaMemcpy(o2i, g->orig2int, n * 4, cudaMemcpyDeviceToHost) != cudaSuccess ||
                       cudaMemcpy(i2o, g->int2orig, ni * 4, cudaMemcpyDeviceToHost) != cudaSuccess ||
                       cudaMemcpy(row, g->row, (ni + 1) * 4, cudaMemcpyDeviceToHost) != cudaSuccess ||
                       (adj && E && cudaMemcpy(adj, g->adj, E * sizeof(uint2), cudaMemcpyDeviceToHost) != cudaSuccess)))
    rc = EIC_ECUDA;
  if (rc == EIC_OK) {
    // rows in original vertex order, each sorted by (weight, original neighbour)
    uint64_t off = 0;
    std::vector<uint64_t> tmpk;
    for (uint64_t u = 0; u < n; ++u) {
      if (row_ptr) row_ptr[u] = off;
      const uint32_t i = o2i[u];
      if (i == 0xFFFFFFFFu) continue;
      const uint32_t b = row[i], e = row[i + 1];
      if (adj) {
        tmpk.resize(e - b);
        for (uint32_t k = b; k < e; ++k) tmpk[k - b] = ((uint64_t)adj[k].y << 32) | i2o[adj[k].x];
        std::sort(tmpk.begin(), tmpk.end());
        for (uint32_t k = 0; k < e - b; ++k) {
          if (nbr) nbr[off + k] = (uint32_t)tmpk[k];
          if (w) w[off + k] = (uint32_t)(tmpk[k] >> 32);
        }
      }
      off += e - b;
    }
    if (row_ptr) row_ptr[n] = off;
  }
  if (rtow && rc == EIC_OK && cudaMemcpy(rtow, g->rtow, EIC_RATIO_NUM * 4, cudaMemcpyDeviceToHost) != cudaSuccess)
    rc = EIC_ECUDA;
  free(o2i);
  free(i2o);
  free(row);
  free(adj);
  (void)cudaGetLastError();
  cudaSetDevice(dev);
  return rc;
}

int eic_graph_export_internal(const eic_graph* g, uint32_t* ni, uint32_t* int2orig, uint32_t* row, uint32_t* nbr,
                              uint32_t* w) {
  if (!g) return EIC_EINVAL;
  if (ni) *ni = g->dg.ni;
  if (!int2orig && !row && !nbr && !w) return EIC_OK;
  int dev = 0;
  cudaGetDevice(&dev);
  cudaSetDevice(g->device);
  int rc = EIC_OK;
  const uint64_t n_int = g->dg.ni, E = g->dg.two_m;
  if (int2orig && n_int && cudaMemcpy(int2orig, g->int2orig, n_int * 4, cudaMemcpyDeviceToHost) != cudaSuccess)
    rc = EIC_ECUDA;
  if (rc == EIC_OK && row && cudaMemcpy(row, g->row, (n_int + 1) * 4, cudaMemcpyDeviceToHost) != cudaSuccess)
    rc = EIC_ECUDA;
  if (rc == EIC_OK && (nbr || w) && E) {
    uint2* adj = (uint2*)malloc(E * sizeof(uint2));
    if (!adj) {
      rc = EIC_ENOMEM;
    } else if (cudaMemcpy(adj, g->adj, E * sizeof(uint2), cudaMemcpyDeviceToHost) != cudaSuccess) {
      rc = EIC_ECUDA;
    } else {
      for (uint64_t k = 0; k < E; ++k) {
        if (nbr) nbr[k] = adj[k].x;
        if (w) w[k] = adj[k].y;
      }
    }
    free(adj);
  }
  (void)cudaGetLastError();
  cudaSetDevice(dev);
  return rc;
}

int eic_graph_memory(const eic_graph* g, uint64_t* graph_bytes, uint64_t* workspace_bytes) {
  if (!g) return EIC_EINVAL;
  if (graph_bytes) *graph_bytes = g->bytes;
  if (workspace_bytes) *workspace_bytes = g->ws.bytes;
  return EIC_OK;
}

int eic_graph_destroy(eic_graph* g) {
  if (!g) return EIC_OK;
  int dev = 0;
  cudaGetDevice(&dev);
  cudaSetDevice(g->device);
  cudaDeviceSynchronize();
  eic_ws_free(&g->ws);
  graph_free_arrays(g);
  (void)cudaGetLastError();
  cudaSetDevice(dev);
  delete g;
  return EIC_OK;
}

}  // extern "C"
