// Shared definitions of libeic's CUDA sources (sm_103a).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/eic.h"

#define EIC_INF_T (((int64_t)1) << 62)
#define EIC_FULL_MASK 0xFFFFFFFFu

#define EIC_CUDA_TRY(expr)                     \
  do {                                         \
    cudaError_t e_ = (expr);                   \
    if (e_ != cudaSuccess) {                   \
      (void)cudaGetLastError();                \
      return e_ == cudaErrorMemoryAllocation   \
                 ? EIC_ENOMEM                  \
                 : EIC_ECUDA;                  \
    }                                          \
  } while (0)

// Read-only view of a device-resident graph (preprocessing of Section 4.1).
// Vertices have internal ids 0..ni-1: the non-isolated vertices ordered by
// (degree descending, original id); orig2int/int2orig translate.
constexpr uint32_t kBigRow = 256;    // a longer row is taken by a whole warp when parents are looked for
constexpr uint32_t kCursorMin = 16;  // rows longer than this keep a window cursor

struct DevGraph {
  uint32_t n;             // vertices in the caller's numbering
  uint32_t ni;            // internal vertices (degree >= 1)
  const uint32_t* orig2int;  // [n] internal id, or 0xFFFFFFFF for an isolated vertex
  const uint32_t* int2orig;  // [ni]
  uint64_t two_m;         // directed entries, sum of degrees
  uint64_t m;             // undirected edges
  const uint32_t* row;    // [ni + 1] row offsets (2m < 2^32)
  const uint2* adj;       // [two_m] {neighbour, weight}, rows sorted by (weight, neighbour)
  const uint32_t* dvals;  // [D] distinct degrees >= 1, ascending
  const uint32_t* dcnt0;  // [D] number of vertices with degree dvals[r]
  const uint32_t* dfirst;  // [D] first internal id of degree dvals[r] (decreasing in r: ids run by degree descending)
  const uint2* dhint;      // [ni / 4096 + 1] {rank of the block's last id, rank of its first id} per 4096 ids
  const uint4* drow;       // [D] {first internal id of degree dvals[r], its row offset, dvals[r], 0}
  uint32_t D;
  const uint32_t* rtow;   // [EIC_RATIO_NUM] maxW(G, i / (RATIO_NUM - 1))
  const uint4* nz;        // [nz_count = ni] {internal id, smallest row weight, row begin, row end}, by (weight, id)
  uint32_t nz_count;
  const uint32_t* nz_lt;  // [nz_lt_len] nz_lt[t] = number of nz entries with smallest weight < t
  uint32_t nz_lt_len;
  uint32_t maxw, minw, max_deg, highd0;
  uint32_t nbig, big_end;  // internal vertices of degree > kBigRow: ids [0, nbig), entries [0, big_end)
  uint32_t nlong;         // internal vertices of degree > kCursorMin: ids [0, nlong), the rows with a window cursor
};

// Rank (index into dvals) of internal vertex x's degree: internal ids run by
// degree descending, so it is the smallest r with dfirst[r] <= x. A search in
// a small table that stays in L1, narrowed to the ranks of x's block of 4096
// ids, in place of a random row[x], row[x + 1].
__device__ __forceinline__ uint32_t degree_rank(const DevGraph& G, uint32_t x) {
  const uint2 h = __ldg(&G.dhint[x >> 12]);  // the ranks in x's block of 4096 ids: one rank in most blocks
  uint32_t lo = h.x, hi = h.y;
  while (lo < hi) {
    const uint32_t mid = (lo + hi) >> 1;
    if (__ldg(&G.dfirst[mid]) <= x)
      hi = mid;
    else
      lo = mid + 1;
  }
  return lo;
}

// Row of internal vertex x as {begin, length}: the rows of one degree follow
// each other in id order, so both come from the id (three reads of small
// tables that stay in L1) in place of a random read of row[x], row[x + 1].
__device__ __forceinline__ uint2 row_of(const DevGraph& G, uint32_t x) {
  const uint4 t = __ldg(&G.drow[degree_rank(G, x)]);
  return make_uint2(t.y + (x - t.x) * t.z, t.z);
}

// ------------------------------------------------------------ warp helpers

__device__ __forceinline__ uint32_t lane_id() { return threadIdx.x & 31u; }

__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t x) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    uint32_t y = __shfl_up_sync(EIC_FULL_MASK, x, o);
    if ((int)lane_id() >= o) x += y;
  }
  return x;
}

__device__ __forceinline__ uint64_t warp_sum_u64(uint64_t x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(EIC_FULL_MASK, x, o);
  return x;
}

// Warp-aggregated append of `item` for each lane with want != 0 to
// list[*counter ...]; returns the slot or UINT32_MAX. All lanes must call.
__device__ __forceinline__ uint32_t warp_append(bool want, uint32_t* counter) {
  uint32_t mask = __ballot_sync(EIC_FULL_MASK, want);
  if (mask == 0) return UINT32_MAX;
  uint32_t leader = __ffs(mask) - 1;
  uint32_t base = 0;
  if (lane_id() == leader) base = atomicAdd(counter, (uint32_t)__popc(mask));
  base = __shfl_sync(EIC_FULL_MASK, base, leader);
  return want ? base + __popc(mask & ((1u << lane_id()) - 1u)) : UINT32_MAX;
}

__device__ __forceinline__ uint32_t ld_acquire_u32(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ int ld_volatile_int(const int* p) { return *(const volatile int*)p; }

// Release/acquire primitives of the barrier (gpu scope).
__device__ __forceinline__ void red_release_add_u32(uint32_t* p, uint32_t v) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// ---------------------------------------------------- bounded grid barrier

struct GridBarrier {
  unsigned long long arrived;  // arrivals since the launch (or query) started; kBarrierError once a block gave up
};
constexpr unsigned long long kBarrierError = 1ull << 63;

__device__ __forceinline__ void red_release_add_u64(unsigned long long* p, unsigned long long v) {
  asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

__device__ __forceinline__ unsigned long long ld_acquire_gpu_u64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

// A wait ran out: the status says so, and every block leaves at its next barrier.
__device__ __forceinline__ void barrier_fail(GridBarrier* bar, int* status) {
  atomicCAS(status, 0, EIC_ETIMEOUT);
  __threadfence();
  atomicOr(&bar->arrived, kBarrierError);
}

// Software barrier over nblocks co-resident (cooperatively launched) blocks:
// the whole grid, or one block group of it. The arrival count only grows while
// the launch runs (its preparation zeroes it), so a block arrives with one
// release add that returns nothing and waits, with acquire loads, until the
// count reaches its own next multiple of nblocks: no block has to see the last
// arrival and publish a new generation. ticket: the block's barriers passed so
// far times nblocks. Every wait is bounded: after max_spin polls the block
// reports EIC_ETIMEOUT. Returns false when the blocks must stop: the error bit
// is part of the word that is polled, so that a passing barrier costs one trip
// to L2 after the last arrival (a separate status word read behind the
// acquire cost a second one, about 0.4 us of the 3.8 us of an empty round).
__device__ __forceinline__ bool grid_barrier(GridBarrier* bar, unsigned long long* ticket, uint32_t nblocks,
                                             uint64_t max_spin, int* status) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned long long target = *ticket + nblocks;
    red_release_add_u64(&bar->arrived, 1ull);
    uint64_t spins = 0;
    unsigned long long seen;
    while ((seen = ld_acquire_gpu_u64(&bar->arrived)) < target) {
      if (++spins > max_spin) {
        barrier_fail(bar, status);
        seen = kBarrierError;
        break;
      }
      __nanosleep(64);
    }
    *ticket = target;
    s_ok = (seen & kBarrierError) == 0;
  }
  __syncthreads();
  return s_ok != 0;
}
