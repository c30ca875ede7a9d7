// Single-source query by Algorithm 1 of the EIC method: steps with
// scheduling pairs <lb, ub> (dynamic stepping, Eq. 1-3), a selection
// threshold st per step (traversal optimisation, Function 2) and rounds of
// window-filtered edge relaxations (Function 1 and the inner loop of
// Algorithm 1), as one persistent cooperative kernel on sm_103a.
//
// Device layout per query (workspace, reused across queries of one graph):
//   dist[ni]     distances in internal ids (non-isolated vertices by degree,
//                densest first), u32, +inf = 0xFFFFFFFF, updated by atomicMin;
//                copied to the caller's buffer in the original numbering at the end
//   fbits[2][n/32]  frontier bitmaps by round parity: the SAP of Algorithm 1 inserts
//                a vertex into the next frontier only if its bit was clear
//   cursor[n]    where the last window relaxed from a vertex ended (offset in its row)
//   q[2][n]      frontier queues, one per round parity
//   sid/sd/scur  settled list in settling order (vertex, final distance, window
//                cursor); step k owns [step_off[k], step_off[k+1])
//   touched[n]   first-step insertions (the first step's ub shrinks, so its
//                tentative distances >= the final ub are reset to +inf)
//   sbits[n/32]  settled bitmap: the pull set of Function 1 is the unsettled part of
//                a prefix of the non-isolated vertices ordered by smallest row weight
//   hist[D]      unsettled vertices per distinct degree (for highD)
//   ring[R]      degree sums of settled vertices by distance mod R (for the
//                sumD differences of Function 2's candidates, while maxW < 2^20;
//                wider weights sum them exactly from the settled list)
//   tasks[]      windows longer than heavy_min, cut into 64-entry tasks for the grid
//
// Phases (one grid barrier each): a round (the first round of a step runs
// Function 1's push set and pull), an optional task phase, and per step one
// statistics pass after which block 0 evaluates Eq. 1-3 and Function 2 and
// publishes the next <st, lb, ub> (with weights of 2^20 and above, after all
// blocks have filled Function 2's bins). In a round each warp takes up to 32
// items at a time (warp-strided, its next items' records loaded ahead); each
// lane finds its item's window in the weight-sorted row, and the warp relaxes
// the concatenation of its lanes' windows, windows longer than heavy_min
// becoming 64-entry tasks for the task phase. A pull set of at least half the
// vertices is swept in vertex order over the unsettled vertices only,
// compacted from the settled bitmap up to 512 vertices at a time. A round with
// few items is fused with those that follow it in the step (fused_round).
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "graph.h"
#include "pool.h"
#include "search.h"
#include "serve.h"
#include "stats.cuh"

using namespace eic;

namespace {

constexpr uint32_t kModePush = 0;     // frontier or push-set vertex: relax its window
constexpr uint32_t kModePull = 2;     // unsettled vertex pulling over its light prefix
constexpr uint32_t kKindNone = 0, kKindVertex = 1, kKindPush = 2, kKindPull = 3;  // a lane's item in a round
constexpr uint32_t kNone = 0xFFFFFFFFu;
constexpr int kShRanks = 1024;
constexpr int kShRing = 2048;
constexpr int64_t kRingNarrow = 16;  // statistics windows up to this width aggregate ring updates per warp

struct KArgs {
  DevGraph G;
  uint32_t* dist;  // internal ids
  uint32_t* out;   // caller's buffer, original ids
  uint32_t* fbits;  // two bitmaps of fwords words
  uint32_t fwords;
  uint32_t* cursor;
  uint32_t* q0;
  uint32_t* q1;
  uint32_t* sid;
  uint32_t* sd;
  uint32_t* scur;
  uint32_t* touched;
  uint32_t* sbits;  // settled bitmap
  uint32_t* hist;
  uint32_t* ring;
  Task* tasks;
  int64_t* step_ub;
  uint32_t* step_off;
  eic_step* trace;
  Ctl* ctl;
  int* status_out;
  uint32_t s;
  uint32_t alpha;
  double beta;
  uint32_t st_num;
  uint32_t gap_shift;
  uint32_t heavy_min;
  uint64_t max_spin;
  uint32_t flags;
  uint32_t ring_mask, ring_shift;
  uint32_t step_cap, trace_cap;
  unsigned long long* timeline;  // NULL unless the caller asked for it
  uint32_t timeline_cap;
  uint32_t nb;  // blocks working on this query: the grid, or one block group of a batch
  uint32_t sweep_words;  // see sweep_chunk
  uint32_t fuse;  // rounds of at most this many items per warp are fused (see fuse_items; 0: none)
};

// Index of the block within the blocks that work on its query.
__device__ __forceinline__ uint32_t qblock(const KArgs& A) { return blockIdx.x % A.nb; }

constexpr uint32_t kMaxBlock = 512;
constexpr uint32_t kMaxWarps = kMaxBlock / 32;
constexpr uint32_t kTaskLen = 64;     // adjacency entries per grid task
// Round-phase shapes (pull prefix entries a lane answers itself, window
// entries a lane relaxes at a time), per kernel: more of each is faster while
// registers last; the batch and serving kernels hold more state.
constexpr uint32_t kPullFastSingle = 8, kRelaxIlpSingle = 2;  // k_eic
constexpr uint32_t kPullFastGroup = 4, kRelaxIlpGroup = 1;    // k_eic_batch, k_eic_serve
constexpr uint32_t kSweepNum = 1, kSweepDen = 2;  // sweep the pull set when it holds >= 1/2 of the vertices
// Settled-bitmap words a warp takes at a time in a sweep: 16 (512 vertices, at
// most 32 words), or fewer on a small graph so that every warp gets four
// chunks: with 16, 90 k vertices kept 178 of 4864 warps busy for 16 batches each.
constexpr uint32_t kSweepChunk = 16;
__host__ __device__ inline uint32_t sweep_chunk(uint32_t ni, uint32_t blocks, uint32_t block_threads) {
  const uint32_t w = (ni / 32 + 1) / (4 * blocks * (block_threads / 32));
  return w < 1 ? 1 : w < kSweepChunk ? w : kSweepChunk;
}
constexpr uint32_t kStageT = 1024;    // tasks staged per block
constexpr uint32_t kWarpStage = 256;  // next-frontier / settled-list appends staged per warp

struct WarpScr {  // one warp's small windows
  uint32_t beg[32];
  uint32_t excl[32];
  uint32_t val[32];  // source distance (push) or best candidate (pull)
  uint32_t u[32];
  uint32_t mode[32];
};

struct RoundScr {
  WarpScr w[kMaxWarps];
};

// Appends gathered in shared memory. Next-frontier and settled-list entries
// are staged per warp and written by the warp with one global atomic per
// kWarpStage entries (no block synchronisation); tasks are staged per block
// and written at the end of a phase.
// A fused round has neither tasks nor a staged next frontier: the local
// queues of its warp groups take their place.
// Warps that share a local queue: 1, 4, 8 and 16 took 13.3, 7.8, 7.2 and 7.3 ms
// on a 1531 x 977 grid at gap_shift 4 (long waves: sharing evens out the work)
// and 123, 117, 119 and 121 ms on a 4096^2 grid (short ones: less to wait for).
constexpr uint32_t kFuseWarps = 8;
constexpr uint32_t kFusePop = 8;      // queued vertices a warp takes at a time
// Graphs with long rows: the longest window of a wave, and the 32-entry
// iterations after which a warp's group hands on what is left. RMAT 250 k with
// wide weights, 1.48 ms without fused rounds: 1.41, 1.47 and 1.50 ms at 6, 16
// and 32 iterations; windows of 64 and 256 entries differ by 2% either way.
constexpr uint32_t kFuseLong = 64;
constexpr uint32_t kFuseIters = 6;
// Road-like graphs hand on after kRoadWaves waves (a step of a grid has some
// tens), fewer where a wave may be long: it takes at most as many iterations as
// the largest degree. The limit is for a chain that one group walks alone while
// every other block waits at the barrier, whose wait is bounded (a path of 10^7
// vertices in one step would outlast it): 1024 waves take 1.2 to 10 ms. The
// group then queues nothing more, which costs the 4096^2 grid 0.1%; its queue
// handed on as below cost 0.6%.
constexpr uint32_t kRoadWaves = 1024, kRoadWavesMin = 64, kRoadIters = 8 * kRoadWaves;
constexpr uint32_t kFuseQueue = 128 * kFuseWarps;  // entries of a local queue (a power of two)
constexpr uint32_t kFuseGroups = (kMaxWarps + kFuseWarps - 1) / kFuseWarps;
static_assert(kFuseGroups <= 15, "a group synchronises on named barrier 1 + its index; 0 is the block barrier");
struct Stage {
  uint32_t tn, tbase;
  union {
    struct {
      Task tbuf[kStageT];
      uint32_t wq[kMaxWarps][kWarpStage];
    };
    uint4 fq[kFuseGroups][kFuseQueue];  // {vertex, distance, row begin, degree}
  };
  uint32_t fcnt[kFuseGroups][3];   // entries pushed to the local queue, by wave mod 3
  uint32_t fstop[kFuseGroups][3];  // set: the group hands on its queue after the wave, by wave mod 3
  uint32_t wf[kMaxWarps][kWarpStage];
};

// One warp's append stage for one list. n is warp-uniform.
struct WarpList {
  uint32_t* buf;    // shared memory, kWarpStage entries
  uint32_t n;       // entries held
  uint32_t* gcnt;   // the list's global count
  uint32_t* glist;  // the list
};

__device__ __forceinline__ void warp_flush(WarpList& W) {
  if (W.n == 0) return;
  uint32_t base = 0;
  if (lane_id() == 0) base = atomicAdd(W.gcnt, W.n);
  base = __shfl_sync(EIC_FULL_MASK, base, 0);
  __syncwarp();
  for (uint32_t k = lane_id(); k < W.n; k += 32) __stcg(&W.glist[base + k], W.buf[k]);
  __syncwarp();
  W.n = 0;
}

// Warp-collective append of v for the lanes with want.
__device__ __forceinline__ void warp_push(WarpList& W, bool want, uint32_t v) {
  const uint32_t mask = __ballot_sync(EIC_FULL_MASK, want);
  if (mask == 0) return;
  const uint32_t cnt = __popc(mask);
  if (W.n + cnt > kWarpStage) warp_flush(W);
  if (want) W.buf[W.n + __popc(mask & ((1u << lane_id()) - 1u))] = v;
  __syncwarp();
  W.n += cnt;
}

struct S2Scr {
  uint32_t hist[kShRanks];
  uint32_t ring[kShRing];
};

constexpr uint32_t kSufMax = 4096;  // Function 2: suffix sums (or bins of wide weights) held in shared memory
constexpr uint32_t kCandMax = 512;  // Function 2: candidates listed for the double-precision evaluation

// A thread sums a run of 8 consecutive words: one word in 9 left free keeps the
// runs of a warp's lanes in different banks (8 lanes met in one: 0.7 us a step,
// 4096^2 grid 99.0 -> 96.1 ms).
__device__ __forceinline__ uint32_t suf_at(uint32_t q) { return q + (q >> 3); }

struct S3Scr {
  uint32_t suf[kSufMax + kSufMax / 8 + 1];
  uint32_t ck[kCandMax], cd[kCandMax];  // a listed candidate and its degree sum
  uint32_t part[kMaxBlock];
  unsigned long long bp[32];  // per warp: the best profit's key (see block_argmax)
  uint32_t bk[32];
};

union PhaseScr {
  RoundScr r;
  S2Scr s2;
  S3Scr s3;
};

// Control values every block holds between barriers.
struct Local {
  int64_t lb, ub, st, lb0;
  uint32_t step, rid, qsel, cur_cnt, s_int;
  uint32_t push_beg, push_end, pull_on, pull_cnt, pull_sweep, extra_s, step_off_cur, done;
};

// State of the step controller, kept in block 0's shared memory across steps.
constexpr uint32_t kStepHist = 128;  // recent steps whose ub and list offset the controller keeps at hand
struct BState {
  int64_t st0, st1, gap_lb, max_settled;
  uint64_t sumd_lb, highd_lb;
  unsigned long long rounds;
  int64_t hub[kStepHist];    // ub of step j at j % kStepHist
  uint32_t hoff[kStepHist];  // step j's first settled-list entry
  uint32_t j0;
  // a boundary that waits for f2_bins
  uint64_t p_sumd;
  int64_t p_gap, p_st0, p_st1;
  uint32_t p_highd, p_settled;
};

struct Counters {  // one thread's counts over the query (added to the 64-bit totals at its end)
  uint32_t frontier, trav, pulls, improved, heavy, pitems;
};

__device__ __forceinline__ void tl_mark(const KArgs& A, uint32_t kind, uint32_t rid) {
  if (!A.timeline) return;
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  uint32_t i = atomicAdd(&A.ctl->tl_len, 1u);
  if (i < A.timeline_cap) {
    A.timeline[2 * i] = t;
    A.timeline[2 * i + 1] = ((unsigned long long)kind << 32) | rid;
  }
}

constexpr uint32_t kFlagBlockTimeline = 1u << 30;  // diagnostic: per-block phase marks

// per-block mark: kind 6 item phase done, 7 task phase done (tag has the block id)
__device__ __forceinline__ void tl_block(const KArgs& A, uint32_t kind, uint32_t rid) {
  if (!A.timeline || !(A.flags & kFlagBlockTimeline) || threadIdx.x != 0) return;
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  uint32_t i = atomicAdd(&A.ctl->tl_len, 1u);
  if (i < A.timeline_cap) {
    A.timeline[2 * i] = t;
    A.timeline[2 * i + 1] = ((unsigned long long)kind << 32) | ((unsigned long long)qblock(A) << 48) | rid;
  }
}

// position of the k-th (from 0) set bit of m; m has more than k set bits
__device__ __forceinline__ uint32_t kth_set_bit(uint32_t m, uint32_t k) {
  uint32_t p = 0;
#pragma unroll
  for (uint32_t half = 16; half >= 1; half >>= 1) {
    const uint32_t low = (uint32_t)__popc(m & ((1u << (p + half)) - 1u));  // set bits below p + half
    if (low <= k) p += half;
  }
  return p;
}

__device__ __forceinline__ int64_t d64(uint32_t d) { return d == EIC_INF ? EIC_INF_T : (int64_t)d; }

// Streaming reads (adjacency entries, the pull list) carry an L2 evict-first
// policy, so that the per-vertex arrays (dist, row offsets, bitmaps, cursors)
// stay in L2 while the adjacency streams past.
__device__ __forceinline__ uint64_t stream_policy() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}

__device__ __forceinline__ uint2 ld_stream(const uint2* p) {
  uint2 v;
  asm("ld.global.nc.L2::cache_hint.v2.u32 {%0, %1}, [%2], %3;" : "=r"(v.x), "=r"(v.y) : "l"(p), "l"(stream_policy()));
  return v;
}

__device__ __forceinline__ uint32_t ld_stream_w(const uint2* p) {
  uint32_t v;
  asm("ld.global.nc.L2::cache_hint.u32 %0, [%1], %2;" : "=r"(v) : "l"(&p->y), "l"(stream_policy()));
  return v;
}

// The same for lists written earlier in the kernel (frontier queue, settled
// list, tasks): L2 only (no L1 copy that another block's write could leave
// stale), evict-first.
__device__ __forceinline__ uint32_t ld_list(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.global.cg.L2::cache_hint.u32 %0, [%1], %2;" : "=r"(v) : "l"(p), "l"(stream_policy()));
  return v;
}

__device__ __forceinline__ uint4 ld_list4(const void* p) {
  uint4 v;
  asm volatile("ld.global.cg.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p), "l"(stream_policy()));
  return v;
}

__device__ __forceinline__ uint4 ld_stream4(const uint4* p) {
  uint4 v;
  asm("ld.global.nc.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
      : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
      : "l"(p), "l"(stream_policy()));
  return v;
}

__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// The window searches (search.h) over the adjacency's weights.
struct AdjWeight {
  const uint2* __restrict__ adj;
  __device__ __forceinline__ uint32_t operator()(uint32_t i) const { return ld_stream_w(&adj[i]); }
};

__device__ __forceinline__ uint32_t lower_bound_w(const uint2* adj, uint32_t b, uint32_t e, int64_t t) {
  return lower_bound(AdjWeight{adj}, b, e, t);
}

__device__ __forceinline__ uint32_t gallop_w(const uint2* adj, uint32_t p, uint32_t e, int64_t t) {
  return gallop(AdjWeight{adj}, p, e, t);
}

__device__ __forceinline__ uint32_t gallop4_w(const uint2* adj, uint32_t p, uint32_t e, int64_t t) {
  return gallop4(AdjWeight{adj}, p, e, t);
}

struct RoundCtx {
  int64_t lb, ub, ub_eff, st, lb0;
  uint32_t rid;
  uint32_t* fbits;  // this round's insertion bitmap
  bool step1;
  uint32_t* qout;
  uint32_t* qcnt_out;
  uint32_t* first_list;
  uint32_t* first_cnt;
  uint32_t* tcnt;
  uint32_t* plain_out;  // set: the next round must be a plain one
};

// Flush the block's task stage to the global list (block-uniform call).
__device__ __forceinline__ void stage_flush(Stage& T, const RoundCtx& R, Task* tasks) {
  __syncthreads();
  if (T.tn == 0) return;  // (next written after the grid barrier)
  __syncthreads();
  if (threadIdx.x == 0) {
    const uint32_t tn = min(T.tn, kStageT);
    T.tn = tn;
    T.tbase = tn ? atomicAdd(R.tcnt, tn) : 0;
  }
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < T.tn; i += blockDim.x) tasks[T.tbase + i] = T.tbuf[i];
  __syncthreads();
  if (threadIdx.x == 0) T.tn = 0;
}

// Cut the window [b, b + len) of vertex u into kTaskLen-entry tasks, staged in
// the block (or written straight to the global list when the stage is full).
__device__ __forceinline__ void emit_tasks(const KArgs& A, const RoundCtx& R, Stage& T, uint32_t b, uint32_t len,
                                           uint32_t u, uint32_t d) {
  const uint32_t nt = (len + kTaskLen - 1) / kTaskLen;
  const uint32_t pos = atomicAdd(&T.tn, nt);
  const uint32_t in_stage = pos < kStageT ? min(nt, kStageT - pos) : 0;
  // the rest goes straight to the global list; capacity covers 2m / 16 tasks per round
  const uint32_t gpos = nt > in_stage ? atomicAdd(R.tcnt, nt - in_stage) : 0;
  for (uint32_t k = 0; k < nt; ++k) {
    Task t;
    t.beg = b + k * kTaskLen;
    t.len = min(kTaskLen, len - k * kTaskLen);
    t.u = u;
    t.d = d;
    if (k < in_stage)
      T.tbuf[pos + k] = t;
    else
      A.tasks[gpos + (k - in_stage)] = t;
  }
}

// The same by a whole warp, for windows of more than kLaneTasks tasks: a lane
// that writes the 10,000 tasks of a hub's window alone keeps its warp, and the
// round, waiting (RMAT 2^25 2.97 -> 2.86 ms, 15 M log-normal 2.00 -> 1.91 ms).
constexpr uint32_t kLaneTasks = 4;
__device__ __forceinline__ void emit_tasks_warp(const KArgs& A, const RoundCtx& R, Stage& T, uint32_t b, uint32_t len,
                                                uint32_t u, uint32_t d) {
  const uint32_t nt = (len + kTaskLen - 1) / kTaskLen;
  uint32_t pos = 0, gpos = 0;
  if (lane_id() == 0) {
    pos = atomicAdd(&T.tn, nt);
    const uint32_t in = pos < kStageT ? min(nt, kStageT - pos) : 0;
    if (nt > in) gpos = atomicAdd(R.tcnt, nt - in) - in;
  }
  pos = __shfl_sync(EIC_FULL_MASK, pos, 0);
  gpos = __shfl_sync(EIC_FULL_MASK, gpos, 0);
  const uint32_t in_stage = pos < kStageT ? min(nt, kStageT - pos) : 0;
  for (uint32_t k = lane_id(); k < nt; k += 32) {
    const Task t = {b + k * kTaskLen, min(kTaskLen, len - k * kTaskLen), u, d};
    if (k < in_stage)
      T.tbuf[pos + k] = t;
    else
      A.tasks[gpos + k] = t;
  }
}

// Sets v's bit in the round's insertion bitmap; true when this call set it.
__device__ __forceinline__ bool claim_bit(const RoundCtx& R, uint32_t v) {
  const uint32_t bit = 1u << (v & 31);
  return !(atomicOr(&R.fbits[v >> 5], bit) & bit);
}

// After a relaxation of v to nd (old = its previous distance): v into the next
// frontier when sap (its insertion bit was set by this lane), into the settled
// (or first-step) list when it had no distance, and in the first step the
// running min over high-degree vertices that becomes ub (Algorithm 1).
// Warp-collective: every lane calls it; the appends go through the warp's stages.
__device__ __forceinline__ void on_claimed(const KArgs& A, const RoundCtx& R, bool ok, bool sap, uint32_t v,
                                           uint32_t nd, uint32_t old, Counters& C, WarpList& Q, WarpList& F) {
  const bool first = ok && old == EIC_INF;
  warp_push(Q, sap, v);
  warp_push(F, first, v);
  if (R.step1 && ok) {
    const uint32_t dg = __ldg(&A.G.row[v + 1]) - __ldg(&A.G.row[v]);
    if (dg >= A.G.highd0) atomicMin(&A.ctl->ub_cand, nd);
  }
  C.improved += ok ? 1 : 0;
}

// The same for a relaxation (ok: it lowered v's distance) whose bit is not yet claimed.
__device__ __forceinline__ void on_success(const KArgs& A, const RoundCtx& R, bool ok, uint32_t v, uint32_t nd,
                                           uint32_t old, Counters& C, WarpList& Q, WarpList& F) {
  const bool sap = ok && claim_bit(R, v);
  on_claimed(A, R, ok, sap, v, nd, old, C, Q, F);
}

// One round over nitems items. Items are frontier vertices (queue qin), or in
// a step's first round Function 1's push set (a settled-list range), its pull
// set and, once, the source. The pull set is a prefix of the weight-ordered
// non-isolated vertices (listed), or, when that prefix holds at least half of
// them, every unsettled vertex (swept in vertex order). Warp by warp without
// block synchronisation, each lane finds its item's window in the
// weight-sorted row; windows up to heavy_min entries are relaxed by the warp
// over their concatenation, kRelaxIlp entries per lane at a time, longer ones
// become grid tasks. A pull reads the prefix of its vertex's row with weight
// < ub - st: its first kPullFast entries in the lane, the rest by the warp.
// Next-frontier and settled-list appends are staged per warp in shared
// memory; tasks per block.
template <uint32_t kPullFast, uint32_t kRelaxIlp>
__device__ void round_phase(const KArgs& A, const RoundCtx& R, const Local& L, RoundScr& S, Stage& T,
                            uint32_t nitems, bool round1, const uint32_t* qin, Counters& C) {
  const uint32_t tid = threadIdx.x, nt = blockDim.x, lane = lane_id(), warp = tid >> 5;
  const uint32_t np = round1 ? L.push_end - L.push_beg : 0;
  const bool sweep = round1 && L.pull_sweep;  // the pull set is every unsettled vertex, swept below
  const uint32_t npp = np + (sweep ? 0u : L.pull_cnt);
  const uint32_t nlisted = sweep ? nitems - L.pull_cnt : nitems;  // items of the listed part
  const uint32_t nwarps = A.nb * (nt >> 5);
  // items a warp takes at a time: 32, or fewer so that a small round reaches every warp, the blocks in turn
  const uint32_t per = nlisted >= 32 * nwarps ? 32u : max(1u, (nlisted + nwarps - 1) / nwarps);
  const uint32_t gwarp = per == 32 ? qblock(A) * (nt >> 5) + warp : warp * A.nb + qblock(A);
  const int64_t pull_bound = R.ub - R.st;
  WarpScr& W = S.w[warp];
  WarpList Qw = {T.wq[warp], 0u, R.qcnt_out, R.qout};
  WarpList Fw = {T.wf[warp], 0u, R.first_cnt, R.first_list};
  // An item's record: {vertex, dist, row begin, row end} for a frontier
  // vertex or the source, {dist, row begin, row end, cursor} for the push set
  // (from the settled list), the nz entry for a listed pull. Records are loaded one
  // warp iteration ahead, a frontier vertex's queue entry two ahead.
  // (the push set's settled-list vertices come in the same way, two ahead).
  // Row bounds are computed from the id: a random read of two offsets per
  // item became three of tables that stay in L1 (RMAT 2^25 2.86 -> 2.77 ms,
  // 15 M log-normal 1.91 -> 1.86 ms).
  auto fetch_id = [&](uint32_t ii) -> uint32_t {
    if (ii >= nlisted) return 0u;
    if (!round1) return ld_list(&qin[ii]);
    return ii < np ? ld_list(&A.sid[L.push_beg + ii]) : 0u;
  };
  auto fetch = [&](uint32_t ii, uint32_t id) -> uint4 {
    if (ii >= nlisted) return make_uint4(0u, 0u, 0u, 0u);
    if (!round1 || ii >= npp) {  // frontier vertex (or the source, once)
      const uint32_t u = round1 ? L.s_int : id;
      const uint2 rr = row_of(A.G, u);
      return make_uint4(u, __ldcg(&A.dist[u]), rr.x, rr.x + rr.y);
    }
    if (ii < np) {
      const uint2 rr = row_of(A.G, id);
      return make_uint4(ld_list(&A.sd[L.push_beg + ii]), rr.x, rr.x + rr.y, ld_list(&A.scur[L.push_beg + ii]));
    }
    return ld_stream4(&A.G.nz[ii - np]);
  };
  // one warp iteration: each lane's item (kind kKindNone: no item)
  auto step_items = [&](const uint4 rec, const uint32_t i, const uint32_t kind) {
    uint32_t u = 0, val = EIC_INF, b = 0, len = 0, mode = kModePush;
    uint32_t pfast = EIC_INF;       // best pull candidate of the lane's vertex
    uint32_t du = EIC_INF;          // the pulled vertex's distance when its pull started
    bool plong = false;             // its prefix is longer than kPullFast entries
    if (kind != kKindNone) {
      if (kind == kKindVertex) {  // frontier vertex (or the source, once)
        u = rec.x;
        const uint32_t d = rec.y, rb = rec.z, re = rec.w;
        val = d;
        if (d != EIC_INF && !(d > 0 && re - rb == 1)) {  // Paths excludes leaves (Algorithm 1)
          C.frontier += 1;
          const int64_t hi = R.ub_eff - (int64_t)d;
          if (hi > 0) {
            b = lower_bound_w(A.G.adj, rb, re, R.lb - (int64_t)d);
            const uint32_t e = gallop4_w(A.G.adj, b, re, hi);
            if (re - rb > kCursorMin) __stcg(&A.cursor[u], e - rb);
            len = e - b;
          }
        }
      } else if (kind == kKindPush) {  // push set: settled, lb0 <= dist <= st (all from the settled list)
        const uint32_t idx = L.push_beg + i;
        const uint32_t d = rec.x;
        val = d;
        if ((int64_t)d >= R.lb0 && (int64_t)d <= R.st) {
          const uint32_t rb = rec.y, re = rec.z;
          if (!(d > 0 && re - rb == 1)) {
            C.frontier += 1;
            const uint32_t cur = rec.w;
            // windows of consecutive steps are contiguous: resume at the cursor
            b = cur == kNone ? lower_bound_w(A.G.adj, rb, re, R.lb - (int64_t)d)
                             : gallop4_w(A.G.adj, rb + cur, re, R.lb - (int64_t)d);
            const uint32_t e = gallop4_w(A.G.adj, b, re, R.ub_eff - (int64_t)d);
            __stcg(&A.scur[idx], e - rb);
            len = e - b;
          }
        }
      } else {  // pull set: unsettled, smallest weight < ub - st (Function 1)
        const uint4 z = rec;  // {vertex, lightest weight or settled word, row begin, row end}
        u = z.x;
        mode = kModePull;
        const uint32_t bits = L.pull_sweep ? z.y : __ldcg(&A.sbits[u >> 5]);
        if (!((bits >> (u & 31)) & 1u)) {  // unsettled: its row's first kPullFast entries, together
          const uint32_t rl = z.w - z.z;
          du = __ldcg(&A.dist[u]);
          uint2 ent[kPullFast];
  #pragma unroll
          for (uint32_t k = 0; k < kPullFast; ++k)
            ent[k] = k < rl ? ld_stream(&A.G.adj[z.z + k]) : make_uint2(0u, EIC_INF);
          uint32_t c = 0;  // the prefix with w < ub - st (rows are weight-sorted)
  #pragma unroll
          for (uint32_t k = 0; k < kPullFast; ++k) c += (k < rl && (int64_t)ent[k].y < pull_bound) ? 1u : 0u;
          C.pitems += c > 0 ? 1 : 0;  // in the pull set iff its lightest edge is below the bound
          plong = c == kPullFast && rl > kPullFast;  // the prefix goes on: the warp scans the rest
          {  // the loaded part of the prefix, answered in the lane
            uint32_t dv[kPullFast];
  #pragma unroll
            for (uint32_t k = 0; k < kPullFast; ++k) dv[k] = k < c ? __ldcg(&A.dist[ent[k].x]) : EIC_INF;
  #pragma unroll
            for (uint32_t k = 0; k < kPullFast; ++k) {
              if (k >= c) continue;
              C.trav += 1;
              C.pulls += 1;
              const int64_t dvv = dv[k];
              if (dv[k] != EIC_INF && dvv >= R.st && dvv < R.lb && dvv + ent[k].y < R.ub)
                pfast = min(pfast, (uint32_t)(dvv + ent[k].y));
            }
          }
          if (plong) {  // the prefix goes on past the lane's entries: find its end, then the rest
                        // is a window like a push window (the warp's concatenation, or grid tasks)
            b = z.z + kPullFast;
            const uint32_t e = pull_bound > (int64_t)A.G.maxw ? z.w : gallop4_w(A.G.adj, b, z.w, pull_bound);
            len = e - b;
          }
        }
      }
    }
    if (len > A.heavy_min && len <= kLaneTasks * kTaskLen) {
      emit_tasks(A, R, T, b, len, u, mode == kModePull ? kNone : val);
      C.heavy += (len + kTaskLen - 1) / kTaskLen;
      len = 0;
    }
    uint32_t big = __ballot_sync(EIC_FULL_MASK, len > A.heavy_min);
    while (big) {  // a long window's tasks are written by the whole warp
      const int src = __ffs(big) - 1;
      big &= big - 1;
      emit_tasks_warp(A, R, T, __shfl_sync(EIC_FULL_MASK, b, src), __shfl_sync(EIC_FULL_MASK, len, src),
                      __shfl_sync(EIC_FULL_MASK, u, src),
                      __shfl_sync(EIC_FULL_MASK, mode == kModePull ? kNone : val, src));
    }
    if (len > A.heavy_min) {
      C.heavy += (len + kTaskLen - 1) / kTaskLen;
      len = 0;
    }
    const uint32_t incl = warp_incl_scan(len);
    const uint32_t total = __shfl_sync(EIC_FULL_MASK, incl, 31);
    W.beg[lane] = b;
    W.excl[lane] = incl - len;
    W.val[lane] = mode == kModePull ? pfast : val;
    W.u[lane] = u;
    W.mode[lane] = mode;
    __syncwarp();
    // the concatenated windows, kRelaxIlp entries per lane at a time (their
    // loads in flight together)
    for (uint32_t g0 = 0; g0 < total; g0 += 32 * kRelaxIlp) {
      uint32_t own[kRelaxIlp], dv[kRelaxIlp], nd[kRelaxIlp], old[kRelaxIlp];
      uint2 ent[kRelaxIlp];
      bool act[kRelaxIlp], push[kRelaxIlp], ok[kRelaxIlp], sap[kRelaxIlp];
#pragma unroll
      for (uint32_t h = 0; h < kRelaxIlp; ++h) {
        const uint32_t g = g0 + h * 32 + lane;
        act[h] = g < total;
        own[h] = 0;
        ent[h] = make_uint2(0u, 0u);
        if (act[h]) {
          uint32_t lo = 0, hi = 31;
          while (lo < hi) {  // last lane whose window starts at or before g
            const uint32_t mid = (lo + hi + 1) >> 1;
            if (W.excl[mid] <= g)
              lo = mid;
            else
              hi = mid - 1;
          }
          own[h] = lo;
          ent[h] = ld_stream(&A.G.adj[W.beg[lo] + (g - W.excl[lo])]);
        }
      }
#pragma unroll
      for (uint32_t h = 0; h < kRelaxIlp; ++h) {
        push[h] = act[h] && W.mode[own[h]] != kModePull;
        // a pull entry is a request answered by a settled v with st <= dist[v] < lb
        act[h] = push[h] || (act[h] && (int64_t)ent[h].y < pull_bound);
        dv[h] = act[h] ? __ldcg(&A.dist[ent[h].x]) : EIC_INF;
      }
#pragma unroll
      for (uint32_t h = 0; h < kRelaxIlp; ++h) {
        ok[h] = false;
        sap[h] = false;
        nd[h] = 0;
        old[h] = 0;
        if (push[h]) {
          C.trav += 1;
          nd[h] = W.val[own[h]] + ent[h].y;  // inside [lb, min(ub, 2^32-1)) by the window bounds
          if (nd[h] < dv[h]) {
            // The insertion bit is claimed together with the atomicMin, not
            // after it. Should the atomicMin find a value <= nd, another
            // relaxation lowered dist[v] in this round after the read above
            // (distances only fall, and the round sees every earlier round's
            // writes), so v is in the next frontier either way and whichever
            // lane set the bit queues it.
            old[h] = atomicMin(&A.dist[ent[h].x], nd[h]);
            sap[h] = claim_bit(R, ent[h].x);
            ok[h] = nd[h] < old[h];
          }
        } else if (act[h]) {
          C.trav += 1;
          C.pulls += 1;
          const int64_t dvv = dv[h];
          if (dv[h] != EIC_INF && dvv >= R.st && dvv < R.lb && dvv + ent[h].y < R.ub)
            atomicMin(&W.val[own[h]], (uint32_t)(dvv + ent[h].y));
        }
      }
#pragma unroll
      for (uint32_t h = 0; h < kRelaxIlp; ++h) on_claimed(A, R, ok[h], sap[h], ent[h].x, nd[h], old[h], C, Qw, Fw);
    }
    __syncwarp();
    bool pok = false, psap = false;
    uint32_t pold = 0;
    const uint32_t pbest = W.val[lane];
    if (mode == kModePull && pbest < du) {  // du was read in this round: the insertion bit is
                                            // claimed with the atomicMin, as for pushes
      pold = atomicMin(&A.dist[u], pbest);
      psap = claim_bit(R, u);
      pok = pbest < pold;
    }
    on_claimed(A, R, pok, psap, u, pbest, pold, C, Qw, Fw);
    __syncwarp();
  };
  const uint32_t stride = nwarps * per;
  auto item = [&](uint32_t base) -> uint32_t { return lane < per ? base + lane : kNone; };
  uint4 pre = fetch(item(gwarp * per), fetch_id(item(gwarp * per)));
  uint32_t idn = fetch_id(item(gwarp * per + stride));
  for (uint32_t base = gwarp * per; base < nlisted; base += stride) {
    const uint32_t i = item(base);
    const uint4 rec = pre;
    pre = fetch(item(base + stride), idn);
    idn = fetch_id(item(base + 2 * stride));
    step_items(rec, i, i >= nlisted ? kKindNone : (!round1 || i >= npp) ? kKindVertex : i < np ? kKindPush : kKindPull);
  }
  if (sweep) {
    // Function 1's pull set swept in vertex order, compacted: a warp takes
    // kSweepChunk settled-bitmap words (32 vertices each) at a time and hands
    // its lanes only the unsettled vertices, 32 per iteration, the next
    // batch's row bounds loaded while the current one runs
    const uint32_t ni = A.G.ni, nwords = (ni + 31) >> 5, nchunks = (nwords + A.sweep_words - 1) / A.sweep_words;
    uint32_t ch = gwarp, m = 0, off = 0, tot = 0, r0 = 0, wn = ~0u;
    auto word_at = [&](uint32_t c) -> uint32_t {
      const uint32_t wi = c * A.sweep_words + lane;
      return c < nchunks && lane < A.sweep_words && wi < nwords ? __ldcg(&A.sbits[wi]) : ~0u;
    };
    auto open_chunk = [&](uint32_t word) {  // this lane's unsettled mask, its exclusive rank, the chunk total
      const uint32_t wi = ch * A.sweep_words + lane;
      uint32_t mm = lane < A.sweep_words && wi < nwords ? ~word : 0u;
      if (wi == nwords - 1 && (ni & 31u)) mm &= (1u << (ni & 31u)) - 1u;
      m = mm;
      const uint32_t c = __popc(mm), inc = warp_incl_scan(c);
      off = inc - c;
      tot = __shfl_sync(EIC_FULL_MASK, inc, 31);
      r0 = 0;
    };
    if (ch < nchunks) {
      open_chunk(word_at(ch));
      wn = word_at(ch + nwarps);
    }
    auto next_batch = [&](bool& ok) -> uint4 {
      while (r0 >= tot && ch < nchunks) {  // warp-uniform: skip to the next chunk with unsettled vertices
        ch += nwarps;
        if (ch >= nchunks) break;
        open_chunk(wn);
        wn = word_at(ch + nwarps);
      }
      ok = false;
      if (ch >= nchunks) return make_uint4(0u, 0u, 0u, 0u);
      const uint32_t r = r0 + lane;
      r0 += 32;
      uint32_t l = 0;  // the last word whose exclusive rank is <= r
#pragma unroll
      for (uint32_t h = 16; h > 0; h >>= 1) {
        const uint32_t o = __shfl_sync(EIC_FULL_MASK, off, l + h);
        if (o <= r) l += h;
      }
      const uint32_t ml = __shfl_sync(EIC_FULL_MASK, m, l), ol = __shfl_sync(EIC_FULL_MASK, off, l);
      if (r >= tot) return make_uint4(0u, 0u, 0u, 0u);
      ok = true;
      const uint32_t v = ((ch * A.sweep_words + l) << 5) + kth_set_bit(ml, r - ol);
      const uint2 rr = row_of(A.G, v);
      return make_uint4(v, 0u, rr.x, rr.x + rr.y);  // {vertex, settled word 0, row}
    };
    bool okc = false;
    uint4 cur = next_batch(okc);
    while (__any_sync(EIC_FULL_MASK, okc)) {
      bool okn = false;
      const uint4 nx = next_batch(okn);
      step_items(cur, 0u, okc ? kKindPull : kKindNone);
      cur = nx;
      okc = okn;
    }
  }
  warp_flush(Qw);
  warp_flush(Fw);
  tl_block(A, 6, R.rid);
  stage_flush(T, R, A.tasks);
}

// The round's tasks, one warp per task of at most 64 entries.
// With kAhead, a warp loads its next task while it runs the current one and
// relaxes a push task's two entries per lane with their loads in flight
// together (the single-query kernel's shape).
template <bool kAhead>
__device__ void task_phase(const KArgs& A, const RoundCtx& R, uint32_t ntasks, Stage& T, Counters& C) {
  const uint32_t lane = lane_id();
  const uint32_t wpb = blockDim.x >> 5;
  const uint32_t nwarps = A.nb * wpb;
  WarpList Qw = {T.wq[threadIdx.x >> 5], 0u, R.qcnt_out, R.qout};
  WarpList Fw = {T.wf[threadIdx.x >> 5], 0u, R.first_cnt, R.first_list};
  const int64_t pull_bound = R.ub - R.st;
  const uint32_t t0 = qblock(A) * wpb + (threadIdx.x >> 5);
  uint4 tnext = make_uint4(0u, 0u, 0u, 0u);
  if constexpr (kAhead) {
    if (t0 < ntasks) tnext = ld_list4(&A.tasks[t0]);
  }
  for (uint32_t t = t0; t < ntasks; t += nwarps) {
    uint4 tv;
    if constexpr (kAhead) {
      tv = tnext;
      if (t + nwarps < ntasks) tnext = ld_list4(&A.tasks[t + nwarps]);
    } else {
      tv = ld_list4(&A.tasks[t]);
    }
    const Task tk = {tv.x, tv.y, tv.z, tv.w};
    if (kAhead && tk.d != kNone) {  // push, both entries' loads in flight together
      uint2 ent[2];
      uint32_t dv[2], nd[2], old[2];
      bool act[2], ok[2], sap[2];
      if (!(tk.beg & 1u)) {  // the task starts on a 16-byte boundary: a lane loads its two entries as one pair
        const uint32_t j = 2 * lane;
        uint4 pr = make_uint4(0u, 0u, 0u, 0u);
        if (j < tk.len) pr = ld_stream4(reinterpret_cast<const uint4*>(A.G.adj + tk.beg + j));  // (2 spare entries)
        act[0] = j < tk.len;
        act[1] = j + 1 < tk.len;
        ent[0] = make_uint2(pr.x, pr.y);
        ent[1] = act[1] ? make_uint2(pr.z, pr.w) : make_uint2(0u, 0u);
      } else {
#pragma unroll
        for (uint32_t h = 0; h < 2; ++h) {
          act[h] = lane + 32 * h < tk.len;
          ent[h] = act[h] ? ld_stream(&A.G.adj[tk.beg + lane + 32 * h]) : make_uint2(0u, 0u);
        }
      }
#pragma unroll
      for (uint32_t h = 0; h < 2; ++h) dv[h] = act[h] ? __ldcg(&A.dist[ent[h].x]) : 0u;
#pragma unroll
      for (uint32_t h = 0; h < 2; ++h) {
        ok[h] = false;
        sap[h] = false;
        old[h] = 0;
        nd[h] = tk.d + ent[h].y;
        if (act[h]) {
          C.trav += 1;
          if (nd[h] < dv[h]) {  // the insertion bit claimed together with the atomicMin, as in the rounds
            old[h] = atomicMin(&A.dist[ent[h].x], nd[h]);
            sap[h] = claim_bit(R, ent[h].x);
            ok[h] = nd[h] < old[h];
          }
        }
      }
#pragma unroll
      for (uint32_t h = 0; h < 2; ++h) on_claimed(A, R, ok[h], sap[h], ent[h].x, nd[h], old[h], C, Qw, Fw);
    } else if (tk.d != kNone) {  // push
#pragma unroll
      for (uint32_t h = 0; h < 2; ++h) {
        const uint32_t j = lane + 32 * h;
        bool ok = false;
        uint32_t v = 0, nd = 0, old = 0;
        if (j < tk.len) {
          const uint2 ent = ld_stream(&A.G.adj[tk.beg + j]);
          v = ent.x;
          nd = tk.d + ent.y;
          C.trav += 1;
          const uint32_t dv = __ldcg(&A.dist[v]);
          if (nd < dv) {
            old = atomicMin(&A.dist[v], nd);
            ok = nd < old;
          }
        }
        on_success(A, R, ok, v, nd, old, C, Qw, Fw);
      }
    } else {  // pull request over a row segment
      uint32_t best = EIC_INF;
#pragma unroll
      for (uint32_t h = 0; h < 2; ++h) {
        const uint32_t j = lane + 32 * h;
        if (j < tk.len) {
          const uint2 ent = ld_stream(&A.G.adj[tk.beg + j]);
          if ((int64_t)ent.y < pull_bound) {
            C.trav += 1;
            C.pulls += 1;
            const uint32_t dv = __ldcg(&A.dist[ent.x]);
            const int64_t dvv = dv;
            if (dv != EIC_INF && dvv >= R.st && dvv < R.lb && dvv + ent.y < R.ub)
              best = min(best, (uint32_t)(dvv + ent.y));
          }
        }
      }
      for (int o = 16; o > 0; o >>= 1) best = min(best, __shfl_xor_sync(EIC_FULL_MASK, best, o));
      bool ok = false;
      uint32_t old = 0;
      if (lane == 0 && best != EIC_INF) {
        old = atomicMin(&A.dist[tk.u], best);
        ok = best < old;
      }
      on_success(A, R, ok, tk.u, best, old, C, Qw, Fw);
    }
  }
  warp_flush(Qw);
  warp_flush(Fw);
  tl_block(A, 7, R.rid);
  stage_flush(T, R, A.tasks);
}

// The first candidate index with the largest positive profit over the block
// (ties: the smaller index), or 0xFFFFFFFF when no profit is positive. The
// reduction compares integer keys: a positive double's bit pattern orders as
// the double does, and a profit <= 0 gets key 0 (this GPU's double-precision
// units are few, and a block of double compares queues on them).
__device__ __forceinline__ uint32_t block_argmax(S3Scr& S, double best, uint32_t bk) {
  const uint32_t t = threadIdx.x, nt = blockDim.x;
  unsigned long long key = best > 0.0 ? (unsigned long long)__double_as_longlong(best) : 0ull;
  if (!key) bk = 0xFFFFFFFFu;
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long ok = __shfl_down_sync(EIC_FULL_MASK, key, o);
    const uint32_t okk = __shfl_down_sync(EIC_FULL_MASK, bk, o);
    if (ok > key || (ok == key && okk < bk)) {
      key = ok;
      bk = okk;
    }
  }
  __syncthreads();
  if ((t & 31) == 0) {
    S.bp[t >> 5] = key;
    S.bk[t >> 5] = bk;
  }
  __syncthreads();
  if (t < 32) {
    key = t < (nt >> 5) ? S.bp[t] : 0ull;
    bk = t < (nt >> 5) ? S.bk[t] : 0xFFFFFFFFu;
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long ok = __shfl_down_sync(EIC_FULL_MASK, key, o);
      const uint32_t okk = __shfl_down_sync(EIC_FULL_MASK, bk, o);
      if (ok > key || (ok == key && okk < bk)) {
        key = ok;
        bk = okk;
      }
    }
    if (t == 0) S.bk[0] = key ? bk : 0xFFFFFFFFu;
  }
  __syncthreads();
  const uint32_t k = S.bk[0];
  __syncthreads();
  return k;
}

// The candidate grid x_k = st0 + floor(k span / ST_NUM) (Section 4.1): a
// shift when ST_NUM is a power of two (the paper's 1024), else a division.
__device__ __forceinline__ int64_t st_candidate(uint32_t k, uint64_t span, uint32_t st_num, uint32_t sh, int64_t st0) {
  const uint64_t q = (uint64_t)k * span;
  return st0 + (int64_t)(sh < 32 ? q >> sh : q / st_num);
}


// Function 2 for weights of 2^20 and above, with D(x') summed exactly from the
// settled list: over the entries of the steps that end above wl, the vertex at
// distance d >= wl adds its degree to bin 1 + k_d, k_d the last candidate k
// with x_k <= d (-1 if none); after a suffix sum, D(x_k) is bin 1 + k for x_k >=
// wl and bin 0 for a candidate clamped to wl. All blocks of the query fill the
// bins (the ring's words, unused for such weights) between two grid barriers:
// one block alone took 95, 185 and 271 us in three steps of an RMAT graph of
// 250 k vertices. A block counts in shared memory first when it has at least
// as many entries as there are bins.
__device__ __forceinline__ void f2_bins(const KArgs& A, S3Scr& S, const Ctl* c) {
  const uint32_t t = threadIdx.x, nt = blockDim.x, n0 = qblock(A) * nt, stride = A.nb * nt;
  const uint32_t beg = __ldcg(&c->f2_beg), end = __ldcg(&c->f2_end);
  const int64_t wl = __ldcg(&c->f2_wl), st0 = __ldcg(&c->f2_st0);
  const uint64_t span = __ldcg(&c->f2_span);
  const uint32_t nbins = A.st_num + 2;
  const bool sh = nbins <= kSufMax && (end - beg) / A.nb >= nbins;
  if (sh)
    for (uint32_t q = t; q < nbins; q += nt) S.suf[q] = 0u;
  __syncthreads();
  for (uint32_t i = beg + n0 + t; i < end; i += stride) {
    const int64_t d = ld_list(&A.sd[i]);
    if (d < wl) continue;
    const uint32_t dg = __ldg(&A.G.dvals[degree_rank(A.G, ld_list(&A.sid[i]))]);
    uint64_t cnt;  // how many x_k are <= d: the k with k (st1 - st0) < (d - st0 + 1) ST_NUM
    if (d < st0)
      cnt = 0;
    else if (span == 0)
      cnt = nbins - 1;
    else
      cnt = min(((uint64_t)(d - st0 + 1) * A.st_num + span - 1) / span, (uint64_t)nbins - 1);
    atomicAdd(sh ? &S.suf[cnt] : &A.ring[cnt], dg);  // (a degree sum is at most 2m < 2^32)
  }
  __syncthreads();
  if (sh) {
    for (uint32_t q = t; q < nbins; q += nt)
      if (S.suf[q]) atomicAdd(&A.ring[q], S.suf[q]);
    __syncthreads();
  }
}

// The same out of line for the batch and serving kernels, which hold their
// arguments in shared memory: inlined there it costs their query loop registers.
__device__ __noinline__ void f2_bins_call(const KArgs& A, S3Scr& S, const Ctl* c) { f2_bins(A, S, c); }

// The candidate of the bins for an ST_NUM above the shared-memory window (one
// block): suffix sums in place, every profit in double precision.
__device__ __noinline__ int64_t block_st_bins(uint32_t* bins, uint32_t st_num, uint32_t maxw, uint64_t two_m, S3Scr& S,
                                              int64_t ub, uint64_t sumd_ub, int64_t y, int64_t st0, int64_t st1) {
  const uint32_t t = threadIdx.x, nt = blockDim.x;
  const int64_t wl = ub - (int64_t)maxw > 0 ? ub - (int64_t)maxw : 0;
  const uint64_t nbins = (uint64_t)st_num + 2, span = (uint64_t)(st1 - st0);
  // suffix sums: chunk totals, a scan over the chunks, then within the chunks
  const uint64_t cs = (nbins + nt - 1) / nt;
  const uint64_t q0 = min(nbins, t * cs), q1 = min(nbins, q0 + cs);
  uint32_t mine = 0;
  for (uint64_t q = q0; q < q1; ++q) mine += __ldcg(&bins[q]);
  S.part[t] = mine;
  __syncthreads();
  for (uint32_t o = 1; o < nt; o <<= 1) {
    const uint32_t v = t + o < nt ? S.part[t + o] : 0;
    __syncthreads();
    S.part[t] += v;
    __syncthreads();
  }
  uint32_t acc = t + 1 < nt ? S.part[t + 1] : 0;
  for (uint64_t q = q1; q > q0; --q) {
    acc += __ldcg(&bins[q - 1]);
    __stcg(&bins[q - 1], acc);
  }
  __syncthreads();
  double best = 0.0;
  uint32_t bk = 0xFFFFFFFFu;
  const uint32_t gsh = (st_num & (st_num - 1)) == 0 ? __ffs(st_num) - 1 : 32u;
  for (uint32_t k = t; k <= st_num; k += nt) {
    const int64_t x = st_candidate(k, span, st_num, gsh, st0);
    if (x >= ub) continue;
    const uint32_t dsum = __ldcg(&bins[x >= wl ? (uint64_t)k + 1 : 0]);
    const double p = dev_profit(x, ub, y, dsum, sumd_ub, maxw, two_m);
    if (p > best) {
      best = p;
      bk = k;
    }
  }
  const uint32_t k = block_argmax(S, best, bk);
  return k == 0xFFFFFFFFu ? ub : st_candidate(k, span, st_num, gsh, st0);
}

// A fused round: the FUSED local iterations of Section 4.1 (bucket fusion), in
// a step's rounds after the first (and its first round too when the step has
// no pull) that have few enough items (fuse_items). The round's
// frontier vertices (or the push set, whose windows start at their cursors)
// are dealt evenly to groups of kFuseWarps warps all over the query's blocks.
// A group relaxes its vertices' windows; every vertex it improves goes into
// the group's local queue (shared memory, kFuseQueue entries) and is relaxed
// in a later wave of the group, until the local queue is empty. The groups
// advance independently, with no grid barrier between waves: the round
// replaces the step's remaining rounds. A queued vertex that has a smaller
// distance by the time its wave comes is dropped: whoever lowered it queued it
// too (within a step any order of the relaxations is exact). What a full
// local queue cannot take goes to the next round's queue through the round's
// SAP bitmap, as in a plain round.
//
// A wave is bound by its chain of dependent accesses, so the chain is two
// long: the row's entries, then the atomicMin on the neighbours. Row bounds
// come from the vertex id (row_of) before the vertex is queued, the check of
// a queued vertex's distance flies with its row's entries, and a neighbour's
// row is prefetched into L2 while its atomicMin is under way. Measured against
// the earlier form (32 items to a warp, one local queue per warp, a chain of
// row bounds, entries, distance, atomicMin): a round of the 4096^2 grid went
// from 26.1 to 14.4 us, its query from 168 to 118 ms, and the 1531 x 977 grid
// at gap_shift 4 from 18.7 to 7.2 ms.
//
// kRoad: no window is longer than heavy_min (every degree of the graph is at
// most that). Otherwise a window may be too long for one warp: an item's then
// becomes grid tasks, a vertex improved in the round waits for the next, plain
// round. A group that has spent its waves (kRoad) or kFuseIters iterations
// leaves the rest to the next round, where it is dealt to all warps again (34
// items whose subtree of 5000 vertices stayed in 34 groups took 220 us, plain
// rounds 130 us). On graphs with long rows fusion saves the 8 us of each small
// round: uniform 2^14 vertices 488 -> 394 us, RMAT 131 k 579 -> 518 us, RMAT
// 2^22 1029 -> 990 us, RMAT 2^25 3.03 -> 2.94 ms a query.
template <bool kRoad>
__device__ void fused_round(const KArgs& A, const RoundCtx& R, const Local& L, Stage& T, uint32_t nitems, bool round1,
                            const uint32_t* qin, Counters& C) {
  const uint32_t lane = lane_id(), warp = threadIdx.x >> 5;
  const uint32_t wpb = blockDim.x >> 5, gpb = (wpb + kFuseWarps - 1) / kFuseWarps;
  const uint32_t grp = warp / kFuseWarps, gw = warp - grp * kFuseWarps;  // the group, the warp's place in it
  const uint32_t gn = min(kFuseWarps, wpb - grp * kFuseWarps);           // its warps
  auto group_sync = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(grp + 1), "r"(gn * 32) : "memory"); };
  uint4* fq = T.fq[grp];  // the local queue: a ring of kFuseQueue entries
  // Written in a wave, read by all between its barrier and the next one, and
  // cleared after that: a warp that is ahead writes the next wave's.
  uint32_t *fcnt = T.fcnt[grp], *fstop = T.fstop[grp];
  WarpList Fw = {T.wf[warp], 0u, R.first_cnt, R.first_list};
  // the group's share of the items: one block's groups are a grid stride
  // apart, so that few items still reach every SM
  const uint32_t per = (nitems + A.nb * gpb - 1) / (A.nb * gpb);
  uint32_t i0 = min(nitems, (grp * A.nb + qblock(A)) * per);
  const uint32_t i1 = min(nitems, i0 + per);
  const uint32_t np = round1 ? L.push_end - L.push_beg : 0;
  if (gw == 0 && lane < 3) fcnt[lane] = fstop[lane] = 0;
  group_sync();
  uint32_t spent = 0;  // the warp's iterations
  uint32_t waves = kRoad ? min(kRoadWaves, max(kRoadWavesMin, kRoadIters / A.G.max_deg)) : 0u;  // the group's waves left
  uint32_t lh = 0, lt = 0, wave = 0;  // the ring's head and tail, the wave mod 3 (the same in every thread of the group)
  while (i0 < i1 || lh != lt) {
    uint32_t d = EIC_INF, b = 0, len = 0, u = 0, rb = 0, deg = 0;
    uint32_t now = EIC_INF;  // a queued vertex's distance as its wave begins
    bool vertex = false;     // a frontier vertex (or the source): its window starts at its row
    bool seed = false;       // one of the round's items
    uint32_t room = kFuseQueue - (lt - lh);
    if (kRoad) {  // its waves spent, the group queues nothing more: what it improves goes to the next round
      if (waves == 0)
        room = 0;
      else
        --waves;
    }
    if (i0 < i1) {
      const uint32_t take = min(i1 - i0, 32 * gn), each = (take + gn - 1) / gn;
      const uint32_t i = i0 + gw * each + lane;
      const bool mine = lane < each && gw * each + lane < take;
      i0 += take;
      if (mine && i < np) {  // push set entry: settled, lb0 <= dist <= st (Function 1)
        const uint32_t idx = L.push_beg + i;
        d = ld_list(&A.sd[idx]);
        u = ld_list(&A.sid[idx]);
        const uint32_t cur = ld_list(&A.scur[idx]);
        const uint2 rr = row_of(A.G, u);
        if ((int64_t)d >= R.lb0 && (int64_t)d <= R.st && !(d > 0 && rr.y == 1)) {
          C.frontier += 1;
          b = rr.x;
          len = rr.y;  // a short row: read whole, filtered by the window
          if (rr.y > kCursorMin) {
            b = cur == kNone ? lower_bound_w(A.G.adj, rr.x, rr.x + rr.y, R.lb - (int64_t)d)
                             : gallop_w(A.G.adj, rr.x + cur, rr.x + rr.y, R.lb - (int64_t)d);
            const uint32_t e = gallop_w(A.G.adj, b, rr.x + rr.y, R.ub_eff - (int64_t)d);
            __stcg(&A.scur[idx], e - rr.x);
            len = e - b;
          }
          now = d;
        }
        seed = true;
      } else if (mine) {  // a frontier vertex, or in a step's first round the source, once
        u = round1 ? L.s_int : ld_list(&qin[i]);
        const uint2 rr = row_of(A.G, u);
        rb = rr.x;
        deg = rr.y;
        d = now = __ldcg(&A.dist[u]);
        vertex = d != EIC_INF && !(d > 0 && deg == 1);  // Paths excludes leaves (Algorithm 1)
        seed = true;
      }
    } else {
      const uint32_t take = min(lt - lh, kFusePop * gn), each = (take + gn - 1) / gn;
      if (lane < each && gw * each + lane < take) {
        const uint4 q = fq[(lh + gw * each + lane) & (kFuseQueue - 1)];
        u = q.x;
        d = q.y;
        rb = q.z;
        deg = q.w;
        now = __ldcg(&A.dist[u]);
        vertex = true;
      }
      lh += take;
    }
    if (vertex && (int64_t)d < R.ub_eff) {
      // d >= lb: the window is the row's prefix with weight < ub - d; rows are
      // short, so the whole row is read and filtered (a search only for rows
      // that keep a cursor)
      b = rb;
      len = deg;
      if (deg > kCursorMin) {
        const uint32_t e = gallop_w(A.G.adj, rb, rb + deg, R.ub_eff - (int64_t)d);
        __stcg(&A.cursor[u], e - rb);
        if ((int64_t)d < R.lb) b = lower_bound_w(A.G.adj, rb, e, R.lb - (int64_t)d);  // (the source)
        len = e - b;
      }
    }
    if (!kRoad && __any_sync(EIC_FULL_MASK, len > kFuseLong)) {
      // Windows too long for a wave. An item's becomes grid tasks, once per
      // vertex and round (what the task list is sized for); a vertex improved
      // in this round goes to the next one, which is then a plain round.
      const bool lng = len > kFuseLong;
      uint32_t emit = __ballot_sync(EIC_FULL_MASK, lng && seed);
      while (emit) {
        const int src = __ffs(emit) - 1;
        emit &= emit - 1;
        const uint32_t tb = __shfl_sync(EIC_FULL_MASK, b, src), tl = __shfl_sync(EIC_FULL_MASK, len, src);
        const uint32_t tu = __shfl_sync(EIC_FULL_MASK, u, src), td = __shfl_sync(EIC_FULL_MASK, d, src);
        const uint32_t ntask = (tl + kTaskLen - 1) / kTaskLen;
        uint32_t at = 0;
        if (lane == 0) at = atomicAdd(R.tcnt, ntask);
        at = __shfl_sync(EIC_FULL_MASK, at, 0);
        for (uint32_t k = lane; k < ntask; k += 32)
          A.tasks[at + k] = Task{tb + k * kTaskLen, min(kTaskLen, tl - k * kTaskLen), tu, td};
        if (lane == 0) C.heavy += ntask;
      }
      const bool sap = lng && !seed && claim_bit(R, u);
      const uint32_t slot = warp_append(sap, R.qcnt_out);
      if (sap) {
        __stcg(&R.qout[slot], u);
        __stcg(R.plain_out, 1u);
      }
      if (lng && !seed) vertex = false;  // (relaxed, and counted, in the next round)
      if (lng) len = 0;
    }
    const uint32_t incl = warp_incl_scan(len);
    const uint32_t total = __shfl_sync(EIC_FULL_MASK, incl, 31);
    const uint32_t excl = incl - len, full = __ballot_sync(EIC_FULL_MASK, len != 0);  // lanes with a window
    uint32_t live = 0;  // lanes whose vertex still has the distance it was queued with
    if (!kRoad && total == 0) C.frontier += vertex && now == d ? 1 : 0;
    if (!kRoad) {
      spent += (total + 31) / 32;
      if (spent > kFuseIters && lane == 0) fstop[wave] = 1;
    }
    for (uint32_t g0 = 0; g0 < total; g0 += 32) {
      const uint32_t g = g0 + lane;
      // the window that holds g: the last one that starts at or before it, from the lanes' votes (a search of
      // their offsets in shared memory was five dependent reads a wave: 4096^2 grid 100.9 -> 99.3 ms)
      const uint32_t at = excl - g0;
      const uint32_t starts = __reduce_or_sync(EIC_FULL_MASK, len != 0 && excl >= g0 && at < 32 ? 1u << at : 0u);
      const uint32_t before = g0 ? __popc(__ballot_sync(EIC_FULL_MASK, len != 0 && excl < g0)) : 0u;
      const uint32_t own = kth_set_bit(full, before + __popc(starts & (0xFFFFFFFFu >> (31 - lane))) - 1);
      const uint32_t first_at = __shfl_sync(EIC_FULL_MASK, b - excl, own), du = __shfl_sync(EIC_FULL_MASK, d, own);
      uint2 ent = make_uint2(0u, 0u);
      if (g < total) ent = ld_stream(&A.G.adj[first_at + g]);
      if (g0 == 0) {
        live = __ballot_sync(EIC_FULL_MASK, now == d);
        if (!kRoad) C.frontier += vertex && now == d ? 1 : 0;
      }
      bool ok = false, first = false;
      uint32_t nd = 0;
      uint2 rr = make_uint2(0u, 0u);
      const uint32_t v = ent.x;
      if (g < total && ((live >> own) & 1u)) {
        const int64_t t = (int64_t)du + ent.y;
        if (t >= R.lb && t < R.ub_eff) {  // in the window [lb - d, ub - d)
          C.trav += 1;
          nd = (uint32_t)t;
          const uint32_t old = atomicMin(&A.dist[v], nd);
          rr = row_of(A.G, v);
          prefetch_l2(&A.G.adj[rr.x]);
          ok = nd < old;
          first = ok && old == EIC_INF;
        }
      }
      C.improved += ok ? 1 : 0;
      // into the local queue while it has room, else into the next round's queue (SAP); leaves are not relaxed from
      const bool go = ok && rr.y > 1;
      const uint32_t m = __ballot_sync(EIC_FULL_MASK, go);
      if (m) {
        uint32_t pos = 0;
        if (lane == 0) pos = atomicAdd(&fcnt[wave], (uint32_t)__popc(m));
        pos = __shfl_sync(EIC_FULL_MASK, pos, 0) + __popc(m & ((1u << lane) - 1u));
        if (go && pos < room) fq[(lt + pos) & (kFuseQueue - 1)] = make_uint4(v, nd, rr.x, rr.y);
        const bool over = go && pos >= room;
        if (__any_sync(EIC_FULL_MASK, over)) {
          const bool sap = over && claim_bit(R, v);
          const uint32_t slot = warp_append(sap, R.qcnt_out);
          if (sap) __stcg(&R.qout[slot], v);
        }
      }
      warp_push(Fw, first, v);
    }
    if (kRoad) C.frontier += vertex && now == d ? 1 : 0;  // (here and not with the entries: 3% on
                                                            // grids, by the kernel's registers)
    group_sync();  // the wave's pushes are complete
    lt += min(fcnt[wave], room);
    const bool stop = !kRoad && fstop[wave] && i0 >= i1;
    const uint32_t last = wave == 0 ? 2 : wave - 1;  // read by all before this barrier, next used two waves on
    if (gw == 0 && lane == 0) fcnt[last] = fstop[last] = 0;
    wave = wave == 2 ? 0 : wave + 1;
    if (stop) {  // long enough alone: the rest goes to the next round
      for (uint32_t i = lh + gw * 32; i < lt; i += gn * 32) {
        const bool in = i + lane < lt;
        const uint32_t v = in ? fq[(i + lane) & (kFuseQueue - 1)].x : 0u;
        const bool sap = in && claim_bit(R, v);
        const uint32_t slot = warp_append(sap, R.qcnt_out);
        if (sap) __stcg(&R.qout[slot], v);
      }
      break;
    }
  }
  warp_flush(Fw);
  tl_block(A, 6, R.rid);
}

// Function 2's window [wl, ub) of the ring (one slot per distance), in at most
// kSufMax chunks of cs slots.
struct F2Window {
  int64_t wl;
  uint32_t slots, cs, chunks;
};

__device__ __forceinline__ F2Window f2_window(int64_t ub, int64_t maxw) {
  F2Window w;
  w.wl = ub > maxw ? ub - maxw : 0;
  w.slots = (uint32_t)(ub - w.wl);
  w.cs = (w.slots + kSufMax - 1) / kSufMax;
  w.chunks = w.cs > 1 ? (w.slots + w.cs - 1) / w.cs : w.slots;
  return w;
}

// The chunk sums of the window to shared memory (block-wide, no barrier).
__device__ __forceinline__ void f2_load(const KArgs& A, S3Scr& S, const F2Window& w) {
  if (w.cs <= 1) {
#pragma unroll 4
    for (uint32_t q = threadIdx.x; q < w.slots; q += blockDim.x)
      S.suf[suf_at(q)] = __ldcg(&A.ring[(uint32_t)(w.wl + q) & A.ring_mask]);
  } else {
    for (uint32_t q = threadIdx.x; q < w.chunks; q += blockDim.x) {
      const uint32_t b = q * w.cs, e = min(w.slots, b + w.cs);
      uint32_t sum = 0;
#pragma unroll 4
      for (uint32_t i = b; i < e; ++i) sum += __ldcg(&A.ring[(uint32_t)(w.wl + i) & A.ring_mask]);
      S.suf[suf_at(q)] = sum;
    }
  }
}

// Function 2 over the ST_NUM grid of candidates x_k = st0 + floor(k (st1 - st0)
// / ST_NUM) < ub (one whole block; every thread gets the result): the first
// candidate with the largest positive profit, or ub. D(x') = sumD(x') -
// sumD(ub), the degree sum of the settled vertices with x' <= dist < ub, x' =
// max(x, ub - maxW), is a suffix sum of the ring (one slot per distance: maxW <
// 2^20), or, for wider weights, of f2_bins' bins (w.cs = 0: one chunk per bin).
//
// The profit is specified in double precision, of which this GPU has two
// operations per clock and SM: ST_NUM candidates with three divisions each cost
// 10 us. Only candidates that can win are evaluated in it: those with pushed >
// pulled, an exact integer comparison (each double operation rounds
// monotonically, so pushed <= pulled there means profit <= 0 here), and, of
// these, those whose single-precision estimate comes within twice its error
// bound of the best. The estimate's error is at most 26 roundings of
// 2^-24 of pushed <= pushed(x = wl), which bounds every term; e takes 32.
// Function 2 went from 5.6 to 2.5 us a step on a uniform graph of 2^14 vertices.
__device__ int64_t block_compute_st(const KArgs& A, S3Scr& S, const F2Window& w, int64_t ub, uint64_t sumd_ub,
                                    int64_t y, int64_t st0, int64_t st1, uint32_t wsuf, uint32_t* s_rw) {
  __shared__ uint32_t s_best, s_cnt;
  const uint32_t t = threadIdx.x, nt = blockDim.x, lane = lane_id(), warp = t >> 5, nw = nt >> 5;
  const int64_t maxw = A.G.maxw;
  {  // suffix sums in place: this thread's run of chunks behind all later threads'
    uint32_t x = lane < nw ? s_rw[lane] : 0u;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t z = __shfl_down_sync(EIC_FULL_MASK, x, o);
      if (lane + o < 32) x += z;
    }
    uint32_t run = __shfl_sync(EIC_FULL_MASK, x, (warp + 1) & 31);
    if (warp + 1 >= nw) run = 0;
    const uint32_t later = __shfl_down_sync(EIC_FULL_MASK, wsuf, 1);
    if (lane < 31) run += later;
    const uint32_t per = (w.chunks + nt - 1) / nt, b = min(w.chunks, t * per), e = min(w.chunks, b + per);
    for (uint32_t q = e; q > b; --q) {
      run += S.suf[suf_at(q - 1)];
      S.suf[suf_at(q - 1)] = run;
    }
    if (t == 0) {
      S.suf[suf_at(w.chunks)] = 0;
      s_best = 0;
      s_cnt = 0;
    }
  }
  __syncthreads();
  const uint64_t span = (uint64_t)(st1 - st0);
  const uint32_t gsh = (A.st_num & (A.st_num - 1)) == 0 ? __ffs(A.st_num) - 1 : 32u;
  const int64_t lo = ub - maxw;
  const uint32_t push_w = (uint32_t)((y < ub + maxw ? y : ub + maxw) - ub);  // ub0 - lb <= maxW
  const float inv = 1.0f / (float)maxw, inv2m = 1.0f / (float)A.G.two_m, fsumd = (float)sumd_ub;
  const float e = (float)push_w * (float)S.suf[suf_at(0)] * inv * (1.0f / 524288.0f);  // 2^-19 pushed(wl)
  // candidate k: false when it cannot be the answer, else its degree sum and estimate + e
  auto estimate = [&](uint32_t k, uint32_t& dsum, float& v) -> bool {
    const int64_t x = st_candidate(k, span, A.st_num, gsh, st0);
    if (x >= ub) return false;
    const int64_t xc = x > lo ? x : lo;
    if (k > 0) {  // the profit depends on x' only: the first candidate of each x' decides the argmax
      const int64_t xp = st_candidate(k - 1, span, A.st_num, gsh, st0);
      if ((xp > lo ? xp : lo) == xc) return false;
    }
    const uint32_t i = (uint32_t)(xc - w.wl);
    if (w.cs == 0) {
      dsum = S.suf[suf_at(x >= w.wl ? k + 1 : 0)];
    } else if (w.cs == 1) {
      dsum = S.suf[suf_at(i)];
    } else {
      const uint32_t c = i / w.cs, ce = min(w.slots, (c + 1) * w.cs);
      dsum = S.suf[suf_at(c + 1)];
      for (uint32_t q = i; q < ce; ++q) dsum += __ldcg(&A.ring[(uint32_t)(w.wl + q) & A.ring_mask]);
    }
    const uint32_t pull_w = (uint32_t)((y < xc + maxw ? y : xc + maxw) - xc);  // ub1 - x' <= maxW
    if ((uint64_t)push_w * dsum <= (uint64_t)pull_w * sumd_ub) return false;
    const float pushed = (float)push_w * (float)dsum * inv, pulled = (float)pull_w * fsumd * inv;
    v = pushed - pulled * (float)dsum * inv2m - pulled + e;
    return v > 0.0f;
  };
  uint32_t mine = 0;  // (a positive float's bits order as the float)
  for (uint32_t k = t; k <= A.st_num; k += nt) {
    uint32_t dsum;
    float v;
    if (estimate(k, dsum, v)) mine = max(mine, __float_as_uint(v));
  }
  mine = __reduce_max_sync(EIC_FULL_MASK, mine);
  if (lane == 0 && mine) atomicMax(&s_best, mine);
  __syncthreads();
  if (s_best == 0) return ub;
  const float least = __uint_as_float(s_best) - 2.0f * e;
  for (uint32_t k = t; k <= A.st_num; k += nt) {
    uint32_t dsum;
    float v;
    if (estimate(k, dsum, v) && v >= least) {
      const uint32_t at = atomicAdd(&s_cnt, 1u);
      if (at < kCandMax) {
        S.ck[at] = k;
        S.cd[at] = dsum;
      }
    }
  }
  __syncthreads();
  const uint32_t cnt = s_cnt;
  double best = 0.0;
  uint32_t bk = 0xFFFFFFFFu;
  if (cnt <= kCandMax) {
    for (uint32_t i = t; i < cnt; i += nt) {
      const uint32_t k = S.ck[i];
      const double p = dev_profit(st_candidate(k, span, A.st_num, gsh, st0), ub, y, S.cd[i], sumd_ub, A.G.maxw, A.G.two_m);
      if (p > best || (p == best && p > 0.0 && k < bk)) {
        best = p;
        bk = k;
      }
    }
  } else {  // more than the list holds (a flat profit): each thread its own
    for (uint32_t k = t; k <= A.st_num; k += nt) {
      uint32_t dsum;
      float v;
      if (!estimate(k, dsum, v) || v < least) continue;
      const double p = dev_profit(st_candidate(k, span, A.st_num, gsh, st0), ub, y, dsum, sumd_ub, A.G.maxw, A.G.two_m);
      if (p > best) {
        best = p;
        bk = k;
      }
    }
  }
  const uint32_t k = block_argmax(S, best, bk);
  return k == 0xFFFFFFFFu ? ub : st_candidate(k, span, A.st_num, gsh, st0);
}

// Step boundary, executed by block 0 once every block finished the
// statistics pass: sumD(ub), highD(ub), gap(ub) (Eq. 1-3), termination
// (Algorithm 1), computeST (Function 2) and the push/pull sets of the next
// step's Function 1. Publishes the new control values before the grid barrier.
// The whole query waits for it, so it is laid out for latency: what depends on
// <lb, ub> alone (the counters, the degree histogram, Function 2's window of
// the ring) is loaded at once, highD and the window's sums share their
// barriers, and double precision is used only where a single-precision
// estimate cannot decide. A boundary went from 10.8 to 7.2 us on the 4096^2
// grid, from 10.9 to 5.8 us on a uniform graph of 2^14 vertices.
//
// With weights of 2^20 and above and Function 2 to be evaluated, it stops
// before that and asks all blocks for f2_bins (c->f2); it then runs again with
// `second` set and goes on from there.
template <bool kWide>
__device__ void step_boundary(const KArgs& A, PhaseScr& P, BState& B, const Local& L, uint32_t rounds_in_step,
                              bool second) {
  Ctl* c = A.ctl;
  __shared__ HighdScr s_h;
  __shared__ uint32_t s_rw[32];
  __shared__ uint64_t s_sumd;
  __shared__ uint32_t s_settled, s_done;
  __shared__ int64_t s_gap;
  const DevGraph& G = A.G;
  S3Scr& S = P.s3;
  const uint32_t t = threadIdx.x, nt = blockDim.x, lane = lane_id(), warp = t >> 5;
  const int64_t lb = L.lb, ub = L.ub, maxw = G.maxw;
  const uint32_t k = L.step;
  uint32_t settled_now = 0, maxd1 = 0, highd_ub;
  unsigned long long acc = 0;
  uint64_t sumd_ub;
  int64_t gap_raw, st0, st1, nst = ub;
  // this thread's run of the window's chunk sums, summed from the end of the warp
  auto window_sums = [&](const F2Window& w) -> uint32_t {
    const uint32_t per = (w.chunks + nt - 1) / nt, b = min(w.chunks, t * per), e = min(w.chunks, b + per);
    uint32_t x = 0;
    for (uint32_t q = b; q < e; ++q) x += S.suf[suf_at(q)];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t z = __shfl_down_sync(EIC_FULL_MASK, x, o);
      if (lane + o < 32) x += z;
    }
    if (lane == 0) s_rw[warp] = x;
    return x;
  };
  if (kWide && second) {
    sumd_ub = B.p_sumd;
    highd_ub = B.p_highd;
    gap_raw = B.p_gap;
    st0 = B.p_st0;
    st1 = B.p_st1;
    F2Window w;
    w.wl = ub > maxw ? ub - maxw : 0;
    w.slots = 0;
    w.cs = 0;
    w.chunks = A.st_num + 2;
    const int64_t y = ub + (gap_raw << A.gap_shift);
    if (w.chunks <= kSufMax) {
      for (uint32_t q = t; q < w.chunks; q += nt) S.suf[suf_at(q)] = __ldcg(&A.ring[q]);
      __syncthreads();
      const uint32_t wsuf = window_sums(w);
      __syncthreads();
      nst = block_compute_st(A, S, w, ub, sumd_ub, y, st0, st1, wsuf, s_rw);
    } else {
      nst = block_st_bins(A.ring, A.st_num, G.maxw, G.two_m, S, ub, sumd_ub, y, st0, st1);
    }
  } else {
  if (t == 0) {
    settled_now = __ldcg(&c->settled_cnt);
    acc = __ldcg(&c->acc_deg);
    maxd1 = __ldcg(&c->acc_maxd1);
  }
  const int64_t gap_lb = B.gap_lb;
  const bool ring = A.ring_shift == 0 && !(A.flags & EIC_FLAG_NO_PULL) && gap_lb != maxw;
  const F2Window w = f2_window(ub, maxw);
  const bool early = ring && w.cs <= 1;  // (a longer window is loaded only once it is needed)
  if (early) f2_load(A, S, w);
  const HighdPart hp = highd_sums(A.hist, G.dvals, G.D, s_h);
  if (t == 0) {
    if (maxd1 && (int64_t)(maxd1 - 1) > B.max_settled) B.max_settled = maxd1 - 1;
    const int64_t maxs = B.max_settled;
    // termination / overflow (Algorithm 1): max{finite dist} + maxW(G,1) < lb
    uint32_t done = 0;
    if (maxs + maxw >= (int64_t)EIC_INF) {
      atomicCAS(&c->status, 0, EIC_EOVERFLOW);
      done = 1;
    } else if (maxs + maxw < ub) {
      done = 1;
    } else if (k + 1 >= A.step_cap) {
      atomicCAS(&c->status, 0, EIC_ENOMEM);
      done = 1;
    }
    s_done = done;
    s_sumd = B.sumd_lb - acc;
    s_settled = settled_now;
    A.step_ub[k] = ub;
    B.hub[k % kStepHist] = ub;
    B.rounds += rounds_in_step;
    c->cnt_rounds = B.rounds;
    c->trace_len = k;
    if (k <= A.trace_cap && A.trace) {
      eic_step r;
      r.lb = lb;
      r.ub = ub;
      r.st = L.st;
      r.gap_lb = gap_lb;
      r.sumd_lb = B.sumd_lb;
      r.highd_lb = B.highd_lb;
      r.rounds = rounds_in_step;
      r.settled = settled_now - L.step_off_cur;
      r.flags = (L.pull_on ? EIC_STEP_PULL : 0u) | (L.pull_on && L.pull_sweep ? EIC_STEP_SWEPT : 0u);
      r.reserved = 0;
      A.trace[k - 1] = r;
    }
  }
  __syncthreads();
  sumd_ub = s_sumd;
  if (s_done) {
    if (t == 0) {
      c->done = 1;
      c->s2_done = 0;  // published by the grid barrier's release
    }
    return;
  }
  highd_cross(A.hist, G.dvals, G.D, hp, s_h);
  uint32_t wsuf = early ? window_sums(w) : 0u;
  __syncthreads();
  highd_ub = s_h.highd;
  gap_raw = dev_gap_quick(sumd_ub, highd_ub, G.two_m, A.alpha, A.beta, G.rtow);
  if (gap_raw < 0) {  // (the same in every thread)
    if (t == 0) s_gap = dev_gap(sumd_ub, highd_ub, G.two_m, A.alpha, A.beta, G.rtow);
    __syncthreads();
    gap_raw = s_gap;
  }
  st0 = k == 1 ? ub : B.st0;
  st1 = B.st1 < 0 && sumd_ub <= G.m ? ub : B.st1;
  if (!(A.flags & EIC_FLAG_NO_PULL) && sumd_ub < G.m && gap_lb != maxw) {
    if (gap_raw == maxw) {
      nst = ub - maxw;
    } else if (!kWide || A.ring_shift == 0) {
      if (!early) {
        f2_load(A, S, w);
        __syncthreads();
        wsuf = window_sums(w);
        __syncthreads();
      }
      nst = block_compute_st(A, S, w, ub, sumd_ub, ub + (gap_raw << A.gap_shift), st0, st1, wsuf, s_rw);
    } else {  // ask for the bins: the settled steps j that end above wl
      for (uint32_t q = t; q < A.st_num + 2; q += nt) __stcg(&A.ring[q], 0u);
      __syncthreads();  // every thread is done with the controller's state
      if (t == 0) {
        B.p_sumd = sumd_ub;
        B.p_highd = highd_ub;
        B.p_gap = gap_raw;
        B.p_st0 = st0;
        B.p_st1 = st1;
        B.p_settled = s_settled;
        const int64_t wl = ub > maxw ? ub - maxw : 0;
        uint32_t j = B.j0;
        while (j <= k && __ldcg(&A.step_ub[j]) <= wl) ++j;
        c->f2_beg = j <= k ? __ldcg(&A.step_off[j]) : s_settled;
        c->f2_end = s_settled;
        c->f2_wl = wl;
        c->f2_st0 = st0;
        c->f2_span = (uint64_t)(st1 - st0);
        c->s2_done = 0;
        c->f2 = 1;
      }
      return;
    }
  }
  }
  const int64_t nlb = ub, nub = ub + (gap_raw << A.gap_shift);
  if (t >= 32) {
    if (A.ring_shift == 0) {  // zero the ring slots the next statistics pass fills: [max(nlb, nub - maxW), nub)
      const int64_t zl = nub - maxw > nlb ? nub - maxw : nlb;
      for (int64_t q = zl + (t - 32); q < nub; q += nt - 32) __stcg(&A.ring[(uint32_t)q & A.ring_mask], 0u);
    }
  } else if (t == 0) {
    settled_now = kWide && second ? B.p_settled : s_settled;
    A.step_off[k + 1] = settled_now;
    B.hoff[(k + 1) % kStepHist] = settled_now;
    uint32_t scnt = settled_now;
    uint32_t extra = 0;
    if (k == 1 && ub == 0) {  // the source itself was not settled by the first step
      A.sid[scnt] = L.s_int;
      A.sd[scnt] = 0;
      A.scur[scnt] = kNone;
      ++scnt;
      extra = 1;
    }
    // Function 1's push set {lb0 <= dist <= st}: the settled steps j with
    // ub_j > lb0 (j0, moving forward only) and lb_j <= st (j1, from the back);
    // the last kStepHist steps are in shared memory
    auto ub_of = [&](uint32_t j) -> int64_t {
      return j + kStepHist > k ? B.hub[j % kStepHist] : __ldcg(&A.step_ub[j]);
    };
    auto off_of = [&](uint32_t j) -> uint32_t {
      return j + kStepHist > k + 1 ? B.hoff[j % kStepHist] : __ldcg(&A.step_off[j]);
    };
    const int64_t lb0 = nlb - maxw > 0 ? nlb - maxw : 0;
    uint32_t pb = 0, pe = 0;
    uint32_t j0 = B.j0;
    while (j0 <= k && ub_of(j0) <= lb0) ++j0;
    B.j0 = j0;
    if (nst >= lb0) {
      uint32_t j1 = k;
      int64_t lbj = lb;  // lb_k
      while (j1 >= 1 && lbj > nst) {
        --j1;
        lbj = j1 >= 2 ? ub_of(j1 - 1) : 0;
      }
      if (j0 <= j1 && j1 >= 1) {
        pb = off_of(j0);
        pe = j1 == k ? settled_now : off_of(j1 + 1);
      }
    }
    // Function 1's pull: unsettled vertices with an edge lighter than ub - st,
    // a prefix of the weight-ordered non-isolated vertices
    const uint32_t pull_on = nst < nlb ? 1u : 0u;
    uint32_t pull_cnt = 0;
    if (pull_on) {
      const int64_t bound = nub - nst;  // smallest weight < bound
      if (bound >= (int64_t)G.nz_lt_len) {
        if ((uint64_t)bound > G.maxw) {
          pull_cnt = G.nz_count;
        } else {
          uint32_t lo = 0, hi = G.nz_count;
          while (lo < hi) {
            const uint32_t mid = (lo + hi) >> 1;
            if ((int64_t)__ldg(&G.nz[mid].y) < bound)
              lo = mid + 1;
            else
              hi = mid;
          }
          pull_cnt = lo;
        }
      } else if (bound > 0) {
        pull_cnt = __ldg(&G.nz_lt[bound]);
      }
    }
    c->settled_cnt = scnt;
    c->lb = nlb;
    c->ub = nub;
    c->st = nst;
    c->lb0 = lb0;
    c->step = k + 1;
    c->push_beg = pb;
    c->push_end = pe;
    c->pull_on = pull_on;
    // a pull set of most vertices is swept in vertex order: rows are read in
    // address order across the grid (the weight-ordered list would make one
    // pass per weight value), and what the round inserts comes out in
    // vertex order, which the next round and the statistics pass read
    const uint32_t sweep = pull_on && (uint64_t)pull_cnt * kSweepDen >= (uint64_t)G.ni * kSweepNum ? 1u : 0u;
    c->pull_sweep = sweep;
    c->pull_cnt = sweep ? G.ni : pull_cnt;
    c->extra_s = extra;
    c->step_off_cur = settled_now;
    c->acc_deg = 0;
    c->acc_maxd1 = 0;
    c->s2_done = 0;
    c->f2 = 0;
    c->done = 0;  // the control values are published by the grid barrier's release
  }
  __syncthreads();  // every thread is done with the controller's state of this step
  if (t == 0) {
    B.st0 = st0;
    B.st1 = st1;
    B.sumd_lb = sumd_ub;
    B.highd_lb = highd_ub;
    B.gap_lb = gap_raw;
  }
}

// All threads: control values published before the last barrier (one thread
// loads them from L2, the block shares them).
__device__ void read_ctl(const Ctl* c, Local& L) {
  __shared__ Local sL;
  if (threadIdx.x == 0) {
    sL.lb = __ldcg(&c->lb);
    sL.ub = __ldcg(&c->ub);
    sL.st = __ldcg(&c->st);
    sL.lb0 = __ldcg(&c->lb0);
    sL.step = __ldcg(&c->step);
    sL.push_beg = __ldcg(&c->push_beg);
    sL.push_end = __ldcg(&c->push_end);
    sL.pull_on = __ldcg(&c->pull_on);
    sL.pull_cnt = __ldcg(&c->pull_cnt);
    sL.pull_sweep = __ldcg(&c->pull_sweep);
    sL.extra_s = __ldcg(&c->extra_s);
    sL.step_off_cur = __ldcg(&c->step_off_cur);
    sL.done = __ldcg(&c->done);
    sL.s_int = __ldcg(&c->s_int);
  }
  __syncthreads();
  const uint32_t rid = L.rid, qsel = L.qsel;
  L = sL;
  L.rid = rid;
  L.qsel = qsel;
  L.cur_cnt = 0;
  __syncthreads();
}

// Block sum of several counters; thread 0 receives the totals.
template <int K>
__device__ __forceinline__ void block_sums(unsigned long long (&v)[K], unsigned long long (*sh)[K]) {
#pragma unroll
  for (int j = 0; j < K; ++j) v[j] = warp_sum_u64(v[j]);
  if ((threadIdx.x & 31) == 0)
#pragma unroll
    for (int j = 0; j < K; ++j) sh[threadIdx.x >> 5][j] = v[j];
  __syncthreads();
  if (threadIdx.x == 0) {
    for (uint32_t w = 1; w < (blockDim.x >> 5); ++w)
#pragma unroll
      for (int j = 0; j < K; ++j) v[j] += sh[w][j];
  }
  __syncthreads();
}

// Shared-memory scratch of one block in the query loop.
struct QueryShared {
  PhaseScr P;
  Stage T;
  BState B;
  unsigned long long red[32][7];
  unsigned long long snap[4];
  uint32_t last, red2[2];
};

// The query loop of Algorithm 1 run by the A.nb blocks of one query: rounds
// of a step (item phase, task phase), statistics pass, step boundary, until
// termination. ticket is the block's arrival ticket of the query's barrier.
// kWide: the query's graph may have weights of 2^20 and above. Without that
// code the other graphs' queries are 2 to 4% faster (registers).
template <uint32_t kPullFast, uint32_t kRelaxIlp, bool kWide>
__device__ void run_query(const KArgs& A, QueryShared& Q, unsigned long long& ticket) {
  PhaseScr& P = Q.P;
  Stage& T = Q.T;
  BState& B = Q.B;
  auto& sh_red = Q.red;
  auto& sh_snap = Q.snap;
  uint32_t& sh_last = Q.last;
  auto& sh_red2 = Q.red2;
  Ctl* c = A.ctl;
  const uint32_t qb = qblock(A);
  Local L;
  L.rid = 0;
  L.qsel = 0;
  read_ctl(c, L);
  L.cur_cnt = 1;  // the first round's frontier is {s}
  Counters C = {0, 0, 0, 0, 0, 0};
  if (threadIdx.x == 0) {
    T.tn = 0;
    B.st0 = -1;
    B.st1 = -1;
    B.gap_lb = __ldcg(&c->gap_lb);
    B.max_settled = -1;
    B.sumd_lb = A.G.two_m;
    B.highd_lb = A.G.highd0;
    B.rounds = 0;
    B.hub[0] = 0;
    B.hoff[1] = 0;
    B.j0 = 1;
  }
  if (qb == 0 && threadIdx.x == 0) tl_mark(A, 0, L.rid);
  bool alive = !L.done;  // an isolated source has nothing to relax
  constexpr uint32_t kMaxRounds = 1u << 22;  // every block counts the same rounds (L.rid) and stops together
  while (alive) {
    // ------------------------------------------------ rounds of one step
    uint32_t rin = 0;
    bool plain = false;                    // the round must be a plain one
    constexpr uint32_t kStayPlainShift = 2;
    for (;;) {
      if (++L.rid > kMaxRounds) {
        if (threadIdx.x == 0) atomicCAS(&c->status, 0, EIC_ETIMEOUT);
        alive = false;
        break;
      }
      const bool round1 = (L.step >= 2 && rin == 0);
      // counters of round rid+1 were last read two barriers ago: clear them now
      if (qb == 0 && threadIdx.x == 0) {
        __stcg(&c->rcnt[(L.rid + 1) % 3], make_uint4(0u, 0u, 0u, 0u));
      }
      if (L.cur_cnt) {  // the other bitmap served round rid-1 (which set a bit per vertex it queued) and is
                        // next used in round rid+1: clear it now
        uint32_t* other = A.fbits + ((L.rid + 1) & 1u) * A.fwords;
        for (uint32_t wi = qb * blockDim.x + threadIdx.x; wi < A.fwords; wi += A.nb * blockDim.x)
          __stcg(&other[wi], 0u);
      }
      RoundCtx R;
      R.fbits = A.fbits + (L.rid & 1u) * A.fwords;
      R.lb = L.lb;
      R.ub = L.ub;
      R.ub_eff = L.ub < (int64_t)EIC_INF ? L.ub : (int64_t)EIC_INF;
      R.st = L.st;
      R.lb0 = L.lb0;
      R.rid = L.rid;
      R.step1 = L.step == 1;
      R.qout = L.qsel ? A.q0 : A.q1;
      R.qcnt_out = &c->rcnt[L.rid % 3].x;
      R.first_list = R.step1 ? A.touched : A.sid;
      R.first_cnt = R.step1 ? &c->touched_cnt : &c->settled_cnt;
      R.tcnt = &c->rcnt[L.rid % 3].y;
      R.plain_out = &c->rcnt[L.rid % 3].z;
      const uint32_t* qin = L.qsel ? A.q1 : A.q0;
      Local LL = L;
      if (!L.pull_on) LL.pull_cnt = 0;
      const uint32_t nitems = round1 ? (LL.push_end - LL.push_beg) + LL.pull_cnt + LL.extra_s : L.cur_cnt;
      if (qb == 0 && threadIdx.x == 0) tl_mark(A, 8, nitems);  // diagnostic: the round's items
      if (!R.step1 && (!round1 || !LL.pull_on) && !plain && nitems <= A.fuse * A.nb * (blockDim.x >> 5)) {
        if (A.fuse == kFuseRoad)
          fused_round<true>(A, R, LL, T, nitems, round1, qin, C);
        else
          fused_round<false>(A, R, LL, T, nitems, round1, qin, C);
      } else {
        round_phase<kPullFast, kRelaxIlp>(A, R, LL, P.r, T, nitems, round1, qin, C);
      }
      if (!grid_barrier(&c->bar, &ticket, A.nb, A.max_spin, &c->status)) {
        alive = false;
        break;
      }
      if (threadIdx.x == 0) {
        const uint4 rc = __ldcg(&c->rcnt[L.rid % 3]);
        sh_snap[0] = rc.y | (unsigned long long)rc.z << 32;
        sh_snap[1] = rc.x;
        sh_snap[2] = __ldcg(&c->ub_cand);
        sh_snap[3] = __ldcg(R.first_cnt);
        if (qb == 0) tl_mark(A, 1, L.rid);
      }
      __syncthreads();
      const uint32_t hp = (uint32_t)sh_snap[0];
      const bool plain_next = sh_snap[0] >> 32;
      L.cur_cnt = (uint32_t)sh_snap[1];
      uint32_t uc = (uint32_t)sh_snap[2];
      __syncthreads();
      if (hp != 0) {
        if (qb == 0 && threadIdx.x == 0) tl_mark(A, 9, hp);  // diagnostic: the round's tasks
        task_phase<(kRelaxIlp >= 2)>(A, R, hp, T, C);
        if (!grid_barrier(&c->bar, &ticket, A.nb, A.max_spin, &c->status)) {
          alive = false;
          break;
        }
        if (qb == 0 && threadIdx.x == 0) tl_mark(A, 2, L.rid);
        if (threadIdx.x == 0) {
          sh_snap[1] = __ldcg(&c->rcnt[L.rid % 3].x);
          sh_snap[2] = __ldcg(&c->ub_cand);
          sh_snap[3] = __ldcg(R.first_cnt);
        }
        __syncthreads();
        L.cur_cnt = (uint32_t)sh_snap[1];
        uc = (uint32_t)sh_snap[2];
        __syncthreads();
      }
      if (R.step1 && uc != EIC_INF && (int64_t)uc < L.ub) L.ub = uc;
      L.qsel ^= 1u;
      // A wide step that meets hubs meets more of them: its next rounds stay plain (at gap_shift 2, 3 and 6 RMAT
      // 131 k 524, 544, 811 -> 484, 493, 650 us, 512 k with wide weights 905, 961, 1820 -> 729, 822, 1738; at the
      // paper's width the rounds in between are worth fusing: 536 against 562 us).
      plain = plain_next || (plain && A.gap_shift >= kStayPlainShift);
      ++rin;
      if (L.cur_cnt == 0) break;
    }
    if (!alive) break;
    // ------------------------------------------------ statistics pass
    {
      S2Scr& S = P.s2;
      const bool step1 = L.step == 1;
      const uint32_t* list = step1 ? A.touched : A.sid;
      const uint32_t lbeg = step1 ? 0 : L.step_off_cur;
      const uint32_t lend = (uint32_t)sh_snap[3];  // (read behind the last round's barrier)
      const bool has = lbeg + qb * blockDim.x < lend;  // this block has settled vertices to count
      const int64_t wlo = L.ub - (int64_t)A.G.maxw > L.lb ? L.ub - (int64_t)A.G.maxw : L.lb;
      // The ring's first slots are counted in shared memory when a block settles at least as many vertices as that
      // has slots (else clearing and flushing them costs more than the vertices' own atomics: 2 us a step on a
      // grid). Distances beyond them go to the ring at once: in a window of 65535 most vertices share the first
      // hundreds of slots, and a step of 2 M vertices took 288 us on those slots' atomics.
      const uint32_t nset = lend - lbeg, per_block = max(min(nset, blockDim.x), nset / A.nb);
      const uint32_t wslots = A.ring_shift == 0 && L.ub < EIC_INF_T ? (uint32_t)min((int64_t)kShRing, L.ub - wlo) : 0u;
      const bool ring_sh = wslots && wslots <= per_block;
      const bool ring_narrow = ring_sh && (L.ub - wlo) <= kRingNarrow && A.G.max_deg < (1u << 27);  // (in shared memory)
      const uint32_t ranks = min(A.G.D, (uint32_t)kShRanks);
      if (has) {
        for (uint32_t r = threadIdx.x; r < ranks; r += blockDim.x) S.hist[r] = 0;
        if (ring_sh)
          for (uint32_t r = threadIdx.x; r < wslots; r += blockDim.x) S.ring[r] = 0;
        if (threadIdx.x < 2) sh_red2[threadIdx.x] = 0;
      }
      __syncthreads();
      uint32_t bdeg = 0, bmax1 = 0;  // degree sum (at most 2m < 2^32), 1 + the largest distance (0: none)
      const uint32_t nthreads = A.nb * blockDim.x;
      uint32_t xnext = 0;  // the single-query shape loads the next list entry one iteration ahead
      if constexpr (kRelaxIlp >= 2) {
        if (lbeg + qb * blockDim.x + threadIdx.x < lend) xnext = ld_list(&list[lbeg + qb * blockDim.x + threadIdx.x]);
      }
      for (uint32_t base = lbeg + qb * blockDim.x; base < lend; base += nthreads) {
        const uint32_t idx = base + threadIdx.x;
        bool take = false;
        uint32_t x = 0, d = 0, r = EIC_INF, dg = 0, cx = kNone;
        uint32_t xcur = 0;
        if constexpr (kRelaxIlp >= 2) {
          xcur = xnext;
          if (idx + nthreads < lend) xnext = ld_list(&list[idx + nthreads]);
        }
        if (idx < lend) {
          if constexpr (kRelaxIlp >= 2)
            x = xcur;
          else
            x = ld_list(&list[idx]);
          d = __ldcg(&A.dist[x]);
          cx = x < A.G.nlong ? __ldcg(&A.cursor[x]) : kNone;  // (a long row by its id: loaded with dist)
          r = degree_rank(A.G, x);  // (the degree from the id: no random row read)
          dg = __ldg(&A.G.dvals[r]);
          take = true;
          if (step1 && d64(d) >= L.ub) {  // first step: keep only what is final
            if (x != L.s_int) __stcg(&A.dist[x], EIC_INF);
            take = false;
          }
        }
        if (step1) {
          const uint32_t slot = warp_append(take, &c->settled_cnt);
          if (take) {
            __stcg(&A.sid[slot], x);
            __stcg(&A.sd[slot], d);
            __stcg(&A.scur[slot], kNone);  // the first step's windows used a larger ub
          }
        }
        if (take) {
          atomicOr(&A.sbits[x >> 5], 1u << (x & 31));
          if (!step1) {
            __stcg(&A.sd[idx], d);
            __stcg(&A.scur[idx], cx);
          }
          bdeg += dg;
          bmax1 = max(bmax1, d + 1);
        }
        // degree histogram (internal vertices all have degree >= 1)
        if (!take) r = EIC_INF;
        if (r < (uint32_t)kShRanks)
          atomicAdd(&S.hist[r], 1u);
        else if (r != EIC_INF)
          atomicSub(&A.hist[r], 1u);
        // D(x) ring: in a narrow window the step's settled vertices share few
        // distances; then one atomic per distinct slot in the warp, with the
        // group's degree sum (32-bit while 32 degrees cannot overflow it)
        const bool rk = take && (int64_t)d >= wlo && A.ring_shift == 0;  // (wide weights: Function 2 sums exactly)
        const uint32_t slot = rk ? (uint32_t)(d - wlo) : EIC_INF;
        if (ring_narrow) {
          const uint32_t rg = __match_any_sync(EIC_FULL_MASK, slot);
          const uint32_t sum = __reduce_add_sync(rg, rk ? dg : 0u);
          if (rk && lane_id() == (uint32_t)__ffs(rg) - 1) atomicAdd(&S.ring[slot], sum);
        } else if (rk) {
          if (ring_sh && slot < wslots)
            atomicAdd(&S.ring[slot], dg);
          else
            atomicAdd(&A.ring[d & A.ring_mask], dg);
        }
      }
      if (has) {  // block totals: one atomic each
        bdeg = __reduce_add_sync(EIC_FULL_MASK, bdeg);
        bmax1 = __reduce_max_sync(EIC_FULL_MASK, bmax1);
        if (lane_id() == 0 && bmax1) {
          atomicAdd(&sh_red2[0], bdeg);
          atomicMax(&sh_red2[1], bmax1);
        }
      }
      __syncthreads();
      if (has) {
        for (uint32_t r = threadIdx.x; r < ranks; r += blockDim.x)
          if (S.hist[r]) atomicSub(&A.hist[r], S.hist[r]);
        for (uint32_t r = threadIdx.x; ring_sh && r < wslots; r += blockDim.x)
          if (S.ring[r]) atomicAdd(&A.ring[(uint32_t)(wlo + r) & A.ring_mask], S.ring[r]);
        if (threadIdx.x == 0 && sh_red2[1]) {
          atomicAdd(&c->acc_deg, (unsigned long long)sh_red2[0]);
          atomicMax(&c->acc_maxd1, sh_red2[1]);
        }
        __syncthreads();
      }
    }
    // The boundary, by block 0 once every block has released its part. With wide weights it may first ask all
    // blocks for Function 2's bins.
    for (bool second = false;; second = true) {
      if (threadIdx.x == 0) red_release_add_u32(&c->s2_done, 1u);
      if (qb == 0) {  // block 0 waits (bounded) for every block's part
        if (threadIdx.x == 0) {
          uint64_t spins = 0;
          sh_last = 1;
          while (ld_acquire_u32(&c->s2_done) < A.nb) {
            if (++spins > A.max_spin || ((spins & 15) == 0 && ld_volatile_int(&c->status) != 0)) {
              barrier_fail(&c->bar, &c->status);
              sh_last = 0;
              break;
            }
          }
          tl_mark(A, 4, L.rid);
        }
        __syncthreads();
        if (sh_last) step_boundary<kWide>(A, P, B, L, rin, second);
        if (threadIdx.x == 0) tl_mark(A, 5, L.rid);
      }
      alive = grid_barrier(&c->bar, &ticket, A.nb, A.max_spin, &c->status);
      if (!kWide || !alive || A.ring_shift == 0) break;
      if (threadIdx.x == 0) sh_last = __ldcg(&c->f2);
      __syncthreads();
      if (!sh_last) break;
      if constexpr (kRelaxIlp >= 2)
        f2_bins(A, P.s3, c);
      else
        f2_bins_call(A, P.s3, c);
    }
    if (!alive) break;
    if (qb == 0 && threadIdx.x == 0) tl_mark(A, 3, L.rid);
    read_ctl(c, L);
    if (L.done) break;
  }
  {  // the query's counters, once per block
    unsigned long long v[7] = {C.frontier, C.trav, C.pulls, C.improved, C.heavy, C.pitems, 0ull};
    block_sums<7>(v, sh_red);
    if (threadIdx.x == 0) {
      atomicAdd(&c->cnt_frontier, v[0]);
      atomicAdd(&c->cnt_trav, v[1]);
      atomicAdd(&c->cnt_pulls, v[2]);
      atomicAdd(&c->cnt_improved, v[3]);
      atomicAdd(&c->cnt_heavy, v[4]);
      atomicAdd(&c->cnt_pitems, v[5]);
    }
  }
  if (qb == 0 && threadIdx.x == 0 && A.status_out) *A.status_out = ld_volatile_int(&c->status);
}

template <bool kWide>
__global__ void __launch_bounds__(kMaxBlock, 2) k_eic(KArgs A) {
  __shared__ QueryShared Q;
  unsigned long long ticket = 0;  // (k_init zeroed the arrival count)
  run_query<kPullFastSingle, kRelaxIlpSingle, kWide>(A, Q, ticket);
}

// Control block of a new query (one thread): the source's distance, the
// first round's frontier {s}, step 1 = <0, +inf> with st = 0, and gap(0).
__device__ void ctl_init(const KArgs& A, bool set_source) {
  Ctl* c = A.ctl;
  const DevGraph& G = A.G;
  const uint32_t si = G.orig2int[A.s];
  c->s_int = si;
  uint32_t dgs = 0;
  if (si != EIC_INF) {
    if (set_source) A.dist[si] = 0;
    A.q0[0] = si;
    A.touched[0] = si;
    dgs = G.row[si + 1] - G.row[si];
  }
  A.step_off[1] = 0;
  A.step_ub[0] = 0;
  c->lb = 0;
  c->ub = EIC_INF_T;
  c->st = 0;
  c->lb0 = 0;
  c->step = 1;
  c->f2 = 0;
  c->done = si == EIC_INF ? 1u : 0u;
  c->push_beg = c->push_end = 0;
  c->pull_on = c->pull_cnt = c->extra_s = 0;
  c->pull_sweep = 0;
  c->step_off_cur = 0;
  c->gap_lb = dev_gap(G.two_m, G.highd0, G.two_m, A.alpha, A.beta, G.rtow);
  c->trace_len = 0;
  c->tl_len = 0;
  c->rcnt[0] = c->rcnt[1] = c->rcnt[2] = make_uint4(0u, 0u, 0u, 0u);
  c->settled_cnt = 0;
  c->touched_cnt = 1;
  c->ub_cand = (G.highd0 > 0 && dgs >= G.highd0) ? 0u : EIC_INF;
  c->s2_done = 0;
  c->ptasks = 0;
  c->acc_maxd1 = 0;
  c->acc_deg = 0;
  c->cnt_rounds = c->cnt_frontier = c->cnt_trav = c->cnt_pulls = c->cnt_improved = c->cnt_heavy = 0;
  c->cnt_pitems = 0;
}

// The query's scratch at its starting values, in one launch (three memsets
// before it cost a small query 6 us). Every array starts on 256 bytes and is
// padded to them: 16-byte stores may run over its last word.
__global__ void k_init(KArgs A) {
  const DevGraph& G = A.G;
  const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x, stride = gridDim.x * blockDim.x;
  const uint32_t si = __ldg(&G.orig2int[A.s]);
  for (uint32_t i = t; i < (G.ni + 3) / 4; i += stride) {
    uint4 v = make_uint4(EIC_INF, EIC_INF, EIC_INF, EIC_INF);
    if (i == si / 4) (&v.x)[si & 3u] = 0u;  // the source (EIC_INF when isolated: no such word)
    reinterpret_cast<uint4*>(A.dist)[i] = v;
  }
  const uint4 z = make_uint4(0u, 0u, 0u, 0u);
  for (uint32_t i = t; i < (A.fwords + 3) / 4; i += stride) reinterpret_cast<uint4*>(A.sbits)[i] = z;
  for (uint32_t i = t; i < (2 * A.fwords + 3) / 4; i += stride) reinterpret_cast<uint4*>(A.fbits)[i] = z;
  for (uint32_t r = t; r < G.D; r += stride) A.hist[r] = G.dcnt0[r];
  if (A.ring_shift == 0)  // (wide weights: Function 2 clears the bins it uses)
    for (uint32_t r = t; r <= A.ring_mask; r += stride) A.ring[r] = 0;
  if (t == 0) {
    ctl_init(A, false);
    A.ctl->bar.arrived = 0;
    A.ctl->status = 0;
  }
}

// Distances in the caller's numbering: out[u] = dist[orig2int[u]], +inf for
// isolated vertices, 0 for the source.
// Each thread has kOutIlp independent gathers in flight.
constexpr uint32_t kOutIlp = 4;
__global__ void k_output(DevGraph G, const uint32_t* __restrict__ idist, uint32_t s, uint32_t* out) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t u0 = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; u0 < G.n; u0 += kOutIlp * stride) {
    uint32_t i[kOutIlp], d[kOutIlp];
#pragma unroll
    for (uint32_t k = 0; k < kOutIlp; ++k) {
      const uint64_t u = u0 + k * stride;
      i[k] = u < G.n ? __ldg(&G.orig2int[u]) : EIC_INF;
    }
#pragma unroll
    for (uint32_t k = 0; k < kOutIlp; ++k) d[k] = i[k] == EIC_INF ? EIC_INF : __ldcg(&idist[i[k]]);
#pragma unroll
    for (uint32_t k = 0; k < kOutIlp; ++k) {
      const uint64_t u = u0 + k * stride;
      if (u < G.n) out[u] = u == s ? 0u : d[k];
    }
  }
}

// parent[v] = smallest original id u with dist[u] + w(u, v) == dist[v]; parent[s]
// = s, +inf where unreachable. Only the prefix of v's row with weight <= dist[v]
// can hold u. Bound by the chain id -> distance -> entries -> their distances of
// every vertex, and by the longest prefix: eight lanes take a row (a warp's 32
// mostly idled); a row of more than kBigRow entries (these come first) is taken
// by a warp, 128 entries at a time, and what its prefix holds beyond kParentAlone
// is shared out over the grid in pieces. With parents a query of a dense graph
// (32 k vertices, 256 M entries) takes 22 us longer, of RMAT graphs of 250 k
// vertices 29, of 2^22 236, of 2^25 1.60 ms; 592, 37, 395 us and 3.19 ms when
// every entry of the big rows was read, 23, 43, 582 us and 6.28 ms when a warp
// took every row. kBigRow 128, 256 and 512: rows of 500 entries (5 k vertices,
// unit weights) 18, 18 and 45 us, rows of 128 (512 k vertices) 137, 94 and 92.
constexpr uint32_t kParentLanes = 8;
constexpr uint32_t kParentAlone = 512;
constexpr uint32_t kParentPiece = 256;
static_assert(kParentAlone >= kParentPiece && kParentPiece >= kHeavyMinFloor,
              "a row has at most length / kParentPiece pieces, and the task list 2m / kHeavyMinFloor entries");

// The smallest parent among kIlp entries per lane of the row part [at, at + len); last: the weight of the last entry
// looked at (all ones past the part's end).
template <uint32_t kIlp>
__device__ __forceinline__ uint32_t parent_of(const DevGraph& G, const uint32_t* __restrict__ idist, uint32_t at,
                                              uint32_t len, uint32_t dv, uint32_t* last) {
  const uint32_t lane = lane_id();
  uint2 ent[kIlp];
  uint32_t du[kIlp], best = EIC_INF;
#pragma unroll
  for (uint32_t j = 0; j < kIlp; ++j)
    ent[j] = 32 * j + lane < len ? ld_stream(&G.adj[at + 32 * j + lane]) : make_uint2(0u, EIC_INF);
#pragma unroll
  for (uint32_t j = 0; j < kIlp; ++j) du[j] = ent[j].y <= dv ? __ldg(&idist[ent[j].x]) : EIC_INF;
#pragma unroll
  for (uint32_t j = 0; j < kIlp; ++j)
    if (du[j] != EIC_INF && (uint64_t)du[j] + ent[j].y == dv) best = min(best, __ldg(&G.int2orig[ent[j].x]));
  *last = __shfl_sync(EIC_FULL_MASK, ent[kIlp - 1].y, 31);
  return best;
}

// best[vi] for the vertices with big rows, from the first kParentAlone entries; the rest of their prefixes to tasks.
__global__ void __launch_bounds__(256) k_parent_big(DevGraph G, const uint32_t* __restrict__ idist, uint32_t* best,
                                                    Task* tasks, uint32_t* count) {
  const uint32_t lane = lane_id(), nw = gridDim.x * (blockDim.x >> 5);
  for (uint32_t vi = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); vi < G.nbig; vi += nw) {
    const uint32_t dv = __ldg(&idist[vi]), end = __ldg(&G.row[vi + 1]);
    uint32_t at = __ldg(&G.row[vi]), mine = EIC_INF, last = 0;
    bool more = dv != EIC_INF;  // the prefix goes on at `at`
    for (uint32_t k = 0; more && k < kParentAlone; k += 128) {
      mine = min(mine, parent_of<4>(G, idist, at, end - at, dv, &last));
      more = last <= dv;  // (then all 128 entries were there)
      at += more ? 128u : 0u;
    }
    mine = __reduce_min_sync(EIC_FULL_MASK, mine);
    if (lane == 0) best[vi] = mine;
    if (!more) continue;
    uint32_t lo = at, hi = end;  // the prefix's end, by 32 probes at a time
    while (hi - lo > 32) {
      const uint32_t step = (hi - lo + 32) / 33, off = (lane + 1) * step;
      const uint32_t in = __popc(__ballot_sync(EIC_FULL_MASK, off < hi - lo && ld_stream_w(&G.adj[lo + off]) <= dv));
      hi = in < 32 && (in + 1) * step < hi - lo ? lo + (in + 1) * step : hi;
      lo += in ? in * step + 1 : 0u;
    }
    lo += __popc(__ballot_sync(EIC_FULL_MASK, lane < hi - lo && ld_stream_w(&G.adj[lo + lane]) <= dv));
    const uint32_t len = lo - at, nt = (len + kParentPiece - 1) / kParentPiece;
    uint32_t slot = 0;
    if (lane == 0 && nt) slot = atomicAdd(count, nt);
    slot = __shfl_sync(EIC_FULL_MASK, slot, 0);
    for (uint32_t k = lane; k < nt; k += 32)
      tasks[slot + k] = Task{at + k * kParentPiece, min(kParentPiece, len - k * kParentPiece), vi, dv};
  }
}

__global__ void __launch_bounds__(256) k_parent_pieces(DevGraph G, const uint32_t* __restrict__ idist,
                                                       const Task* __restrict__ tasks,
                                                       const uint32_t* __restrict__ count, uint32_t* best) {
  const uint32_t nw = gridDim.x * (blockDim.x >> 5), n = __ldg(count);
  for (uint32_t k = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); k < n; k += nw) {
    const uint4 t = __ldg(reinterpret_cast<const uint4*>(&tasks[k]));
    uint32_t last;
    const uint32_t mine = __reduce_min_sync(EIC_FULL_MASK, parent_of<kParentPiece / 32>(G, idist, t.x, t.y, t.w, &last));
    if (lane_id() == 0 && mine != EIC_INF) atomicMin(&best[t.z], mine);
  }
}

__global__ void k_parent(DevGraph G, const uint32_t* __restrict__ idist, const uint32_t* __restrict__ big, uint32_t s,
                         uint32_t* parent) {
  const uint32_t sub = threadIdx.x % kParentLanes;
  const uint32_t mask = ((1u << kParentLanes) - 1u) << (lane_id() - sub);
  const uint64_t step = (uint64_t)gridDim.x * (blockDim.x / kParentLanes);
  for (uint64_t v = (uint64_t)blockIdx.x * (blockDim.x / kParentLanes) + threadIdx.x / kParentLanes; v < G.n; v += step) {
    const uint32_t vi = __ldg(&G.orig2int[v]);
    uint32_t best = EIC_INF;
    if (vi != EIC_INF && v != s) {
      if (vi < G.nbig) {
        best = __ldg(&big[vi]);
      } else {
        const uint32_t dv = __ldg(&idist[vi]);
        const uint2 rr = dv != EIC_INF ? row_of(G, vi) : make_uint2(0u, 0u);
        for (uint32_t k = sub; k < rr.y; k += kParentLanes) {  // (an entry's index plus the step may wrap)
          const uint2 ent = __ldg(&G.adj[rr.x + k]);
          if (ent.y > dv) break;  // (rows are in weight order)
          const uint32_t du = __ldg(&idist[ent.x]);
          if (du != EIC_INF && (uint64_t)du + ent.y == dv) best = min(best, __ldg(&G.int2orig[ent.x]));
        }
      }
    }
    best = __reduce_min_sync(mask, best);
    if (sub == 0) parent[v] = v == s ? s : best;
  }
}

// ------------------------------------------------------------- batched queries

struct BatchArgs {
  const BatchQuery* q;    // [nq], in the order groups claim them
  const BatchSlot* slot;  // [gridDim.x / nb]
  int* status;            // [nq]; a query no group finished keeps EIC_EABORT
  uint32_t* queue;        // next unclaimed query
  uint32_t nq, nb;        // queries; blocks per group
  uint32_t alpha;
  double beta;
  uint32_t st_num, gap_shift, heavy_min, flags, step_cap;
  uint64_t max_spin;
};

// The query's scratch at its starting values (what the single-query path
// does with memsets and k_init), by the group's blocks.
__device__ bool query_setup(const KArgs& A, unsigned long long& ticket) {
  const DevGraph& G = A.G;
  const uint32_t stride = A.nb * blockDim.x, t0 = qblock(A) * blockDim.x + threadIdx.x;
  for (uint32_t i = t0; i < G.ni; i += stride) __stcg(&A.dist[i], EIC_INF);
  for (uint32_t i = t0; i < 2 * A.fwords; i += stride) __stcg(&A.fbits[i], 0u);
  for (uint32_t i = t0; i < A.fwords; i += stride) __stcg(&A.sbits[i], 0u);
  for (uint32_t r = t0; r < G.D; r += stride) __stcg(&A.hist[r], __ldg(&G.dcnt0[r]));
  if (A.ring_shift == 0)
    for (uint32_t r = t0; r <= A.ring_mask; r += stride) __stcg(&A.ring[r], 0u);
  if (!grid_barrier(&A.ctl->bar, &ticket, A.nb, A.max_spin, &A.ctl->status)) return false;
  if (qblock(A) == 0 && threadIdx.x == 0) ctl_init(A, true);
  return grid_barrier(&A.ctl->bar, &ticket, A.nb, A.max_spin, &A.ctl->status);
}

// Distances in the caller's numbering (as k_output), by the group's blocks.
__device__ void query_output(const KArgs& A) {
  const DevGraph& G = A.G;
  const uint64_t stride = (uint64_t)A.nb * blockDim.x;
  for (uint64_t u = (uint64_t)qblock(A) * blockDim.x + threadIdx.x; u < G.n; u += stride) {
    const uint32_t i = __ldg(&G.orig2int[u]);
    A.out[u] = u == A.s ? 0u : (i == EIC_INF ? EIC_INF : __ldcg(&A.dist[i]));
  }
}

// Many queries in one cooperative launch. The grid is cut into groups of nb
// blocks; each group claims the next query from a device counter, runs it
// with its own scratch and a barrier over its nb blocks, writes the output,
// and claims again. A group stops at its first query with a non-OK status
// (its barrier state is then unreliable); the other groups carry on.
template <bool kWide>
__global__ void __launch_bounds__(kMaxBlock, 2) k_eic_batch(BatchArgs P) {
  __shared__ QueryShared Q;
  __shared__ KArgs sA;
  __shared__ uint32_t sh_qi;
  const uint32_t grp = blockIdx.x / P.nb, qb = blockIdx.x % P.nb;
  const BatchSlot& W = P.slot[grp];
  Ctl* c = W.ctl;
  unsigned long long ticket = 0;  // (the launch's preparation zeroed the arrival count)
  uint32_t qi = 0xFFFFFFFFu;
  for (;;) {
    if (qb == 0 && threadIdx.x == 0) c->next_q = ld_volatile_int(&c->status) == 0 ? atomicAdd(P.queue, 1u) : P.nq;
    if (!grid_barrier(&c->bar, &ticket, P.nb, P.max_spin, &c->status)) break;
    if (threadIdx.x == 0) sh_qi = __ldcg(&c->next_q);
    __syncthreads();
    qi = sh_qi;
    if (qi >= P.nq) break;
    if (threadIdx.x == 0) {
      const BatchQuery& bq = P.q[qi];
      sA.G = bq.G;
      sA.dist = W.idist;
      sA.out = bq.out;
      sA.fbits = W.fbits;
      sA.fwords = bq.G.ni / 32 + 2;
      sA.cursor = W.cursor;
      sA.q0 = W.q0;
      sA.q1 = W.q1;
      sA.sid = W.sid;
      sA.sd = W.sd;
      sA.scur = W.scur;
      sA.touched = W.touched;
      sA.sbits = W.sbits;
      sA.hist = W.hist;
      sA.ring = W.ring;
      sA.tasks = W.tasks;
      sA.step_ub = W.step_ub;
      sA.step_off = W.step_off;
      sA.trace = nullptr;
      sA.ctl = c;
      sA.status_out = &P.status[qi];
      sA.s = bq.s;
      sA.alpha = P.alpha;
      sA.beta = P.beta;
      sA.st_num = P.st_num;
      sA.gap_shift = bq.gap_shift;
      sA.heavy_min = bq.heavy_min;
      sA.max_spin = P.max_spin;
      sA.flags = P.flags;
      sA.ring_mask = bq.ring_mask;
      sA.ring_shift = bq.ring_shift;
      sA.step_cap = P.step_cap;
      sA.trace_cap = 0;
      sA.timeline = nullptr;
      sA.timeline_cap = 0;
      sA.nb = P.nb;
      sA.fuse = bq.fuse;
      sA.sweep_words = sweep_chunk(bq.G.ni, P.nb, blockDim.x);
    }
    __syncthreads();
    if (!query_setup(sA, ticket)) break;
    run_query<kPullFastGroup, kRelaxIlpGroup, kWide>(sA, Q, ticket);
    __syncthreads();
    if (ld_volatile_int(&c->status) != 0) break;
    query_output(sA);
  }
  // the query a group stopped in reports the group's status
  if (qb == 0 && threadIdx.x == 0 && qi < P.nq) {
    const int st = ld_volatile_int(&c->status);
    if (st != 0) P.status[qi] = st;
  }
}

// Starting state of every group's barrier and status, of the work queue and
// of the per-query statuses (EIC_EABORT until a group finishes the query).
__global__ void k_batch_prep(BatchArgs P, uint32_t groups) {
  const uint32_t g = blockIdx.x * blockDim.x + threadIdx.x;
  if (g < groups) {
    P.slot[g].ctl->bar.arrived = 0;
    P.slot[g].ctl->status = 0;
  }
  if (g < P.nq) P.status[g] = EIC_EABORT;
  if (g == 0) *P.queue = 0;
}

// ------------------------------------------------------------- serving kernel

__device__ __forceinline__ unsigned long long ld_acquire_sys_u64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.sys.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ unsigned long long ld_relaxed_sys_u64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.sys.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ uint32_t ld_relaxed_sys_u32(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.relaxed.sys.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void st_release_sys_u64(unsigned long long* p, unsigned long long v) {
  asm volatile("st.release.sys.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

__device__ __forceinline__ unsigned long long globaltimer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

constexpr unsigned long long kNoTicket = ~0ull;      // the group leaves
constexpr unsigned long long kRetry = ~0ull - 1;      // nothing yet: the group waits again

// Continuous batching: the grid is cut into groups of nb blocks; each group's
// first thread claims the next admitted request from the ring, the group runs
// it with its own scratch, writes the result into the request's buffer and
// publishes the completion, then claims again. A first thread with nothing to
// claim waits at most poll_ns at a time (its group then passes its barrier
// and waits again, so no barrier wait comes near its bound). After idle_ns
// without work, once no group runs a request, a group registers as idle; when
// every group is registered they all leave together (the host relaunches the
// kernel when work arrives). They also leave when the host sets stop, and,
// in a launch with fewer groups than the server has, once widen_at admitted
// requests wait unclaimed (each after its current request; the host then
// relaunches with more groups). A group stops at its first failing request
// (whose completion carries the error) and counts as idle from then on.
template <bool kWide>
__global__ void __launch_bounds__(kMaxBlock, 2) k_eic_serve(ServeArgs P) {
  __shared__ QueryShared Q;
  __shared__ KArgs sA;
  __shared__ unsigned long long sh_t;
  const uint32_t grp = blockIdx.x / P.nb, qb = blockIdx.x % P.nb;
  const BatchSlot& W = P.slot[grp];
  Ctl* c = W.ctl;
  unsigned long long* claim = &P.claim[0];
  unsigned long long* finished = &P.claim[1];
  unsigned long long* idle_groups = &P.claim[2];
  unsigned long long* leave = &P.claim[3];
  unsigned long long ticket = 0;  // (the launch's preparation zeroed the arrival count)
  unsigned long long mine = kNoTicket;  // first thread: the request it claimed last
  bool reported = true;                 // first thread: that request's completion is published
  bool registered = false;              // first thread: this group counts as idle
  for (;;) {
    if (qb == 0 && threadIdx.x == 0) {
      unsigned long long got = kRetry;
      if (ld_volatile_int(&c->status) != 0) got = kNoTicket;
      const unsigned long long t0 = globaltimer_ns();
      while (got == kRetry) {  // bounded: poll_ns per pass
        if (*(volatile uint32_t*)&P.ring->stop || atomicAdd(leave, 0ull) != 0) {
          got = kNoTicket;
          break;
        }
        const unsigned long long head = ld_acquire_sys_u64(&P.ring->head);
        const unsigned long long cur = atomicAdd(claim, 0ull);
        if (P.widen_at && cur < head && head - cur >= P.widen_at) {  // a backlog: make room for more groups
          atomicExch(leave, 1ull);
          got = kNoTicket;
          break;
        }
        if (cur < head) {
          if (atomicCAS(claim, cur, cur + 1) == cur) {
            got = cur;
            if (registered) {
              atomicAdd(idle_groups, ~0ull);  // minus one
              registered = false;
            }
          }
          continue;
        }
        const unsigned long long waited = globaltimer_ns() - t0;
        if (!registered && waited > P.idle_ns && atomicAdd(finished, 0ull) == cur) {
          atomicAdd(idle_groups, 1ull);
          registered = true;
        }
        if (registered && atomicAdd(idle_groups, 0ull) >= P.groups) {
          atomicExch(leave, 1ull);
          got = kNoTicket;
          break;
        }
        if (waited > P.poll_ns) break;  // kRetry
        __nanosleep(256);
      }
      c->next_ticket = got;
      if (got != kNoTicket && got != kRetry) {
        mine = got;
        reported = false;
      }
    }
    if (!grid_barrier(&c->bar, &ticket, P.nb, P.max_spin, &c->status)) break;
    if (threadIdx.x == 0) sh_t = __ldcg(&c->next_ticket);
    __syncthreads();
    const unsigned long long t = sh_t;
    if (t == kNoTicket) break;
    if (t == kRetry) continue;
    const uint32_t e = (uint32_t)(t & (P.cap - 1));
    if (threadIdx.x == 0) {  // the entry was published before head (host release, leader acquire)
      const ServeRequest* rq = &P.req[e];
      const uint32_t gi = ld_relaxed_sys_u32(&rq->graph);
      const uint32_t src = ld_relaxed_sys_u32(&rq->source);
      uint32_t* out = (uint32_t*)ld_relaxed_sys_u64((const unsigned long long*)&rq->out);
      const BatchQuery& bq = P.graphs[gi < P.num_graphs ? gi : 0];  // the host admits valid ids only
      sA.G = bq.G;
      sA.dist = W.idist;
      sA.out = out;
      sA.fbits = W.fbits;
      sA.fwords = bq.G.ni / 32 + 2;
      sA.cursor = W.cursor;
      sA.q0 = W.q0;
      sA.q1 = W.q1;
      sA.sid = W.sid;
      sA.sd = W.sd;
      sA.scur = W.scur;
      sA.touched = W.touched;
      sA.sbits = W.sbits;
      sA.hist = W.hist;
      sA.ring = W.ring;
      sA.tasks = W.tasks;
      sA.step_ub = W.step_ub;
      sA.step_off = W.step_off;
      sA.trace = nullptr;
      sA.ctl = c;
      sA.status_out = nullptr;
      sA.s = src;
      sA.alpha = P.alpha;
      sA.beta = P.beta;
      sA.st_num = P.st_num;
      sA.gap_shift = bq.gap_shift;
      sA.heavy_min = bq.heavy_min;
      sA.max_spin = P.max_spin;
      sA.flags = P.flags;
      sA.ring_mask = bq.ring_mask;
      sA.ring_shift = bq.ring_shift;
      sA.step_cap = P.step_cap;
      sA.trace_cap = 0;
      sA.timeline = nullptr;
      sA.timeline_cap = 0;
      sA.nb = P.nb;
      sA.fuse = bq.fuse;
      sA.sweep_words = sweep_chunk(bq.G.ni, P.nb, blockDim.x);
    }
    __syncthreads();
    if (!query_setup(sA, ticket)) break;
    run_query<kPullFastGroup, kRelaxIlpGroup, kWide>(sA, Q, ticket);
    __syncthreads();
    if (ld_volatile_int(&c->status) != 0) break;
    query_output(sA);
    // every block's part of the result is written before the group reports
    if (!grid_barrier(&c->bar, &ticket, P.nb, P.max_spin, &c->status)) break;
    if (qb == 0 && threadIdx.x == 0) {
      __threadfence_system();
      P.done[e].status = EIC_OK;
      st_release_sys_u64(&P.done[e].ticket_plus1, t + 1);
      atomicAdd(finished, 1ull);
      reported = true;
    }
  }
  if (qb == 0 && threadIdx.x == 0) {
    if (!reported) {  // a request the group claimed and stopped in reports the group's error
      const unsigned long long t = mine;
      const uint32_t e = (uint32_t)(t & (P.cap - 1));
      const int st = ld_volatile_int(&c->status);
      __threadfence_system();
      P.done[e].status = st != 0 ? st : EIC_ETIMEOUT;
      st_release_sys_u64(&P.done[e].ticket_plus1, t + 1);
      atomicAdd(finished, 1ull);
    }
    // a group that stopped early counts as idle, so the others can leave
    if (!registered && atomicAdd(leave, 0ull) == 0) atomicAdd(idle_groups, 1ull);
  }
}

// Starting state of every group's barrier and status, and of the idle vote.
__global__ void k_serve_prep(const BatchSlot* slot, uint32_t groups, unsigned long long* claim) {
  const uint32_t g = blockIdx.x * blockDim.x + threadIdx.x;
  if (g < groups) {
    slot[g].ctl->bar.arrived = 0;
    slot[g].ctl->status = 0;
  }
  if (g == 0) {
    claim[2] = 0;
    claim[3] = 0;
  }
}

}  // namespace

// ------------------------------------------------------------------ host

namespace {

constexpr uint32_t kStepCap = 1u << 20;     // steps per query
constexpr uint32_t kTraceCap = 1u << 16;    // trace rows kept on the device
constexpr uint32_t kTimelineCap = 1u << 16; // diagnostic timeline events
constexpr uint32_t kHeavyMinCeil = 4096;
constexpr uint32_t kDefaultHeavyMin = 32;
constexpr int kDefaultBlock = 512;
constexpr uint32_t kDefaultSpinLog2 = 22;
constexpr uint32_t kStNumMax = 1u << 16;  // Function 2's candidate bins fit the 2^20-slot ring of wide weights

int resolve_params(const eic_params* in, eic_params* out) {
  if (in) {
    *out = *in;
  } else {
    eic_params_default(out);
  }
  if (!(out->beta > 0.0 && out->beta < 1.0)) return EIC_EINVAL;
  if (out->st_num == 0 || out->st_num > kStNumMax) return EIC_EINVAL;
  if (out->gap_shift > 16) return EIC_EINVAL;
  if (out->block_threads != 0 &&
      (out->block_threads % 32 != 0 || out->block_threads < 128 || out->block_threads > kMaxBlock))
    return EIC_EINVAL;
  if (out->heavy_min == 0) out->heavy_min = kDefaultHeavyMin;
  if (out->heavy_min < kHeavyMinFloor || out->heavy_min > kHeavyMinCeil) return EIC_EINVAL;
  if (out->max_spin_log2 == 0) out->max_spin_log2 = kDefaultSpinLog2;
  if (out->max_spin_log2 > 40) return EIC_EINVAL;
  return EIC_OK;
}

struct DeviceGuard {
  int prev = 0;
  bool ok = false;
  explicit DeviceGuard(int dev) {
    if (cudaGetDevice(&prev) == cudaSuccess && cudaSetDevice(dev) == cudaSuccess) ok = true;
    (void)cudaGetLastError();
  }
  ~DeviceGuard() { cudaSetDevice(prev); }
};

// Blocks a query runs on, of the sms * per_sm that fit: all of them, or 512
// threads on every SM for a query that is a chain of small steps, where a
// second block on the SM only slows the first one's chain (whether 152, 76 or 38
// blocks remain makes no difference to such a query). Measured with 304 and
// 152 blocks: RMAT 4 k 441, 376 us; 250 k 593, 564; 1 M vertices (650 k not
// isolated) 698, 672; 2 M 806, 804; 4 M 957, 1034; uniform 16 k 399, 368; 131 k
// 506, 509; 1 M 813, 841; grids 1024^2 24.1, 23.1 ms; 2048^2 46.9, 44.6; at
// gap_shift 4 1000^2 4.95, 4.80, 3000^2 15.6, 15.8.
// A dense graph with few distinct weights is no chain of small steps however
// few its vertices: the rows' entries of one weight, about 2m / maxW, all fall
// into the same step. 8 k to 260 k vertices with 41, 46, 50, 83, 132 and 208 M
// entries of weight 1: 560, 509, 485, 593, 801, 1114 us with 304 blocks and 467,
// 504, 604, 805, 1139, 1714 with 152; 266 M of weights up to 4: 641, 915; up to
// 8 (33 M each): 299, 317; up to 255: 302, 294. Nor is a graph of small degrees
// whose average is above 8 (no road network's is): 1 M vertices of degree 30
// without pulls 694, 744; 2 M 1019, 1047; 4 M of degree 16 1489, 1600.
int query_blocks(const DevGraph& G, const eic_params& p, int block, int sms, int per_sm) {
  const uint64_t vertices = (uint64_t)G.ni << p.gap_shift;  // (wider steps settle more at a time)
  const bool road = fuse_items(G, p.heavy_min, p.flags) == kFuseRoad && G.two_m <= 8ull * G.ni;
  if (vertices > (road ? 1ull << 26 : 3ull << 18) || (!road && G.two_m / G.maxw > 45u << 20)) return sms * per_sm;
  return sms * std::min(per_sm, std::max(1, kDefaultBlock / block));
}

// The cooperative grid of the query kernel, cached per workspace for the block
// size last used.
int launch_shape(Workspace* ws, int block) {
  if (ws->grid && ws->block == block) return EIC_OK;
  int dev = 0, sms = 0, per_sm = 0, coop = 0;
  EIC_CUDA_TRY(cudaGetDevice(&dev));
  EIC_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  EIC_CUDA_TRY(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
  if (!coop) return EIC_ECUDA;
  const bool wide = ws->ring_shift != 0;
  EIC_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, wide ? k_eic<true> : k_eic<false>, block, 0));
  if (per_sm < 1) return EIC_ECUDA;
  ws->grid = sms * per_sm;
  ws->sms = sms;
  ws->block = block;
  return EIC_OK;
}

// Blocks of k_init: a few 16-byte stores per thread, at most four blocks an SM.
int init_grid(const KArgs& A) {
  const uint64_t words = (uint64_t)A.G.ni + A.ring_mask + 1;
  return (int)std::min<uint64_t>(608, words / 2048 + 16);
}

KArgs make_args(eic_graph* g, uint32_t s, uint32_t* dist, const eic_params& p, int* status_out, int grid) {
  Workspace& w = g->ws;
  KArgs A;
  A.G = g->dg;
  A.dist = w.idist;
  A.out = dist;
  A.fbits = w.fbits;
  A.fwords = (uint32_t)(g->dg.ni / 32 + 2);
  A.cursor = w.cursor;
  A.q0 = w.q[0];
  A.q1 = w.q[1];
  A.sid = w.sid;
  A.sd = w.sd;
  A.scur = w.scur;
  A.touched = w.touched;
  A.sbits = w.sbits;
  A.hist = w.hist;
  A.ring = w.ring;
  A.tasks = w.tasks;
  A.step_ub = w.step_ub;
  A.step_off = w.step_off;
  A.trace = w.trace;
  A.ctl = w.ctl;
  A.status_out = status_out;
  A.s = s;
  A.alpha = p.alpha;
  A.beta = p.beta;
  A.st_num = p.st_num;
  A.gap_shift = p.gap_shift;
  A.heavy_min = p.heavy_min;
  A.max_spin = spin_limit(p.max_spin_log2);
  A.flags = p.flags;
  A.ring_mask = (1u << w.ring_bits) - 1u;
  A.ring_shift = w.ring_shift;
  A.step_cap = w.step_cap;
  A.trace_cap = kTraceCap;
  A.timeline = nullptr;
  A.timeline_cap = 0;
  A.nb = (uint32_t)grid;
  A.fuse = fuse_items(g->dg, p.heavy_min, p.flags);
  A.sweep_words = sweep_chunk(g->dg.ni, (uint32_t)grid, p.block_threads ? p.block_threads : kDefaultBlock);
  return A;
}

// Enqueue one query: dist <- +inf, init, persistent kernel, optional parent.
int enqueue_query(eic_graph* g, uint32_t s, uint32_t* dist, uint32_t* parent, const eic_params& p, int* status_out,
                  cudaStream_t st, bool timeline = false, cudaEvent_t ev0 = nullptr, cudaEvent_t ev1 = nullptr) {
  Workspace& w = g->ws;
  const int block = p.block_threads ? (int)p.block_threads : kDefaultBlock;
  int rc = launch_shape(&w, block);
  if (rc) return rc;
  const int grid = query_blocks(g->dg, p, block, w.sms, w.grid / w.sms);
  KArgs A = make_args(g, s, dist, p, status_out, grid);
  if (timeline) {
    A.timeline = w.timeline;
    A.timeline_cap = kTimelineCap;
  }
  k_init<<<init_grid(A), 256, 0, st>>>(A);
  EIC_CUDA_TRY(cudaGetLastError());
  void* args[] = {&A};
  if (ev0) EIC_CUDA_TRY(cudaEventRecord(ev0, st));
  EIC_CUDA_TRY(cudaLaunchCooperativeKernel(w.ring_shift ? (const void*)k_eic<true> : (const void*)k_eic<false>, dim3(grid),
                                           dim3(block), args, 0, st));
  if (ev1) EIC_CUDA_TRY(cudaEventRecord(ev1, st));
  k_output<<<4 * w.grid, 256, 0, st>>>(g->dg, w.idist, s, dist);
  EIC_CUDA_TRY(cudaGetLastError());
  if (parent) {
    if (g->dg.nbig) {  // (the queue's words and the tasks have served)
      k_parent_big<<<std::min(8 * (unsigned)w.sms, g->dg.nbig / 8 + 1), 256, 0, st>>>(g->dg, w.idist, w.q[0], w.tasks,
                                                                                     &w.ctl->ptasks);
      k_parent_pieces<<<std::min(8 * (unsigned)w.sms, g->dg.big_end / (8 * kParentPiece) + 1), 256, 0, st>>>(
          g->dg, w.idist, w.tasks, &w.ctl->ptasks, w.q[0]);
    }
    k_parent<<<(unsigned)std::min<uint64_t>(8 * w.sms, (uint64_t)g->dg.n / 32 + 1), 256, 0, st>>>(g->dg, w.idist, w.q[0],
                                                                                                  s, parent);
    EIC_CUDA_TRY(cudaGetLastError());
  }
  return EIC_OK;
}

// A graph without edges: only the source is reachable (its own parent).
__global__ void k_trivial(uint32_t n, uint32_t s, uint32_t* dist, uint32_t* parent) {
  for (uint64_t u = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; u < n; u += (uint64_t)gridDim.x * blockDim.x) {
    dist[u] = u == s ? 0u : EIC_INF;
    if (parent) parent[u] = u == s ? s : EIC_INF;
  }
}

int trivial_query(eic_graph* g, uint32_t s, uint32_t* dist, uint32_t* parent, cudaStream_t st) {
  k_trivial<<<256, 256, 0, st>>>(g->dg.n, s, dist, parent);
  EIC_CUDA_TRY(cudaGetLastError());
  EIC_CUDA_TRY(cudaStreamSynchronize(st));
  return EIC_OK;
}

// The device's address of an output array of the graph's GPU: its device
// memory, managed memory, or page-locked host memory mapped for the device
// (written across the host link). Anything else is rejected before launch.
int output_view(int dev, uint32_t* p, uint32_t** out) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    (void)cudaGetLastError();
    return EIC_EINVAL;
  }
  switch (a.type) {
    case cudaMemoryTypeDevice:
      if (a.device != dev) return EIC_EINVAL;
      *out = p;
      return EIC_OK;
    case cudaMemoryTypeManaged:
      *out = p;
      return EIC_OK;
    case cudaMemoryTypeHost:
      if (!a.devicePointer) return EIC_EINVAL;
      *out = (uint32_t*)a.devicePointer;
      return EIC_OK;
    default:
      return EIC_EINVAL;
  }
}

}  // namespace

namespace {
PinnedSlots g_mirrors[kMaxDevices];
}  // namespace

void eic_ws_free(Workspace* w) {
  cudaFree(w->base);
  if (w->ctl_pool)
    w->ctl_pool->put(w->ctl_host, w->ctl_epoch);
  else if (w->ctl_host)
    cudaFreeHost(w->ctl_host);
  if (w->ev[0]) cudaEventDestroy(w->ev[0]);
  if (w->ev[1]) cudaEventDestroy(w->ev[1]);
  *w = Workspace();
}

int eic_ws_ensure(eic_graph* g, int) {
  Workspace* w = &g->ws;
  if (w->ctl) return EIC_OK;
  const DevGraph& G = g->dg;
  w->ring_bits = ring_layout(G.maxw, &w->ring_shift);
  w->step_cap = kStepCap;
  w->n = G.ni;  // per-vertex arrays cover the internal (non-isolated) vertices
  SlotCaps caps;
  caps.ni = G.ni;
  caps.two_m = G.two_m;
  caps.D = G.D;
  caps.ring_bits = w->ring_bits;
  const SlotLayout L = slot_layout(caps, kStepCap);  // one allocation: 19 of them took 0.5 ms, and freeing them as long
  const uint64_t trace = L.bytes, timeline = trace + ((kTraceCap * sizeof(eic_step) + 255) & ~255ull);
  const uint64_t bytes = timeline + 2ull * kTimelineCap * 8;
  if (cudaMalloc((void**)&w->base, bytes) != cudaSuccess) {
    (void)cudaGetLastError();
    *w = Workspace();
    return EIC_ENOMEM;
  }
  unsigned char* b = w->base;
  w->bytes = bytes;
  w->idist = (uint32_t*)(b + L.idist);
  w->fbits = (uint32_t*)(b + L.fbits);
  w->cursor = (uint32_t*)(b + L.cursor);
  w->q[0] = (uint32_t*)(b + L.q0);
  w->q[1] = (uint32_t*)(b + L.q1);
  w->sid = (uint32_t*)(b + L.sid);
  w->sd = (uint32_t*)(b + L.sd);
  w->scur = (uint32_t*)(b + L.scur);
  w->touched = (uint32_t*)(b + L.touched);
  w->sbits = (uint32_t*)(b + L.sbits);
  w->hist = (uint32_t*)(b + L.hist);
  w->ring = (uint32_t*)(b + L.ring);
  w->tasks = (Task*)(b + L.tasks);
  w->step_ub = (int64_t*)(b + L.step_ub);
  w->step_off = (uint32_t*)(b + L.step_off);
  w->ctl = (Ctl*)(b + L.ctl);
  w->trace = (eic_step*)(b + trace);
  w->timeline = (unsigned long long*)(b + timeline);
  static_assert(sizeof(Ctl) <= PinnedSlots::kBytes, "a control block fits a slot");
  PinnedSlots* pool = g->device >= 0 && g->device < kMaxDevices ? &g_mirrors[g->device] : nullptr;
  w->ctl_host = pool ? (Ctl*)pool->get(&w->ctl_epoch) : nullptr;
  w->ctl_pool = w->ctl_host ? pool : nullptr;
  if (!w->ctl_host && cudaMallocHost((void**)&w->ctl_host, sizeof(Ctl)) != cudaSuccess) {
    (void)cudaGetLastError();
    eic_ws_free(w);
    return EIC_ENOMEM;
  }
  return EIC_OK;
}

extern "C" {

int eic_sssp(const eic_graph* gc, uint32_t source, uint32_t* dist, uint32_t* parent, const eic_params* params,
             eic_stats* stats, void* stream) {
  eic_graph* g = const_cast<eic_graph*>(gc);
  if (!g || !dist) return EIC_EINVAL;
  if (source >= g->dg.n) return EIC_EINVAL;
  eic_params p;
  int rc = resolve_params(params, &p);
  if (rc) return rc;
  std::lock_guard<std::mutex> lock(g->mu);
  DeviceGuard dg(g->device);
  if (!dg.ok) return EIC_ECUDA;
  cudaStream_t st = (cudaStream_t)stream;
  if ((rc = output_view(g->device, dist, &dist)) || (parent && (rc = output_view(g->device, parent, &parent))))
    return rc;
  eic_step* trace = stats ? stats->trace : nullptr;
  const uint64_t trace_cap = stats ? stats->trace_cap : 0;
  uint64_t* tl = stats ? stats->timeline : nullptr;
  const uint64_t tl_cap = stats ? stats->timeline_cap : 0;
  if (stats) {
    memset(stats, 0, sizeof(*stats));
    stats->trace = trace;
    stats->trace_cap = trace_cap;
    stats->timeline = tl;
    stats->timeline_cap = tl_cap;
  }
  if (g->dg.two_m == 0) return trivial_query(g, source, dist, parent, st);
  if ((rc = eic_ws_ensure(g, 0))) return rc;
  Workspace& w = g->ws;
  if (stats && !w.ev[0]) {
    if (cudaEventCreate(&w.ev[0]) != cudaSuccess || cudaEventCreate(&w.ev[1]) != cudaSuccess) {
      (void)cudaGetLastError();
      return EIC_ECUDA;
    }
  }
  if ((rc = enqueue_query(g, source, dist, parent, p, nullptr, st, tl && tl_cap, stats ? w.ev[0] : nullptr,
                          stats ? w.ev[1] : nullptr))) {
    cudaStreamSynchronize(st);
    (void)cudaGetLastError();
    return rc;
  }
  EIC_CUDA_TRY(cudaMemcpyAsync(w.ctl_host, w.ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, st));
  EIC_CUDA_TRY(cudaStreamSynchronize(st));
  const Ctl& h = *w.ctl_host;
  if (stats) {
    stats->steps = h.trace_len;
    stats->rounds = h.cnt_rounds;
    stats->frontier = h.cnt_frontier;
    stats->traversed = h.cnt_trav;
    stats->pulls = h.cnt_pulls;
    stats->improved = h.cnt_improved;
    stats->heavy = h.cnt_heavy;
    stats->pull_items = h.cnt_pitems;
    stats->trace_len = h.trace_len;
    float kms = 0.f;
    if (cudaEventElapsedTime(&kms, w.ev[0], w.ev[1]) == cudaSuccess) stats->kernel_ms = kms;
    (void)cudaGetLastError();
    if (trace && trace_cap) {
      uint64_t rows = h.trace_len < trace_cap ? h.trace_len : trace_cap;
      if (rows > kTraceCap) rows = kTraceCap;
      if (rows) EIC_CUDA_TRY(cudaMemcpy(trace, w.trace, rows * sizeof(eic_step), cudaMemcpyDeviceToHost));
    }
    if (tl && tl_cap) {
      uint64_t ev = h.tl_len < tl_cap ? h.tl_len : tl_cap;
      if (ev > kTimelineCap) ev = kTimelineCap;
      stats->timeline_len = h.tl_len;
      if (ev) EIC_CUDA_TRY(cudaMemcpy(tl, w.timeline, ev * 16, cudaMemcpyDeviceToHost));
    }
  }
  return h.status;
}

}  // extern "C"

// ------------------------------------------------------------ batch host side

namespace {

int batch_grid(int block, bool wide, uint32_t* grid) {
  int dev = 0, sms = 0, per_sm = 0, coop = 0;
  EIC_CUDA_TRY(cudaGetDevice(&dev));
  EIC_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  EIC_CUDA_TRY(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
  if (!coop) return EIC_ECUDA;
  EIC_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, wide ? k_eic_batch<true> : k_eic_batch<false>,
                                                             block, 0));
  if (per_sm < 1) return EIC_ECUDA;
  *grid = (uint32_t)(sms * per_sm);
  return EIC_OK;
}

SlotPool g_pool[kMaxDevices];  // scratch reused by eic_sssp_batch, per device
std::mutex g_pool_mu;

}  // namespace

// A prepared batch: the query table in claim order (largest graphs first),
// the trivial queries (graphs without edges), the launch configuration and,
// once run, the CUDA graph that replays it.
struct eic_batch {
  int device = 0;
  uint32_t nq = 0;
  eic_params p{};
  std::vector<uint32_t> order;  // claim position -> caller's query index
  std::vector<const eic_graph*> qgraph;  // claim position -> graph, source, output
  std::vector<uint32_t> qsource;
  std::vector<uint32_t*> qdist;
  std::vector<BatchQuery> hq;
  struct Trivial {
    uint32_t* dist;
    uint32_t n, s, index;
  };
  std::vector<Trivial> trivial;
  SlotCaps caps;
  uint32_t groups = 0, nb = 0, block = 0, grid_max = 0;
  SlotPool own;
  SlotPool* pool = &own;
  BatchQuery* d_q = nullptr;
  int* d_status = nullptr;
  int* h_status = nullptr;
  uint32_t* d_queue = nullptr;
  bool use_graph = true;
  bool wide = false;  // a graph of the batch has weights of 2^20 and above
  cudaGraphExec_t exec = nullptr;
  double tuned_ms = 0.0;
};

namespace {

// Largest group count whose scratch fits in the share of free memory.
uint32_t groups_that_fit(eic_batch* b, uint32_t want) {
  size_t fr = 0, tot = 0;
  if (cudaMemGetInfo(&fr, &tot) != cudaSuccess) {
    (void)cudaGetLastError();
    return want;
  }
  const uint64_t per = slot_layout(b->caps).bytes;
  const uint64_t held = b->pool->base ? (uint64_t)b->pool->count * b->pool->slot_bytes : 0;
  const uint64_t avail = (uint64_t)((double)(fr + held) * kBatchMemFrac);
  const uint64_t fit = per ? avail / per : want;
  return (uint32_t)(fit < want ? fit : want);
}

// groups -> blocks per group for the current block shape; nb_force (when
// nonzero) fixes the blocks per group instead, and the groups then fill at
// most the co-resident grid.
int batch_configure(eic_batch* b, uint32_t groups, uint32_t block, uint32_t nb_force = 0) {
  uint32_t gmax = 0;
  int rc = batch_grid((int)block, b->wide, &gmax);
  if (rc) return rc;
  if (nb_force) {
    if (nb_force > gmax) nb_force = gmax;
    if (groups == 0 || groups > gmax / nb_force) groups = gmax / nb_force;
  }
  const uint32_t nrun = (uint32_t)b->hq.size();
  if (groups == 0) {  // library choice: about 8 blocks per group, more for graphs above 2^27 entries
    const uint64_t per = b->caps.two_m >> 24;
    const uint32_t nb = per < 8 ? 8 : (per > gmax ? gmax : (uint32_t)per);
    groups = gmax / nb;
  }
  if (groups > nrun) groups = nrun ? nrun : 1;
  if (groups > gmax) groups = gmax;
  groups = groups_that_fit(b, groups);
  if (groups == 0) return EIC_ENOMEM;
  if ((rc = b->pool->ensure(b->caps, groups))) return rc;
  if (b->exec && (b->groups != groups || b->block != block)) {
    cudaGraphExecDestroy(b->exec);
    b->exec = nullptr;
  }
  b->groups = groups;
  b->block = block;
  b->grid_max = gmax;
  b->nb = nb_force ? nb_force : gmax / groups;
  return EIC_OK;
}

// The host query table to the device (per-query parameters changed), before any later launch on any stream.
int batch_upload(eic_batch* b, cudaStream_t st) {
  if (b->hq.empty()) return EIC_OK;
  EIC_CUDA_TRY(cudaMemcpyAsync(b->d_q, b->hq.data(), b->hq.size() * sizeof(BatchQuery), cudaMemcpyHostToDevice, st));
  EIC_CUDA_TRY(cudaStreamSynchronize(st));
  if (b->exec) {
    cudaGraphExecDestroy(b->exec);
    b->exec = nullptr;
  }
  return EIC_OK;
}

BatchArgs batch_args(const eic_batch* b) {
  BatchArgs P;
  P.q = b->d_q;
  P.slot = b->pool->d_slots;
  P.status = b->d_status;
  P.queue = b->d_queue;
  P.nq = (uint32_t)b->hq.size();
  P.nb = b->nb;
  P.alpha = b->p.alpha;
  P.beta = b->p.beta;
  P.st_num = b->p.st_num;
  P.gap_shift = b->p.gap_shift;
  P.heavy_min = b->p.heavy_min;
  P.flags = b->p.flags;
  P.step_cap = kBatchStepCap;
  P.max_spin = spin_limit(b->p.max_spin_log2);
  return P;
}

int batch_enqueue(eic_batch* b, cudaStream_t st) {
  if (!b->hq.empty()) {
    BatchArgs P = batch_args(b);
    const uint32_t nrun = P.nq, cover = b->groups > nrun ? b->groups : nrun;
    k_batch_prep<<<(cover + 255) / 256, 256, 0, st>>>(P, b->groups);
    EIC_CUDA_TRY(cudaGetLastError());
    void* args[] = {&P};
    EIC_CUDA_TRY(cudaLaunchCooperativeKernel(b->wide ? (const void*)k_eic_batch<true> : (const void*)k_eic_batch<false>,
                                             dim3(b->groups * b->nb), dim3(b->block), args, 0, st));
  }
  for (const auto& t : b->trivial) {  // no edges: only the source is reachable
    EIC_CUDA_TRY(cudaMemsetAsync(t.dist, 0xFF, (uint64_t)t.n * 4, st));
    EIC_CUDA_TRY(cudaMemsetAsync(t.dist + t.s, 0, 4, st));
  }
  return EIC_OK;
}

void batch_free(eic_batch* b) {
  if (b->exec) cudaGraphExecDestroy(b->exec);
  b->own.release();
  cudaFree(b->d_q);
  cudaFree(b->d_status);
  cudaFree(b->d_queue);
  if (b->h_status) cudaFreeHost(b->h_status);
  delete b;
}

// The query table is copied on st, which orders it before launches there.
int batch_create(const eic_graph* const* graphs, const uint32_t* sources, uint32_t nq, uint32_t* const* dists,
                 const eic_params* params, SlotPool* shared_pool, cudaStream_t st, eic_batch** out) {
  *out = nullptr;
  if (nq == 0 || !graphs || !sources || !dists) return EIC_EINVAL;
  eic_params p;
  int rc = resolve_params(params, &p);
  if (rc) return rc;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    (void)cudaGetLastError();
    return EIC_ECUDA;
  }
  for (uint32_t i = 0; i < nq; ++i)
    if (!graphs[i] || !dists[i] || sources[i] >= graphs[i]->dg.n || graphs[i]->device != dev) return EIC_EINVAL;
  eic_batch* b = new eic_batch();
  b->device = dev;
  b->nq = nq;
  b->p = p;
  if (shared_pool) b->pool = shared_pool;
  std::vector<uint32_t> idx;
  for (uint32_t i = 0; i < nq; ++i) {
    const DevGraph& G = graphs[i]->dg;
    if (G.two_m == 0) {
      b->trivial.push_back({dists[i], G.n, sources[i], i});
      continue;
    }
    idx.push_back(i);
  }
  // largest graphs are claimed first (longest-processing-time order)
  std::stable_sort(idx.begin(), idx.end(),
                   [&](uint32_t a, uint32_t c) { return graphs[a]->dg.two_m > graphs[c]->dg.two_m; });
  for (uint32_t i : idx) {
    const DevGraph& G = graphs[i]->dg;
    BatchQuery q;
    q.G = G;
    q.out = dists[i];
    q.s = sources[i];
    uint32_t shift = 0;
    const uint32_t bits = ring_layout(G.maxw, &shift);
    b->wide |= shift != 0;
    q.ring_mask = (1u << bits) - 1u;
    q.ring_shift = shift;
    q.gap_shift = p.gap_shift;
    q.heavy_min = p.heavy_min;
    q.fuse = fuse_items(G, p.heavy_min, p.flags);
    b->hq.push_back(q);
    b->order.push_back(i);
    b->qgraph.push_back(graphs[i]);
    b->qsource.push_back(sources[i]);
    b->qdist.push_back(dists[i]);
    SlotCaps& c = b->caps;
    c.ni = G.ni > c.ni ? G.ni : c.ni;
    c.two_m = G.two_m > c.two_m ? G.two_m : c.two_m;
    c.D = G.D > c.D ? G.D : c.D;
    c.ring_bits = bits > c.ring_bits ? bits : c.ring_bits;
  }
  const uint64_t nrun = b->hq.size();
  if (nrun) {
    if (cudaMalloc((void**)&b->d_q, nrun * sizeof(BatchQuery)) != cudaSuccess ||
        cudaMalloc((void**)&b->d_status, nrun * sizeof(int)) != cudaSuccess ||
        cudaMalloc((void**)&b->d_queue, sizeof(uint32_t)) != cudaSuccess ||
        cudaMallocHost((void**)&b->h_status, nrun * sizeof(int)) != cudaSuccess) {
      (void)cudaGetLastError();
      batch_free(b);
      return EIC_ENOMEM;
    }
    if (cudaMemcpyAsync(b->d_q, b->hq.data(), nrun * sizeof(BatchQuery), cudaMemcpyHostToDevice, st) != cudaSuccess) {
      (void)cudaGetLastError();
      batch_free(b);
      return EIC_ECUDA;
    }
    const uint32_t block = p.block_threads ? p.block_threads : (uint32_t)kDefaultBlock;
    if ((rc = batch_configure(b, p.batch_groups, block))) {
      batch_free(b);
      return rc;
    }
  }
  *out = b;
  return EIC_OK;
}

int batch_run(eic_batch* b, cudaStream_t st) {
  if (b->use_graph && !b->exec) {  // capture the launch sequence once, replay it afterwards
    cudaStream_t cs = nullptr;
    cudaGraph_t graph = nullptr;
    bool ok = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking) == cudaSuccess &&
              cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal) == cudaSuccess;
    if (ok) {
      const int rc = batch_enqueue(b, cs);
      ok = cudaStreamEndCapture(cs, &graph) == cudaSuccess && rc == EIC_OK && graph &&
           cudaGraphInstantiate(&b->exec, graph, 0) == cudaSuccess;
    }
    if (graph) cudaGraphDestroy(graph);
    if (cs) cudaStreamDestroy(cs);
    if (!ok) {  // capture unavailable: launch directly from now on
      (void)cudaGetLastError();
      b->exec = nullptr;
      b->use_graph = false;
    }
  }
  if (b->exec) {
    EIC_CUDA_TRY(cudaGraphLaunch(b->exec, st));
    return EIC_OK;
  }
  return batch_enqueue(b, st);
}

int batch_wait(eic_batch* b, cudaStream_t st, int* statuses) {
  const uint64_t nrun = b->hq.size();
  if (nrun) EIC_CUDA_TRY(cudaMemcpyAsync(b->h_status, b->d_status, nrun * sizeof(int), cudaMemcpyDeviceToHost, st));
  EIC_CUDA_TRY(cudaStreamSynchronize(st));
  std::vector<int> all(b->nq, EIC_OK);
  for (uint64_t k = 0; k < nrun; ++k) all[b->order[k]] = b->h_status[k];
  int first = EIC_OK;
  for (uint32_t i = 0; i < b->nq; ++i) {
    if (statuses) statuses[i] = all[i];
    if (first == EIC_OK) first = all[i];
  }
  return first;
}

// Device time of one whole batch run (ms), or a negative value on error.
double batch_time(eic_batch* b, cudaStream_t st) {
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
    (void)cudaGetLastError();
    return -1.0;
  }
  double ms = -1.0;
  float t = 0.f;
  if (cudaEventRecord(e0, st) == cudaSuccess && batch_enqueue(b, st) == EIC_OK &&
      cudaEventRecord(e1, st) == cudaSuccess && cudaEventSynchronize(e1) == cudaSuccess &&
      cudaEventElapsedTime(&t, e0, e1) == cudaSuccess && batch_wait(b, st, nullptr) == EIC_OK)
    ms = t;
  (void)cudaGetLastError();
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  return ms;
}

}  // namespace

extern "C" {

int eic_sssp_batch(const eic_graph* const* graphs, const uint32_t* sources, uint32_t num_queries,
                   uint32_t* const* dists, const eic_params* params, int* statuses, void* stream) {
  if (num_queries == 0) return EIC_OK;
  if (!graphs || !sources || !dists) return EIC_EINVAL;
  if (!graphs[0]) return EIC_EINVAL;
  DeviceGuard guard(graphs[0]->device);
  if (!guard.ok || graphs[0]->device < 0 || graphs[0]->device >= kMaxDevices) return EIC_ECUDA;
  std::lock_guard<std::mutex> lock(g_pool_mu);
  eic_batch* b = nullptr;
  cudaStream_t st = (cudaStream_t)stream;
  int rc = batch_create(graphs, sources, num_queries, dists, params, &g_pool[graphs[0]->device], st, &b);
  if (rc) {
    if (statuses)
      for (uint32_t i = 0; i < num_queries; ++i) statuses[i] = rc;
    return rc;
  }
  b->use_graph = false;  // one-shot: launch directly
  rc = batch_enqueue(b, st);
  if (rc == EIC_OK) {
    rc = batch_wait(b, st, statuses);
  } else {
    cudaStreamSynchronize(st);
    (void)cudaGetLastError();
    if (statuses)
      for (uint32_t i = 0; i < num_queries; ++i) statuses[i] = rc;
  }
  batch_free(b);
  return rc;
}

int eic_batch_create(const eic_graph* const* graphs, const uint32_t* sources, uint32_t num_queries,
                     uint32_t* const* dists, const eic_params* params, eic_batch** out) {
  if (!out) return EIC_EINVAL;
  *out = nullptr;
  if (!graphs || !graphs[0]) return EIC_EINVAL;
  DeviceGuard guard(graphs[0]->device);
  if (!guard.ok) return EIC_ECUDA;
  const int rc = batch_create(graphs, sources, num_queries, dists, params, nullptr, nullptr, out);
  if (rc != EIC_OK || cudaStreamSynchronize(nullptr) == cudaSuccess) return rc;
  (void)cudaGetLastError();
  batch_free(*out);
  *out = nullptr;
  return EIC_ECUDA;
}

int eic_batch_run(eic_batch* b, void* stream) {
  if (!b) return EIC_EINVAL;
  DeviceGuard guard(b->device);
  if (!guard.ok) return EIC_ECUDA;
  return batch_run(b, (cudaStream_t)stream);
}

int eic_batch_wait(eic_batch* b, void* stream, int* statuses) {
  if (!b) return EIC_EINVAL;
  DeviceGuard guard(b->device);
  if (!guard.ok) return EIC_ECUDA;
  return batch_wait(b, (cudaStream_t)stream, statuses);
}

int eic_batch_tune(eic_batch* b, void* stream, eic_batch_config* best) {
  if (!b) return EIC_EINVAL;
  DeviceGuard guard(b->device);
  if (!guard.ok) return EIC_ECUDA;
  cudaStream_t st = (cudaStream_t)stream;
  if (!b->hq.empty()) {
    const uint32_t nrun = (uint32_t)b->hq.size();
    int rc = EIC_OK;
    uint32_t best_g = b->groups, best_block = b->block, best_hm = b->p.heavy_min;
    double best_ms = 1e300;
    // one configuration: a warm-up run, then a timed one when the warm-up was
    // within 2x of the best so far
    auto trial = [&](uint32_t g, uint32_t block, uint32_t hm, double* ms_out) -> int {
      for (auto& q : b->hq) {
        q.heavy_min = hm;
        q.fuse = fuse_items(q.G, hm, b->p.flags);
      }
      b->p.heavy_min = hm;
      int r = batch_upload(b, st);
      if (r) return r;
      if ((r = batch_configure(b, g, block))) return r;
      double ms = batch_time(b, st);
      if (ms < 0) return EIC_ECUDA;
      if (ms < 2.0 * best_ms) {
        const double ms2 = batch_time(b, st);
        if (ms2 < 0) return EIC_ECUDA;
        ms = ms2 < ms ? ms2 : ms;
      }
      if (ms < best_ms) {
        best_ms = ms;
        best_g = b->groups;
        best_block = b->block;
        best_hm = hm;
      }
      if (ms_out) *ms_out = ms;
      return EIC_OK;
    };
    uint32_t gmax = 0;
    if ((rc = batch_grid((int)b->block, b->wide, &gmax))) return rc;
    // pass 1: group counts (divisors of the grid and powers of two), from the
    // most groups down, until two in a row are 20% slower than the best
    std::vector<uint32_t> cand;
    for (uint32_t g = gmax; g >= 1; --g)
      if (g <= nrun && (gmax % g == 0 || (g & (g - 1)) == 0)) cand.push_back(g);
    uint32_t worse = 0;
    for (uint32_t g : cand) {
      double ms = 0;
      if ((rc = trial(g, b->block, best_hm, &ms))) return rc;
      worse = ms > 1.2 * best_ms ? worse + 1 : 0;
      if (worse >= 2) break;
    }
    // pass 2: each graph's step-width scaling (exact for every value), timed on
    // a sub-batch of that graph's queries at the chosen blocks per group:
    // gap_shift + 1, + 2, ... while it helps by 2% (up to 8)
    if ((rc = batch_configure(b, best_g, best_block))) return rc;
    const uint32_t nb = b->nb;
    std::vector<const eic_graph*> seen;
    for (uint32_t k = 0; k < nrun; ++k) {
      const eic_graph* g = b->qgraph[k];
      if (std::find(seen.begin(), seen.end(), g) != seen.end()) continue;
      seen.push_back(g);
      std::vector<uint32_t> pos;
      for (uint32_t j = 0; j < nrun; ++j)
        if (b->qgraph[j] == g) pos.push_back(j);
      std::vector<const eic_graph*> sg(pos.size(), g);
      std::vector<uint32_t> ss;
      std::vector<uint32_t*> sd;
      for (uint32_t j : pos) {
        ss.push_back(b->qsource[j]);
        sd.push_back(b->qdist[j]);
      }
      eic_batch* sub = nullptr;
      if ((rc = batch_create(sg.data(), ss.data(), (uint32_t)pos.size(), sd.data(), &b->p, nullptr, st, &sub)))
        return rc;
      rc = batch_configure(sub, (uint32_t)pos.size(), best_block, nb);
      uint32_t gs_best = b->hq[k].gap_shift;
      double t_best = -1.0;
      for (uint32_t gs = gs_best; rc == EIC_OK && gs <= 8; ++gs) {
        for (auto& q : sub->hq) q.gap_shift = gs;
        if ((rc = batch_upload(sub, st))) break;
        double t = batch_time(sub, st);
        const double t2 = batch_time(sub, st);
        if (t < 0 || t2 < 0) {
          rc = EIC_ECUDA;
          break;
        }
        t = t2 < t ? t2 : t;
        if (t_best < 0 || t < 0.98 * t_best) {
          t_best = t;
          gs_best = gs;
        } else {
          break;
        }
      }
      batch_free(sub);
      if (rc) return rc;
      for (uint32_t j : pos) b->hq[j].gap_shift = gs_best;
    }
    best_ms = 1e300;
    if ((rc = trial(best_g, best_block, best_hm, nullptr))) return rc;
    // pass 3 at the best group count: the window-class threshold, then a
    // 256-thread block
    const uint32_t hm0 = best_hm;
    for (uint32_t hm : {64u, 256u})
      if ((rc = trial(best_g, best_block, hm, nullptr))) return rc;
    if ((rc = trial(best_g, 256, best_hm, nullptr))) return rc;
    (void)hm0;
    // keep the winner; the scratch shrinks to its group count
    for (auto& q : b->hq) {
      q.heavy_min = best_hm;
      q.fuse = fuse_items(q.G, best_hm, b->p.flags);
    }
    b->p.heavy_min = best_hm;
    if ((rc = batch_upload(b, st))) return rc;
    if (b->pool == &b->own && b->own.count > best_g) b->own.release();
    if ((rc = batch_configure(b, best_g, best_block))) return rc;
    if (b->exec) {
      cudaGraphExecDestroy(b->exec);
      b->exec = nullptr;
    }
    b->tuned_ms = best_ms;
  }
  return best ? eic_batch_info(b, best) : EIC_OK;
}

int eic_batch_info(const eic_batch* b, eic_batch_config* out) {
  if (!b || !out) return EIC_EINVAL;
  memset(out, 0, sizeof(*out));
  out->groups = b->groups;
  out->blocks_per_group = b->nb;
  out->block_threads = b->block;
  out->cuda_graph = b->exec ? 1u : 0u;
  out->gap_shift = b->p.gap_shift;
  for (const auto& q : b->hq) out->gap_shift = q.gap_shift > out->gap_shift ? q.gap_shift : out->gap_shift;
  out->heavy_min = b->p.heavy_min;
  out->queries = b->nq;
  out->scratch_bytes = (uint64_t)b->pool->count * b->pool->slot_bytes;
  out->tuned_ms = b->tuned_ms;
  return EIC_OK;
}

int eic_batch_gap_shifts(const eic_batch* b, uint32_t* gap_shifts) {
  if (!b || !gap_shifts) return EIC_EINVAL;
  for (uint32_t i = 0; i < b->nq; ++i) gap_shifts[i] = b->p.gap_shift;  // graphs without edges keep the batch's
  for (size_t k = 0; k < b->hq.size(); ++k) gap_shifts[b->order[k]] = b->hq[k].gap_shift;
  return EIC_OK;
}

int eic_batch_destroy(eic_batch* b) {
  if (!b) return EIC_OK;
  DeviceGuard guard(b->device);
  batch_free(b);
  return EIC_OK;
}

}  // extern "C"


// ------------------------------------------------ allocation-free entry point
//
// The query scratch of eic_sssp_noalloc: one file-scope device array carved
// into the workspace arrays of a graph with at most kNaN vertices, kNaE
// adjacency entries, weights below 2^16 and kNaD distinct degrees. Every GPU
// that loads the library holds it until the process exits.
namespace {

constexpr uint64_t kNaN = EIC_NOALLOC_MAX_VERTICES;
constexpr uint64_t kNaE = EIC_NOALLOC_MAX_ENTRIES;
constexpr uint64_t kNaD = EIC_NOALLOC_MAX_DEGREES;
constexpr uint64_t kNaS = EIC_NOALLOC_MAX_STEPS;
constexpr uint32_t kNaRingBits = 16;  // 2^16 > EIC_NOALLOC_MAX_WEIGHT
constexpr uint64_t kNaTasks = kNaE / kHeavyMinFloor + 2;

constexpr uint64_t na_align(uint64_t x) { return (x + 255) & ~255ull; }
constexpr uint64_t kNaIdist = 0;
constexpr uint64_t kNaFbits = kNaIdist + na_align(kNaN * 4);
constexpr uint64_t kNaCursor = kNaFbits + na_align(2 * (kNaN / 32 + 2) * 4);
constexpr uint64_t kNaQ0 = kNaCursor + na_align(kNaN * 4);
constexpr uint64_t kNaQ1 = kNaQ0 + na_align(kNaN * 4);
constexpr uint64_t kNaSid = kNaQ1 + na_align(kNaN * 4);
constexpr uint64_t kNaSd = kNaSid + na_align((kNaN + 2) * 4);
constexpr uint64_t kNaScur = kNaSd + na_align((kNaN + 2) * 4);
constexpr uint64_t kNaTouched = kNaScur + na_align((kNaN + 2) * 4);
constexpr uint64_t kNaSbits = kNaTouched + na_align((kNaN + 1) * 4);
constexpr uint64_t kNaHist = kNaSbits + na_align((kNaN / 32 + 2) * 4);
constexpr uint64_t kNaRing = kNaHist + na_align(kNaD * 4);
constexpr uint64_t kNaTaskOff = kNaRing + na_align((1ull << kNaRingBits) * 4);
constexpr uint64_t kNaStepUb = kNaTaskOff + na_align(kNaTasks * sizeof(Task));
constexpr uint64_t kNaStepOff = kNaStepUb + na_align((kNaS + 2) * 8);
constexpr uint64_t kNaCtl = kNaStepOff + na_align((kNaS + 2) * 4);
constexpr uint64_t kNaBytes = kNaCtl + na_align(sizeof(Ctl));
static_assert(kNaBytes > 13100000 && kNaBytes < 13250000, "the header states the scratch size as about 13.1 MB");

static __device__ __align__(256) unsigned char g_na_scratch[kNaBytes];

struct NaDevice {
  bool ready = false;
  unsigned char* base = nullptr;  // device address of g_na_scratch on this device
  int grid = 0, sms = 0;
};
NaDevice g_na[kMaxDevices];
std::mutex g_na_mu;

// Once per device, with that device current: the scratch's device address
// (the symbol's host-side name is not a device pointer), a cleared control
// block, and the cooperative grid shape.
int na_setup(NaDevice& d, cudaStream_t st) {
  void* ptr = nullptr;
  EIC_CUDA_TRY(cudaGetSymbolAddress(&ptr, g_na_scratch));
  if (!ptr) return EIC_ECUDA;
  int dev = 0, sms = 0, per_sm = 0, coop = 0;
  EIC_CUDA_TRY(cudaGetDevice(&dev));
  EIC_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  EIC_CUDA_TRY(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
  if (!coop) return EIC_ECUDA;
  EIC_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_eic<false>, kDefaultBlock, 0));
  if (per_sm < 1) return EIC_ECUDA;
  unsigned char* base = (unsigned char*)ptr;
  EIC_CUDA_TRY(cudaMemsetAsync(base + kNaCtl, 0, sizeof(Ctl), st));
  EIC_CUDA_TRY(cudaStreamSynchronize(st));
  d.base = base;
  d.grid = sms * per_sm;
  d.sms = sms;
  d.ready = true;
  return EIC_OK;
}

}  // namespace

extern "C" int eic_sssp_noalloc(const eic_graph* gc, uint32_t source, uint32_t* dist, void* stream) {
  if (!gc || !dist) return EIC_EINVAL;
  const DevGraph& G = gc->dg;
  if (source >= G.n) return EIC_EINVAL;
  if (G.n > kNaN || G.two_m > kNaE || G.maxw > EIC_NOALLOC_MAX_WEIGHT || G.D > kNaD) return EIC_ESIZE;
  cudaStream_t st = (cudaStream_t)stream;
  std::lock_guard<std::mutex> lock(g_na_mu);
  DeviceGuard guard(gc->device);
  if (!guard.ok || gc->device < 0 || gc->device >= kMaxDevices) return EIC_ECUDA;
  NaDevice& nd = g_na[gc->device];
  int rc;
  if (!nd.ready && (rc = na_setup(nd, st))) return rc;
  if (G.two_m == 0) {  // no edges: only the source is reachable
    EIC_CUDA_TRY(cudaMemsetAsync(dist, 0xFF, (uint64_t)G.n * 4, st));
    EIC_CUDA_TRY(cudaMemsetAsync(dist + source, 0, 4, st));
    EIC_CUDA_TRY(cudaStreamSynchronize(st));
    return EIC_OK;
  }
  unsigned char* b = nd.base;
  Ctl* ctl = (Ctl*)(b + kNaCtl);
  KArgs A;
  A.G = G;
  A.dist = (uint32_t*)(b + kNaIdist);
  A.out = dist;
  A.fbits = (uint32_t*)(b + kNaFbits);
  A.fwords = (uint32_t)(G.ni / 32 + 2);
  A.cursor = (uint32_t*)(b + kNaCursor);
  A.q0 = (uint32_t*)(b + kNaQ0);
  A.q1 = (uint32_t*)(b + kNaQ1);
  A.sid = (uint32_t*)(b + kNaSid);
  A.sd = (uint32_t*)(b + kNaSd);
  A.scur = (uint32_t*)(b + kNaScur);
  A.touched = (uint32_t*)(b + kNaTouched);
  A.sbits = (uint32_t*)(b + kNaSbits);
  A.hist = (uint32_t*)(b + kNaHist);
  A.ring = (uint32_t*)(b + kNaRing);
  A.tasks = (Task*)(b + kNaTaskOff);
  A.step_ub = (int64_t*)(b + kNaStepUb);
  A.step_off = (uint32_t*)(b + kNaStepOff);
  A.trace = nullptr;
  A.ctl = ctl;
  A.status_out = nullptr;
  A.s = source;
  A.alpha = 3;
  A.beta = 0.9;
  A.st_num = 1024;
  A.gap_shift = 0;
  A.heavy_min = kDefaultHeavyMin;
  A.max_spin = spin_limit(kDefaultSpinLog2);
  A.flags = 0;
  A.ring_mask = (1u << kNaRingBits) - 1u;
  A.ring_shift = 0;
  A.step_cap = (uint32_t)kNaS;
  A.trace_cap = 0;
  A.timeline = nullptr;
  A.timeline_cap = 0;
  A.fuse = fuse_items(G, A.heavy_min, A.flags);
  eic_params p;
  eic_params_default(&p);
  p.heavy_min = A.heavy_min;
  const int grid = query_blocks(G, p, kDefaultBlock, nd.sms, nd.grid / nd.sms);
  A.nb = (uint32_t)grid;
  A.sweep_words = sweep_chunk(G.ni, (uint32_t)grid, kDefaultBlock);
  // Once anything is enqueued, every return waits for the stream first: the
  // next call may reuse the scratch only when this call's work has finished.
  auto enqueue = [&]() -> int {
    k_init<<<init_grid(A), 256, 0, st>>>(A);
    EIC_CUDA_TRY(cudaGetLastError());
    void* args[] = {&A};
    EIC_CUDA_TRY(cudaLaunchCooperativeKernel((const void*)k_eic<false>, dim3(grid), dim3(kDefaultBlock), args, 0, st));
    k_output<<<4 * nd.grid, 256, 0, st>>>(G, A.dist, source, dist);
    EIC_CUDA_TRY(cudaGetLastError());
    return EIC_OK;
  };
  int status = 0;
  rc = enqueue();
  if (rc == EIC_OK && cudaMemcpyAsync(&status, &ctl->status, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess)
    rc = EIC_ECUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess && rc == EIC_OK) rc = EIC_ECUDA;
  (void)cudaGetLastError();
  if (rc) return rc;
  return status;
}

// ------------------------------------------------------------ serving launch

int eic_serve_grid(int block, bool wide, uint32_t* grid) {
  int dev = 0, sms = 0, per_sm = 0, coop = 0;
  EIC_CUDA_TRY(cudaGetDevice(&dev));
  EIC_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  EIC_CUDA_TRY(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
  if (!coop) return EIC_ECUDA;
  EIC_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, wide ? k_eic_serve<true> : k_eic_serve<false>,
                                                             block, 0));
  if (per_sm < 1) return EIC_ECUDA;
  *grid = (uint32_t)(sms * per_sm);
  return EIC_OK;
}

int eic_serve_launch(const ServeArgs& args, uint32_t groups, uint32_t block, cudaStream_t stream) {
  k_serve_prep<<<(groups + 255) / 256, 256, 0, stream>>>(args.slot, groups, args.claim);
  EIC_CUDA_TRY(cudaGetLastError());
  ServeArgs a = args;
  void* kargs[] = {&a};
  EIC_CUDA_TRY(cudaLaunchCooperativeKernel(args.wide ? (const void*)k_eic_serve<true> : (const void*)k_eic_serve<false>,
                                           dim3(groups * args.nb), dim3(block), kargs, 0, stream));
  return EIC_OK;
}

int eic_tune_step_width(const eic_graph* g, uint32_t source, uint32_t copies, uint32_t nb, const eic_params& p,
                        uint32_t from, cudaStream_t stream, uint32_t* best_shift, double* best_ms) {
  if (!g || copies == 0 || source >= g->dg.n) return EIC_EINVAL;
  *best_shift = from;
  *best_ms = 0.0;
  if (g->dg.two_m == 0) return EIC_OK;
  uint32_t* buf = nullptr;
  const uint64_t n = g->dg.n;
  if (cudaMalloc((void**)&buf, n * 4 * copies) != cudaSuccess) {
    (void)cudaGetLastError();
    return EIC_ENOMEM;
  }
  std::vector<const eic_graph*> gs(copies, g);
  std::vector<uint32_t> ss(copies, source);
  std::vector<uint32_t*> ds;
  for (uint32_t k = 0; k < copies; ++k) ds.push_back(buf + n * k);
  eic_batch* b = nullptr;
  int rc = batch_create(gs.data(), ss.data(), copies, ds.data(), &p, nullptr, stream, &b);
  if (rc == EIC_OK) rc = batch_configure(b, copies, p.block_threads ? p.block_threads : kDefaultBlock, nb);
  double t_best = -1.0;
  for (uint32_t shift = from; rc == EIC_OK && shift <= 8; ++shift) {
    for (auto& q : b->hq) q.gap_shift = shift;
    if ((rc = batch_upload(b, stream))) break;
    double t = batch_time(b, stream);
    const double t2 = batch_time(b, stream);
    if (t < 0 || t2 < 0) {
      rc = EIC_ECUDA;
      break;
    }
    t = t2 < t ? t2 : t;
    if (t_best < 0 || t < 0.98 * t_best) {
      t_best = t;
      *best_shift = shift;
    } else {
      break;
    }
  }
  if (b) batch_free(b);
  cudaFree(buf);
  *best_ms = t_best;
  return rc;
}
