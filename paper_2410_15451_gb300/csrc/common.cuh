// Device-side helpers shared by the kernels of the GB300 dynamic Leiden
// library.  Internal header: not part of the C ABI.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

typedef __int128 i128;
typedef unsigned __int128 u128;

#define LD_FULL 0xffffffffu
#define LD_EMPTY_KEY (-1)

// ---------------------------------------------------------------- counters
// One block of device counters per handle, mirrored to pinned host memory at
// the few host synchronisation points of a call.
// Counters of one sub-sweep.  A local-moving iteration uses one set per class,
// so that all are cleared together before it (SUB_RING classes at a time).
struct SubCounters {
  int32_t bin_count[4];           // vertices in each degree bin
  int32_t movers;                 // deferred moves (SYNC)
  int32_t big_movers;             // moved hubs whose neighbours are marked by a kernel of their own
  int32_t pad[2];
};
constexpr int SUB_RING = 16;

struct DevCounters {
  // a local-moving iteration: dq .. sub are cleared together
  unsigned long long dq[2];       // sum of accepted gains g (int128, two's complement)
  int64_t moves;                  // local-moving moves of the iteration
  SubCounters sub[SUB_RING];
  SubCounters ref;                // bins of a refinement round or of aggregation
  int32_t accepted;               // refinement moves applied in this round
  int32_t cand_count[2];          // refinement candidate lists (ping-pong)
  // error .. refine_marks: cleared together at the start of a call
  int32_t error;                  // batch validation error
  int32_t overflow;               // a touched CSR row outgrew its capacity and the spill arena
  int32_t list_count;             // generic list length
  int32_t max_count;              // max degree (level), max community degree
  int32_t large_count;            // batch apply: touched rows merged in chunks
  int32_t mid_count;              // batch apply: touched rows merged by one block each
  int32_t tr_occ;                 // tracking: filled slots of the pair table
  int32_t tr_flagged;             // tracking: old communities without a majority candidate
  int32_t hub_big;                // local moving: listed hubs whose tables are read in pieces
  int32_t max_row;                // batch apply: longest touched row
  int32_t warp_count;             // batch apply: touched rows merged by one warp with a large stage
  int64_t processed;              // local-moving vertex visits
  int64_t arcs;                   // local-moving arcs scanned
  int64_t ref_processed;          // refinement vertex visits
  int64_t ref_arcs;               // refinement arcs scanned
  int64_t lmk_visits[3];          // local moving per timed kernel (warp range, block bin, hub scan):
  int64_t lmk_arcs[3];            //   vertex visits, arcs scanned and algorithmic bytes
  int64_t lmk_bytes[3];
  int64_t sigma_intra;            // modularity: intra-community arc weight
  unsigned long long sq[2];       // modularity: sum of Sigma_c^2 (int128)
  int64_t batch_dw;               // batch: change of 2m
  int64_t slot_change;            // batch: change of huge_slots by the touched rows
  int64_t huge_slots;             // table slots the vertices above the block bin need
  int64_t bcounts[8];             // batch apply: unique deletions, unique insertions, new arcs,
                                  //   touched rows, merge-buffer arcs
  int64_t affected;               // |dV|: vertices flagged affected (counted into the frontier)
  int64_t split_arcs;             // splitting: arcs of the vertices listed for splitting,
  int32_t split_count;            //   these vertices,
  int32_t big_count;              //   and long rows (also of the row kernels) left to a chunked one
  int64_t deg_sum;                // degree sum of the level scanned by level_maxdeg (its arcs)
  int64_t xk_bytes[3];            // algorithmic bytes of the other timed kernels (split sampling,
                                  //   giant-community aggregation scan, block merge of touched rows)
  int64_t agg_tables[2];          // aggregation's per-community global tables: [0] hashed, [1] indexed
                                  //   by the key (the table has a slot per community)
  int64_t refine_marks;           // batch: not 0 when a community is marked for refinement
  // kept between calls
  int64_t m2;                     // 2m (sum of arc weights), device copy
  int64_t arena_used;             // next free arc slot of G^t (relocated rows go here)
};

// ---------------------------------------------------------------- checked build
// Built with -DLEIDEN_CHECKED, the kernels test conditions the algorithm
// guarantees -- an open-addressing probe ends within its table, neighbour and
// community ids lie in [0, n), a union-find chain is shorter than n -- and
// where one fails they record its code in a device word of their source
// file, skip the access and go on.  A broken invariant then ends the call
// with LEIDEN_ERR_STATE instead of a fault, a trap or an endless loop.  The
// default build compiles every test away (ld_ok is then always true).
enum { LD_CHK_PROBE = 1, LD_CHK_COL = 2, LD_CHK_COMM = 3, LD_CHK_CHAIN = 4, LD_CHK_SELFTEST = 0x5e1f };
#ifdef LEIDEN_CHECKED
static __device__ unsigned int ld_check_word;
__device__ __forceinline__ bool ld_ok(bool cond, unsigned int code) {
  if (!cond) atomicCAS(&ld_check_word, 0u, code);
  return cond;
}
// Host: the file's check word (after a stream sync), reset to 0.
#define LD_CHECK_WORD_READER(fn)                                      \
  unsigned int fn() {                                                 \
    unsigned int v = 0, z = 0;                                        \
    if (cudaMemcpyFromSymbol(&v, ld_check_word, sizeof(v)) != cudaSuccess) { cudaGetLastError(); return 0; } \
    cudaMemcpyToSymbol(ld_check_word, &z, sizeof(z));                 \
    return v;                                                         \
  }
#else
__device__ __forceinline__ bool ld_ok(bool, unsigned int) { return true; }
#define LD_CHECK_WORD_READER(fn) \
  unsigned int fn() { return 0; }
#endif

// ---------------------------------------------------------------- hashing
// SplitMix64 output function (Steele, Lea, Flood, OOPSLA 2014).
__host__ __device__ __forceinline__ uint64_t ld_splitmix64(uint64_t x) {
  uint64_t z = x + 0x9E3779B97F4A7C15ULL;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}

// Sub-sweep class of a vertex in the snapshot schedule.
__device__ __forceinline__ int ld_class_of(int64_t v, int classes_mask) {
  return (int)(ld_splitmix64((uint64_t)v) & (uint64_t)classes_mask);
}

// Multiplicative hash of a community id into a power-of-two table.
__device__ __forceinline__ uint32_t ld_hash32(uint32_t k) {
  k *= 0x9E3779B1u;
  return k ^ (k >> 15);
}

// ---------------------------------------------------------------- int128
__device__ __forceinline__ void ld_atomic_add_i128(unsigned long long *p, i128 v) {
  unsigned long long lo = (unsigned long long)(u128)v;
  unsigned long long hi = (unsigned long long)((u128)v >> 64);
  if (lo == 0 && hi == 0) return;
  unsigned long long old = atomicAdd(&p[0], lo);
  unsigned long long carry = (old + lo < old) ? 1ull : 0ull;
  if (hi + carry) atomicAdd(&p[1], hi + carry);
}

__device__ __forceinline__ i128 ld_shfl_xor_i128(i128 v, int mask) {
  long long lo = (long long)(unsigned long long)(u128)v;
  long long hi = (long long)((u128)v >> 64);
  lo = __shfl_xor_sync(LD_FULL, lo, mask);
  hi = __shfl_xor_sync(LD_FULL, hi, mask);
  return (i128)(((u128)(unsigned long long)hi << 64) | (u128)(unsigned long long)lo);
}

// Candidate (value, community) ordered by larger value, then smaller id.
// c < 0 means "no candidate".
__device__ __forceinline__ bool ld_better(i128 v1, int32_t c1, i128 v2, int32_t c2) {
  if (c1 < 0) return false;
  if (c2 < 0) return true;
  return v1 > v2 || (v1 == v2 && c1 < c2);
}

__device__ __forceinline__ int64_t ld_warp_sum_i64(int64_t v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(LD_FULL, v, o);
  return v;
}

// Sum over the lanes that share a key (peers = __match_any_sync of the
// key).  Every lane of the warp must call it (full-mask shuffles); each
// lane receives its group's sum.  (The warp reduction unit, __reduce_add_sync
// with one mask per group, measured about twice as slow here: it serialises
// over the distinct masks of a warp.)
__device__ __forceinline__ int64_t ld_group_sum_i64(uint32_t peers, int64_t v) {
  int64_t s = 0;
#pragma unroll
  for (int k = 0; k < 32; k++) {
    int64_t x = __shfl_sync(LD_FULL, v, k);
    if ((peers >> k) & 1u) s += x;
  }
  return s;
}
// True in the lowest lane of the group.
__device__ __forceinline__ bool ld_group_leader(uint32_t peers) {
  return (__ffs(peers) - 1) == (int)(threadIdx.x & 31);
}

// ---------------------------------------------------------------- sums by community
// Tables of (community, weight sum).  NARROW tables hold 32-bit sums and are
// used when the graph's total weight 2m is below 2^32, which bounds every sum
// of arc weights; WIDE ones hold the low and the high halves apart, so that
// the shared-memory adds are 32-bit in both (the high half is only touched by
// a carry or a weight above 2^32; 64-bit shared atomics cost more than twice
// as much).  The sums are exact in both.

// The gain term m2 * kv - Ki * S as an exact 128-bit integer.  NARROW: all four
// below 2^32, so each product is one 32 x 32 multiplication.
template <bool WIDE>
__device__ __forceinline__ i128 ld_gain(int64_t m2, int64_t kv, int64_t Ki, int64_t S) {
  if (WIDE) return (i128)m2 * kv - (i128)Ki * S;
  uint64_t a = (uint64_t)(uint32_t)m2 * (uint32_t)kv, b = (uint64_t)(uint32_t)Ki * (uint32_t)S;
  return (i128)a - (i128)b;
}

// Lane holding the largest v among the lanes with c >= 0, ties to the
// smallest c; -1 if there is none.  All lanes call it.  The warp's reduction
// unit takes the value word by word (a butterfly of shuffles moves every
// field of a candidate through every step).
template <bool WIDE>
__device__ __forceinline__ int ld_warp_argmax(i128 v, int32_t c) {
  bool has = c >= 0;
  if (!__any_sync(LD_FULL, has)) return -1;
  // (every lane takes part in every reduction; `has` only selects its input)
  if (WIDE) {
    int32_t w3 = (int32_t)(v >> 96), m3 = __reduce_max_sync(LD_FULL, has ? w3 : INT32_MIN);
    has = has && w3 == m3;
    uint32_t w2 = (uint32_t)((u128)v >> 64), m2 = __reduce_max_sync(LD_FULL, has ? w2 : 0u);
    has = has && w2 == m2;
  } else {  // |v| < 2^64: the upper half is the sign
    int32_t w2 = (int32_t)(v >> 64), m2 = __reduce_max_sync(LD_FULL, has ? w2 : INT32_MIN);
    has = has && w2 == m2;
  }
  uint32_t w1 = (uint32_t)((u128)v >> 32), m1 = __reduce_max_sync(LD_FULL, has ? w1 : 0u);
  has = has && w1 == m1;
  uint32_t w0 = (uint32_t)(u128)v, m0 = __reduce_max_sync(LD_FULL, has ? w0 : 0u);
  has = has && w0 == m0;
  int32_t cm = __reduce_min_sync(LD_FULL, has ? c : INT32_MAX);
  return __ffs(__ballot_sync(LD_FULL, has && c == cm)) - 1;
}

// Sum over the lanes of a warp of values whose total is a sum of arc weights.
template <bool WIDE>
__device__ __forceinline__ int64_t ld_warp_weight(int64_t v) {
  if (WIDE) return ld_warp_sum_i64(v);
  return (int64_t)__reduce_add_sync(LD_FULL, (uint32_t)v);
}

// A table in global memory (a vertex's or a community's slice of the handle's
// table scratch): open addressing on the community id, or, when it has a slot
// per community (dense), indexed by it.  Slots filled are listed (count in
// *occ), so the reader visits only those and empties them again.  NARROW: key
// + 1 and sum share one 64-bit word of `vals` (0 = empty), so an insertion
// touches one sector (emission of the giant communities' tables, R-MAT 21
// static: 2525 -> 570 us per launch, its loads four deep; chunked scan 2259 ->
// 1438 us); WIDE: key in `keys` (-1 = empty), sum in `vals`.  Both
// leave keys all -1 and vals all 0.
struct GTable {
  int32_t *keys;
  int64_t *vals;
  int32_t *list;
  int32_t *occ;
  int mask;
  bool dense;
};

// Find or claim the slot of c and add w; the claimed slot if it was empty,
// else -1.  A slot's key only goes from empty to a key while a table is in
// use, so a plain read from L2 decides every probe but the claim of an empty
// slot.
template <bool WIDE>
__device__ __forceinline__ int32_t gt_add(const GTable &T, int32_t c, int64_t w) {
  uint32_t s = T.dense ? (uint32_t)c : ld_hash32((uint32_t)c) & (uint32_t)T.mask;
  for (uint32_t probe = 0; ld_ok(probe <= (uint32_t)T.mask, LD_CHK_PROBE); probe++) {
    if (WIDE) {
      int32_t k = __ldcg(&T.keys[s]);
      bool claimed = false;
      if (k == LD_EMPTY_KEY) {
        k = atomicCAS(&T.keys[s], LD_EMPTY_KEY, c);
        claimed = k == LD_EMPTY_KEY;
      }
      if (claimed || k == c) {
        atomicAdd((unsigned long long *)&T.vals[s], (unsigned long long)w);
        return claimed ? (int32_t)s : -1;
      }
    } else {
      unsigned long long *p = (unsigned long long *)&T.vals[s];
      unsigned long long key = (unsigned long long)((uint32_t)c + 1u) << 32, x = __ldcg(p);
      if (x == 0) {
        x = atomicCAS(p, 0ull, key | (uint32_t)w);
        if (x == 0) return (int32_t)s;
      }
      if ((x >> 32) == (key >> 32)) {
        atomicAdd(p, (unsigned long long)(uint32_t)w);
        return -1;
      }
    }
    s = (s + 1) & (uint32_t)T.mask;
  }
  return -1;
}

// One lane: add and list.
template <bool WIDE>
__device__ __forceinline__ void gt_insert(const GTable &T, int32_t c, int64_t w) {
  int32_t s = gt_add<WIDE>(T, c, w);
  if (s >= 0) T.list[atomicAdd(T.occ, 1)] = s;
}

// All 32 lanes, each with at most one key: the slots claimed by the warp are
// listed with one atomic on the fill count.
template <bool WIDE>
__device__ __forceinline__ void gt_insert_warp(const GTable &T, bool has, int32_t c, int64_t w) {
  int lane = threadIdx.x & 31;
  int32_t s = has ? gt_add<WIDE>(T, c, w) : -1;
  uint32_t m = __ballot_sync(LD_FULL, s >= 0);
  if (!m) return;
  int leader = __ffs(m) - 1;
  int32_t p0 = 0;
  if (lane == leader) p0 = atomicAdd(T.occ, __popc(m));
  p0 = __shfl_sync(LD_FULL, p0, leader);
  if (s >= 0) T.list[p0 + __popc(m & ((1u << lane) - 1u))] = s;
}

// Read slot s; leave it empty.
template <bool WIDE>
__device__ __forceinline__ void gt_read(const GTable &T, int32_t s, int32_t &c, int64_t &w) {
  int64_t x = T.vals[s];
  c = WIDE ? T.keys[s] : (int32_t)((uint64_t)x >> 32) - 1;
  w = WIDE ? x : (int64_t)(uint32_t)x;
}
template <bool WIDE>
__device__ __forceinline__ void gt_empty(const GTable &T, int32_t s) {
  if (WIDE) T.keys[s] = LD_EMPTY_KEY;
  T.vals[s] = 0;
}

// Shared staging table of one block (local moving and refinement of the
// block bin): STAGE_SLOTS open-addressing slots, at most STAGE_FILL keys.
constexpr int STAGE_SLOTS = 2048;
constexpr int STAGE_FILL = 1024;  // distinct keys per use at most (load <= 1/2)

// Warp-private shared table: only the lanes of one warp touch it.  Flushed
// into a global table before it passes half full.
constexpr int WT_SLOTS = 256;
constexpr int WT_LIMIT = WT_SLOTS / 2 - 32;  // flush above this many keys

// `hi` of a NARROW table is one unused word.
template <bool WIDE, int SLOTS, int FILL, typename Slot>
struct STable {
  int32_t keys[SLOTS];
  uint32_t lo[SLOTS];
  uint32_t hi[WIDE ? SLOTS : 1];
  Slot list[FILL];
};
template <bool WIDE>
struct WarpTable : STable<WIDE, WT_SLOTS, WT_SLOTS / 2, uint8_t> {
  int32_t count;
};

template <typename T>
__device__ __forceinline__ void st_clear(T &t, int first, int stride, int slots) {
  for (int s = first; s < slots; s += stride) {
    t.keys[s] = LD_EMPTY_KEY;
    t.lo[s] = 0;
    if (sizeof(t.hi) > 4) t.hi[s] = 0;
  }
}

template <bool WIDE, int SLOTS, int FILL, typename Slot>
__device__ __forceinline__ void st_add(STable<WIDE, SLOTS, FILL, Slot> &t, uint32_t s, int64_t w) {
  uint32_t a = (uint32_t)w;
  if (!WIDE) {
    atomicAdd(&t.lo[s], a);
  } else {
    uint32_t old = atomicAdd(&t.lo[s], a), h = (uint32_t)((uint64_t)w >> 32) + (old + a < old ? 1u : 0u);
    if (h) atomicAdd(&t.hi[s], h);
  }
}

// Add (c, w); a newly filled slot is listed with the fill count *count.
// Lanes of one warp or of one block may call it at once.
template <bool WIDE, int SLOTS, int FILL, typename Slot>
__device__ __forceinline__ void st_insert(STable<WIDE, SLOTS, FILL, Slot> &t, int32_t *count, int32_t c, int64_t w) {
  uint32_t s = ld_hash32((uint32_t)c) & (uint32_t)(SLOTS - 1);
  for (int probe = 0; ld_ok(probe < SLOTS, LD_CHK_PROBE); probe++) {
    int32_t k = t.keys[s];
    if (k == LD_EMPTY_KEY) {
      k = atomicCAS(&t.keys[s], LD_EMPTY_KEY, c);
      if (k == LD_EMPTY_KEY) {
        t.list[atomicAdd(count, 1)] = (Slot)s;
        k = c;
      }
    }
    if (k == c) {
      st_add(t, s, w);
      return;
    }
    s = (s + 1) & (uint32_t)(SLOTS - 1);
  }
}

// Read the listed slot q and leave it empty.
template <bool WIDE, int SLOTS, int FILL, typename Slot>
__device__ __forceinline__ void st_take(STable<WIDE, SLOTS, FILL, Slot> &t, int q, int32_t &c, int64_t &w) {
  uint32_t s = t.list[q];
  c = t.keys[s];
  w = (int64_t)t.lo[s];
  t.keys[s] = LD_EMPTY_KEY;
  t.lo[s] = 0;
  if (WIDE) {
    w |= (int64_t)((uint64_t)t.hi[s] << 32);
    t.hi[s] = 0;
  }
}

template <bool WIDE>
__device__ __forceinline__ void wt_init(WarpTable<WIDE> &T) {
  st_clear(T, threadIdx.x & 31, 32, WT_SLOTS);
  if ((threadIdx.x & 31) == 0) T.count = 0;
  __syncwarp();
}

// All 32 lanes: move the pairs into a global table and empty the warp table.
template <bool WIDE>
__device__ __forceinline__ void wt_flush(WarpTable<WIDE> &T, const GTable &G) {
  int lane = threadIdx.x & 31;
  __syncwarp();
  int n = T.count;
  for (int q0 = 0; q0 < n; q0 += 32) {  // warp-uniform
    bool has = q0 + lane < n;
    int32_t c = 0;
    int64_t w = 0;
    if (has) st_take(T, q0 + lane, c, w);
    gt_insert_warp<WIDE>(G, has, c, w);
  }
  __syncwarp();
  if (lane == 0) T.count = 0;
  __syncwarp();
}

// All 32 lanes, before each adds at most one key: room for them.  The flush is a
// collective, so all lanes must take the same side: each reads the fill count and
// then votes, and no lane adds a key before all have voted (a lane that ran ahead
// on its own reading would send the lanes behind it into a flush that it does not
// join).  The lane that added last reads the whole count.  A read between two warp
// barriers decides the same: R-MAT 20, rollback of 0.1 of its edges, 26.6 ms, with
// the vote 25.7; R-MAT 21 static 53.2 and 52.8.
template <bool WIDE>
__device__ __forceinline__ void wt_make_room(WarpTable<WIDE> &T, const GTable &G) {
  int filled = *(volatile int32_t *)&T.count;
  if (__any_sync(LD_FULL, filled > WT_LIMIT)) wt_flush(T, G);
}

// ---------------------------------------------------------------- block appends
// A block of 256 threads appends its items to up to CATS lists at once, one
// atomic per list and step: one atomic per warp on a list's length costs more
// than the sweep itself (4.19M vertices: 131k of them on one word).  An item
// is a set of categories (bit q: list q); each thread has APPEND_UNROLL items
// per step.  All threads call it; at[u][q] is the item's place in list q.
constexpr int APPEND_UNROLL = 4;
constexpr int APPEND_STEP = 256 * APPEND_UNROLL;
template <int CATS>
struct BlockAppend {
  int32_t off[CATS][APPEND_UNROLL * 8];
};
template <int CATS>
__device__ __forceinline__ void block_append(BlockAppend<CATS> &B, const uint32_t *cats, int32_t *const *lengths,
                                             int32_t (*at)[CATS]) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const uint32_t below = (1u << lane) - 1u;
  __syncthreads();  // the places of the step before are read
#pragma unroll
  for (int u = 0; u < APPEND_UNROLL; u++)
#pragma unroll
    for (int q = 0; q < CATS; q++) {
      uint32_t m = __ballot_sync(LD_FULL, cats[u] >> q & 1);
      at[u][q] = __popc(m & below);
      if (lane == 0) B.off[q][u * 8 + wid] = __popc(m);
    }
  __syncthreads();
  for (int q = wid; q < CATS; q += 8) {  // a warp per list: 32 counts
    int32_t v = B.off[q][lane], incl = v, base = 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int32_t y = __shfl_up_sync(LD_FULL, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31 && incl) base = atomicAdd(lengths[q], incl);
    B.off[q][lane] = __shfl_sync(LD_FULL, base, 31) + incl - v;
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < APPEND_UNROLL; u++)
#pragma unroll
    for (int q = 0; q < CATS; q++) at[u][q] += B.off[q][u * 8 + wid];
}

// Per-graph sums of a batched handle: every lane of the warp calls these;
// lanes with `has` add v into arr[g].  When the whole warp is on one graph
// (the common case: lists follow vertex order) one lane adds the warp's sum.
__device__ __forceinline__ void ld_graph_add_i64(int64_t *arr, bool has, int32_t g, int64_t v) {
  int32_t g0 = __shfl_sync(LD_FULL, has ? g : -1, __ffs(__ballot_sync(LD_FULL, has) | 0x80000000u) - 1);
  if (__all_sync(LD_FULL, !has || g == g0)) {
    int64_t s = has ? v : 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(LD_FULL, s, o);
    if ((threadIdx.x & 31) == 0 && g0 >= 0 && s) atomicAdd((unsigned long long *)&arr[g0], (unsigned long long)s);
  } else if (has && v) {
    atomicAdd((unsigned long long *)&arr[g], (unsigned long long)v);
  }
}
__device__ __forceinline__ void ld_graph_add_i32(int32_t *arr, bool has, int32_t g, int32_t v) {
  int32_t g0 = __shfl_sync(LD_FULL, has ? g : -1, __ffs(__ballot_sync(LD_FULL, has) | 0x80000000u) - 1);
  if (__all_sync(LD_FULL, !has || g == g0)) {
    int32_t s = has ? v : 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(LD_FULL, s, o);
    if ((threadIdx.x & 31) == 0 && g0 >= 0 && s) atomicAdd(&arr[g0], s);
  } else if (has && v) {
    atomicAdd(&arr[g], v);
  }
}
__device__ __forceinline__ void ld_graph_add_i128(unsigned long long *arr, bool has, int32_t g, i128 v) {
  int32_t g0 = __shfl_sync(LD_FULL, has ? g : -1, __ffs(__ballot_sync(LD_FULL, has) | 0x80000000u) - 1);
  if (__all_sync(LD_FULL, !has || g == g0)) {
    i128 s = has ? v : 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += ld_shfl_xor_i128(s, o);
    if ((threadIdx.x & 31) == 0 && g0 >= 0 && s != 0) ld_atomic_add_i128(&arr[2 * g0], s);
  } else if (has && v != 0) {
    ld_atomic_add_i128(&arr[2 * g], v);
  }
}

// ---------------------------------------------------------------- bitmaps
__device__ __forceinline__ bool ld_bit_test(const uint32_t *bm, int64_t i) {
  return (bm[i >> 5] >> (i & 31)) & 1u;
}
// Sets bit i; returns true if it was clear.
__device__ __forceinline__ bool ld_bit_set(uint32_t *bm, int64_t i) {
  uint32_t m = 1u << (i & 31);
  return (atomicOr(&bm[i >> 5], m) & m) == 0;
}

// ---------------------------------------------------------------- rows by windows
// A warp takes the arcs of up to 32 rows as one flat range: lane i holds row
// i's first flat position s (non-decreasing over the lanes) and arc(x) =
// ab + x of that row, so that consecutive lanes read consecutive arcs
// whatever the rows' lengths.  A warp per row leaves 31 lanes idle on a short
// row and one warp alone on a hub; longer rows than ROWS_BIG are therefore
// cut into chunks by the callers.
constexpr int ROWS_BIG = 2048;

// The row (lane) that holds flat position x: the last one with s <= x.  All
// lanes call it; positions of one call rise with the lane, so when the first
// and last fall into one row (a long row) the search is two ballots (and the
// result true).
template <int U>
__device__ __forceinline__ bool ld_window_rows(int s, int x0, int lane, int *k) {
  int first = 31 - __clz(__ballot_sync(LD_FULL, s <= x0));
  int last = 31 - __clz(__ballot_sync(LD_FULL, s <= x0 + 32 * U - 1));
#pragma unroll
  for (int u = 0; u < U; u++) k[u] = first;
  if (first == last) return true;  // warp-uniform
#pragma unroll
  for (int u = 0; u < U; u++) {
    int x = x0 + 32 * u + lane, r = 0;
#pragma unroll
    for (int step = 16; step > 0; step >>= 1) {
      int sc = __shfl_sync(LD_FULL, s, r + step);
      if (sc <= x) r += step;
    }
    k[u] = r;
  }
  return false;
}

// Inclusive sum over the lanes.
__device__ __forceinline__ int64_t ld_warp_incl_i64(int64_t v) {
  int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int64_t y = __shfl_up_sync(LD_FULL, v, o);
    if (lane >= o) v += y;
  }
  return v;
}
__device__ __forceinline__ int ld_warp_incl_i32(int v) {
  int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int y = __shfl_up_sync(LD_FULL, v, o);
    if (lane >= o) v += y;
  }
  return v;
}

// The part of each lane's row [s, e) in 32 flat positions xb .. xb + 31 that
// hold one value per lane (v): the values summed over the overlap.
__device__ __forceinline__ int64_t ld_window_part(int s, int e, int xb, int64_t v) {
  int64_t p = ld_warp_incl_i64(v);
  int lo = s > xb ? s - xb : 0, hi = e < xb + 32 ? e - xb : 32;  // [lo, hi) of the step
  int64_t a = __shfl_sync(LD_FULL, p, (lo - 1) & 31), b = __shfl_sync(LD_FULL, p, (hi - 1) & 31);
  return lo < hi ? b - (lo > 0 ? a : 0) : 0;
}

// Item k of a chunk plan (ch_off[k] <= t < ch_off[k+1], ch_off[0] = 0): a 32-way
// search by the whole warp (t the same in all lanes), three dependent loads for
// 32k items where a binary search takes fifteen.
__device__ __forceinline__ int64_t ld_chunk_item(const int64_t *ch_off, int64_t count, int64_t t) {
  const int lane = threadIdx.x & 31;
  int64_t lo = 0, span = count;
  while (span > 1) {  // warp-uniform; ch_off[lo] <= t throughout
    int64_t step = (span + 31) >> 5, p = lo + lane * step;
    bool le = p < lo + span && ch_off[p] <= t;
    uint32_t m = __ballot_sync(LD_FULL, le);
    int k = m ? 31 - __clz(m) : 0;
    lo += k * step;
    span = span - k * step < step ? span - k * step : step;
  }
  return lo;
}

// ---------------------------------------------------------------- programmatic launches
// A kernel launched by launch_after (internal.h) may start while the kernel
// before it on the stream still runs; it calls this before it touches memory:
// the wait ends when that kernel has completed and its writes are visible.  It
// first lets the kernel after itself start (and wait) in turn.
__device__ __forceinline__ void ld_after_previous() {
  cudaTriggerProgrammaticLaunchCompletion();
  cudaGridDependencySynchronize();
}

// Grid-stride helpers.
__device__ __forceinline__ int64_t ld_gtid() { return (int64_t)blockIdx.x * blockDim.x + threadIdx.x; }
__device__ __forceinline__ int64_t ld_gstride() { return (int64_t)gridDim.x * blockDim.x; }
