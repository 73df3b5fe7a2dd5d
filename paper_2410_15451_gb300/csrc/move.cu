// Local-moving phase (Alg. "leidenlm") and refinement phase (Alg.
// "leidenre") of Leiden on one level of the dendrogram.
//
// Each vertex scans its neighbours' communities into an open-addressing
// table (K_{i->c}), takes the community with the largest delta-modularity
// (Eq. 2 times 2m^2, exact in int128; ties to the lowest community id) and
// moves when the gain is positive.  Vertices are binned by degree: a warp
// with a shared-memory table (<= 128 arcs), a block with a shared table
// (<= 1024 arcs); larger ones are cut into chunks for all blocks, with a table in
// global scratch per vertex that a warp, or a block per piece of it, reads to
// decide.
//
// Deterministic mode (snapshot schedule): moves found in a sub-sweep are
// applied by a separate kernel after all decisions, so every decision reads
// the state at the start of the sub-sweep.  Asynchronous mode applies each
// move as soon as it is found.
#include <algorithm>
#include <atomic>
#include <cstddef>

#include "internal.h"

namespace {

constexpr int WARPS_PER_BLOCK = 8;
constexpr int BLOCK_THREADS = 128;
constexpr int HUGE_THREADS = 256;  // a hub's decision reads only its distinct communities

enum Kind { KIND_MOVE = 0, KIND_REFINE = 1 };

struct Args {
  // level graph
  int64_t n;
  const int64_t *off;
  const int32_t *deg;
  const int32_t *col;
  const void *w;
  // state
  int32_t *C;
  int64_t *S;
  const int64_t *K;
  int32_t *size;
  const int32_t *CB;     // refinement bounds
  int32_t *prop;         // refinement proposals / async states
  uint8_t *dS;           // split flags (local moving, dynamic)
  uint32_t *unproc;      // bitmap
  const uint8_t *in_range;
  int32_t *movers, *mtarget;
  int32_t *big_movers;   // moved hubs whose neighbours the apply kernel marks
  const int32_t *list;   // bin list
  const int32_t *count;  // bin count (device)
  const int32_t *list_tiny;   // bin 3 list (degree <= 8), used with bin 0
  const int32_t *count_tiny;
  int64_t m2;                 // 2m of the level graph (one graph)
  // batched handles (null otherwise): graph of each vertex, 2m per graph,
  // the gain of each deferred move, per-graph refinement counters
  const int32_t *gid;
  const int64_t *m2g;
  const uint8_t *lm_on;
  int64_t *mgain;
  int32_t *accg;
  uint8_t *refg;
  DevCounters *cnt;
  SubCounters *sub;      // of this sub-sweep
  int dynamic;
  int async_mode;
  int classes_mask;
  // global scratch for the huge bin
  int32_t *gkeys;
  int64_t *gvals;
  int32_t *glist;  // filled slots of each table
  int32_t *gocc;   // number of filled slots of each listed vertex
};

// 2m of the graph vertex i belongs to.
__device__ __forceinline__ int64_t m2_of(const Args &A, int64_t i) { return A.gid ? A.m2g[A.gid[i]] : A.m2; }

__device__ __forceinline__ void mark_neighbours(const Args &A, int64_t i, int64_t base, int64_t dg, int t0,
                                                int stride) {
  for (int64_t a = t0; a < dg; a += stride) {
    int32_t j = A.col[base + a];
    if (j == i) continue;
    if (A.in_range && !A.in_range[j]) continue;
    ld_bit_set(A.unproc, j);
  }
}

__device__ __forceinline__ void add_counters(DevCounters *cnt, int kind, int64_t visits, int64_t arcs, int64_t moves,
                                             i128 dq) {
  if (kind == KIND_MOVE) {
    if (visits) atomicAdd((unsigned long long *)&cnt->processed, (unsigned long long)visits);
    if (arcs) atomicAdd((unsigned long long *)&cnt->arcs, (unsigned long long)arcs);
    if (moves) atomicAdd((unsigned long long *)&cnt->moves, (unsigned long long)moves);
    if (dq != 0) ld_atomic_add_i128(cnt->dq, dq);
  } else {
    if (visits) atomicAdd((unsigned long long *)&cnt->ref_processed, (unsigned long long)visits);
    if (arcs) atomicAdd((unsigned long long *)&cnt->ref_arcs, (unsigned long long)arcs);
  }
}

// Work counters of the timed local-moving kernels (algorithmic bytes as
// stated in the C header).
__device__ __forceinline__ void add_lmk(DevCounters *cnt, int k, int64_t visits, int64_t arcs, int64_t bytes) {
  if (visits) atomicAdd((unsigned long long *)&cnt->lmk_visits[k], (unsigned long long)visits);
  if (arcs) atomicAdd((unsigned long long *)&cnt->lmk_arcs[k], (unsigned long long)arcs);
  if (bytes) atomicAdd((unsigned long long *)&cnt->lmk_bytes[k], (unsigned long long)bytes);
}

// ---------------------------------------------------------------- bins 3 and 0: warp range
// The best candidate community of a vertex with what its decision needs:
// K_{i->c}, Sigma_c, and K_{i->d} of the vertex's own community.
struct BestX {
  i128 v;
  int32_t c;
  int32_t szc;  // size of c (local moving; read for the winner only)
  int64_t kc;
  int64_t kd;
  int64_t sc;   // Sigma of c
};

__device__ __forceinline__ void bestx_merge(BestX &a, const BestX &b) {
  if (ld_better(b.v, b.c, a.v, a.c)) { a.v = b.v; a.c = b.c; a.kc = b.kc; a.sc = b.sc; }
  a.kd += b.kd;
}

// The warp's best candidate and summed K_{i->d}, in every lane.
template <bool WIDE>
__device__ __forceinline__ BestX warp_bestx(BestX b) {
  b.kd = ld_warp_weight<WIDE>(b.kd);
  int win = ld_warp_argmax<WIDE>(b.v, b.c);
  int src = win < 0 ? 0 : win;
  uint64_t lo = __shfl_sync(LD_FULL, (unsigned long long)(u128)b.v, src);
  int64_t hi = __shfl_sync(LD_FULL, (long long)(b.v >> 64), src);
  b.v = (i128)(((u128)(uint64_t)hi << 64) | lo);
  b.c = __shfl_sync(LD_FULL, b.c, src);
  b.kc = __shfl_sync(LD_FULL, b.kc, src);
  b.sc = __shfl_sync(LD_FULL, b.sc, src);
  if (win < 0) b.c = -1;
  return b;
}

// The block's best and summed K_{i->d}, in every thread (sb: one per warp).
template <bool WIDE>
__device__ __forceinline__ BestX block_bestx(BestX b, BestX *sb) {
  b = warp_bestx<WIDE>(b);
  if ((threadIdx.x & 31) == 0) sb[threadIdx.x >> 5] = b;
  __syncthreads();
  BestX r = sb[0];
  for (int q = 1; q < (int)(blockDim.x >> 5); q++) bestx_merge(r, sb[q]);
  __syncthreads();
  return r;
}

// The best over aligned groups of eight lanes, by a butterfly over (value,
// community, lane); the other fields are read from the winner once.
__device__ __forceinline__ BestX group_bestx(BestX b) {
  i128 v = b.v;
  int32_t c = b.c;
  int at = threadIdx.x & 31;
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) {
    i128 tv = ld_shfl_xor_i128(v, o);
    int32_t tc = __shfl_xor_sync(LD_FULL, c, o);
    int ta = __shfl_xor_sync(LD_FULL, at, o);
    if (ld_better(tv, tc, v, c)) { v = tv; c = tc; at = ta; }
    b.kd += __shfl_xor_sync(LD_FULL, b.kd, o);
  }
  b.v = v;
  b.c = c;
  b.kc = __shfl_sync(LD_FULL, b.kc, at);
  b.sc = __shfl_sync(LD_FULL, b.sc, at);
  return b;
}

// The decision of vertex i in community d (K_i, Sigma_d, size_d given) for
// the reduced candidate b.  Returns the gain (Eq. 2 times 2m^2) when i moves
// (local moving) or proposes (refinement), else 0; the caller records a
// deferred move.  Refinement runs in proposal/accept rounds in both modes: an
// in-place CAS scheme (pin the target, then leave) never merges mutual best
// pairs, because both pin each other before either can leave, and such
// pairs are common since the gain of joining a singleton is symmetric.
template <int KIND>
__device__ __forceinline__ i128 decide_x(const Args &A, int64_t i, int32_t d, int64_t Ki, int64_t Sd, int32_t szd,
                                         int64_t m2, BestX b) {
  if (b.c < 0) return 0;
  if (KIND == KIND_MOVE && A.async_mode) {
    // in-place moves: read the totals again, as late as possible
    Sd = A.S[d];
    b.sc = A.S[b.c];
    szd = A.size[d];
    b.szc = A.size[b.c];
  }
  i128 g = (i128)m2 * (b.kc - b.kd) - (i128)Ki * ((i128)Ki + b.sc - Sd);
  if (g <= 0) return 0;
  if (KIND == KIND_MOVE) {
    if (szd == 1 && b.szc == 1 && b.c > d) return 0;
    if (A.async_mode) {
      A.C[i] = b.c;
      atomicAdd((unsigned long long *)&A.S[d], (unsigned long long)(-Ki));
      atomicAdd((unsigned long long *)&A.S[b.c], (unsigned long long)Ki);
      atomicSub(&A.size[d], 1);
      atomicAdd(&A.size[b.c], 1);
    }
    if (A.dynamic) A.dS[d] = 1;
    return g;
  } else {
    if (A.C[b.c] != b.c) return 0;  // the representative of c* left it
    A.prop[i] = b.c;
    return g;
  }
}

// The outcome of decide_x<KIND_MOVE> in the snapshot schedule, without its
// writes: a pure function of the sub-sweep's starting state, so every
// thread of a group can evaluate it.
__device__ __forceinline__ bool would_move(int32_t d, int64_t Ki, int64_t Sd, int32_t szd, int64_t m2,
                                           const BestX &b) {
  if (b.c < 0) return false;
  i128 g = (i128)m2 * (b.kc - b.kd) - (i128)Ki * ((i128)Ki + b.sc - Sd);
  if (g <= 0) return false;
  return !(szd == 1 && b.szc == 1 && b.c > d);
}

// Deferred moves of the lanes with `mv` set (snapshot schedule): one
// counter update per warp.
__device__ __forceinline__ void record_movers(const Args &A, bool mv, int32_t i, int32_t c, i128 g) {
  uint32_t m = __ballot_sync(LD_FULL, mv);
  if (!m) return;
  int lane = threadIdx.x & 31;
  int32_t p0 = 0;
  if (lane == __ffs(m) - 1) p0 = atomicAdd(&A.sub->movers, __popc(m));
  p0 = __shfl_sync(LD_FULL, p0, __ffs(m) - 1);
  if (mv) {
    int32_t slot = p0 + __popc(m & ((1u << lane) - 1u));
    A.movers[slot] = i;
    A.mtarget[slot] = c;
    if (A.mgain) { A.mgain[2 * slot] = (int64_t)(u128)g; A.mgain[2 * slot + 1] = (int64_t)((u128)g >> 64); }
  }
}

// One thread's deferred move.
__device__ __forceinline__ void record_mover(const Args &A, int32_t i, int32_t c, i128 g) {
  int32_t slot = atomicAdd(&A.sub->movers, 1);
  A.movers[slot] = i;
  A.mtarget[slot] = c;
  if (A.mgain) { A.mgain[2 * slot] = (int64_t)(u128)g; A.mgain[2 * slot + 1] = (int64_t)((u128)g >> 64); }
}

struct Tally {
  int64_t visits = 0, arcs = 0, moves = 0;
  i128 dq = 0;
};

// Per-block sums of the lanes' tallies, then one set of counter updates; with
// kt >= 0 also the work counters of that timed kernel (local moving;
// algorithmic bytes: per visit the list entry, off, deg, C[i], K[i],
// Sigma[C[i]], size[C[i]], 40 B; per arc col, C[j] and the weight).
template <int KIND>
__device__ __forceinline__ void flush_tally(const Args &A, Tally t, int kt = -1, int wbytes = 0) {
  __shared__ unsigned long long sacc[6];
  if (threadIdx.x < 6) sacc[threadIdx.x] = 0;
  __syncthreads();
  int64_t v = ld_warp_sum_i64(t.visits), a = ld_warp_sum_i64(t.arcs), m = ld_warp_sum_i64(t.moves);
  i128 q = t.dq;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) q += ld_shfl_xor_i128(q, o);
  if ((threadIdx.x & 31) == 0 && v) {
    atomicAdd(&sacc[0], (unsigned long long)v);
    atomicAdd(&sacc[1], (unsigned long long)a);
    atomicAdd(&sacc[2], (unsigned long long)m);
    ld_atomic_add_i128(&sacc[3], q);
  }
  __syncthreads();
  if (threadIdx.x == 0 && sacc[0]) {
    i128 dq = (i128)(((u128)sacc[4] << 64) | (u128)sacc[3]);
    add_counters(A.cnt, KIND, (int64_t)sacc[0], (int64_t)sacc[1], (int64_t)sacc[2], dq);
    if (KIND == KIND_MOVE && kt >= 0)
      add_lmk(A.cnt, kt, (int64_t)sacc[0], (int64_t)sacc[1], 40 * (int64_t)sacc[0] + (8 + wbytes) * (int64_t)sacc[1]);
  }
}

constexpr int TINY_LANES = 8;  // lanes per vertex of degree <= BIN_TINY_MAX (one arc each)

// Four vertices of degree <= 8 per warp, one arc per lane: lanes whose
// neighbours share a community find each other with __match_any_sync, so
// no table is built; each group's leader lanes hold K_{i->c} and Sigma_c.
template <typename W, int KIND, bool WIDE>
__device__ __forceinline__ void tiny_step(const Args &A, int64_t item, int64_t ntiny, int lane, Tally &tl) {
  const W *w = (const W *)A.w;
  int grp = lane >> 3, sub = lane & 7, gl = lane & ~7;
  int64_t k = item * 4 + grp;
  bool has = k < ntiny;
  int32_t i = has ? A.list_tiny[k] : 0;
  int64_t base = 0, Ki = 0, Sd = 0, wj = 0, m2 = A.m2;
  int32_t dg = 0, d = 0, szd = 0, bi = 0, j = -1;
  if (has) {
    base = A.off[i];
    dg = A.deg[i];
    d = A.C[i];
    Ki = A.K[i];
    if (A.gid) m2 = A.m2g[A.gid[i]];
    if (KIND == KIND_REFINE) bi = A.CB[i];
  }
  bool arc = has && sub < dg;
  if (arc) { j = A.col[base + sub]; wj = (int64_t)w[base + sub]; }
  arc = arc && ld_ok((uint64_t)j < (uint64_t)A.n, LD_CHK_COL);
  if (has) {
    Sd = A.S[d];
    if (KIND == KIND_MOVE) szd = A.size[d];
  }
  bool valid = arc && j != i && (KIND != KIND_REFINE || A.CB[j] == bi);
  int32_t c = valid ? A.C[j] : 0;
  valid = valid && ld_ok((uint64_t)c < (uint64_t)A.n, LD_CHK_COMM);
  unsigned long long key = valid ? (((unsigned long long)grp << 32) | (uint32_t)c)
                                 : (0xffffffff00000000ull | (unsigned)lane);
  uint32_t peers = __match_any_sync(LD_FULL, key);
  int64_t kv = 0;  // peers lie within the lane's group of eight
#pragma unroll
  for (int q = 0; q < TINY_LANES; q++) {
    int64_t x = __shfl_sync(LD_FULL, wj, gl + q);
    if ((peers >> (gl + q)) & 1u) kv += x;
  }
  BestX b{0, -1, 0, 0, 0, 0};
  if (valid && ld_group_leader(peers)) {
    if (c == d) {
      b.kd = kv;
    } else {
      b.sc = A.S[c];
      b.v = ld_gain<WIDE>(m2, kv, Ki, b.sc);
      b.c = c;
      b.kc = kv;
    }
  }
  b = group_bestx(b);
  i128 g = 0;
  if (has && sub == 0) {
    // the winner's size matters only to the singleton rule (size_d == 1)
    if (KIND == KIND_MOVE && !A.async_mode && b.c > d && szd == 1) b.szc = A.size[b.c];
    g = decide_x<KIND>(A, i, d, Ki, Sd, szd, m2, b);
  }
  bool mv = g > 0;
  if (KIND == KIND_MOVE && !A.async_mode) record_movers(A, mv, i, b.c, g);
  int moved = __shfl_sync(LD_FULL, mv ? 1 : 0, gl);
  if (KIND == KIND_MOVE && moved && arc && j != i && (!A.in_range || A.in_range[j])) ld_bit_set(A.unproc, j);
  if (has && sub == 0) { tl.visits++; tl.arcs += dg; tl.moves += mv; tl.dq += g; }
}

// One vertex of degree 9..128 per warp with a warp-private shared table that
// records its filled slots and is emptied by the reads (so it is cleared
// once per launch, not per vertex).  Every lane keeps its up to four arcs in
// flight: their col, weight and C[j] loads are independent, and so are the
// Sigma loads of the up to four candidates each lane reads back.
//
// Arcs into the vertex's own community and into one more community seen in
// the first step (`hot`) are summed in registers: the neighbours of a vertex
// fall mostly into a few communities, and every lane of the warp would add to
// the same table slot, one after the other.  With the 32-bit sums and the
// reduction by words, alone on the GPU: warp range 86 -> 72 us per launch
// (R-MAT 20, all vertices), block bin 79 -> 58 us (30 -> 9 us on the web-like
// graph).  Loading a segment's vertex records ahead of the rows was slower in
// both (registers: 72 -> 75 and 58 -> 70 us).
constexpr int WARP_UNROLL = BIN_WARP_MAX / 32;

// A community other than d among the lanes' first arcs, or -1.
__device__ __forceinline__ int32_t hot_community(bool valid, int32_t c, int32_t d) {
  uint32_t m = __ballot_sync(LD_FULL, valid && c != d);
  int32_t h = __shfl_sync(LD_FULL, c, m ? __ffs(m) - 1 : 0);
  return m ? h : -1;
}

template <typename W, int KIND, bool WIDE>
__device__ __forceinline__ void warp_step(const Args &A, int32_t i, int lane, WarpTable<WIDE> &T, Tally &tl) {
  const W *w = (const W *)A.w;
  int64_t base = A.off[i];
  int32_t dg = A.deg[i];
  int32_t d = A.C[i];
  int64_t Ki = A.K[i];
  int64_t Sd = A.S[d];
  int32_t szd = KIND == KIND_MOVE ? A.size[d] : 0;
  int32_t bi = KIND == KIND_REFINE ? A.CB[i] : 0;
  int64_t m2 = m2_of(A, i);
  int32_t j[WARP_UNROLL], c[WARP_UNROLL];
  int64_t wa[WARP_UNROLL];
  bool v[WARP_UNROLL];
#pragma unroll
  for (int u = 0; u < WARP_UNROLL; u++) {
    int a = lane + 32 * u;
    v[u] = a < dg;
    j[u] = v[u] ? A.col[base + a] : i;
    wa[u] = v[u] ? (int64_t)w[base + a] : 0;
  }
#pragma unroll
  for (int u = 0; u < WARP_UNROLL; u++) {
    v[u] = v[u] && j[u] != i && ld_ok((uint64_t)j[u] < (uint64_t)A.n, LD_CHK_COL);
    if (KIND == KIND_REFINE) v[u] = v[u] && A.CB[j[u]] == bi;
  }
#pragma unroll
  for (int u = 0; u < WARP_UNROLL; u++) {
    c[u] = v[u] ? A.C[j[u]] : 0;
    v[u] = v[u] && ld_ok((uint64_t)c[u] < (uint64_t)A.n, LD_CHK_COMM);
  }
  BestX b{0, -1, 0, 0, 0, 0};
  int32_t hot = hot_community(v[0], c[0], d);
  int64_t sh = hot >= 0 ? A.S[hot] : 0, kh = 0;
#pragma unroll
  for (int u = 0; u < WARP_UNROLL; u++) {
    if (!v[u]) continue;
    if (c[u] == d) b.kd += wa[u];
    else if (c[u] == hot) kh += wa[u];
    else st_insert(T, &T.count, c[u], wa[u]);
  }
  __syncwarp();
  int n = T.count;
  int32_t cc[WARP_UNROLL];
  int64_t kv[WARP_UNROLL], sc[WARP_UNROLL];
#pragma unroll
  for (int u = 0; u < WARP_UNROLL; u++) {
    int q = lane + 32 * u;
    cc[u] = -1;
    kv[u] = 0;
    if (q < n) st_take(T, q, cc[u], kv[u]);
  }
  __syncwarp();
  if (lane == 0) T.count = 0;
  __syncwarp();
#pragma unroll
  for (int u = 0; u < WARP_UNROLL; u++) sc[u] = cc[u] >= 0 ? A.S[cc[u]] : 0;
  kh = ld_warp_weight<WIDE>(kh);
  if (lane == 31 && hot >= 0) {  // the last lane has the fewest candidates of its own
    b.v = ld_gain<WIDE>(m2, kh, Ki, sh);
    b.c = hot;
    b.kc = kh;
    b.sc = sh;
  }
#pragma unroll
  for (int u = 0; u < WARP_UNROLL; u++) {
    if (cc[u] < 0) continue;
    i128 val = ld_gain<WIDE>(m2, kv[u], Ki, sc[u]);
    if (ld_better(val, cc[u], b.v, b.c)) { b.v = val; b.c = cc[u]; b.kc = kv[u]; b.sc = sc[u]; }
  }
  b = warp_bestx<WIDE>(b);
  i128 g = 0;
  if (lane == 0) {
    // the winner's size matters only to the singleton rule (size_d == 1)
    if (KIND == KIND_MOVE && !A.async_mode && b.c > d && szd == 1) b.szc = A.size[b.c];
    g = decide_x<KIND>(A, i, d, Ki, Sd, szd, m2, b);
  }
  bool mv = g > 0;
  if (KIND == KIND_MOVE && !A.async_mode) record_movers(A, mv, i, b.c, g);
  int moved = __shfl_sync(LD_FULL, mv ? 1 : 0, 0);
  if (KIND == KIND_MOVE && moved) {
#pragma unroll
    for (int u = 0; u < WARP_UNROLL; u++)
      if (j[u] != i && (!A.in_range || A.in_range[j[u]])) ld_bit_set(A.unproc, j[u]);
  }
  if (lane == 0) { tl.visits++; tl.arcs += dg; tl.moves += mv; tl.dq += g; }
}

// Bins 3 (degree <= 8, groups of 8 lanes) and 0 (degree <= 128, a warp
// each) in one launch: items [0, ceil(n3/4)) are groups of four tiny
// vertices, the rest one warp-bin vertex each.
template <typename W, int KIND, bool WIDE>
__global__ void __launch_bounds__(WARPS_PER_BLOCK * 32, 4) k_decide_warp(Args A) {
  ld_after_previous();
  __shared__ WarpTable<WIDE> WT[WARPS_PER_BLOCK];
  int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int64_t ntiny = *A.count_tiny, nwarp = *A.count;
  int64_t ngroups = (ntiny + 3) / 4, total = ngroups + nwarp;
  if ((int64_t)blockIdx.x * WARPS_PER_BLOCK >= total) return;
  int64_t gw = (int64_t)blockIdx.x * WARPS_PER_BLOCK + wid, nw = (int64_t)gridDim.x * WARPS_PER_BLOCK;
  wt_init(WT[wid]);
  Tally tl;
  for (int64_t t = gw; t < total; t += nw) {
    if (t < ngroups) tiny_step<W, KIND, WIDE>(A, t, ntiny, lane, tl);
    else warp_step<W, KIND, WIDE>(A, A.list[t - ngroups], lane, WT[wid], tl);
  }
  flush_tally<KIND>(A, tl, KT_WARP, (int)sizeof(W));
}

// ---------------------------------------------------------------- bin 1: block, shared stage
// One vertex of degree 129..1024 per block of BLOCK_THREADS.  Each thread
// keeps BLOCK_UNROLL arcs in flight (their col, weight and C[j] loads are
// independent), adds them into a shared open-addressing stage with shared
// atomics, and the block then reads the candidates from the stage's
// filled-slot list (the distinct neighbour communities only), emptying
// each slot as it reads it.
//
// Two barriers per vertex: B1 after the inserts, B2 after the per-warp
// candidates are posted.  The filled-slot count alternates between two
// words by vertex parity: the count of vertex k is read between B1(k) and
// B2(k) and reset by thread 0 after B2(k); it is next used by vertex k+2,
// whose inserts begin after B2(k+1).  The slots read (and emptied) for
// vertex k are all emptied before B2(k), so the inserts of vertex k+1 find
// the stage empty.
//
// As in the warp bin, arcs into the vertex's own community and into one more
// per warp are summed in registers (the second is added to the stage once).
constexpr int BLOCK_UNROLL = 4;
template <bool WIDE>
struct BlockStage : STable<WIDE, STAGE_SLOTS, STAGE_FILL, uint16_t> {
  int32_t count[2];
};

template <typename W, int KIND, bool WIDE>
__global__ void __launch_bounds__(BLOCK_THREADS) k_decide_block(Args A) {
  ld_after_previous();
  __shared__ BlockStage<WIDE> S;
  __shared__ BestX sb[BLOCK_THREADS / 32];
  __shared__ int moved_s;
  const int64_t count = *A.count;
  if (blockIdx.x >= count) return;
  st_clear(S, threadIdx.x, BLOCK_THREADS, STAGE_SLOTS);
  if (threadIdx.x < 2) S.count[threadIdx.x] = 0;
  __syncthreads();
  const W *w = (const W *)A.w;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  int64_t visits = 0, arcs = 0, moves = 0;
  i128 dq = 0;
  int par = 0;
  for (int64_t t = blockIdx.x; t < count; t += gridDim.x, par ^= 1) {
    int32_t i = A.list[t];
    int64_t base = A.off[i];
    int32_t dg = A.deg[i];
    int32_t d = A.C[i];
    int64_t Ki = A.K[i];
    int64_t Sd = A.S[d];
    int32_t szd = KIND == KIND_MOVE ? A.size[d] : 0;
    int32_t bi = KIND == KIND_REFINE ? A.CB[i] : 0;
    int64_t m2 = m2_of(A, i);
    int32_t *cnt = &S.count[par];
    BestX b{0, -1, 0, 0, 0, 0};
    int32_t hot = -1;
    int64_t kh = 0;
    for (int r0 = 0; r0 < dg; r0 += BLOCK_THREADS * BLOCK_UNROLL) {
      int32_t j[BLOCK_UNROLL], c[BLOCK_UNROLL];
      int64_t wa[BLOCK_UNROLL];
      bool v[BLOCK_UNROLL];
#pragma unroll
      for (int u = 0; u < BLOCK_UNROLL; u++) {
        int a = r0 + u * BLOCK_THREADS + tid;
        v[u] = a < dg;
        j[u] = v[u] ? A.col[base + a] : i;
        wa[u] = v[u] ? (int64_t)w[base + a] : 0;
      }
#pragma unroll
      for (int u = 0; u < BLOCK_UNROLL; u++) {
        v[u] = v[u] && j[u] != i && ld_ok((uint64_t)j[u] < (uint64_t)A.n, LD_CHK_COL);
        if (KIND == KIND_REFINE) v[u] = v[u] && A.CB[j[u]] == bi;
      }
#pragma unroll
      for (int u = 0; u < BLOCK_UNROLL; u++) {
        c[u] = v[u] ? A.C[j[u]] : 0;
        v[u] = v[u] && ld_ok((uint64_t)c[u] < (uint64_t)A.n, LD_CHK_COMM);
      }
      if (r0 == 0) hot = hot_community(v[0], c[0], d);
#pragma unroll
      for (int u = 0; u < BLOCK_UNROLL; u++) {
        if (!v[u]) continue;
        if (c[u] == d) b.kd += wa[u];
        else if (c[u] == hot) kh += wa[u];
        else st_insert(S, cnt, c[u], wa[u]);
      }
    }
    kh = ld_warp_weight<WIDE>(kh);
    if (lane == 0 && kh) st_insert(S, cnt, hot, kh);
    __syncthreads();  // B1: the stage holds K_{i->c} for every neighbour community c but d
    int n = *cnt;
    for (int q0 = 0; q0 < n; q0 += BLOCK_THREADS * BLOCK_UNROLL) {
      int32_t cc[BLOCK_UNROLL];
      int64_t kv[BLOCK_UNROLL], sc[BLOCK_UNROLL];
#pragma unroll
      for (int u = 0; u < BLOCK_UNROLL; u++) {
        int q = q0 + u * BLOCK_THREADS + tid;
        cc[u] = -1;
        kv[u] = 0;
        if (q < n) st_take(S, q, cc[u], kv[u]);
      }
#pragma unroll
      for (int u = 0; u < BLOCK_UNROLL; u++) sc[u] = cc[u] >= 0 ? A.S[cc[u]] : 0;
#pragma unroll
      for (int u = 0; u < BLOCK_UNROLL; u++) {
        if (cc[u] < 0) continue;
        i128 val = ld_gain<WIDE>(m2, kv[u], Ki, sc[u]);
        if (ld_better(val, cc[u], b.v, b.c)) { b.v = val; b.c = cc[u]; b.kc = kv[u]; b.sc = sc[u]; }
      }
    }
    b = warp_bestx<WIDE>(b);
    if (lane == 0) sb[wid] = b;
    __syncthreads();  // B2: every warp's best is posted, every read slot emptied
    if (tid == 0) S.count[par] = 0;
    BestX r = sb[0];
#pragma unroll
    for (int k = 1; k < BLOCK_THREADS / 32; k++) bestx_merge(r, sb[k]);
    // the winner's size matters only to the singleton rule (size_d == 1)
    if (KIND == KIND_MOVE && !A.async_mode && r.c > d && szd == 1) r.szc = A.size[r.c];
    bool mv;
    if (A.async_mode) {
      // in-place moves change the totals under the decision: one thread
      // decides and applies, the block learns the outcome
      if (tid == 0) {
        i128 g = decide_x<KIND>(A, i, d, Ki, Sd, szd, m2, r);
        moved_s = g > 0;
        visits++; arcs += dg; moves += g > 0; dq += g;
      }
      __syncthreads();
      mv = moved_s;
    } else {
      // snapshot schedule: the decision reads only the state at the start
      // of the sub-sweep, so every thread reaches the same one; thread 0
      // writes it
      i128 g = 0;
      if (tid == 0) {
        g = decide_x<KIND>(A, i, d, Ki, Sd, szd, m2, r);
        if (KIND == KIND_MOVE && g > 0) record_mover(A, i, r.c, g);
        visits++; arcs += dg; moves += g > 0; dq += g;
      }
      mv = KIND == KIND_MOVE && would_move(d, Ki, Sd, szd, m2, r);
    }
    if (KIND == KIND_MOVE && mv) mark_neighbours(A, i, base, dg, tid, BLOCK_THREADS);
  }
  if (tid == 0) add_counters(A.cnt, KIND, visits, arcs, moves, dq);
  if (KIND == KIND_MOVE && tid == 0)
    add_lmk(A.cnt, KT_BLOCK, visits, arcs, 40 * visits + (8 + (int64_t)sizeof(W)) * arcs);
}

// ---------------------------------------------------------------- bin 2, split across blocks
// Vertices above BIN_BLOCK_MAX arcs: each gets its own table of
// pow2 >= 2*degree slots in global scratch and its arcs are cut into chunks
// of HUGE_CHUNK that any block may take, so one hub no longer runs on one SM.
constexpr int HUGE_CHUNK = TABLE_CHUNK;
constexpr int HUGE_UNROLL = 4;

// Global tables start clean and are cleaned again by the kernel that reads
// them; each records the slots it fills in a list (occ[k] entries at
// tab_off[k] in A.glist), so the decision visits only the distinct
// communities instead of the whole table.
__device__ __forceinline__ GTable hub_table(const Args &A, const int64_t *tab_off, int64_t k) {
  int64_t o = tab_off[k];
  return GTable{A.gkeys + o, A.gvals + o, A.glist + o, &A.gocc[k], (int)(tab_off[k + 1] - o - 1), false};
}

template <typename W, int KIND, bool WIDE>
__global__ void __launch_bounds__(256) k_huge_scan(Args A, const int64_t *tab_off, const int64_t *ch_off) {
  ld_after_previous();
  // Each warp sums its arcs per community in a private shared table first
  // (the neighbours of a hub fall into few communities), then each distinct
  // community updates the vertex's global table once per flush.  The hub's
  // own community and one more are summed in registers, as in the other bins.
  __shared__ WarpTable<WIDE> WT[8];
  WarpTable<WIDE> &T8 = WT[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  int64_t count = *A.count;
  int64_t nch = ch_off[count];
  if (blockIdx.x >= nch) return;
  wt_init(T8);
  for (int64_t t = blockIdx.x; t < nch; t += gridDim.x) {
    int64_t lo = ld_chunk_item(ch_off, count, t);
    int64_t i = A.list[lo];
    int64_t first = (t - ch_off[lo]) * HUGE_CHUNK;
    int64_t full = A.deg[i];
    int64_t last = first + HUGE_CHUNK < full ? first + HUGE_CHUNK : full;
    GTable G = hub_table(A, tab_off, lo);
    const W *w = (const W *)A.w;
    int64_t base = A.off[i] + first;
    int len = (int)(last - first);
    int32_t bi = KIND == KIND_REFINE ? A.CB[i] : 0, d = A.C[i], hot = -1;
    int64_t kd = 0, kh = 0;
    // HUGE_UNROLL arcs per lane in flight: their col, weight and C[j] loads
    // are independent; the inserts follow one by one
    for (int a0 = threadIdx.x & ~31; a0 < len; a0 += (int)blockDim.x * HUGE_UNROLL) {  // warp-uniform
      int32_t j[HUGE_UNROLL], c[HUGE_UNROLL];
      int64_t wa[HUGE_UNROLL];
      bool valid[HUGE_UNROLL];
#pragma unroll
      for (int u = 0; u < HUGE_UNROLL; u++) {
        int a = a0 + u * (int)blockDim.x + lane;
        valid[u] = a < len;
        j[u] = valid[u] ? A.col[base + a] : (int32_t)i;
        wa[u] = valid[u] ? (int64_t)w[base + a] : 0;
      }
#pragma unroll
      for (int u = 0; u < HUGE_UNROLL; u++) {
        valid[u] = valid[u] && j[u] != i && ld_ok((uint64_t)j[u] < (uint64_t)A.n, LD_CHK_COL);
        if (KIND == KIND_REFINE) valid[u] = valid[u] && A.CB[j[u]] == bi;
      }
#pragma unroll
      for (int u = 0; u < HUGE_UNROLL; u++) {
        c[u] = valid[u] ? A.C[j[u]] : 0;
        valid[u] = valid[u] && ld_ok((uint64_t)c[u] < (uint64_t)A.n, LD_CHK_COMM);
      }
      if (hot < 0) hot = hot_community(valid[0], c[0], d);
#pragma unroll
      for (int u = 0; u < HUGE_UNROLL; u++) {
        wt_make_room(T8, G);
        if (!valid[u]) continue;
        if (c[u] == d) kd += wa[u];
        else if (c[u] == hot) kh += wa[u];
        else st_insert(T8, &T8.count, c[u], wa[u]);
      }
    }
    wt_flush(T8, G);
    kd = ld_warp_weight<WIDE>(kd);
    kh = ld_warp_weight<WIDE>(kh);
    gt_insert_warp<WIDE>(G, lane == 0 ? kd != 0 : lane == 1 && kh != 0, lane == 0 ? d : hot, lane == 0 ? kd : kh);
    if (KIND == KIND_MOVE && threadIdx.x == 0)
      add_lmk(A.cnt, KT_HUGE_SCAN, first == 0 ? 1 : 0, len, (8 + (int64_t)sizeof(W)) * len);
  }
}

// Decisions of the hubs, from their tables: a warp per hub of at most BIG_KEYS
// slots (a hub's decision is a chain of dependent loads; a block per hub has
// an eighth as many of them in flight and waits at its barriers), a block per
// piece of BIG_PIECE slots of the others, because at the first aggregated
// level a hub has a slot per neighbour.  Each piece of several leaves its best
// candidate behind the hub's slot list (which has at least twice as many
// words as slots), and the block that finishes a hub's last piece decides.
// R-MAT 21, static: 120 -> 89 us per launch (a block per hub, the moved hubs'
// neighbours marked by their block).
constexpr int PIECE_WORDS = 12;  // a BestX without szc, padded

__device__ __forceinline__ void piece_put(volatile int32_t *p, const BestX &b) {
  int32_t x[11] = {(int32_t)(uint32_t)(u128)b.v,
                   (int32_t)(uint32_t)((u128)b.v >> 32),
                   (int32_t)(uint32_t)((u128)b.v >> 64),
                   (int32_t)(uint32_t)((u128)b.v >> 96),
                   b.c,
                   (int32_t)b.kc, (int32_t)(b.kc >> 32), (int32_t)b.kd, (int32_t)(b.kd >> 32),
                   (int32_t)b.sc, (int32_t)(b.sc >> 32)};
#pragma unroll
  for (int q = 0; q < 11; q++) p[q] = x[q];
}
__device__ __forceinline__ int64_t join64(int32_t lo, int32_t hi) {
  return (int64_t)(((uint64_t)(uint32_t)hi << 32) | (uint32_t)lo);
}
__device__ __forceinline__ BestX piece_get(const int32_t *p) {
  int32_t x[11];
#pragma unroll
  for (int q = 0; q < 11; q++) x[q] = __ldcg(p + q);
  BestX b{0, x[4], 0, join64(x[5], x[6]), join64(x[7], x[8]), join64(x[9], x[10])};
  b.v = (i128)(((u128)(uint64_t)join64(x[2], x[3]) << 64) | (uint64_t)join64(x[0], x[1]));
  return b;
}

// One thread's best of the listed slots q0, q0 + step, ... below q1 of a hub's
// table, emptied as they are read.
template <bool WIDE>
__device__ __forceinline__ BestX hub_best(const Args &A, const GTable &G, int q0, int step, int q1, int32_t d,
                                          int64_t m2, int64_t Ki) {
  BestX b{0, -1, 0, 0, 0, 0};
  for (; q0 < q1; q0 += step * HUGE_UNROLL) {
    int32_t sl[HUGE_UNROLL], cc[HUGE_UNROLL];  // (loads before the stores that empty the slots)
    int64_t kv[HUGE_UNROLL], sc[HUGE_UNROLL];
#pragma unroll
    for (int u = 0; u < HUGE_UNROLL; u++) {
      int q = q0 + u * step;
      sl[u] = q < q1 ? G.list[q] : -1;
    }
#pragma unroll
    for (int u = 0; u < HUGE_UNROLL; u++) {
      cc[u] = -1;
      kv[u] = 0;
      if (sl[u] >= 0) gt_read<WIDE>(G, sl[u], cc[u], kv[u]);
    }
#pragma unroll
    for (int u = 0; u < HUGE_UNROLL; u++)
      if (sl[u] >= 0) gt_empty<WIDE>(G, sl[u]);
#pragma unroll
    for (int u = 0; u < HUGE_UNROLL; u++) sc[u] = cc[u] >= 0 && cc[u] != d ? A.S[cc[u]] : 0;
#pragma unroll
    for (int u = 0; u < HUGE_UNROLL; u++) {
      if (cc[u] < 0) continue;
      if (cc[u] == d) { b.kd += kv[u]; continue; }
      i128 v = ld_gain<WIDE>(m2, kv[u], Ki, sc[u]);
      if (ld_better(v, cc[u], b.v, b.c)) { b.v = v; b.c = cc[u]; b.kc = kv[u]; b.sc = sc[u]; }
    }
  }
  return b;
}

struct Hub {
  int32_t i, occ, d, dg, szd;
  int64_t m2, Ki, Sd, base;
  GTable G;
};
template <int KIND>
__device__ __forceinline__ Hub hub_load(const Args &A, const int64_t *tab_off, int64_t k) {
  Hub H;
  H.i = A.list[k];
  H.G = hub_table(A, tab_off, k);
  H.occ = *H.G.occ;
  H.d = A.C[H.i];
  H.Ki = A.K[H.i];
  H.m2 = m2_of(A, H.i);
  H.dg = A.deg[H.i];
  H.base = A.off[H.i];
  H.Sd = A.S[H.d];
  H.szd = KIND == KIND_MOVE ? A.size[H.d] : 0;
  return H;
}

// The decision of hub H, by one thread: whether it moved.  The neighbours of a
// moved hub are marked by its caller, or, above MARK_INLINE arcs in the
// snapshot schedule, by a kernel of their own.
constexpr int MARK_INLINE = 2048;
template <int KIND>
__device__ __forceinline__ bool hub_decide(const Args &A, const Hub &H, BestX b, Tally &tl) {
  // the winner's size matters only to the singleton rule (size_d == 1)
  if (KIND == KIND_MOVE && !A.async_mode && b.c > H.d && H.szd == 1) b.szc = A.size[b.c];
  i128 g = decide_x<KIND>(A, H.i, H.d, H.Ki, H.Sd, H.szd, H.m2, b);
  bool mv = g > 0;
  if (KIND == KIND_MOVE && !A.async_mode && mv) {
    record_mover(A, H.i, b.c, g);
    if (H.dg > MARK_INLINE) A.big_movers[atomicAdd(&A.sub->big_movers, 1)] = H.i;
  }
  tl.visits++; tl.arcs += H.dg; tl.moves += mv; tl.dq += g;
  return mv && (A.async_mode || H.dg <= MARK_INLINE);
}

template <int KIND, bool WIDE>
__global__ void __launch_bounds__(HUGE_THREADS, 4) k_huge_decide(Args A, const int64_t *tab_off, BigTables big) {
  ld_after_previous();
  __shared__ BestX sb[HUGE_THREADS / 32];
  __shared__ int flag_s;
  const int lane = threadIdx.x & 31;
  const int64_t count = *A.count, nbig = *big.count, npc = nbig ? big.pieces[nbig] : 0;
  Tally tl;
  for (int64_t t = blockIdx.x; t < npc; t += gridDim.x) {  // block-uniform
    int64_t at = ld_chunk_item(big.pieces, nbig, t), k = big.items[at], p = t - big.pieces[at];
    Hub H = hub_load<KIND>(A, tab_off, k);
    const int pieces = (H.occ + BIG_PIECE - 1) / BIG_PIECE;
    int q0 = (int)p * BIG_PIECE, q1 = q0 + BIG_PIECE < H.occ ? q0 + BIG_PIECE : H.occ;
    BestX b = block_bestx<WIDE>(
        hub_best<WIDE>(A, H.G, q0 + (int)threadIdx.x, HUGE_THREADS, q1, H.d, H.m2, H.Ki), sb);
    if (pieces > 1) {  // block-uniform
      int32_t *part = H.G.list + H.occ;
      if (threadIdx.x == 0) {
        piece_put(part + p * PIECE_WORDS, b);
        __threadfence();
        flag_s = atomicAdd(&big.ticket[k], 1) == pieces - 1;
        __threadfence();
      }
      __syncthreads();
      if (!flag_s) continue;
      b = BestX{0, -1, 0, 0, 0, 0};
      for (int q = threadIdx.x; q < pieces; q += HUGE_THREADS) bestx_merge(b, piece_get(part + q * PIECE_WORDS));
      b = block_bestx<WIDE>(b, sb);
    }
    if (threadIdx.x == 0) flag_s = hub_decide<KIND>(A, H, b, tl);
    __syncthreads();
    if (KIND == KIND_MOVE && flag_s) mark_neighbours(A, H.i, H.base, H.dg, threadIdx.x, HUGE_THREADS);
    __syncthreads();
  }
  for (int64_t k = ld_gtid() >> 5; k < count; k += ld_gstride() >> 5) {  // warp-uniform
    if (A.gocc[k] > BIG_KEYS) continue;  // read in pieces
    Hub H = hub_load<KIND>(A, tab_off, k);
    BestX b = warp_bestx<WIDE>(hub_best<WIDE>(A, H.G, lane, 32, H.occ, H.d, H.m2, H.Ki));
    int mark = 0;
    if (lane == 0) mark = hub_decide<KIND>(A, H, b, tl);
    mark = __shfl_sync(LD_FULL, mark, 0);
    if (KIND == KIND_MOVE && mark) mark_neighbours(A, H.i, H.base, H.dg, lane, 32);
  }
  flush_tally<KIND>(A, tl);
}

// ---------------------------------------------------------------- collection
// The bin of a degree.
__device__ __forceinline__ int bin_of(int dg, const leiden_tuning &tn) {
  return dg <= tn.tiny_max ? BIN_TINY : dg <= tn.warp_max ? BIN_WARP : dg <= tn.block_max ? BIN_BLOCK : BIN_HUGE;
}

struct CollectArgs {
  int cls;
  int32_t *bins;
  SubCounters *sub;
  const int64_t *loff;
  leiden_tuning tn;
};

// The bin of frontier vertex v in this sub-sweep: a bin, NBINS (taken, but not
// listed: out of range, or without arcs, whose taking is its visit), or -1 (of
// another class, or of a batched graph whose iterations ended; the class of
// such a vertex is taken on its id within its graph).
__device__ __forceinline__ int collect_bin(const Args &A, const CollectArgs &Q, int64_t v) {
  int64_t vl = A.gid ? v - Q.loff[A.gid[v]] : v;
  if (ld_class_of(vl, A.classes_mask) != Q.cls || (A.gid && !A.lm_on[A.gid[v]])) return -1;
  if (A.in_range && !A.in_range[v]) return NBINS;
  int dg = A.deg[v];
  return dg == 0 ? NBINS : bin_of(dg, Q.tn);
}

// Take the unprocessed vertices of class `cls` (clearing their bits) and
// append the in-range ones to the degree bins.  Dense frontiers (all vertices,
// or more than an eighth of them, see lm_iteration): a block takes 32 bitmap
// words at a time, a lane per bit, so that the degrees are loaded side by
// side, and appends with one atomic per bin.  Sparse ones: a warp takes 32
// words, a lane per word, and a scan over the lanes' counts places every
// vertex with one atomic per bin and warp.  Us per launch, sparse and dense
// form: R-MAT 22 DF, 64,154 edges (1 bit in 40) 11.6 and 22.4; R-MAT 20 ND 12.5
// and 10.4; a rolled back batch of 0.1 of its edges 12.3 and 5.7 (a lane
// walking a full word waits for 32 degrees one after the other).
__device__ __forceinline__ void collect_sparse(const Args &A, const CollectArgs &Q) {
  int lane = threadIdx.x & 31;
  int64_t n = A.n, nwords = (n + 31) >> 5;
  int64_t warp = ld_gtid() >> 5, nwarps = ld_gstride() >> 5;
  for (int64_t w0 = warp * 32; w0 < nwords; w0 += nwarps * 32) {  // warp-uniform
    int64_t wi = w0 + lane;
    uint32_t word = wi < nwords ? A.unproc[wi] : 0u, taken = 0u;
    uint32_t bm[NBINS];
#pragma unroll
    for (int b = 0; b < NBINS; b++) bm[b] = 0u;
    for (uint32_t rest = word; rest; rest &= rest - 1u) {
      int bit = __ffs(rest) - 1;
      int bin = collect_bin(A, Q, (wi << 5) + bit);
      if (bin >= 0) taken |= 1u << bit;
#pragma unroll
      for (int b = 0; b < NBINS; b++)
        if (bin == b) bm[b] |= 1u << bit;
    }
#pragma unroll
    for (int b = 0; b < NBINS; b++) {
      int k = __popc(bm[b]), incl = ld_warp_incl_i32(k);
      int total = __shfl_sync(LD_FULL, incl, 31);
      if (total == 0) continue;  // warp-uniform
      int32_t pos0 = 0;
      if (lane == 31) pos0 = atomicAdd(&Q.sub->bin_count[b], total);
      pos0 = __shfl_sync(LD_FULL, pos0, 31) + incl - k;
      int32_t *dst = Q.bins + (int64_t)b * n + pos0;
      for (uint32_t m = bm[b]; m; m &= m - 1u) *dst++ = (int32_t)((wi << 5) + __ffs(m) - 1);
    }
    if (taken) A.unproc[wi] = word & ~taken;
  }
}
__device__ __forceinline__ void collect_dense(const Args &A, const CollectArgs &Q) {
  __shared__ BlockAppend<NBINS> B;
  int32_t *const lengths[NBINS] = {&Q.sub->bin_count[0], &Q.sub->bin_count[1], &Q.sub->bin_count[2],
                                   &Q.sub->bin_count[3]};
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t n = A.n, nwords = (n + 31) >> 5;
  for (int64_t w0 = (int64_t)blockIdx.x * 32; w0 < nwords; w0 += (int64_t)gridDim.x * 32) {  // block-uniform
    uint32_t word[APPEND_UNROLL], cats[APPEND_UNROLL];
#pragma unroll
    for (int u = 0; u < APPEND_UNROLL; u++) {
      int64_t wi = w0 + 8 * u + wid;
      word[u] = wi < nwords ? A.unproc[wi] : 0u;
    }
    bool some = false;
#pragma unroll
    for (int u = 0; u < APPEND_UNROLL; u++) {
      int64_t wi = w0 + 8 * u + wid;
      int bin = word[u] >> lane & 1u ? collect_bin(A, Q, (wi << 5) + lane) : -1;
      uint32_t taken = __ballot_sync(LD_FULL, bin >= 0);
      if (lane == 0 && taken) A.unproc[wi] = word[u] & ~taken;
      cats[u] = bin >= 0 && bin < NBINS ? 1u << bin : 0u;
      some = some || cats[u];
    }
    if (!__syncthreads_or(some)) continue;
    int32_t at[APPEND_UNROLL][NBINS];
    block_append<NBINS>(B, cats, lengths, at);
#pragma unroll
    for (int u = 0; u < APPEND_UNROLL; u++)
#pragma unroll
      for (int b = 0; b < NBINS; b++)
        if (cats[u] >> b & 1) Q.bins[(int64_t)b * n + at[u][b]] = (int32_t)(((w0 + 8 * u + wid) << 5) + lane);
  }
}

// Deferred moves of a sub-sweep (deterministic mode).  Batched handles also
// sum the gains and moves per graph (gid non-null).
__device__ __forceinline__ void apply_moves(const Args &A, unsigned long long *dqg, int64_t *movesg) {
  const int32_t *gid = A.gid;
  int64_t m = A.sub->movers;
  for (int64_t t0 = (ld_gtid() & ~31ll); t0 < m; t0 += ld_gstride()) {  // warp-uniform trip count
    int64_t t = t0 + (threadIdx.x & 31);
    bool has = t < m;
    int32_t i = 0, gi = 0;
    i128 gain = 0;
    if (has) {
      i = A.movers[t];
      int32_t c = A.mtarget[t];
      int32_t d = A.C[i];
      int64_t k = A.K[i];
      A.C[i] = c;
      atomicAdd((unsigned long long *)&A.S[d], (unsigned long long)(-k));
      atomicAdd((unsigned long long *)&A.S[c], (unsigned long long)k);
      atomicSub(&A.size[d], 1);
      atomicAdd(&A.size[c], 1);
      if (gid) {
        gi = gid[i];
        gain = (i128)(((u128)(uint64_t)A.mgain[2 * t + 1] << 64) | (u128)(uint64_t)A.mgain[2 * t]);
      }
    }
    if (gid) {
      ld_graph_add_i128(dqg, has, gi, gain);
      ld_graph_add_i64(movesg, has, gi, 1);
    }
  }
}

// Between two sub-sweeps: the moves of one are applied and the vertices of the
// next are collected (they touch different arrays).  `apply`: there was one
// before; Q.cls < 0: there is none after.
template <bool DENSE>
__global__ void __launch_bounds__(256)
    k_apply_collect(Args A, bool apply, unsigned long long *dqg, int64_t *movesg, CollectArgs Q) {
  ld_after_previous();
  if (apply) apply_moves(A, dqg, movesg);
  if (Q.cls < 0) return;
  if (DENSE) collect_dense(A, Q);
  else collect_sparse(A, Q);
}

// The neighbours of the moved hubs above MARK_INLINE arcs, each hub cut into
// MARK_PARTS for as many warps (before the next vertices are collected).
constexpr int MARK_PARTS = 32;
__global__ void k_mark_hubs(Args A) {
  ld_after_previous();
  int64_t parts = (int64_t)A.sub->big_movers * MARK_PARTS;
  for (int64_t t = ld_gtid() >> 5; t < parts; t += ld_gstride() >> 5) {  // warp-uniform
    int32_t i = A.big_movers[t / MARK_PARTS];
    int64_t dg = A.deg[i], len = (dg + MARK_PARTS - 1) / MARK_PARTS, a = (t % MARK_PARTS) * len;
    if (a < dg) mark_neighbours(A, i, A.off[i] + a, dg - a < len ? dg - a : len, threadIdx.x & 31, 32);
  }
}

// Community sizes; lanes with the same community add once (giant
// communities would otherwise serialise on one counter).
__global__ void k_sizes(const int32_t *C, int64_t n, int32_t *size) {
  ld_after_previous();
  int lane = threadIdx.x & 31;
  for (int64_t base = (ld_gtid() & ~31ll); base < n; base += ld_gstride()) {
    int64_t i = base + lane;
    int32_t c = i < n ? C[i] : -1 - lane;
    uint32_t peers = __match_any_sync(LD_FULL, c);
    if (i < n && ld_group_leader(peers)) atomicAdd(&size[c], __popc(peers));
  }
}

// ---- refinement
// The bounds C'_B = C', and the vertices of refined bounds reset to singletons
// and listed.
__global__ void __launch_bounds__(256) k_refine_reset(int64_t n, int32_t *CB, const uint8_t *dR, int32_t *C, int64_t *S,
                                                      const int64_t *K, int32_t *prop, int32_t *cand, DevCounters *cnt,
                                                      const int32_t *gid, uint8_t *refg) {
  ld_after_previous();
  __shared__ BlockAppend<1> B;
  int32_t *const lengths[1] = {&cnt->cand_count[0]};
  for (int64_t b0 = (int64_t)blockIdx.x * APPEND_STEP; b0 < n; b0 += (int64_t)gridDim.x * APPEND_STEP) {
    uint32_t cats[APPEND_UNROLL];
    int32_t at[APPEND_UNROLL][1];
#pragma unroll
    for (int u = 0; u < APPEND_UNROLL; u++) {
      int64_t i = b0 + 256 * u + threadIdx.x;
      cats[u] = 0;
      if (i >= n) continue;
      int32_t c = C[i];
      bool r = dR[c];
      CB[i] = c;
      prop[i] = r ? 0 : -1;
      if (r) { C[i] = (int32_t)i; S[i] = K[i]; }
      if (r && gid) refg[gid[i]] = 1;  // the graph has a vertex in a refined bound
      cats[u] = r;
    }
    block_append<1>(B, cats, lengths, at);
#pragma unroll
    for (int u = 0; u < APPEND_UNROLL; u++)
      if (cats[u]) cand[at[u][0]] = (int32_t)(b0 + 256 * u + threadIdx.x);
  }
}

// Keep the candidates that are still alone in their community and bin them
// by degree; reset their proposals.
__global__ void __launch_bounds__(256) k_refine_collect(const int32_t *cand_in, const int32_t *count_in,
                                                        int32_t *cand_out, int32_t *count_out, int64_t n,
                                                        const int32_t *C, const int64_t *S, const int64_t *K,
                                                        const int32_t *deg, int32_t *prop, int32_t *bins,
                                                        SubCounters *sub, leiden_tuning tn) {
  ld_after_previous();
  __shared__ BlockAppend<NBINS + 1> B;
  int32_t *const lengths[NBINS + 1] = {&sub->bin_count[0], &sub->bin_count[1], &sub->bin_count[2], &sub->bin_count[3],
                                       count_out};
  int64_t m = *count_in;
  for (int64_t b0 = (int64_t)blockIdx.x * APPEND_STEP; b0 < m; b0 += (int64_t)gridDim.x * APPEND_STEP) {
    uint32_t cats[APPEND_UNROLL];
    int32_t at[APPEND_UNROLL][NBINS + 1], v[APPEND_UNROLL];
#pragma unroll
    for (int u = 0; u < APPEND_UNROLL; u++) {
      int64_t t = b0 + 256 * u + threadIdx.x;
      cats[u] = 0;
      v[u] = t < m ? cand_in[t] : -1;
    }
#pragma unroll
    for (int u = 0; u < APPEND_UNROLL; u++) {
      int32_t i = v[u];
      if (i < 0) continue;
      prop[i] = -1;
      if (S[C[i]] != K[i]) continue;
      int dg = deg[i];  // without arcs: no proposal (prop stays -1)
      cats[u] = (1u << NBINS) | (dg ? 1u << bin_of(dg, tn) : 0u);
    }
    block_append<NBINS + 1>(B, cats, lengths, at);
#pragma unroll
    for (int u = 0; u < APPEND_UNROLL; u++) {
      if (!cats[u]) continue;
      cand_out[at[u][NBINS]] = v[u];
#pragma unroll
      for (int b = 0; b < NBINS; b++)
        if (cats[u] >> b & 1) bins[(int64_t)b * n + at[u][b]] = v[u];
    }
  }
}

// Snapshot rounds: i -> c* applies iff i does not hold and c* holds, where
// v holds when it proposed nothing, or when v and prop[v] chose each other
// and v has the smaller id.
__device__ __forceinline__ bool holds(const int32_t *prop, int32_t v) {
  int32_t t = prop[v];
  return t < 0 || (prop[t] == v && v < t);
}
__global__ void k_refine_accept(const int32_t *cand, const int32_t *count, const int32_t *prop, int32_t *C, int64_t *S,
                                const int64_t *K, DevCounters *cnt, const int32_t *gid, int32_t *accg) {
  ld_after_previous();
  int64_t m = *count;
  int32_t acc = 0;
  for (int64_t t0 = (ld_gtid() & ~31ll); t0 < m; t0 += ld_gstride()) {  // warp-uniform trip count
    int64_t t = t0 + (threadIdx.x & 31);
    bool took = false;
    int32_t i = 0;
    if (t < m) {
      i = cand[t];
      int32_t c = prop[i];
      if (c >= 0 && !holds(prop, i) && holds(prop, c)) {
        int32_t d = C[i];
        C[i] = c;
        atomicAdd((unsigned long long *)&S[d], (unsigned long long)(-K[i]));
        atomicAdd((unsigned long long *)&S[c], (unsigned long long)K[i]);
        acc++;
        took = true;
      }
    }
    if (gid) ld_graph_add_i32(accg, took, took ? gid[i] : 0, 1);
  }
  if (acc) atomicAdd(&cnt->accepted, acc);
}

__global__ void k_check_selftest() {
  if (threadIdx.x == 0) ld_ok(false, LD_CHK_SELFTEST);
}

Args make_args(leiden_handle *h, const LevelGraph &g) {
  Args A{};
  A.n = g.n;
  A.off = g.off;
  A.deg = g.deg;
  A.col = g.col;
  A.w = g.w;
  A.C = h->Cp;
  A.S = h->Sp;
  A.K = h->Kc;
  A.size = h->csize;
  A.CB = h->CB;
  A.prop = h->prop;
  A.dS = h->dS;
  A.unproc = h->unproc;
  A.movers = h->movers;
  A.mtarget = h->mtarget;
  A.big_movers = h->ibuf2;
  A.cnt = h->dcnt;
  A.sub = &h->dcnt->ref;
  A.m2 = h->m2;
  if (g.gid) {
    A.gid = g.gid;
    A.m2g = h->gc.m2;
    A.mgain = h->mgain;
    A.lm_on = h->gc.lm_on;
    A.accg = h->gc.accepted;
    A.refg = h->gc.refined;
  }
  A.async_mode = h->p.deterministic ? 0 : 1;
  A.classes_mask = lm_classes(h) - 1;
  return A;
}

// The block-bin kernels ask for the largest shared-memory carveout, so that
// seven stages fit on an SM (set once per device of the process).
template <typename W, int KIND>
void block_carveout_of() {
  int co = cudaSharedmemCarveoutMaxShared;
  cudaFuncSetAttribute(k_decide_block<W, KIND, false>, cudaFuncAttributePreferredSharedMemoryCarveout, co);
  cudaFuncSetAttribute(k_decide_block<W, KIND, true>, cudaFuncAttributePreferredSharedMemoryCarveout, co);
}
void block_kernel_carveout() {
  static std::atomic<uint64_t> done{0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev >= 64) { cudaGetLastError(); return; }
  if (done.load(std::memory_order_relaxed) & (1ull << dev)) return;
  block_carveout_of<int32_t, KIND_MOVE>();
  block_carveout_of<int64_t, KIND_MOVE>();
  block_carveout_of<int32_t, KIND_REFINE>();
  block_carveout_of<int64_t, KIND_REFINE>();
  cudaGetLastError();
  done.fetch_or(1ull << dev, std::memory_order_relaxed);
}

// The bins of one sub-sweep (or refinement round) read the same state and
// write disjoint outputs (deferred moves through one atomic counter,
// frontier bits through atomics), so the block bin and the hub path run on
// the handle's side streams beside the warp bin, joined before the caller
// launches anything else: each of these kernels is bound by the latency of
// its gathers and leaves most of the GPU idle in its tail.
template <typename W, int KIND, bool WIDE>
void launch_bins_of(leiden_handle *h, const LevelGraph &g, Args A) {
  cudaStream_t s = h->stream;
  int sms = h->sm_count;
  bool need_block = g.maxdeg > h->tune.warp_max, need_hub = g.maxdeg > h->tune.block_max;
  // tables for every listed hub at once: at most huge_slots slots (taken
  // before the fork: growing them synchronises and frees)
  if (need_hub && !ensure_hslots(h, g.huge_slots)) {
    h->fatal = LEIDEN_ERR_OOM;
    h->err = "global table scratch";
    return;
  }
  // (the in-place mode keeps the bins in order: there a bin's moves are
  // seen by the bins launched after it)
  bool fork = h->tune.overlap && h->p.deterministic && (need_block || need_hub) && side_streams(h);
  cudaStream_t sblock = s, shub = s;
  if (fork) {
    cudaEventRecord(h->fork_ev, s);
    if (need_block) { sblock = h->side[0]; cudaStreamWaitEvent(sblock, h->fork_ev, 0); }
    if (need_hub) { shub = h->side[1]; cudaStreamWaitEvent(shub, h->fork_ev, 0); }
  }
  auto bin = [&](int b) {
    A.list = h->bins + (int64_t)b * g.n;
    A.count = &A.sub->bin_count[b];
  };
  {
    A.list_tiny = h->bins + (int64_t)BIN_TINY * g.n;
    A.count_tiny = &A.sub->bin_count[BIN_TINY];
    bin(BIN_WARP);
    // default 4: one wave at four resident blocks per SM (a level of few vertices needs less)
    int grid = grid_for(g.n, WARPS_PER_BLOCK, sms * h->tune.warp_blocks_per_sm);
    if (KIND == KIND_MOVE) kt_begin(h, KT_WARP);
    ld_note_launch(), launch_after(k_decide_warp<W, KIND, WIDE>, grid, WARPS_PER_BLOCK * 32, s, A);
    if (KIND == KIND_MOVE) kt_end(h);
  }
  if (need_block) {
    // default 7 blocks per SM, with the carveout set to favour shared memory
    block_kernel_carveout();
    bin(BIN_BLOCK);
    int grid = sms * h->tune.block_blocks_per_sm;
    if (KIND == KIND_MOVE) kt_begin(h, KT_BLOCK, sblock);
    ld_note_launch(), launch_after(k_decide_block<W, KIND, WIDE>, grid, BLOCK_THREADS, sblock, A);
    if (KIND == KIND_MOVE) kt_end(h, sblock);
  }
  if (need_hub) {
    bin(BIN_HUGE);
    A.gkeys = hs_keys(h);
    A.gvals = hs_vals(h);
    A.glist = hs_list(h);
    A.gocc = h->hocc;
    int64_t *tab_off = h->lbuf2, *ch_off = h->lbuf3;
    // keys: communities of the level
    launch_table_plan(A.list, A.count, g.deg, nullptr, g.n, tab_off, ch_off, shub, A.gocc);
    if (KIND == KIND_MOVE) kt_begin(h, KT_HUGE_SCAN, shub);
    int hg = sms * h->tune.hub_blocks_per_sm;
    ld_note_launch(), launch_after(k_huge_scan<W, KIND, WIDE>, hg, 256, shub, A, tab_off, ch_off);
    if (KIND == KIND_MOVE) kt_end(h, shub);
    BigTables big{h->ibuf1, &h->dcnt->hub_big, h->lbuf1, h->ibuf0};
    launch_piece_plan(A.count, A.gocc, big, shub);
    ld_note_launch(), launch_after(k_huge_decide<KIND, WIDE>, sms * 8, HUGE_THREADS, shub, A, tab_off, big);
  }
  if (fork) {
    for (int k = 0; k < 2; k++) {
      if ((k == 0 && !need_block) || (k == 1 && !need_hub)) continue;
      cudaEventRecord(h->join_ev[k], h->side[k]);
      cudaStreamWaitEvent(s, h->join_ev[k], 0);
    }
  }
}

template <int KIND>
void launch_bins(leiden_handle *h, const LevelGraph &g, const Args &A) {
  bool wide = wide_sums(h);
  if (g.w64) wide ? launch_bins_of<int64_t, KIND, true>(h, g, A) : launch_bins_of<int64_t, KIND, false>(h, g, A);
  else wide ? launch_bins_of<int32_t, KIND, true>(h, g, A) : launch_bins_of<int32_t, KIND, false>(h, g, A);
}

}  // namespace

// The side streams and events of a handle, created on first use; false
// (and the bins stay on the handle's stream) if they cannot be had.
bool side_streams(leiden_handle *h) {
  if (h->side[1]) return true;
  if (h->side_failed) return false;
  bool ok = cudaEventCreateWithFlags(&h->fork_ev, cudaEventDisableTiming) == cudaSuccess;
  for (int k = 0; k < 2 && ok; k++)
    ok = cudaStreamCreateWithFlags(&h->side[k], cudaStreamNonBlocking) == cudaSuccess &&
         cudaEventCreateWithFlags(&h->join_ev[k], cudaEventDisableTiming) == cudaSuccess;
  if (!ok) {
    cudaGetLastError();
    for (int k = 0; k < 2; k++) {
      if (h->side[k]) cudaStreamDestroy(h->side[k]);
      if (h->join_ev[k]) cudaEventDestroy(h->join_ev[k]);
      h->side[k] = nullptr;
      h->join_ev[k] = nullptr;
    }
    if (h->fork_ev) cudaEventDestroy(h->fork_ev);
    h->fork_ev = nullptr;
    h->side_failed = true;
  }
  return ok;
}

// Global table scratch of `slots` slots laid out as keys int32[S] | values
// int64[S] | slot lists int32[S] (16 B per slot).  Every user leaves the
// slots it touched empty again, so a new allocation is cleared once.
bool ensure_hslots(leiden_handle *h, int64_t slots) {
  if (slots <= h->hslots) return true;
  int64_t S = (slots + 1023) & ~(int64_t)1023;
  if (h->hscratch) {
    cudaStreamSynchronize(h->stream);
    for (auto &q : h->owned)
      if (q == h->hscratch) { cudaFree(q); q = nullptr; }
  }
  void *p = nullptr;
  if (cudaMalloc(&p, (size_t)S * 16) != cudaSuccess) {
    cudaGetLastError();
    h->hscratch = nullptr;
    h->hscratch_bytes = 0;
    h->hslots = 0;
    return false;
  }
  h->owned.push_back(p);
  h->hscratch = p;
  h->hscratch_bytes = (size_t)S * 16;
  h->hslots = S;
  cudaMemsetAsync(p, 0xff, (size_t)S * 4, h->stream);                   // keys: empty
  cudaMemsetAsync((char *)p + (size_t)S * 4, 0, (size_t)S * 8, h->stream);  // values: 0
  return true;
}

int32_t *hs_keys(leiden_handle *h) { return (int32_t *)h->hscratch; }
int64_t *hs_vals(leiden_handle *h) { return (int64_t *)((char *)h->hscratch + (size_t)h->hslots * 4); }
int32_t *hs_list(leiden_handle *h) { return (int32_t *)((char *)h->hscratch + (size_t)h->hslots * 12); }

void count_sizes(leiden_handle *h, const int32_t *C, int64_t n, int32_t *size) {
  cudaMemsetAsync(size, 0, (size_t)n * sizeof(int32_t), h->stream);
  ld_note_launch(), launch_after(k_sizes, grid_for(n, 256), 256, h->stream, C, n, size);
}

void lm_iteration(leiden_handle *h, const LevelGraph &g, const uint8_t *in_range, int dynamic, bool dense) {
  cudaStream_t s = h->stream;
  const int classes = lm_classes(h);
  const bool deferred = h->p.deterministic;
  Args A = make_args(h, g);
  A.in_range = in_range;
  A.dynamic = dynamic;
  CollectArgs Q{0, h->bins, nullptr, h->d_loff, h->tune};
  auto kernel = dense ? k_apply_collect<true> : k_apply_collect<false>;
  const int grid = grid_for((g.n + 31) / 32, dense ? 32 : 256);  // bitmap words per block
  bool pending = false;  // the moves of the class before wait to be applied
  cudaMemsetAsync(h->dcnt->dq, 0, offsetof(DevCounters, ref), s);
  for (int cls = 0; cls < classes; cls++) {
    Q.cls = cls;
    Q.sub = &h->dcnt->sub[cls % SUB_RING];
    if (cls && cls % SUB_RING == 0) {  // the sets are used again
      if (pending) {
        CollectArgs none = Q;
        none.cls = -1;
        ld_note_launch(), launch_after(kernel, grid, 256, s, A, true, h->gc.dq, h->gc.moves, none);
        pending = false;
      }
      cudaMemsetAsync(h->dcnt->sub, 0, sizeof(h->dcnt->sub), s);
    }
    ld_note_launch(), launch_after(kernel, grid, 256, s, A, pending, h->gc.dq, h->gc.moves, Q);
    A.sub = Q.sub;
    launch_bins<KIND_MOVE>(h, g, A);
    if (deferred && g.maxdeg > h->tune.block_max && g.maxdeg > MARK_INLINE)
      ld_note_launch(), launch_after(k_mark_hubs, h->sm_count * 4, 256, s, A);
    pending = deferred;
  }
  if (pending) {
    Q.cls = -1;
    ld_note_launch(), launch_after(kernel, std::min(grid, h->sm_count * 4), 256, s, A, true, h->gc.dq, h->gc.moves, Q);
  }
}

void refine_reset(leiden_handle *h, const LevelGraph &g) {
  cudaStream_t s = h->stream;
  cudaMemsetAsync(&h->dcnt->cand_count[0], 0, sizeof(int32_t), s);
  ld_note_launch(), launch_after(k_refine_reset, grid_for(g.n, APPEND_STEP), 256, s, g.n, h->CB, h->dR2, h->Cp, h->Sp,
                                 h->Kc, h->prop, h->cand, h->dcnt, g.gid, h->gc.refined);
}

// One round on the candidates of list `slot` (cand + slot*n, count
// cand_count[slot]); the ones still alone go to the other list.
void refine_round(leiden_handle *h, const LevelGraph &g, int slot) {
  cudaStream_t s = h->stream;
  int32_t *in = h->cand + (int64_t)slot * g.n, *out = h->cand + (int64_t)(1 - slot) * g.n;
  int32_t *cin = &h->dcnt->cand_count[slot], *cout = &h->dcnt->cand_count[1 - slot];
  static_assert(offsetof(DevCounters, accepted) == offsetof(DevCounters, ref) + sizeof(SubCounters),
                "cleared together");
  cudaMemsetAsync(&h->dcnt->ref, 0, sizeof(SubCounters) + sizeof(int32_t), s);  // bins, accepted
  cudaMemsetAsync(cout, 0, sizeof(int32_t), s);
  ld_note_launch(), launch_after(k_refine_collect, grid_for(g.n, APPEND_STEP), 256, s, in, cin, out, cout, g.n, h->Cp,
                                 h->Sp, h->Kc, g.deg, h->prop, h->bins, &h->dcnt->ref, h->tune);
  Args A = make_args(h, g);
  launch_bins<KIND_REFINE>(h, g, A);
  ld_note_launch(), launch_after(k_refine_accept, grid_for(g.n, 256, h->sm_count * 4), 256, s, out, cout, h->prop,
                                 h->Cp, h->Sp, h->Kc, h->dcnt, g.gid, h->gc.accepted);
}

LD_CHECK_WORD_READER(check_word_move)

unsigned int check_selftest(cudaStream_t s) {
  ld_note_launch(), k_check_selftest<<<1, 32, 0, s>>>();
  cudaStreamSynchronize(s);
  return check_word_move();
}
