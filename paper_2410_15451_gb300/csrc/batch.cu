// Batch update: canonicalise the batch, apply it to the slack CSR by sorted
// merge, mark affected vertices (ND / DS / DF, Appendix A.1-A.3), update
// K, Sigma and Delta Sigma (Alg. "update"), and mark communities to split /
// refine (Alg. "leidenmk").
#include <algorithm>

#include "internal.h"

namespace {

constexpr int TB = 256;
// Touched rows by new length: a warp with 2 KB of shared staging, a warp with
// 8 KB, a block with 32 KB, and above that chunks over all SMs.  A row is a chain
// of dependent loads (its plan, its place, the row), so what counts is how many
// are in flight: 64, 28 and 7 per SM.
constexpr int MERGE_SMALL = 256;
constexpr int MERGE_WARP = 1024;
constexpr int MERGE_MID = 4096;

__device__ __forceinline__ int64_t lower_bound_i32(const int32_t *a, int64_t n, int32_t x) {
  int64_t lo = 0, hi = n;
  while (lo < hi) {
    int64_t mid = (lo + hi) >> 1;
    if (a[mid] < x) lo = mid + 1; else hi = mid;
  }
  return lo;
}
__device__ __forceinline__ int64_t lower_bound_u64(const uint64_t *a, int64_t n, uint64_t x) {
  int64_t lo = 0, hi = n;
  while (lo < hi) {
    int64_t mid = (lo + hi) >> 1;
    if (a[mid] < x) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// Ids in range, no self-loop, a positive weight to insert, and (batched handles)
// both ends in one graph.
__device__ __forceinline__ bool valid_edge(const leiden_edge &x, bool del, int64_t n, const int32_t *gid0) {
  if (x.u < 0 || x.u >= n || x.v < 0 || x.v >= n || x.u == x.v || (!del && x.w <= 0)) return false;
  return !gid0 || gid0[x.u] == gid0[x.v];
}

// Mirror each undirected edge into two arcs keyed (src << vb) | dst and
// validate it.  error := 1 on any violation.  Deletions and insertions go
// into one array for one sort: the 2*n_del deletion arcs first (weight 0),
// then the insertion arcs with bit 2*vb set, so that after the sort the
// deletions come first and each part is sorted by its keys.
__global__ void k_expand(const leiden_edge *del, int64_t n_del, const leiden_edge *ins, int64_t n_ins,
                         int64_t n, int vb, uint64_t *key, int64_t *w, DevCounters *cnt, const int32_t *gid0) {
  ld_after_previous();
  const uint64_t ins_bit = 1ull << (2 * vb);
  for (int64_t e = ld_gtid(); e < n_del + n_ins; e += ld_gstride()) {
    bool is_del = e < n_del;
    leiden_edge x = is_del ? del[e] : ins[e - n_del];
    if (!valid_edge(x, is_del, n, gid0)) {
      atomicExch(&cnt->error, 1);
      x.u = 0; x.v = 1 % (int32_t)(n > 1 ? n : 1); x.w = 1;
    }
    uint64_t k1 = ((uint64_t)x.u << vb) | (uint64_t)x.v;
    uint64_t k2 = ((uint64_t)x.v << vb) | (uint64_t)x.u;
    uint64_t tag = is_del ? 0ull : ins_bit;
    key[2 * e] = k1 | tag;
    key[2 * e + 1] = k2 | tag;
    w[2 * e] = is_del ? 0 : x.w;
    w[2 * e + 1] = is_del ? 0 : x.w;
  }
}

// Heads of the runs of equal keys over both parts of the sorted batch (the
// insertion tag keeps them apart); IW zeroed for the sums.
__global__ void k_head_flags(const uint64_t *key, int64_t n, int32_t *flag, int64_t *zero, int64_t nzero) {
  ld_after_previous();
  for (int64_t i = ld_gtid(); i < n; i += ld_gstride()) {
    flag[i] = (i == 0 || key[i] != key[i - 1]) ? 1 : 0;
    if (i < nzero) zero[i] = 0;
  }
}

// Unique keys (and summed payload) into out_key/out_w at the scanned positions.
__global__ void k_unique(const uint64_t *key, const int64_t *w, int64_t n, const int32_t *flag, const int64_t *pos,
                         uint64_t *out_key, int64_t *out_w) {
  ld_after_previous();
  for (int64_t i = ld_gtid(); i < n; i += ld_gstride()) {
    int64_t p = pos[i] + flag[i] - 1;
    if (flag[i]) out_key[p] = key[i];
    if (out_w) atomicAdd((unsigned long long *)&out_w[p], (unsigned long long)w[i]);
  }
}

// The same for the batch: deletions collapse (-> dkey), insertions lose their
// tag and add up (-> ikey, iw); counts [0] and [1].
__global__ void k_unique_batch(const uint64_t *key, const int64_t *w, int64_t nda, int64_t nia, const int32_t *flag,
                               const int64_t *pos, uint64_t mask, uint64_t *dkey, uint64_t *ikey, int64_t *iw,
                               int64_t *counts) {
  ld_after_previous();
  const int64_t nd = pos[nda];
  if (ld_gtid() == 0) {
    counts[0] = nd;
    counts[1] = pos[nda + nia] - nd;
  }
  for (int64_t i = ld_gtid(); i < nda + nia; i += ld_gstride()) {
    int64_t p = pos[i] + flag[i] - 1;
    if (i < nda) {
      if (flag[i]) dkey[p] = key[i];
    } else {
      if (flag[i]) ikey[p - nd] = key[i] & mask;
      atomicAdd((unsigned long long *)&iw[p - nd], (unsigned long long)w[i]);
    }
  }
}

// What both batch paths need of the graph and of the handle's parameters.
struct BatchGraph {
  int64_t n;
  const int64_t *off;
  const int32_t *deg, *rcap, *col, *w, *gid0;
  int64_t colcap;
  double slack;
  int min_slack, block_max, vb;
};

// A deletion must name an existing arc: its stored weight (0 and error 2 if not).
__device__ __forceinline__ int64_t deleted_weight(const BatchGraph &G, uint64_t key, DevCounters *cnt) {
  int32_t u = (int32_t)(key >> G.vb), v = (int32_t)(key & ((1ull << G.vb) - 1));
  const int32_t *row = G.col + G.off[u];
  int64_t p = lower_bound_i32(row, G.deg[u], v);
  if (p < G.deg[u] && row[p] == v) return G.w[G.off[u] + p];
  atomicExch(&cnt->error, 2);
  return 0;
}
// The arc an insertion adds to, or -1: a new arc (also when the batch deletes
// the existing one; dkey: its nd sorted deletions).
__device__ __forceinline__ int64_t existing_arc(const BatchGraph &G, uint64_t key, const uint64_t *dkey, int64_t nd) {
  int32_t u = (int32_t)(key >> G.vb), v = (int32_t)(key & ((1ull << G.vb) - 1));
  const int32_t *row = G.col + G.off[u];
  int64_t p = lower_bound_i32(row, G.deg[u], v);
  if (p >= G.deg[u] || row[p] != v) return -1;
  int64_t q = lower_bound_u64(dkey, nd, key);
  return q < nd && dkey[q] == key ? -1 : G.off[u] + p;
}

// Deletions checked (stored weights -> dw), insertions classified: state 1 and
// position of an existing arc, state 0 for a new one, flagged (over the bound
// nia >= ni, zero past ni).  The change of 2m is summed.
__global__ void __launch_bounds__(256) k_check_batch(BatchGraph G, const uint64_t *dkey, const uint64_t *ikey,
                                                     const int64_t *iw, const int64_t *counts, int64_t nda, int64_t nia,
                                                     int64_t *dw, int32_t *state, int64_t *ipos, int32_t *flag,
                                                     DevCounters *cnt) {
  ld_after_previous();
  __shared__ unsigned long long sum;
  if (threadIdx.x == 0) sum = 0;
  __syncthreads();
  const int64_t nd = counts[0], ni = counts[1];
  int64_t acc = 0;
  for (int64_t i = ld_gtid(); i < nda + nia; i += ld_gstride()) {
    if (i < nda) {
      if (i < nd) acc -= dw[i] = deleted_weight(G, dkey[i], cnt);
      continue;
    }
    int64_t k = i - nda;
    flag[k] = 0;
    if (k >= ni) continue;
    int64_t p = existing_arc(G, ikey[k], dkey, nd);
    state[k] = p >= 0;
    ipos[k] = p;
    flag[k] = p < 0;
    acc += iw[k];
  }
  acc = ld_warp_sum_i64(acc);
  if ((threadIdx.x & 31) == 0 && acc) atomicAdd(&sum, (unsigned long long)acc);
  __syncthreads();
  if (threadIdx.x == 0 && sum) atomicAdd((unsigned long long *)&cnt->batch_dw, sum);
}

__global__ void k_compact_new(const uint64_t *ikey, const int64_t *iw, int64_t ni, const int32_t *flag,
                              const int64_t *pos, uint64_t *okey, int64_t *ow, int64_t *count) {
  ld_after_previous();
  if (ld_gtid() == 0) *count = pos[ni];
  for (int64_t i = ld_gtid(); i < ni; i += ld_gstride())
    if (flag[i]) { okey[pos[i]] = ikey[i]; ow[pos[i]] = iw[i]; }
}

// Rows whose structure changes (sources of deletions and of new arcs), each
// listed once, in no particular order: the first arc of a source's run in
// either sorted list sets the source's bit, and the arc that found it clear
// appends the row.  Work is O(batch), not O(n).
__global__ void k_touched_rows(const uint64_t *dkey, const int64_t *nd_p, const uint64_t *nkey, const int64_t *nn_p,
                               int vb, uint32_t *bits, int32_t *rows, int64_t *nrows) {
  ld_after_previous();
  int64_t nd = *nd_p, nn = *nn_p;
  for (int64_t t = ld_gtid(); t < nd + nn; t += ld_gstride()) {
    bool del = t < nd;
    const uint64_t *K = del ? dkey : nkey;
    int64_t k = del ? t : t - nd;
    uint64_t u = K[k] >> vb;
    if (k > 0 && (K[k - 1] >> vb) == u) continue;
    uint32_t bit = 1u << (u & 31);
    if (!(atomicOr(&bits[u >> 5], bit) & bit))
      rows[atomicAdd((unsigned long long *)nrows, 1ull)] = (int32_t)u;
  }
}

// Table slots a hub of d arcs needs (0 below the hub path).
__device__ __forceinline__ int64_t hub_slots(int64_t d, int block_max) {
  return d > block_max ? (int64_t)1 << (64 - __clzll(2 * d - 1)) : 0;
}

// Where the plan of a touched row goes.
struct RowPlan {
  int32_t *dlo, *dhi, *ilo, *ihi;
  int64_t *len, *dst;
  int32_t *newcap, *olddeg, *large, *mid, *warp;
};

// Plan of touched row r = vertex u: its segments in the two arc lists, its new
// length, its class, and a new place at the end of the arc arrays with fresh
// slack if it outgrows its capacity (if the arena is full the whole CSR is
// rebuilt instead: overflow).  A batch already found invalid takes no arena
// space.  Returns the new length; slots: the change of the hub tables' size.
__device__ __forceinline__ int64_t plan_row(const BatchGraph &G, const RowPlan &P, int64_t r, uint64_t u,
                                            const uint64_t *dkey, int64_t nd, const uint64_t *nkey, int64_t nn,
                                            bool invalid, DevCounters *cnt, int64_t &slots) {
  int64_t a = lower_bound_u64(dkey, nd, u << G.vb), b = lower_bound_u64(dkey, nd, (u + 1) << G.vb);
  int64_t c = lower_bound_u64(nkey, nn, u << G.vb), d = lower_bound_u64(nkey, nn, (u + 1) << G.vb);
  P.dlo[r] = (int32_t)a; P.dhi[r] = (int32_t)b; P.ilo[r] = (int32_t)c; P.ihi[r] = (int32_t)d;
  int32_t dg = G.deg[u];
  int64_t L = (int64_t)dg - (b - a) + (d - c), dst = G.off[u];
  int32_t newcap = 0;
  P.len[r] = L;
  P.olddeg[r] = dg;
  if (L > MERGE_MID) P.large[atomicAdd(&cnt->large_count, 1)] = (int32_t)r;
  else if (L > MERGE_WARP) P.mid[atomicAdd(&cnt->mid_count, 1)] = (int32_t)r;
  else if (L > MERGE_SMALL) P.warp[atomicAdd(&cnt->warp_count, 1)] = (int32_t)r;
  if (L > G.rcap[u] && !invalid) {
    int64_t extra = (int64_t)((double)L * G.slack);
    if (extra < G.min_slack) extra = G.min_slack;
    int64_t cap = L + extra;
    dst = (int64_t)atomicAdd((unsigned long long *)&cnt->arena_used, (unsigned long long)cap);
    if (dst + cap > G.colcap) atomicExch(&cnt->overflow, 1);
    newcap = (int32_t)cap;
  }
  P.dst[r] = dst;
  P.newcap[r] = newcap;
  slots += hub_slots(L, G.block_max) - hub_slots(dg, G.block_max);
  return L;
}

// Plans of the touched rows; lengths are written up to the bound nb >= nrows
// (zero past nrows) so that their scan needs no host count.  Leaves the row
// bitmap clear for the next call (every set bit belongs to a listed row).
__global__ void __launch_bounds__(256) k_row_plan(BatchGraph G, RowPlan P, const int32_t *rows, const int64_t *nrows_p,
                                                  int64_t nb, const uint64_t *dkey, const int64_t *nd_p,
                                                  const uint64_t *nkey, const int64_t *nn_p, uint32_t *bits,
                                                  int64_t *total, DevCounters *cnt) {
  ld_after_previous();
  __shared__ unsigned long long sum_s, slots_s;
  __shared__ int max_s;
  if (threadIdx.x == 0) { sum_s = 0; slots_s = 0; max_s = 0; }
  __syncthreads();
  const int64_t nrows = *nrows_p, nd = *nd_p, nn = *nn_p;
  const bool invalid = cnt->error != 0;
  int64_t sum = 0, slots = 0;
  int mx = 0;
  for (int64_t r = ld_gtid(); r < nb; r += ld_gstride()) {
    if (r >= nrows) { P.len[r] = 0; continue; }
    int32_t u = rows[r];
    bits[u >> 5] = 0;
    int64_t L = plan_row(G, P, r, (uint64_t)u, dkey, nd, nkey, nn, invalid, cnt, slots);
    sum += L;
    mx = max(mx, (int)L);
  }
  sum = ld_warp_sum_i64(sum);
  slots = ld_warp_sum_i64(slots);
  mx = __reduce_max_sync(LD_FULL, mx);
  if ((threadIdx.x & 31) == 0) {
    if (sum) atomicAdd(&sum_s, (unsigned long long)sum);
    if (slots) atomicAdd(&slots_s, (unsigned long long)slots);
    if (mx) atomicMax(&max_s, mx);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    if (sum_s) atomicAdd((unsigned long long *)total, sum_s);
    if (slots_s) atomicAdd((unsigned long long *)&cnt->slot_change, slots_s);
    if (max_s) atomicMax(&cnt->max_row, max_s);
  }
}

// ---------------------------------------------------------------- small batches
// A batch of at most SMALL_ARCS arcs is expanded, sorted, deduplicated, checked
// and planned by one block in shared memory: the steps are a chain, and at
// this size each of them costs a launch more than its work (23 launches and
// clears of the path above; 100 edges on 10k vertices: 433 -> 302 us a call,
// the kernel itself 22 us).
constexpr int SMALL_ARCS = 2048;

// Exclusive sums of the threads' values over a block of 1024, the total in *total.
__device__ __forceinline__ int64_t block_excl_1024(int64_t v, int64_t *ws, int64_t *total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int64_t incl = ld_warp_incl_i64(v);
  __syncthreads();
  if (lane == 31) ws[wid] = incl;
  __syncthreads();
  int64_t y = ws[lane], yi = ld_warp_incl_i64(y);
  *total = __shfl_sync(LD_FULL, yi, 31);
  return __shfl_sync(LD_FULL, yi - y, wid) + incl - v;
}

struct SmallOut {
  uint64_t *dkey, *ikey, *nkey;
  int64_t *dw, *iw, *nw, *ipos, *tmp_off;
  int32_t *state, *rows;
};

__global__ void __launch_bounds__(1024) k_small_batch(BatchGraph G, RowPlan P, SmallOut O, const leiden_edge *del,
                                                      int n_del, const leiden_edge *ins, int n_ins, DevCounters *cnt) {
  ld_after_previous();
  __shared__ uint64_t sk[SMALL_ARCS];     // arcs by key, then the unique ones: deletions, insertions
  __shared__ int64_t sw[SMALL_ARCS];      // summed weights of the unique arcs, then the new arcs' keys
  __shared__ int32_t si[SMALL_ARCS];      // input positions, then the touched rows
  __shared__ int64_t ws[32];
  __shared__ int nrows_s, max_s;
  const int tid = threadIdx.x, nda = 2 * n_del, na = 2 * (n_del + n_ins), vb = G.vb;
  const uint64_t mask = (1ull << (2 * vb)) - 1, tag = 1ull << (2 * vb);
  if (tid == 0) { nrows_s = 0; max_s = 0; }
  int N2 = 2;
  while (N2 < na) N2 <<= 1;
  for (int t = tid; t < N2; t += 1024) {
    uint64_t key = ~0ull;  // padding sorts last (its positions are larger)
    if (t < na) {
      int e = t >> 1;
      bool d = e < n_del;
      leiden_edge x = d ? del[e] : ins[e - n_del];
      if (!valid_edge(x, d, G.n, G.gid0)) {
        atomicExch(&cnt->error, 1);
        x.u = 0; x.v = 1 % (int32_t)(G.n > 1 ? G.n : 1);
      }
      key = (t & 1 ? ((uint64_t)x.v << vb) | (uint64_t)x.u : ((uint64_t)x.u << vb) | (uint64_t)x.v) | (d ? 0ull : tag);
    }
    sk[t] = key;
    si[t] = t;
  }
  __syncthreads();
  for (int k = 2; k <= N2; k <<= 1)  // bitonic network
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int t = tid; t < N2; t += 1024) {
        int u = t ^ j;
        if (u <= t) continue;
        uint64_t a = sk[t], b = sk[u];
        if ((a > b) == ((t & k) == 0) && a != b) {
          int32_t x = si[t];
          sk[t] = b; sk[u] = a; si[t] = si[u]; si[u] = x;
        }
      }
      __syncthreads();
    }
  // unique arcs: thread t holds the sorted ones 2t and 2t + 1
  uint64_t key[2];
  int64_t w[2];
  bool head[2];
#pragma unroll
  for (int q = 0; q < 2; q++) {
    int t = 2 * tid + q;
    head[q] = t < na && (t == 0 || sk[t] != sk[t - 1]);
    key[q] = t < na ? sk[t] : 0;
    int e = t < na ? si[t] >> 1 : 0;
    w[q] = t < na && e >= n_del ? ins[e - n_del].w : 0;
  }
  int64_t nu, nd, total;
  int64_t pos = block_excl_1024((int)head[0] + (int)head[1], ws, &nu);
  block_excl_1024((int)(head[0] && key[0] < tag) + (int)(head[1] && key[1] < tag), ws, &nd);
  for (int t = tid; t < SMALL_ARCS; t += 1024) sw[t] = 0;
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 2; q++) {
    pos += head[q];
    if (2 * tid + q < na) {
      if (head[q]) sk[pos - 1] = key[q] & mask;
      if (w[q]) atomicAdd((unsigned long long *)&sw[pos - 1], (unsigned long long)w[q]);
    }
  }
  __syncthreads();
  // deletions checked, insertions classified (unique arcs 2t and 2t + 1)
  const int64_t ni = nu - nd;
  int64_t dsum = 0;
  bool fresh[2] = {false, false};
#pragma unroll
  for (int q = 0; q < 2; q++) {
    int t = 2 * tid + q;
    if (t >= nu) continue;
    key[q] = sk[t];
    w[q] = sw[t];
    if (t < nd) {
      int64_t x = deleted_weight(G, key[q], cnt);
      O.dkey[t] = key[q];
      O.dw[t] = x;
      dsum -= x;
    } else {
      int64_t p = existing_arc(G, key[q], sk, nd);
      O.ikey[t - nd] = key[q];
      O.iw[t - nd] = w[q];
      O.state[t - nd] = p >= 0;
      O.ipos[t - nd] = p;
      fresh[q] = p < 0;
      dsum += w[q];
    }
  }
  int64_t nn, at = block_excl_1024((int)fresh[0] + (int)fresh[1], ws, &nn);  // (its barriers: sw has been read)
  uint64_t *nk = (uint64_t *)sw;
#pragma unroll
  for (int q = 0; q < 2; q++)
    if (fresh[q]) {
      nk[at] = key[q];
      O.nkey[at] = key[q];
      O.nw[at] = w[q];
      at++;
    }
  block_excl_1024(dsum, ws, &total);
  if (tid == 0) cnt->batch_dw = total;
  __syncthreads();
  // touched rows: the heads of the sources' runs, a new arc's only if no deletion has its source
  for (int t = tid; t < nd + nn; t += 1024) {
    const uint64_t *L = t < nd ? sk : nk;
    int64_t k = t < nd ? t : t - nd;
    uint64_t u = L[k] >> vb;
    if (k > 0 && (L[k - 1] >> vb) == u) continue;
    if (t >= nd) {
      int64_t q = lower_bound_u64(sk, nd, u << vb);
      if (q < nd && (sk[q] >> vb) == u) continue;
    }
    si[atomicAdd(&nrows_s, 1)] = (int32_t)u;
  }
  __syncthreads();
  const int nrows = nrows_s;
  const bool invalid = *(volatile int32_t *)&cnt->error != 0;
  int64_t len[2] = {0, 0}, slots = 0;
#pragma unroll
  for (int q = 0; q < 2; q++) {
    int r = 2 * tid + q;
    if (r >= nrows) continue;
    O.rows[r] = si[r];
    len[q] = plan_row(G, P, r, (uint64_t)si[r], sk, nd, nk, nn, invalid, cnt, slots);
  }
  int64_t off = block_excl_1024(len[0] + len[1], ws, &total), st;
#pragma unroll
  for (int q = 0; q < 2; q++) {
    int r = 2 * tid + q;
    if (r < nrows) O.tmp_off[r] = off;
    off += len[q];
    if (r == nrows - 1) O.tmp_off[nrows] = off;
  }
  block_excl_1024(slots, ws, &st);
  int mx = __reduce_max_sync(LD_FULL, (int)max(len[0], len[1]));
  if ((tid & 31) == 0) atomicMax(&max_s, mx);
  __syncthreads();
  if (tid == 0) {
    cnt->bcounts[0] = nd;
    cnt->bcounts[1] = ni;
    cnt->bcounts[2] = nn;
    cnt->bcounts[3] = nrows;
    cnt->bcounts[4] = total;
    cnt->slot_change = st;
    cnt->max_row = max_s;
  }
}

__global__ void k_add_existing(const int64_t *ipos, const int32_t *state, const int64_t *iw, int64_t ni, int32_t *w) {
  ld_after_previous();
  for (int64_t i = ld_gtid(); i < ni; i += ld_gstride())
    if (state[i]) w[ipos[i]] += (int32_t)iw[i];
}

// Warp per touched row: old row minus deletions plus new arcs, by ranks.
__global__ void k_merge_rows(const int32_t *rows, const int64_t *nrows_p, int vb, const uint64_t *dkey,
                             const uint64_t *nkey, const int64_t *nw, const int32_t *dlo, const int32_t *dhi,
                             const int32_t *ilo, const int32_t *ihi, const int64_t *tmp_off, const int64_t *off,
                             const int32_t *deg, const int32_t *col, const int32_t *w, int32_t *tcol, int32_t *tw) {
  ld_after_previous();
  int64_t nrows = *nrows_p;
  int lane = threadIdx.x & 31;
  int64_t warp = ld_gtid() >> 5, nwarps = ld_gstride() >> 5;
  uint64_t mask = (1ull << vb) - 1;
  for (int64_t r = warp; r < nrows; r += nwarps) {
    int32_t u = rows[r];
    const int32_t *row = col + off[u];
    const int32_t *roww = w + off[u];
    int64_t dg = deg[u];
    const uint64_t *D = dkey + dlo[r];
    int64_t nD = dhi[r] - dlo[r];
    const uint64_t *I = nkey + ilo[r];
    const int64_t *IW = nw + ilo[r];
    int64_t nI = ihi[r] - ilo[r];
    int64_t base = tmp_off[r];
    uint64_t ubase = (uint64_t)u << vb;
    for (int64_t p = lane; p < dg; p += 32) {
      int32_t x = row[p];
      int64_t dless = lower_bound_u64(D, nD, ubase | (uint64_t)x);
      if (dless < nD && (D[dless] & mask) == (uint64_t)x) continue;  // deleted
      int64_t iless = lower_bound_u64(I, nI, ubase | (uint64_t)x);
      int64_t o = base + (p - dless) + iless;
      tcol[o] = x;
      tw[o] = roww[p];
    }
    for (int64_t k = lane; k < nI; k += 32) {
      int32_t y = (int32_t)(I[k] & mask);
      int64_t rless = lower_bound_i32(row, dg, y);
      int64_t dless = lower_bound_u64(D, nD, ubase | (uint64_t)y);
      int64_t o = base + k + (rless - dless);
      tcol[o] = y;
      tw[o] = (int32_t)IW[k];
    }
  }
}

// In-place merge of the touched rows that fit their capacity (no overflow).
// Output position of an old element x at p: p - |D < x| + |I < x|; of the
// k-th new arc y: k + |row < y| - |D < y|.  Everything before the first change
// stays where it is (unless the row is relocated); the rest is staged in
// shared memory and written back after all of the row's reads.
constexpr int MERGE_WARPS = 4;

struct MergeArgs {
  const int32_t *rows;
  const int64_t *nrows_p;
  int vb;
  const uint64_t *dkey, *nkey;
  const int64_t *nw;
  const int32_t *dlo, *dhi, *ilo, *ihi;
  const int64_t *len, *tmp_off, *off;
  int32_t *deg, *col, *w, *tcol, *tw;
  const int64_t *dst;     // where the merged row goes (its old place unless relocated)
  const int32_t *newcap;  // capacity of a relocated row, 0 otherwise
  int64_t *off_w;         // row starts (written after a row is relocated)
  int32_t *rcap;          // row capacities
};

// After the row's reads are done: record a relocation.
__device__ __forceinline__ void finish_row(const MergeArgs &A, int64_t r, int32_t u, int64_t L) {
  A.deg[u] = (int32_t)L;
  if (A.newcap[r]) {
    A.off_w[u] = A.dst[r];
    A.rcap[u] = A.newcap[r];
  }
}

// Rows of at most MERGE_SMALL arcs, a warp each, moved whole: the search for the
// first change and the registers of the longer rows' form below cost more than
// the row (R-MAT 22: 60 us, with that form 92).
__device__ __forceinline__ void merge_row_into(const MergeArgs &A, int64_t r, int t0, int stride, int32_t *ocol,
                                               int32_t *ow, const uint64_t *D, const uint64_t *I) {
  uint64_t mask = (1ull << A.vb) - 1;
  int32_t u = A.rows[r];
  const int32_t *row = A.col + A.off[u];
  const int32_t *roww = A.w + A.off[u];
  int64_t dg = A.deg[u];
  int64_t nD = A.dhi[r] - A.dlo[r];
  const int64_t *IW = A.nw + A.ilo[r];
  int64_t nI = A.ihi[r] - A.ilo[r];
  uint64_t ubase = (uint64_t)u << A.vb;
  for (int64_t p = t0; p < dg; p += stride) {
    int32_t x = row[p];
    int64_t dless = nD ? lower_bound_u64(D, nD, ubase | (uint64_t)x) : 0;
    if (dless < nD && (D[dless] & mask) == (uint64_t)x) continue;
    int64_t iless = nI ? lower_bound_u64(I, nI, ubase | (uint64_t)x) : 0;
    int64_t o = (p - dless) + iless;
    ocol[o] = x;
    ow[o] = roww[p];
  }
  for (int64_t k = t0; k < nI; k += stride) {
    int32_t y = (int32_t)(I[k] & mask);
    int64_t rless = lower_bound_i32(row, dg, y);
    int64_t dless = nD ? lower_bound_u64(D, nD, ubase | (uint64_t)y) : 0;
    int64_t o = k + (rless - dless);
    ocol[o] = y;
    ow[o] = (int32_t)IW[k];
  }
}

__global__ void __launch_bounds__(MERGE_WARPS * 32) k_merge_small(MergeArgs A) {
  ld_after_previous();
  __shared__ int32_t scol[MERGE_WARPS][MERGE_SMALL];
  __shared__ int32_t sw[MERGE_WARPS][MERGE_SMALL];
  int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int64_t nrows = *A.nrows_p;
  for (int64_t r = (int64_t)blockIdx.x * MERGE_WARPS + wid; r < nrows; r += (int64_t)gridDim.x * MERGE_WARPS) {
    int64_t L = A.len[r];
    if (L > MERGE_SMALL) continue;
    merge_row_into(A, r, lane, 32, scol[wid], sw[wid], A.dkey + A.dlo[r], A.nkey + A.ilo[r]);
    __syncwarp();
    int32_t u = A.rows[r];
    int64_t o = A.dst[r];
    for (int64_t x = lane; x < L; x += 32) { A.col[o + x] = scol[wid][x]; A.w[o + x] = sw[wid][x]; }
    if (lane == 0) finish_row(A, r, u, L);
    __syncwarp();
  }
}

// Most rows get a handful of arcs: up to MERGE_FEW of either kind are held one
// per lane and counted with shuffles, more are searched.
constexpr int MERGE_FEW = 8;
constexpr int MERGE_UNROLL = 4;

// Row r merged by `threads` threads (whole warps; t0: the thread's index) into
// the stage from its first changed position on (0 for a row that moves).
// Returns its vertex; first: that position.
__device__ __forceinline__ int32_t merge_tail(const MergeArgs &A, int64_t r, int t0, int threads, int32_t *scol,
                                              int32_t *sw, int &first) {
  const int lane = threadIdx.x & 31;
  const uint64_t mask = (1ull << A.vb) - 1;
  const int32_t u = A.rows[r];
  const int64_t b = A.off[u];
  const int dg = A.deg[u], nD = A.dhi[r] - A.dlo[r], nI = A.ihi[r] - A.ilo[r];
  const int32_t *row = A.col + b, *roww = A.w + b;
  const uint64_t *D = A.dkey + A.dlo[r], *I = A.nkey + A.ilo[r];
  const int64_t *IW = A.nw + A.ilo[r];
  const uint64_t ubase = (uint64_t)u << A.vb;
  const bool few = nD <= MERGE_FEW && nI <= MERGE_FEW, one = threads == 32;
  const int32_t dv = lane < nD ? (int32_t)(D[lane] & mask) : 0, iv = lane < nI ? (int32_t)(I[lane] & mask) : 0;
  const int64_t iw = lane < nI ? IW[lane] : 0;
  int below = 0;  // (few, one warp) row elements below this lane's new arc
  first = 0;
  if (!A.newcap[r]) {
    int32_t x = __shfl_sync(LD_FULL, nD ? dv : iv, 0);
    if (nD && nI) x = min(x, __shfl_sync(LD_FULL, iv, 0));
    first = (int)lower_bound_i32(row, dg, x);
    below = first;
  }
  for (int p0 = first + (t0 & ~31); p0 < dg; p0 += threads * MERGE_UNROLL) {  // warp-uniform
    int32_t x[MERGE_UNROLL], xw[MERGE_UNROLL];
#pragma unroll
    for (int q = 0; q < MERGE_UNROLL; q++) {
      int p = p0 + q * threads + lane;
      x[q] = p < dg ? row[p] : INT32_MAX;
      xw[q] = p < dg ? roww[p] : 0;
    }
#pragma unroll
    for (int q = 0; q < MERGE_UNROLL; q++) {
      if (p0 + q * threads >= dg) break;  // warp-uniform
      int p = p0 + q * threads + lane;
      int dless = 0, iless = 0;
      bool gone = false;
      if (few) {
        for (int k = 0; k < nD; k++) {
          int32_t y = __shfl_sync(LD_FULL, dv, k);
          dless += y < x[q];
          gone = gone || y == x[q];
        }
        for (int k = 0; k < nI; k++) {
          int32_t y = __shfl_sync(LD_FULL, iv, k);
          iless += y < x[q];
          int c = __popc(__ballot_sync(LD_FULL, x[q] < y));
          if (lane == k) below += c;
        }
      } else if (p < dg) {
        const uint64_t key = ubase | (uint64_t)x[q];
        dless = (int)lower_bound_u64(D, nD, key);
        gone = dless < nD && D[dless] == key;
        iless = (int)lower_bound_u64(I, nI, key);
      }
      if (p < dg && !gone) {
        int o = p - dless + iless - first;
        scol[o] = x[q];
        sw[o] = xw[q];
      }
    }
  }
  if (few && one) {
    int dless = 0;
    for (int k = 0; k < nD; k++) dless += __shfl_sync(LD_FULL, dv, k) < iv;
    if (lane < nI) {
      int o = lane + below - dless - first;
      scol[o] = iv;
      sw[o] = (int32_t)iw;
    }
    return u;
  }
  for (int k = t0; k < nI; k += threads) {
    int32_t y = (int32_t)(I[k] & mask);
    int o = k + (int)lower_bound_i32(row, dg, y) - (int)lower_bound_u64(D, nD, ubase | (uint64_t)y) - first;
    scol[o] = y;
    sw[o] = (int32_t)IW[k];
  }
  return u;
}

// Rows of MERGE_SMALL+1..MERGE_WARP arcs, a warp each.  With a block each (and a
// search of both arc lists per element), these and the block's rows took 277 us
// (R-MAT 22, 64,154 edges); now 55 and 88.
__global__ void __launch_bounds__(MERGE_WARPS * 32) k_merge_warp(MergeArgs A, const int32_t *list,
                                                                 const int32_t *count_p) {
  ld_after_previous();
  __shared__ int32_t scol[MERGE_WARPS][MERGE_WARP];
  __shared__ int32_t sw[MERGE_WARPS][MERGE_WARP];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t count = *count_p;
  for (int64_t k = (int64_t)blockIdx.x * MERGE_WARPS + wid; k < count; k += (int64_t)gridDim.x * MERGE_WARPS) {
    const int64_t r = list[k];
    const int64_t L = A.len[r];
    int first;
    const int32_t u = merge_tail(A, r, lane, 32, scol[wid], sw[wid], first);
    __syncwarp();
    const int64_t o = A.dst[r] + first;
    const int n = (int)L - first;
    for (int x = lane; x < n; x += 32) { A.col[o + x] = scol[wid][x]; A.w[o + x] = sw[wid][x]; }
    if (lane == 0) finish_row(A, r, u, L);
    __syncwarp();
  }
}

// Rows of MERGE_WARP+1..MERGE_MID arcs: one block each.
__global__ void __launch_bounds__(256) k_merge_mid(MergeArgs A, const int32_t *mid, const int32_t *count_p,
                                                   int64_t *xk_bytes) {
  ld_after_previous();
  __shared__ int32_t scol[MERGE_MID];
  __shared__ int32_t sw[MERGE_MID];
  int64_t count = *count_p;
  int64_t bytes = 0;  // algorithmic bytes (thread 0): the moved part of the row, old and new, its batch arcs
  for (int64_t k = blockIdx.x; k < count; k += gridDim.x) {
    int64_t r = mid[k];
    int64_t L = A.len[r];
    int first;
    const int32_t u = merge_tail(A, r, threadIdx.x, 256, scol, sw, first);
    if (threadIdx.x == 0)
      bytes += 8 * ((int64_t)A.deg[u] + L - 2 * first) + 16 * (A.dhi[r] - A.dlo[r] + A.ihi[r] - A.ilo[r]);
    __syncthreads();
    const int64_t o = A.dst[r] + first;
    const int n = (int)L - first;
    for (int x = threadIdx.x; x < n; x += 256) { A.col[o + x] = scol[x]; A.w[o + x] = sw[x]; }
    if (threadIdx.x == 0) finish_row(A, r, u, L);
    __syncthreads();
  }
  if (threadIdx.x == 0 && bytes) atomicAdd((unsigned long long *)xk_bytes, (unsigned long long)bytes);
}

// Long rows in chunks any block may take (items k of `large`, chunk offsets
// ch_off over the old row): elements go to the merge buffer by rank; the
// first chunk of a row also places its new arcs.
__global__ void __launch_bounds__(256) k_merge_chunks_write(MergeArgs A, const int32_t *large,
                                                            const int32_t *count_p, const int64_t *ch_off) {
  ld_after_previous();
  int64_t count = *count_p;
  int64_t nch = ch_off[count];
  uint64_t mask = (1ull << A.vb) - 1;
  for (int64_t t = blockIdx.x; t < nch; t += gridDim.x) {
    int64_t lo = ld_chunk_item(ch_off, count, t);
    int64_t r = large[lo];
    int32_t u = A.rows[r];
    const int32_t *row = A.col + A.off[u];
    const int32_t *roww = A.w + A.off[u];
    int64_t dg = A.deg[u];
    const uint64_t *D = A.dkey + A.dlo[r];
    int64_t nD = A.dhi[r] - A.dlo[r];
    const uint64_t *I = A.nkey + A.ilo[r];
    const int64_t *IW = A.nw + A.ilo[r];
    int64_t nI = A.ihi[r] - A.ilo[r];
    uint64_t ubase = (uint64_t)u << A.vb;
    int32_t *ocol = A.tcol + A.tmp_off[r];
    int32_t *ow = A.tw + A.tmp_off[r];
    int64_t c = t - ch_off[lo];
    int64_t p0 = c * TABLE_CHUNK, p1 = p0 + TABLE_CHUNK < dg ? p0 + TABLE_CHUNK : dg;
    for (int64_t p = p0 + threadIdx.x; p < p1; p += blockDim.x) {
      int32_t x = row[p];
      int64_t dless = nD ? lower_bound_u64(D, nD, ubase | (uint64_t)x) : 0;
      if (dless < nD && (D[dless] & mask) == (uint64_t)x) continue;
      int64_t iless = nI ? lower_bound_u64(I, nI, ubase | (uint64_t)x) : 0;
      int64_t o = (p - dless) + iless;
      ocol[o] = x;
      ow[o] = roww[p];
    }
    if (c == 0) {
      for (int64_t k = threadIdx.x; k < nI; k += blockDim.x) {
        int32_t y = (int32_t)(I[k] & mask);
        int64_t rless = lower_bound_i32(row, dg, y);
        int64_t dless = nD ? lower_bound_u64(D, nD, ubase | (uint64_t)y) : 0;
        int64_t o = k + (rless - dless);
        ocol[o] = y;
        ow[o] = (int32_t)IW[k];
      }
    }
  }
}

// Copy the merged long rows back (chunks over the new length) and record
// the new degree and any relocation.
__global__ void __launch_bounds__(256) k_merge_chunks_copy(MergeArgs A, const int32_t *large,
                                                           const int32_t *count_p, const int64_t *ch_off) {
  ld_after_previous();
  int64_t count = *count_p;
  int64_t nch = ch_off[count];
  for (int64_t t = blockIdx.x; t < nch; t += gridDim.x) {
    int64_t lo = ld_chunk_item(ch_off, count, t);
    int64_t r = large[lo];
    int64_t L = A.len[r];
    int64_t c = t - ch_off[lo];
    int64_t x0 = c * TABLE_CHUNK, x1 = x0 + TABLE_CHUNK < L ? x0 + TABLE_CHUNK : L;
    int64_t b = A.tmp_off[r], o = A.dst[r];
    for (int64_t x = x0 + threadIdx.x; x < x1; x += blockDim.x) {
      A.col[o + x] = A.tcol[b + x];
      A.w[o + x] = A.tw[b + x];
    }
    if (c == 0 && threadIdx.x == 0) finish_row(A, r, A.rows[r], L);
  }
}

// ----- rebuild with fresh slack (when a row outgrows its capacity)
__global__ void k_row_lengths(const int32_t *deg, int64_t n, int64_t *len) {
  ld_after_previous();
  for (int64_t i = ld_gtid(); i < n; i += ld_gstride()) len[i] = deg[i];
}
__global__ void k_touched_lengths(const int32_t *rows, const int64_t *nrows_p, const int64_t *rlen, int64_t *len) {
  ld_after_previous();
  for (int64_t r = ld_gtid(); r < *nrows_p; r += ld_gstride()) len[rows[r]] = rlen[r];
}
__global__ void k_capacity(const int64_t *len, int64_t n, double slack, int min_slack, int64_t *cap) {
  ld_after_previous();
  for (int64_t i = ld_gtid(); i < n; i += ld_gstride()) {
    int64_t L = len[i];
    int64_t extra = (int64_t)((double)L * slack);
    if (extra < min_slack) extra = min_slack;
    cap[i] = L + extra;
  }
}
// rowsrc[i] = index into the touched-row list, or -1
__global__ void k_copy_rows_rebuild(int64_t n, const int64_t *old_off, const int32_t *old_deg, const int32_t *old_col,
                                    const int32_t *old_w, const int32_t *rowsrc, const int64_t *tmp_off,
                                    const int64_t *rlen, const int32_t *tcol, const int32_t *tw,
                                    const int64_t *new_off, int32_t *new_deg, int32_t *new_col, int32_t *new_w) {
  ld_after_previous();
  int lane = threadIdx.x & 31;
  int64_t warp = ld_gtid() >> 5, nwarps = ld_gstride() >> 5;
  for (int64_t u = warp; u < n; u += nwarps) {
    int32_t r = rowsrc ? rowsrc[u] : -1;
    const int32_t *sc, *sw;
    int64_t L;
    if (r >= 0) { sc = tcol + tmp_off[r]; sw = tw + tmp_off[r]; L = rlen[r]; }
    else { sc = old_col + old_off[u]; sw = old_w + old_off[u]; L = old_deg[u]; }
    int64_t o = new_off[u];
    for (int64_t x = lane; x < L; x += 32) { new_col[o + x] = sc[x]; new_w[o + x] = sw[x]; }
    if (lane == 0) new_deg[u] = (int32_t)L;
  }
}
__global__ void k_set_rcap(const int64_t *cap, int64_t n, int32_t *rcap) {
  ld_after_previous();
  for (int64_t i = ld_gtid(); i < n; i += ld_gstride()) rcap[i] = (int32_t)cap[i];
}
__global__ void k_rowsrc(const int32_t *rows, const int64_t *nrows_p, int32_t *rowsrc) {
  ld_after_previous();
  for (int64_t r = ld_gtid(); r < *nrows_p; r += ld_gstride()) rowsrc[rows[r]] = (int32_t)r;
}

// ----- marking (uses C^{t-1}, and K^{t-1}, Sigma^{t-1}, 2m^{t-1} for DS)
__global__ void k_mark_ds_del(const uint64_t *dkey, int64_t nd, int vb, const int32_t *C, uint8_t *dV, uint8_t *dE,
                              uint8_t *dCf) {
  ld_after_previous();
  uint64_t mask = (1ull << vb) - 1;
  for (int64_t i = ld_gtid(); i < nd; i += ld_gstride()) {
    int32_t u = (int32_t)(dkey[i] >> vb), v = (int32_t)(dkey[i] & mask);
    if (C[u] == C[v]) { dV[u] = 1; dE[u] = 1; dCf[C[v]] = 1; }
  }
}

// (src, C[dst]) keys of the cross-community insertions; same-community
// arcs get the key ~0 and sort last.
__global__ void k_ds_keys(const uint64_t *ikey, const int64_t *iw, int64_t ni, int vb, const int32_t *C,
                          uint64_t *okey, int64_t *ow) {
  ld_after_previous();
  uint64_t mask = (1ull << vb) - 1;
  for (int64_t i = ld_gtid(); i < ni; i += ld_gstride()) {
    int32_t u = (int32_t)(ikey[i] >> vb), v = (int32_t)(ikey[i] & mask);
    if (C[u] != C[v]) { okey[i] = ((uint64_t)u << vb) | (uint64_t)C[v]; ow[i] = iw[i]; }
    else { okey[i] = ~0ull; ow[i] = 0; }
  }
}

// Sorted unique (src, c) pairs with summed weights H; warp per source run:
// c* = argmax 2m*H[c] - K_src*Sigma_c, ties to the lowest c.
__global__ void k_ds_best(const uint64_t *pkey, const int64_t *pw, const int64_t *np_p, int vb, const int64_t *K,
                          const int64_t *Sig, const DevCounters *cnt, uint8_t *dV, uint8_t *dE, uint8_t *dCf,
                          const int32_t *gid0, const int64_t *m2g) {
  ld_after_previous();
  int64_t np = *np_p;
  uint64_t mask = (1ull << vb) - 1;
  for (int64_t i = ld_gtid(); i < np; i += ld_gstride()) {
    if (pkey[i] == ~0ull) continue;
    uint64_t src = pkey[i] >> vb;
    if (i > 0 && (pkey[i - 1] >> vb) == src) continue;  // only the run head works
    int64_t m2 = gid0 ? m2g[gid0[src]] : cnt->m2;  // 2m^{t-1} of the source's graph
    int32_t best = -1;
    i128 bv = 0;
    for (int64_t j = i; j < np && pkey[j] != ~0ull && (pkey[j] >> vb) == src; j++) {
      int32_t c = (int32_t)(pkey[j] & mask);
      i128 v = (i128)m2 * pw[j] - (i128)K[src] * Sig[c];
      if (ld_better(v, c, bv, best)) { bv = v; best = c; }
    }
    dV[src] = 1; dE[src] = 1; dCf[best] = 1;
  }
}

// Neighbours of G^t of the vertices with dE become affected.  Rows by
// windows of up to 32 per warp (see window_rows), the flagged ones flattened; flagged rows above
// ROWS_BIG arcs are listed for the chunked kernel (a warp per vertex of the
// graph spent its time on unflagged rows and on the longest hub: R-MAT 20,
// 15,700 edges: 580 -> 19 us, and 14 us for the hubs' chunks).
__global__ void __launch_bounds__(256) k_ds_expand_neighbours(const uint8_t *dE, int64_t n, const int64_t *off,
                                                              const int32_t *deg, const int32_t *col, uint8_t *dV,
                                                              int32_t *big, DevCounters *cnt, int rows) {
  ld_after_previous();
  const int lane = threadIdx.x & 31;
  int64_t warp = ld_gtid() >> 5, nw = ld_gstride() >> 5;
  for (int64_t r = warp * rows; r < n; r += nw * rows) {  // warp-uniform
    int64_t i = r + lane;
    bool f = lane < rows && i < n && dE[i];
    if (!__any_sync(LD_FULL, f)) continue;
    int d = f ? deg[i] : 0;
    if (d > ROWS_BIG) {
      big[atomicAdd(&cnt->big_count, 1)] = (int32_t)i;
      d = 0;
    }
    int e = ld_warp_incl_i32(d), s = e - d, total = __shfl_sync(LD_FULL, e, 31);
    int64_t ab = (f ? off[i] : 0) - s;
    for (int x0 = 0; x0 < total; x0 += 128) {  // warp-uniform
      int k[4];
      int32_t j[4];
      ld_window_rows<4>(s, x0, lane, k);
#pragma unroll
      for (int u = 0; u < 4; u++) {
        int x = x0 + 32 * u + lane;
        int64_t a = __shfl_sync(LD_FULL, ab, k[u]) + x;
        j[u] = x < total ? col[a] : -1;
      }
#pragma unroll
      for (int u = 0; u < 4; u++)
        if (j[u] >= 0) dV[j[u]] = 1;
    }
  }
}
__global__ void __launch_bounds__(256) k_ds_expand_big(const int32_t *big, const int64_t *ch_off, const int64_t *off,
                                                       const int32_t *deg, const int32_t *col, uint8_t *dV,
                                                       const DevCounters *cnt) {
  ld_after_previous();
  const int64_t count = cnt->big_count;
  if (count == 0) return;
  const int64_t nch = ch_off[count];
  for (int64_t t = blockIdx.x; t < nch; t += gridDim.x) {  // block-uniform
    int64_t k = ld_chunk_item(ch_off, count, t);
    int32_t i = big[k];
    int64_t x0 = (t - ch_off[k]) * TABLE_CHUNK, b = off[i] + x0;
    int len = (int)(deg[i] - x0 < TABLE_CHUNK ? deg[i] - x0 : TABLE_CHUNK);
#pragma unroll 4
    for (int x = threadIdx.x; x < len; x += 256) dV[col[b + x]] = 1;
  }
}
__global__ void k_ds_expand_communities(const uint8_t *dCf, const int32_t *C, int64_t n, uint8_t *dV) {
  ld_after_previous();
  for (int64_t i = ld_gtid(); i < n; i += ld_gstride())
    if (dCf[C[i]]) dV[i] = 1;
}

// Alg. update (updateWeights, updateChanges) on both arc lists, with the DF
// marking (dV non-null; it reads C^{t-1} only).  The arcs of giant communities
// meet on a few words of Sigma and Delta Sigma: a block first adds them up in a
// small shared table (an arc whose slot another community holds adds
// directly), the lanes of the warp's first community in one add
// (R-MAT 20, 1.6M edges: 361 -> 138 us).
constexpr int UPD_SLOTS = 256;
__global__ void __launch_bounds__(256) k_update_weights(const uint64_t *dkey, const int64_t *dw, int64_t nd,
                                                        const uint64_t *ikey, const int64_t *iw, int64_t ni, int vb,
                                                        const int32_t *C, int64_t *K, int64_t *Sig, int64_t *dSig,
                                                        DevCounters *cnt, const int32_t *gid0, int64_t *m2g,
                                                        uint8_t *dV) {
  ld_after_previous();
  __shared__ int32_t hk[UPD_SLOTS];
  __shared__ unsigned long long hs[UPD_SLOTS], hw[UPD_SLOTS];
  for (int t = threadIdx.x; t < UPD_SLOTS; t += 256) { hk[t] = -1; hs[t] = 0; hw[t] = 0; }
  __syncthreads();
  if (ld_gtid() == 0) cnt->m2 += cnt->batch_dw;
  const int lane = threadIdx.x & 31;
  const uint64_t mask = (1ull << vb) - 1;
  auto add = [&](int32_t c, int64_t s, int64_t w) {
    int t = (int)(ld_hash32((uint32_t)c) & (UPD_SLOTS - 1));
    int32_t k = hk[t];
    if (k == -1) {
      k = atomicCAS(&hk[t], -1, c);
      if (k == -1) k = c;
    }
    if (k == c) {
      atomicAdd(&hs[t], (unsigned long long)s);
      atomicAdd(&hw[t], (unsigned long long)w);
    } else {
      atomicAdd((unsigned long long *)&Sig[c], (unsigned long long)s);
      atomicAdd((unsigned long long *)&dSig[c], (unsigned long long)w);
    }
  };
  for (int64_t i0 = (ld_gtid() & ~31ll); i0 < nd + ni; i0 += ld_gstride()) {  // warp-uniform trip count
    int64_t i = i0 + lane;
    bool has = i < nd + ni;
    int64_t s = 0, w = 0;
    int32_t u = 0, c = -1;
    if (has) {
      bool del = i < nd;
      uint64_t k = del ? dkey[i] : ikey[i - nd];
      w = del ? dw[i] : iw[i - nd];
      u = (int32_t)(k >> vb);
      c = C[u];
      s = del ? -w : w;
      atomicAdd((unsigned long long *)&K[u], (unsigned long long)s);
      if (dV && del == (c == C[(int32_t)(k & mask)])) dV[u] = 1;
    }
    int32_t c0 = __shfl_sync(LD_FULL, c, 0);
    bool first = c == c0;
    if (__popc(__ballot_sync(LD_FULL, first)) > 4) {  // warp-uniform
      int64_t ss = ld_warp_sum_i64(first ? s : 0), sw = ld_warp_sum_i64(first ? w : 0);
      if (lane == 0) add(c0, ss, sw);
      if (has && !first) add(c, s, w);
    } else if (has) {
      add(c, s, w);
    }
    // batched: 2m per graph (a signed sum; the helper adds two's-complement values)
    if (gid0) ld_graph_add_i64(m2g, has, has ? gid0[u] : 0, s);
  }
  __syncthreads();
  for (int t = threadIdx.x; t < UPD_SLOTS; t += 256)
    if (hk[t] >= 0) {
      if (hs[t]) atomicAdd((unsigned long long *)&Sig[hk[t]], hs[t]);
      if (hw[t]) atomicAdd((unsigned long long *)&dSig[hk[t]], hw[t]);
    }
}

// Alg. leidenmk: dS for same-community deletions; dR for same-community
// arcs of either list with dSigma/Sigma > tau_re.
__global__ void k_mark_communities(const uint64_t *dkey, int64_t nd, const uint64_t *ikey, int64_t ni, int vb,
                                   const int32_t *C, const int64_t *Sig, const int64_t *dSig, double tau_re,
                                   uint8_t *dS, uint8_t *dR, DevCounters *cnt) {
  ld_after_previous();
  uint64_t mask = (1ull << vb) - 1;
  for (int64_t i = ld_gtid(); i < nd + ni; i += ld_gstride()) {
    bool del = i < nd;
    uint64_t k = del ? dkey[i] : ikey[i - nd];
    int32_t u = (int32_t)(k >> vb), v = (int32_t)(k & mask);
    int32_t c = C[u];
    if (c != C[v]) continue;
    if (del) dS[c] = 1;
    if ((double)dSig[c] / (double)Sig[c] > tau_re) {
      dR[c] = 1;
      cnt->refine_marks = 1;  // (any value but 0: is there one?)
    }
  }
}
__global__ void k_reset_changes(const uint64_t *dkey, int64_t nd, const uint64_t *ikey, int64_t ni, int vb,
                                const int32_t *C, const uint8_t *dR, int64_t *dSig, const DevCounters *cnt) {
  ld_after_previous();
  if (cnt->refine_marks == 0) return;
  for (int64_t i = ld_gtid(); i < nd + ni; i += ld_gstride()) {
    uint64_t k = i < nd ? dkey[i] : ikey[i - nd];
    int32_t c = C[(int32_t)(k >> vb)];
    if (dR[c]) dSig[c] = 0;
  }
}

int bits_for(int64_t n) {
  int b = 1;
  while (((int64_t)1 << b) < n) b++;
  return b;
}

template <typename T>
cudaError_t grow(leiden_handle *h, T **p, int64_t count) {
  void *q = nullptr;
  cudaError_t e = cudaMalloc(&q, (size_t)std::max<int64_t>(count, 1) * sizeof(T));
  if (e != cudaSuccess) return e;
  h->owned.push_back(q);
  *p = (T *)q;
  return cudaSuccess;
}

void release(leiden_handle *h, void *p) {
  if (!p) return;
  for (auto &q : h->owned)
    if (q == p) { cudaFree(q); q = nullptr; }
}

// Buffers that grow with the batch.  A larger set is allocated in full
// before the old one is freed: a failed allocation leaves the handle with its
// old, valid buffers and capacity (and frees what it got).
cudaError_t ensure_batch(leiden_handle *h, int64_t edges) {
  BatchBuffers &b = h->b;
  if (b.cap_edges > 0 && edges <= b.cap_edges) return cudaSuccess;  // the first call always allocates
  // geometric growth: a freed buffer synchronises the whole device, which
  // stalls every other stream of a serving process
  int64_t cap = std::max<int64_t>({edges, 2 * b.cap_edges, (int64_t)1024});
  int64_t arcs = 2 * cap;
  int64_t rows = std::min<int64_t>(2 * arcs, h->n) + 1;
  BatchBuffers nb = b;
  void **slot[] = {(void **)&nb.dkey, (void **)&nb.dkey_alt, (void **)&nb.ikey, (void **)&nb.ikey_alt,
                   (void **)&nb.iw, (void **)&nb.iw_alt, (void **)&nb.dw, (void **)&nb.flag, (void **)&nb.pos,
                   (void **)&nb.ins_state, (void **)&nb.ins_pos, (void **)&nb.rows, (void **)&nb.row_dlo,
                   (void **)&nb.row_dhi, (void **)&nb.row_ilo, (void **)&nb.row_ihi, (void **)&nb.row_len,
                   (void **)&nb.row_tmp_off, (void **)&nb.row_dst, (void **)&nb.row_newcap, (void **)&nb.row_olddeg,
                   (void **)&nb.row_large, (void **)&nb.row_mid, (void **)&nb.row_warp, (void **)&nb.ds_key, (void **)&nb.ds_key_alt,
                   (void **)&nb.ds_w, (void **)&nb.ds_w_alt, (void **)&nb.ds_ukey, (void **)&nb.ds_uw};
  // dkey, dkey_alt, iw, iw_alt, flag and pos hold the deletion and insertion
  // arcs of one sort together (2 * arcs); ikey, ikey_alt and iw_alt's unique part
  // at most one kind
  size_t bytes[] = {16 * (size_t)arcs, 16 * (size_t)arcs, 8 * (size_t)arcs, 8 * (size_t)arcs, 16 * (size_t)arcs,
                    16 * (size_t)arcs, 8 * (size_t)arcs, 4 * (size_t)(2 * arcs + 1), 8 * (size_t)(2 * arcs + 1),
                    4 * (size_t)arcs, 8 * (size_t)arcs, 4 * (size_t)rows, 4 * (size_t)rows, 4 * (size_t)rows,
                    4 * (size_t)rows, 4 * (size_t)rows, 8 * (size_t)(rows + 1), 8 * (size_t)(rows + 1),
                    8 * (size_t)(rows + 1), 4 * (size_t)(rows + 1), 4 * (size_t)(rows + 1), 4 * (size_t)(rows + 1),
                    4 * (size_t)(rows + 1), 4 * (size_t)(rows + 1), 8 * (size_t)arcs, 8 * (size_t)arcs, 8 * (size_t)arcs, 8 * (size_t)arcs,
                    8 * (size_t)arcs, 8 * (size_t)arcs};
  constexpr int NB = sizeof(slot) / sizeof(slot[0]);
  static_assert(NB == sizeof(bytes) / sizeof(bytes[0]), "one size per batch buffer");
  void *fresh[NB] = {};
  cudaError_t e = cudaSuccess;
  for (int k = 0; k < NB && e == cudaSuccess; k++) e = cudaMalloc(&fresh[k], bytes[k]);
  if (e == cudaSuccess && !b.row_bits) {
    int64_t words = (h->n + 31) / 32;
    e = grow(h, &nb.row_bits, words);
    if (e == cudaSuccess)
      e = cudaMemsetAsync(nb.row_bits, 0, (size_t)std::max<int64_t>(words, 1) * sizeof(uint32_t), h->stream);
  }
  if (e != cudaSuccess) {
    cudaGetLastError();
    for (void *q : fresh)
      if (q) cudaFree(q);
    return e;
  }
  void *old[NB];
  for (int k = 0; k < NB; k++) {
    old[k] = *slot[k];
    *slot[k] = fresh[k];
    h->owned.push_back(fresh[k]);
  }
  for (void *q : old) release(h, q);
  nb.counts = h->dcnt->bcounts;
  nb.cap_edges = cap;
  b = nb;
  return cudaSuccess;
}

cudaError_t ensure_scan_tmp(leiden_handle *h, size_t bytes) {
  if (bytes <= h->scan_tmp_bytes) return cudaSuccess;
  void *p = nullptr;
  cudaError_t e = cudaMalloc(&p, bytes);
  if (e != cudaSuccess) { cudaGetLastError(); return e; }  // the old scratch stays
  release(h, h->scan_tmp);
  h->owned.push_back(p);
  h->scan_tmp = p;
  h->scan_tmp_bytes = bytes;
  return cudaSuccess;
}

cudaError_t ensure_tmp_rows(leiden_handle *h, int64_t arcs) {
  BatchBuffers &b = h->b;
  if (arcs <= b.tmp_cap) return cudaSuccess;
  int64_t cap = std::max<int64_t>({arcs, 2 * b.tmp_cap, (int64_t)4096});
  int32_t *col = nullptr, *w = nullptr;
  cudaError_t e = cudaMalloc((void **)&col, (size_t)cap * sizeof(int32_t));
  if (e == cudaSuccess) e = cudaMalloc((void **)&w, (size_t)cap * sizeof(int32_t));
  if (e != cudaSuccess) {  // the old buffers stay
    cudaGetLastError();
    if (col) cudaFree(col);
    return e;
  }
  release(h, b.tmp_col);
  release(h, b.tmp_w);
  h->owned.push_back(col);
  h->owned.push_back(w);
  b.tmp_col = col;
  b.tmp_w = w;
  b.tmp_cap = cap;
  return cudaSuccess;
}

leiden_status fail(leiden_handle *h, leiden_status st, const std::string &msg) {
  h->err = msg;
  return st;
}

}  // namespace

// Rebuild G^t with new capacities: rows keep their content (touched rows
// come from the merge buffer).
static leiden_status rebuild_graph(leiden_handle *h, int64_t nrows_host, const int64_t *nrows_dev) {
  cudaStream_t s = h->stream;
  int64_t n = h->n;
  BatchBuffers &b = h->b;
  int64_t *len = h->lbuf0, *cap = h->lbuf1;
  ld_note_launch(), launch_after(k_row_lengths, grid_for(n, TB), TB, s, h->g_deg, n, len);
  ld_note_launch(), launch_after(k_touched_lengths, grid_for(nrows_host, TB), TB, s, b.rows, nrows_dev, b.row_len, len);
  ld_note_launch(), launch_after(k_capacity, grid_for(n, TB), TB, s, len, n, h->p.slack, h->p.min_slack, cap);
  int64_t *new_off = nullptr;
  if (grow(h, &new_off, n + 1) != cudaSuccess) return fail(h, LEIDEN_ERR_OOM, "rebuild: offsets");
  if (ensure_scan_tmp(h, scan_tmp_bytes(n + 1)) != cudaSuccess) return fail(h, LEIDEN_ERR_OOM, "scan tmp");
  exclusive_scan_i64(cap, new_off, n, h->scan_tmp, s);
  int64_t used = 0;
  cudaMemcpyAsync(&used, new_off + n, sizeof(int64_t), cudaMemcpyDeviceToHost, s);
  cudaStreamSynchronize(s);
  int64_t total = used + spill_arena_size(used, h->p.arena_log2);
  int32_t *new_col = nullptr, *new_w = nullptr, *new_deg = nullptr;
  if (grow(h, &new_col, total) != cudaSuccess || grow(h, &new_w, total) != cudaSuccess ||
      grow(h, &new_deg, n) != cudaSuccess)
    return fail(h, LEIDEN_ERR_OOM, "rebuild: arcs");
  ld_note_launch(), launch_after(k_set_rcap, grid_for(n, TB), TB, s, cap, n, h->g_rcap);
  cudaMemcpyAsync(&h->dcnt->arena_used, &used, sizeof(int64_t), cudaMemcpyHostToDevice, s);
  int32_t *rowsrc = h->ibuf2;
  launch_fill_i32(rowsrc, -1, n, s);
  ld_note_launch(), launch_after(k_rowsrc, grid_for(nrows_host, TB), TB, s, b.rows, nrows_dev, rowsrc);
  ld_note_launch(), launch_after(k_copy_rows_rebuild, grid_for(n * 32, TB), TB, s, n, h->g_off, h->g_deg, h->g_col,
                                 h->g_w, rowsrc, b.row_tmp_off, b.row_len, b.tmp_col, b.tmp_w, new_off, new_deg,
                                 new_col, new_w);
  cudaStreamSynchronize(s);
  release(h, h->g_off);
  release(h, h->g_col);
  release(h, h->g_w);
  release(h, h->g_deg);
  h->g_off = new_off;
  h->g_col = new_col;
  h->g_w = new_w;
  h->g_deg = new_deg;
  h->g_cap = total;
  return LEIDEN_OK;
}

leiden_status batch_apply_and_mark(leiden_handle *h, const leiden_edge *d_del, int64_t n_del,
                                   const leiden_edge *d_ins, int64_t n_ins, int mode) {
  cudaStream_t s = h->stream;
  int64_t n = h->n;
  BatchBuffers &b = h->b;
  int vb = bits_for(n);
  DevCounters *cnt = h->dcnt;
  if (ensure_batch(h, std::max(n_del, n_ins)) != cudaSuccess) return fail(h, LEIDEN_ERR_OOM, "batch buffers");
  int64_t nda = 2 * n_del, nia = 2 * n_ins;
  if (ensure_scan_tmp(h, std::max(sort_tmp_bytes(nda + nia), scan_tmp_bytes(std::max(n, nda + nia) + 1))) != cudaSuccess)
    return fail(h, LEIDEN_ERR_OOM, "scan tmp");
  // [0] nd, [1] ni, [2] new arcs, [3] touched rows, [4] merge-buffer arcs (cleared
  // with the call's counters): they stay on the device until the one host read
  // below; launches are sized by the bounds nda, nia
  int64_t *counts = b.counts;
  uint64_t *DK = b.dkey_alt, *IK = b.ikey_alt;
  int64_t *IW = b.iw_alt, *DW = b.dw;
  uint64_t *NK = b.ikey;  // new insertions, compacted in sorted order
  int64_t *NW = b.iw;      // (the sorted raw arcs there are consumed by then)
  BatchGraph G{n, h->g_off, h->g_deg, h->g_rcap, h->g_col, h->g_w, h->gid0, h->g_cap, h->p.slack, h->p.min_slack,
               h->tune.block_max, vb};
  RowPlan P{b.row_dlo, b.row_dhi, b.row_ilo, b.row_ihi, b.row_len, b.row_dst, b.row_newcap, b.row_olddeg, b.row_large,
            b.row_mid, b.row_warp};
  if (nda + nia == 0) {
  } else if (nda + nia <= SMALL_ARCS) {
    SmallOut O{DK, IK, NK, DW, IW, NW, b.ins_pos, b.row_tmp_off, b.ins_state, b.rows};
    ld_note_launch(), launch_after(k_small_batch, 1, 1024, s, G, P, O, d_del, (int)n_del, d_ins, (int)n_ins, cnt);
  } else {
    // one sort of both: the deletion arcs sorted in dkey[0, nda), the
    // insertion arcs and their weights in dkey, iw [nda, nda + nia)
    ld_note_launch(), launch_after(k_expand, grid_for(n_del + n_ins, TB), TB, s, d_del, n_del, d_ins, n_ins, n, vb,
                                   b.dkey, b.iw, cnt, h->gid0);
    radix_sort_u64(b.dkey, b.dkey_alt, b.iw, b.iw_alt, nda + nia, 2 * vb + 1, h->scan_tmp, s);
    ld_note_launch(), launch_after(k_head_flags, grid_for(nda + nia, TB), TB, s, b.dkey, nda + nia, b.flag, IW, nia);
    exclusive_scan_i32_to_i64(b.flag, b.pos, nda + nia, h->scan_tmp, s);
    ld_note_launch(), launch_after(k_unique_batch, grid_for(nda + nia, TB), TB, s, b.dkey, b.iw, nda, nia, b.flag,
                                   b.pos, (1ull << (2 * vb)) - 1, DK, IK, IW, counts);
    // deletions must exist (stored weight -> DW); insertions: existing or new
    ld_note_launch(), launch_after(k_check_batch, grid_for(nda + nia, TB), TB, s, G, DK, IK, IW, counts, nda, nia, DW,
                                   b.ins_state, b.ins_pos, b.flag, cnt);
    if (nia > 0) {
      exclusive_scan_i32_to_i64(b.flag, b.pos, nia, h->scan_tmp, s);
      ld_note_launch(), launch_after(k_compact_new, grid_for(nia, TB), TB, s, IK, IW, nia, b.flag, b.pos, NK, NW,
                                     counts + 2);
    }
    // rows whose structure changes: sources of deletions and of new arcs
    int64_t nb = std::min<int64_t>(n, nda + nia);  // bound on the touched rows
    ld_note_launch(), launch_after(k_touched_rows, grid_for(nda + nia, TB), TB, s, DK, counts + 0, NK, counts + 2, vb,
                                   b.row_bits, b.rows, counts + 3);
    ld_note_launch(), launch_after(k_row_plan, grid_for(nb, TB), TB, s, G, P, b.rows, counts + 3, nb, DK, counts + 0,
                                   NK, counts + 2, b.row_bits, counts + 4, cnt);
    exclusive_scan_i64(b.row_len, b.row_tmp_off, nb, h->scan_tmp, s);
  }
  // the one host read before the graph changes: counts, validation, overflow
  cudaMemcpyAsync(h->hcnt, h->dcnt, sizeof(DevCounters), cudaMemcpyDeviceToHost, s);
  cudaStreamSynchronize(s);
  if (h->hcnt->error)
    return fail(h, LEIDEN_ERR_BATCH, h->hcnt->error == 2 ? "batch deletes an edge that does not exist"
                                                         : "batch edge out of range, self-loop or weight <= 0");
  const int64_t *hc = h->hcnt->bcounts;
  int64_t nd = hc[0], ni = hc[1], nn = hc[2], nrows = hc[3], tmp_total = hc[4];
  bool overflow = nrows > 0 && h->hcnt->overflow != 0;
  if (ensure_tmp_rows(h, tmp_total) != cudaSuccess) return fail(h, LEIDEN_ERR_OOM, "merge buffer");
  // ---- apply: from here on the handle changes
  if (ni > nn) ld_note_launch(), launch_after(k_add_existing, grid_for(ni, TB), TB, s, b.ins_pos, b.ins_state, IW, ni,
                                              h->g_w);
  if (nrows > 0) {
    if (!overflow) {
      MergeArgs M{b.rows, counts + 3, vb, DK, NK, NW, b.row_dlo, b.row_dhi, b.row_ilo, b.row_ihi, b.row_len,
                  b.row_tmp_off, h->g_off, h->g_deg, h->g_col, h->g_w, b.tmp_col, b.tmp_w,
                  b.row_dst, b.row_newcap, h->g_off, h->g_rcap};
      // the three row classes write disjoint rows and merge-buffer ranges:
      // short rows on the handle's stream, mid rows and long rows on its
      // side streams, joined before the marking below
      const bool some_mid = h->hcnt->mid_count > 0, some_long = h->hcnt->large_count > 0,
                 some_warp = h->hcnt->warp_count > 0,
                 some_small = nrows > (int64_t)h->hcnt->mid_count + h->hcnt->large_count + h->hcnt->warp_count;
      bool fork = (some_mid || some_long) && h->tune.overlap && side_streams(h);
      cudaStream_t smid = s, slong = s;
      if (fork) {
        cudaEventRecord(h->fork_ev, s);
        smid = h->side[0];
        slong = h->side[1];
        if (some_mid) cudaStreamWaitEvent(smid, h->fork_ev, 0);
        if (some_long) cudaStreamWaitEvent(slong, h->fork_ev, 0);
      }
      if (some_warp)
        ld_note_launch(), launch_after(k_merge_warp,
                                       grid_for((h->hcnt->warp_count + MERGE_WARPS - 1) / MERGE_WARPS, 1, h->sm_count * 7),
                                       MERGE_WARPS * 32, s, M, b.row_warp, &cnt->warp_count);
      if (some_small)
        ld_note_launch(), launch_after(k_merge_small,
                                       grid_for((nrows + MERGE_WARPS - 1) / MERGE_WARPS, 1, h->sm_count * 16),
                                       MERGE_WARPS * 32, s, M);
      if (some_mid) {
        kt_begin(h, KT_MERGE_MID, smid);
        ld_note_launch(), launch_after(k_merge_mid, h->sm_count * 7, 256, smid, M, b.row_mid, &cnt->mid_count,  // 32 KB: 7 per SM
                                                                        &cnt->xk_bytes[2]);
        kt_end(h, smid);
      }
      if (some_long) {
        // long rows: chunks over the old row, then chunks over the new row
        int32_t *large = b.row_large;
        const int32_t *nlarge = &cnt->large_count;
        launch_table_plan(large, nlarge, b.row_olddeg, nullptr, INT64_MAX, h->lbuf0, h->lbuf1, slong);
        ld_note_launch(), launch_after(k_merge_chunks_write, h->sm_count * 16, 256, slong, M, large, nlarge, h->lbuf1);
        launch_table_plan(large, nlarge, nullptr, b.row_tmp_off, INT64_MAX, h->lbuf2, h->lbuf3, slong);
        ld_note_launch(), launch_after(k_merge_chunks_copy, h->sm_count * 16, 256, slong, M, large, nlarge, h->lbuf3);
      }
      if (fork) {
        for (int k = 0; k < 2; k++) {
          if (!(k == 0 ? some_mid : some_long)) continue;
          cudaEventRecord(h->join_ev[k], h->side[k]);
          cudaStreamWaitEvent(s, h->join_ev[k], 0);
        }
      }
    } else {
      ld_note_launch(), launch_after(k_merge_rows, grid_for(nrows * 32, TB), TB, s, b.rows, counts + 3, vb, DK, NK, NW,
                                     b.row_dlo, b.row_dhi, b.row_ilo, b.row_ihi, b.row_tmp_off, h->g_off, h->g_deg,
                                     h->g_col, h->g_w, b.tmp_col, b.tmp_w);
      leiden_status st = rebuild_graph(h, nrows, counts + 3);
      h->stats.rebuilds++;
      if (st != LEIDEN_OK) {
        h->broken = true;  // the batch was applied in part
        return st;
      }
    }
  }
  h->g_arcs = h->g_arcs - nd + nn;
  h->stats.batch_arcs = nd + ni;
  h->batch_dw = h->hcnt->batch_dw;
  h->g_maxdeg = std::max(h->g_maxdeg, h->hcnt->max_row);  // (a bound: the longest row may have shrunk)
  h->g_huge_slots += h->hcnt->slot_change;
  // ---- affected vertices (C^{t-1}; DS also K^{t-1}, Sigma^{t-1}, 2m^{t-1}; DF
  // with the weights below), dS and dR (the three flag arrays are neighbours)
  uint8_t *dV = h->dV;
  size_t flags = (size_t)(h->dR - h->dV) + (size_t)n;
  cudaMemsetAsync(dV, 0, flags, s);
  if (mode == LEIDEN_ND) cudaMemsetAsync(dV, 1, (size_t)n, s);
  if (mode == LEIDEN_DS) {
    {
      cudaMemsetAsync(h->dE, 0, (size_t)n, s);
      cudaMemsetAsync(h->dCf, 0, (size_t)n, s);
      if (nd > 0) ld_note_launch(), launch_after(k_mark_ds_del, grid_for(nd, TB), TB, s, DK, nd, vb, h->C, dV, h->dE,
                                                 h->dCf);
      if (ni > 0) {
        // H of each insertion source: (src, C[dst]) pairs, sorted, runs summed
        ld_note_launch(), launch_after(k_ds_keys, grid_for(ni, TB), TB, s, IK, IW, ni, vb, h->C, b.ds_key, b.ds_w);
        radix_sort_u64(b.ds_key, b.ds_key_alt, b.ds_w, b.ds_w_alt, ni, 64, h->scan_tmp, s);
        ld_note_launch(), launch_after(k_head_flags, grid_for(ni, TB), TB, s, b.ds_key, ni, b.flag, nullptr, 0);
        exclusive_scan_i32_to_i64(b.flag, b.pos, ni, h->scan_tmp, s);
        cudaMemsetAsync(b.ds_uw, 0, (size_t)ni * sizeof(int64_t), s);
        ld_note_launch(), launch_after(k_unique, grid_for(ni, TB), TB, s, b.ds_key, b.ds_w, ni, b.flag, b.pos,
                                       b.ds_ukey, b.ds_uw);
        ld_note_launch(), launch_after(k_ds_best, grid_for(ni, TB), TB, s, b.ds_ukey, b.ds_uw, b.pos + ni, vb, h->K,
                                       h->Sig, cnt, dV, h->dE, h->dCf, h->gid0, h->gc.m2);
      }
      cudaMemsetAsync(&cnt->big_count, 0, sizeof(int32_t), s);
      const int wr = window_rows(h);
      ld_note_launch(), launch_after(k_ds_expand_neighbours, window_grid(n, wr), TB, s, h->dE, n, h->g_off, h->g_deg,
                                     h->g_col, dV, h->ibuf0, cnt, wr);
      launch_table_plan(h->ibuf0, &cnt->big_count, h->g_deg, nullptr, 1, h->lbuf0, h->lbuf1, s);
      ld_note_launch(), launch_after(k_ds_expand_big, h->sm_count * 8, TB, s, h->ibuf0, h->lbuf1, h->g_off, h->g_deg,
                                     h->g_col, dV, cnt);
      ld_note_launch(), launch_after(k_ds_expand_communities, grid_for(n, TB), TB, s, h->dCf, h->C, n, dV);
    }
  }
  // ---- Alg. update, then Alg. leidenmk (dS, dR; reset dSigma of refined)
  if (nd + ni > 0) {
    ld_note_launch(), launch_after(k_update_weights, grid_for(nd + ni, TB), TB, s, DK, DW, nd, IK, IW, ni, vb, h->C,
                                   h->K, h->Sig, h->dSig, cnt, h->gid0, h->gc.m2, mode == LEIDEN_DF ? dV : nullptr);
    ld_note_launch(), launch_after(k_mark_communities, grid_for(nd + ni, TB), TB, s, DK, nd, IK, ni, vb, h->C, h->Sig,
                                   h->dSig, h->p.tau_refine, h->dS, h->dR, cnt);
    ld_note_launch(), launch_after(k_reset_changes, grid_for(nd + ni, TB), TB, s, DK, nd, IK, ni, vb, h->C, h->dR,
                                   h->dSig, cnt);
  }
  // Algorithmic bytes of the batch phase: the edge triples read (12 B per
  // edge); per raw arc its expansion and sort (48 B: key and weight written,
  // then read and written once more) and deduplication (24 B); per unique
  // arc the existence check or classification (16 B) and the updates of K,
  // Sigma, Delta Sigma, 2m and the flags (40 B); per touched row its plan
  // (40 B) and per arc of a merged row its read and write (16 B); a full
  // rebuild copies every arc (16 B); marking: dV (1 B per vertex) plus, for
  // DF, both endpoints' communities per unique arc (16 B), for DS the
  // (source, community) pairs of the insertions and their sort (48 B per
  // arc), dE and the community sweep (7 B per vertex); dS and dR (2 B per
  // vertex).
  int64_t A = nda + nia, U = nd + ni;
  int64_t bytes = 12 * (n_del + n_ins) + 72 * A + 56 * U + 40 * nrows + 16 * tmp_total + 3 * n;
  if (overflow) bytes += 16 * h->g_arcs;
  if (mode == LEIDEN_DF) bytes += 16 * U;
  if (mode == LEIDEN_DS) bytes += 48 * ni + 7 * n;
  ph_bytes(h, LEIDEN_PHASE_BATCH, bytes);
  return LEIDEN_OK;
}
