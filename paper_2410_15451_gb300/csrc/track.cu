// Community tracking (Alg. "leidentr"), Sigma recomputation and the terms of
// modularity (Eq. 1).
#include <algorithm>
#include <climits>

#include "internal.h"

namespace {

constexpr int TB = 256;
constexpr uint64_t EMPTY64 = ~0ull;

__device__ __forceinline__ uint64_t hash64(uint64_t k) { return ld_splitmix64(k); }

// Best successor of each old community o: the new community with the largest
// overlap weight W(o, c) = sum of K_i over i with C^{t-1}_i = o and C_i = c,
// ties to the lowest new id.  Most communities keep a strict majority of
// their weight in one new community, and that one is then the unique
// argmax: a candidate (the new label of any member) is checked with two
// coalesced sweeps, and only communities without a majority go through the
// pair table.
// Tracking's per-id arrays in one sweep: best weights -1, best ids INT_MAX,
// candidates -1, use flags and deviant weights 0.
__global__ void k_tr_init(int64_t N, long long *bw, int32_t *bc, long long *ow, int32_t *ob, int32_t *cand,
                          int32_t *used, int64_t *dev) {
  ld_after_previous();
  for (int64_t i = ld_gtid(); i < N; i += ld_gstride()) {
    bw[i] = -1;
    bc[i] = INT_MAX;
    ow[i] = -1;
    ob[i] = INT_MAX;
    cand[i] = -1;
    used[i] = 0;
    dev[i] = 0;
  }
}
__global__ void k_trc_cand(int64_t N, const int32_t *Cold, const int32_t *Cnew, int32_t *cand) {
  ld_after_previous();
  for (int64_t i = ld_gtid(); i < N; i += ld_gstride()) cand[Cold[i]] = Cnew[i];  // any member will do
}
// The weight of an old community is Sigma^{t-1} with K^t (the batch kept it
// current), so only the members whose new label differs from the candidate
// (the deviants) need adding up: ov = tot - deviant weight.
__global__ void k_trc_deviants(int64_t N, const int32_t *Cold, const int32_t *Cnew, const int64_t *K,
                               const int32_t *cand, int64_t *dev) {
  ld_after_previous();
  for (int64_t i = ld_gtid(); i < N; i += ld_gstride()) {
    int32_t o = Cold[i];
    if (Cnew[i] != cand[o]) {
      int64_t k = K[i];
      if (k) atomicAdd((unsigned long long *)&dev[o], (unsigned long long)k);
    }
  }
}
// bw/bc of the majority communities; the others are flagged: 1 = through
// the pair table, 2 = weight 0 (every member has K = 0, e.g. isolated
// vertices): every pair weighs 0, so the lowest new label of a member wins.
__global__ void k_trc_majority(int64_t N, const int32_t *cand, const int64_t *tot, const int64_t *dev,
                               long long *bw, int32_t *bc, int32_t *flag) {
  ld_after_previous();
  for (int64_t o = ld_gtid(); o < N; o += ld_gstride()) {
    int f = 0;
    if (cand[o] >= 0) {
      int64_t ov = tot[o] - dev[o];
      if (tot[o] == 0) { bw[o] = 0; f = 2; }
      else if (2 * ov > tot[o]) { bw[o] = ov; bc[o] = cand[o]; }
      else f = 1;
    }
    flag[o] = f;
  }
}
// Pair weights of the flagged communities.  The table is empty between
// calls; each filled slot is listed (count in *occ) and emptied by its reader.
__global__ void k_trc_insert(int64_t N, const int32_t *Cold, const int32_t *Cnew, const int64_t *K,
                             const int32_t *flag, int32_t *bc, int64_t cap, uint64_t *keys, int64_t *vals,
                             int32_t *list, int32_t *occ) {
  ld_after_previous();
  uint64_t mask = (uint64_t)cap - 1;
  int lane = threadIdx.x & 31;
  for (int64_t base = (ld_gtid() & ~31ll); base < N; base += ld_gstride()) {
    int64_t i = base + lane;
    bool take = false;
    uint64_t key = EMPTY64 - 1 - lane;
    int64_t kw = 0;
    if (i < N) {
      int32_t o = Cold[i];
      int f = flag[o];
      if (f == 1) {
        take = true;
        key = ((uint64_t)(uint32_t)o << 32) | (uint32_t)Cnew[i];
        kw = K[i];
      } else if (f == 2) {
        atomicMin(&bc[o], Cnew[i]);
      }
    }
    if (!__any_sync(LD_FULL, take)) continue;
    uint32_t peers = __match_any_sync(LD_FULL, (unsigned long long)key);
    int64_t sum = ld_group_sum_i64(peers, kw);
    // the warp lists the slots it claims with one atomic on occ
    int32_t claimed = -1;
    if (take && ld_group_leader(peers)) {
      uint64_t sl = hash64(key) & mask;
      for (uint64_t probe = 0; ld_ok(probe <= mask, LD_CHK_PROBE); probe++) {
        unsigned long long k = atomicCAS((unsigned long long *)&keys[sl], EMPTY64, key);
        if (k == EMPTY64) claimed = (int32_t)sl;
        if (k == EMPTY64 || k == key) {
          atomicAdd((unsigned long long *)&vals[sl], (unsigned long long)sum);
          break;
        }
        sl = (sl + 1) & mask;
      }
    }
    uint32_t m = __ballot_sync(LD_FULL, claimed >= 0);
    if (m) {
      int leader = __ffs(m) - 1;
      int32_t p0 = 0;
      if (lane == leader) p0 = atomicAdd(occ, __popc(m));
      p0 = __shfl_sync(LD_FULL, p0, leader);
      if (claimed >= 0) list[p0 + __popc(m & ((1u << lane) - 1u))] = claimed;
    }
  }
}
__global__ void k_trc_best_w(const int32_t *occ, const int32_t *list, const uint64_t *keys, const int64_t *vals,
                             long long *bw) {
  ld_after_previous();
  int64_t m = *occ;
  for (int64_t t = ld_gtid(); t < m; t += ld_gstride()) {
    int32_t sl = list[t];
    atomicMax(&bw[keys[sl] >> 32], (long long)vals[sl]);
  }
}
__global__ void k_trc_best_c(const int32_t *occ, const int32_t *list, uint64_t *keys, int64_t *vals,
                             const long long *bw, int32_t *bc) {
  ld_after_previous();
  int64_t m = *occ;
  for (int64_t t = ld_gtid(); t < m; t += ld_gstride()) {
    int32_t sl = list[t];
    uint64_t key = keys[sl];
    uint32_t o = (uint32_t)(key >> 32);
    if (vals[sl] == bw[o]) atomicMin(&bc[o], (int32_t)(key & 0xffffffffu));
    keys[sl] = EMPTY64;  // leave the table empty
    vals[sl] = 0;
  }
}
// For each new community: among the old communities that picked it, the
// largest overlap, then the lowest old id.
__global__ void k_tr_best_old_w(int64_t N, const int32_t *bc, const long long *bw, long long *ow) {
  ld_after_previous();
  for (int64_t b = ld_gtid(); b < N; b += ld_gstride())
    if (bc[b] != INT_MAX) atomicMax(&ow[bc[b]], bw[b]);
}
__global__ void k_tr_best_old_b(int64_t N, const int32_t *bc, const long long *bw, const long long *ow, int32_t *ob) {
  ld_after_previous();
  for (int64_t b = ld_gtid(); b < N; b += ld_gstride())
    if (bc[b] != INT_MAX && bw[b] == ow[bc[b]]) atomicMin(&ob[bc[b]], (int32_t)b);
}
__global__ void k_tr_new_used(int64_t N, const int32_t *Cnew, int32_t *used) {
  ld_after_previous();
  for (int64_t i = ld_gtid(); i < N; i += ld_gstride()) used[Cnew[i]] = 1;
}
// unmatched[c] (new id used, nobody picked it); free[id] (no old vertex had id)
__global__ void k_tr_flags(int64_t N, const int32_t *new_used, const int32_t *ob, const int32_t *bc,
                           int32_t *unmatched, int32_t *freef) {
  ld_after_previous();
  for (int64_t c = ld_gtid(); c < N; c += ld_gstride()) {
    unmatched[c] = (new_used[c] && ob[c] == INT_MAX) ? 1 : 0;
    freef[c] = bc[c] == INT_MAX ? 1 : 0;
  }
}
__global__ void k_tr_free_list(int64_t N, const int32_t *freef, const int64_t *frank, int32_t *flist) {
  ld_after_previous();
  for (int64_t id = ld_gtid(); id < N; id += ld_gstride())
    if (freef[id]) flist[frank[id]] = (int32_t)id;
}
// The k-th unmatched new community of a graph takes the k-th free id of that
// graph (batched handles: ranks counted from the graph's first id).
__global__ void k_tr_map(int64_t N, const int32_t *new_used, const int32_t *ob, const int64_t *urank,
                         const int64_t *frank, const int32_t *flist, int32_t *map, uint8_t *matched,
                         const int32_t *gid0, const int64_t *voff) {
  ld_after_previous();
  for (int64_t c = ld_gtid(); c < N; c += ld_gstride()) {
    if (!new_used[c]) continue;
    if (ob[c] != INT_MAX) {
      map[c] = ob[c];
      matched[ob[c]] = 1;
    } else if (!gid0) {
      map[c] = flist[urank[c]];
    } else {
      int64_t v0 = voff[gid0[c]];
      map[c] = flist[frank[v0] + urank[c] - urank[v0]];
    }
  }
}
// C^t = map[new label]; Sigma and the member counts follow the vertices
// whose id changes (Sigma^{t-1} is current with K^t, so the others add
// nothing).
__global__ void k_tr_relabel(int64_t N, const int32_t *Cnew, const int32_t *map, const int64_t *K, int32_t *C,
                             int64_t *Sig, int32_t *size) {
  ld_after_previous();
  for (int64_t i = ld_gtid(); i < N; i += ld_gstride()) {
    int32_t c = map[Cnew[i]], o = C[i];
    if (c == o) continue;
    C[i] = c;
    int64_t k = K[i];
    if (k) {
      atomicAdd((unsigned long long *)&Sig[o], (unsigned long long)(-k));
      atomicAdd((unsigned long long *)&Sig[c], (unsigned long long)k);
    }
    atomicSub(&size[o], 1);  // member counts of C^t, for the next call
    atomicAdd(&size[c], 1);
  }
}
__global__ void k_tr_dsig(int64_t N, const uint8_t *matched, int64_t *dSig) {
  ld_after_previous();
  for (int64_t id = ld_gtid(); id < N; id += ld_gstride())
    if (!matched[id]) dSig[id] = 0;
}

// ---------------------------------------------------------------- sums below 2^32
// The same result when 2m < 2^32: a weight and an id share one 64-bit word, so
// "largest weight, then lowest id" is one atomicMax (0 = none).  What else the
// general path spends its time on is left out:
//  - community sizes of C^{t-1} (kept for local moving) say which ids exist, so
//    candidates need no initial value and free ids no sweep over the vertices;
//  - an old community of one vertex has its candidate as its choice whatever
//    its weight (most of an R-MAT graph's ids are isolated vertices);
//  - the new ids are the roots of the last level (C'[c] == c), read in place
//    of marking every vertex's label;
//  - the k-th unmatched community meets the k-th free id through two compact
//    lists built by one pair of kernels;
//  - stores to the words of giant communities, which every warp holds members
//    of, pass a small filter per block first.
// R-MAT 22 (4.19M ids), 64,154 edges: 570 -> 240 us, nine kernels instead of
// twenty-two.
constexpr int TR_FILTER = 512;

__device__ __forceinline__ unsigned long long tr_word(uint32_t w, int32_t id) {
  return ((unsigned long long)w << 32) | (uint32_t)~id;  // never 0: ids are below 2^31
}
__device__ __forceinline__ int32_t tr_id(unsigned long long x) { return (int32_t) ~(uint32_t)x; }

// Candidates, and the zeros that the next kernels add to.  Few blocks with many
// vertices each, so that the filter sees most members of a giant community
// after its first (R-MAT 20, 1M ids: 19.7 us with 2432 blocks, now 7.7); vertices that
// carry their own id (isolated ones, mostly) do not pass through it.
__global__ void __launch_bounds__(256) k_tn_cand(int64_t N, const int32_t *Cold, const int32_t *Cnew, int32_t *cand,
                                                 uint32_t *dev, unsigned long long *match, DevCounters *cnt) {
  ld_after_previous();
  __shared__ int32_t seen[TR_FILTER];
  for (int t = threadIdx.x; t < TR_FILTER; t += 256) seen[t] = -1;
  __syncthreads();
  if (ld_gtid() == 0) { cnt->tr_occ = 0; cnt->tr_flagged = 0; }
  const int64_t step = ld_gstride();
  for (int64_t i0 = ld_gtid(); i0 < N; i0 += 4 * step) {
    int32_t o[4], c[4];
#pragma unroll
    for (int u = 0; u < 4; u++) {
      int64_t i = i0 + u * step;
      o[u] = i < N ? Cold[i] : -1;
      c[u] = i < N ? Cnew[i] : 0;
    }
#pragma unroll
    for (int u = 0; u < 4; u++) {
      int64_t i = i0 + u * step;
      if (i >= N) break;
      dev[i] = 0;
      match[i] = 0;
      if (o[u] != (int32_t)i) {
        int32_t *f = &seen[(uint32_t)o[u] % TR_FILTER];
        if (*f == o[u]) continue;  // a member of this block has stored it (any member will do)
        *f = o[u];
      }
      cand[o[u]] = c[u];
    }
  }
}
// Weight of the members whose new label differs from the candidate.
__global__ void __launch_bounds__(256) k_tn_deviants(int64_t N, const int32_t *Cold, const int32_t *Cnew,
                                                     const int64_t *K, const int32_t *cand, uint32_t *dev) {
  ld_after_previous();
  for (int64_t i = ld_gtid(); i < N; i += ld_gstride()) {
    int32_t o = Cold[i];
    if (Cnew[i] != cand[o]) {
      int64_t k = K[i];
      if (k) atomicAdd(&dev[o], (uint32_t)k);
    }
  }
}
// The choice of every old community with a majority (bc, matched at once);
// the others are flagged: bit set, listed, best word cleared.  choice -1: no
// such community.
__global__ void __launch_bounds__(256) k_tn_majority(int64_t N, const int32_t *size, const int32_t *cand,
                                                     const int64_t *tot, const uint32_t *dev, int32_t *choice,
                                                     unsigned long long *match, uint32_t *bits, int32_t *flagged,
                                                     unsigned long long *best, DevCounters *cnt) {
  ld_after_previous();
  const int lane = threadIdx.x & 31;
  for (int64_t o0 = (ld_gtid() & ~31ll); o0 < N; o0 += ld_gstride()) {  // warp-uniform
    int64_t o = o0 + lane;
    int32_t sz = o < N ? size[o] : 0;
    bool f = false;
    int32_t c = -1;
    if (sz > 0) {
      int64_t t = tot[o], ov = t - (int64_t)dev[o];
      if (sz == 1 || (t > 0 && 2 * ov > t)) {
        c = cand[o];
        unsigned long long w = tr_word((uint32_t)ov, (int32_t)o);
        if (__ldcg(&match[c]) < w) atomicMax(&match[c], w);
      } else {
        f = true;  // no majority, or weight 0 and several members
        best[o] = 0;
      }
    }
    if (o < N) choice[o] = c;
    uint32_t m = __ballot_sync(LD_FULL, f);
    if (lane == 0) bits[o0 >> 5] = m;
    if (!m) continue;
    int32_t p0 = 0;
    if (lane == 0) p0 = atomicAdd(&cnt->tr_flagged, __popc(m));
    p0 = __shfl_sync(LD_FULL, p0, 0);
    if (f) flagged[p0 + __popc(m & ((1u << lane) - 1u))] = (int32_t)o;
  }
}
// Pair weights of the flagged communities (as k_trc_insert); members of a
// community of weight 0 offer their labels at weight 0.
__global__ void __launch_bounds__(256) k_tn_insert(int64_t N, const int32_t *Cold, const int32_t *Cnew,
                                                   const int64_t *K, const int64_t *tot, const uint32_t *bits,
                                                   unsigned long long *best, int64_t cap, uint64_t *keys,
                                                   int64_t *vals, int32_t *list, DevCounters *cnt) {
  ld_after_previous();
  if (cnt->tr_flagged == 0) return;
  uint64_t mask = (uint64_t)cap - 1;
  int lane = threadIdx.x & 31;
  for (int64_t base = (ld_gtid() & ~31ll); base < N; base += ld_gstride()) {  // warp-uniform
    int64_t i = base + lane;
    int32_t o = i < N ? Cold[i] : 0;
    bool take = i < N && ld_bit_test(bits, o);
    if (!__any_sync(LD_FULL, take)) continue;
    uint64_t key = EMPTY64 - 1 - lane;
    int64_t kw = 0;
    if (take && tot[o] == 0) {
      atomicMax(&best[o], tr_word(0, Cnew[i]));
      take = false;
    } else if (take) {
      key = ((uint64_t)(uint32_t)o << 32) | (uint32_t)Cnew[i];
      kw = K[i];
    }
    uint32_t peers = __match_any_sync(LD_FULL, (unsigned long long)key);
    int64_t sum = ld_group_sum_i64(peers, kw);
    int32_t claimed = -1;
    if (take && ld_group_leader(peers)) {
      uint64_t sl = hash64(key) & mask;
      for (uint64_t probe = 0; ld_ok(probe <= mask, LD_CHK_PROBE); probe++) {
        unsigned long long k = __ldcg((const unsigned long long *)&keys[sl]);
        if (k == EMPTY64) {
          k = atomicCAS((unsigned long long *)&keys[sl], EMPTY64, key);
          if (k == EMPTY64) claimed = (int32_t)sl;
        }
        if (k == EMPTY64 || k == key) {
          atomicAdd((unsigned long long *)&vals[sl], (unsigned long long)sum);
          break;
        }
        sl = (sl + 1) & mask;
      }
    }
    uint32_t m = __ballot_sync(LD_FULL, claimed >= 0);
    if (m) {
      int leader = __ffs(m) - 1;
      int32_t p0 = 0;
      if (lane == leader) p0 = atomicAdd(&cnt->tr_occ, __popc(m));
      p0 = __shfl_sync(LD_FULL, p0, leader);
      if (claimed >= 0) list[p0 + __popc(m & ((1u << lane) - 1u))] = claimed;
    }
  }
}
// The flagged communities' best pairs, leaving the table empty.
__global__ void k_tn_best(const DevCounters *cnt, const int32_t *list, uint64_t *keys, int64_t *vals,
                          unsigned long long *best) {
  ld_after_previous();
  int64_t m = cnt->tr_occ;
  for (int64_t t = ld_gtid(); t < m; t += ld_gstride()) {
    int32_t sl = list[t];
    uint64_t key = keys[sl];
    atomicMax(&best[key >> 32], tr_word((uint32_t)vals[sl], (int32_t)(key & 0xffffffffu)));
    keys[sl] = EMPTY64;
    vals[sl] = 0;
  }
}
__global__ void k_tn_match(const DevCounters *cnt, const int32_t *flagged, const unsigned long long *best,
                           int32_t *choice, unsigned long long *match) {
  ld_after_previous();
  int64_t m = cnt->tr_flagged;
  for (int64_t t = ld_gtid(); t < m; t += ld_gstride()) {
    int32_t o = flagged[t];
    unsigned long long b = best[o];
    int32_t c = tr_id(b);
    choice[o] = c;
    atomicMax(&match[c], tr_word((uint32_t)(b >> 32), o));
  }
}

// Flags of id c: 1 = a new community that nobody chose, 2 = an id that no old
// community has, 4 = a new community.
__device__ __forceinline__ uint32_t tn_flags(int64_t c, int64_t N, const uint8_t *used, const int32_t *root,
                                             int64_t nroot, const unsigned long long *match, const int32_t *size) {
  if (c >= N) return 0;
  bool u = used ? used[c] != 0 : c < nroot && root[c] == (int32_t)c;
  return (u && match[c] == 0 ? 1u : 0u) | (size[c] == 0 ? 2u : 0u) | (u ? 4u : 0u);
}
// The ids in tiles of a multiple of TR_STEP, at most TR_TILES_MAX of them (each
// block of the second kernel adds up the tiles before its own); the four ids
// of a thread per step are loaded together.
constexpr int TR_STEP = 1024, TR_TILES_MAX = 4096;
// Tile counts (unmatched, free), and the number of new communities.
__global__ void __launch_bounds__(256) k_tn_tiles(int64_t N, int tile, const uint8_t *used, const int32_t *root,
                                                  int64_t nroot, const unsigned long long *match, const int32_t *size,
                                                  int2 *tiles, DevCounters *cnt) {
  ld_after_previous();
  __shared__ int su, sf, sr;
  if (threadIdx.x == 0) su = sf = sr = 0;
  __syncthreads();
  int nu = 0, nf = 0, nr = 0;
  for (int q = 0; q < tile; q += TR_STEP) {
#pragma unroll
    for (int u = 0; u < 4; u++) {
      uint32_t f = tn_flags((int64_t)blockIdx.x * tile + q + 256 * u + threadIdx.x, N, used, root, nroot, match, size);
      nu += f & 1;
      nf += f >> 1 & 1;
      nr += f >> 2;
    }
  }
  nu = __reduce_add_sync(LD_FULL, nu);
  nf = __reduce_add_sync(LD_FULL, nf);
  nr = __reduce_add_sync(LD_FULL, nr);
  if ((threadIdx.x & 31) == 0) { atomicAdd(&su, nu); atomicAdd(&sf, nf); atomicAdd(&sr, nr); }
  __syncthreads();
  if (threadIdx.x == 0) {
    tiles[blockIdx.x] = make_int2(su, sf);
    if (sr) atomicAdd(&cnt->list_count, sr);
  }
}
// rank[c] of the unmatched ids and the list of the free ones, both in id
// order; batched handles also record both ranks at each graph's first id.
__global__ void __launch_bounds__(256) k_tn_lists(int64_t N, int tile, const uint8_t *used, const int32_t *root,
                                                  int64_t nroot, const unsigned long long *match, const int32_t *size,
                                                  const int2 *tiles, int32_t *rank, int32_t *freel,
                                                  const int32_t *gid0, const int64_t *voff, int2 *granks) {
  ld_after_previous();
  __shared__ int2 wsum[4][8];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int pu = 0, pf = 0;  // in the tiles before this one
#pragma unroll 4
  for (int t = threadIdx.x; t < (int)blockIdx.x; t += 256) { int2 x = tiles[t]; pu += x.x; pf += x.y; }
  pu = __reduce_add_sync(LD_FULL, pu);
  pf = __reduce_add_sync(LD_FULL, pf);
  if (lane == 0) wsum[0][wid] = make_int2(pu, pf);
  __syncthreads();
  pu = pf = 0;
  for (int w = 0; w < 8; w++) { pu += wsum[0][w].x; pf += wsum[0][w].y; }
  const uint32_t below = (1u << lane) - 1u;
  for (int q = 0; q < tile; q += TR_STEP) {
    int64_t c0 = (int64_t)blockIdx.x * tile + q + threadIdx.x;
    uint32_t f[4], mu[4], mf[4];
#pragma unroll
    for (int u = 0; u < 4; u++) f[u] = tn_flags(c0 + 256 * u, N, used, root, nroot, match, size);
    __syncthreads();  // the sums of the step before are read
#pragma unroll
    for (int u = 0; u < 4; u++) {
      mu[u] = __ballot_sync(LD_FULL, f[u] & 1);
      mf[u] = __ballot_sync(LD_FULL, f[u] & 2);
      if (lane == 0) wsum[u][wid] = make_int2(__popc(mu[u]), __popc(mf[u]));
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 4; u++) {
      int ru = pu, rf = pf;
#pragma unroll
      for (int w = 0; w < 8; w++) {
        int2 x = wsum[u][w];
        if (w < wid) { ru += x.x; rf += x.y; }
        pu += x.x;
        pf += x.y;
      }
      ru += __popc(mu[u] & below);
      rf += __popc(mf[u] & below);
      int64_t c = c0 + 256 * u;
      if (f[u] & 1) rank[c] = ru;
      if (f[u] & 2) freel[rf] = (int32_t)c;
      if (gid0 && c < N && voff[gid0[c]] == c) granks[gid0[c]] = make_int2(ru, rf);
    }
  }
}
// The tracked id of new community c.
__device__ __forceinline__ int32_t tn_name(int32_t c, const unsigned long long *match, const int32_t *rank,
                                           const int32_t *freel, const int32_t *gid0, const int2 *granks) {
  unsigned long long m = match[c];
  if (m) return tr_id(m);
  if (!gid0) return freel[rank[c]];
  int2 g = granks[gid0[c]];  // the k-th unmatched of a graph takes its k-th free id
  return freel[g.y + rank[c] - g.x];
}
// C^t, Sigma and the member counts follow the vertices whose id changes; the
// change sums of ids that were not carried over are reset.
__global__ void __launch_bounds__(256) k_tn_relabel(int64_t N, const int32_t *Cnew, const unsigned long long *match,
                                                    const int32_t *rank, const int32_t *freel, const int32_t *choice,
                                                    const int64_t *K, int32_t *C, int64_t *Sig, int32_t *size,
                                                    int64_t *dSig, const int32_t *gid0, const int2 *granks) {
  ld_after_previous();
  for (int64_t i = ld_gtid(); i < N; i += ld_gstride()) {
    int32_t ch = choice[i];
    if (ch < 0 || tr_id(match[ch]) != (int32_t)i) dSig[i] = 0;
    int32_t c = tn_name(Cnew[i], match, rank, freel, gid0, granks), o = C[i];
    if (c == o) continue;
    C[i] = c;
    int64_t k = K[i];
    if (k) {
      atomicAdd((unsigned long long *)&Sig[o], (unsigned long long)(-k));
      atomicAdd((unsigned long long *)&Sig[c], (unsigned long long)k);
    }
    atomicSub(&size[o], 1);
    atomicAdd(&size[c], 1);
  }
}

// ---- modularity
__global__ void k_sig_of(int64_t N, const int32_t *C, const int64_t *K, int64_t *Sig) {
  ld_after_previous();
  int lane = threadIdx.x & 31;
  for (int64_t base = (ld_gtid() & ~31ll); base < N; base += ld_gstride()) {
    int64_t i = base + lane;
    int32_t c = i < N ? C[i] : -1 - lane;
    int64_t k = i < N ? K[i] : 0;
    uint32_t peers = __match_any_sync(LD_FULL, c);
    int64_t s = ld_group_sum_i64(peers, k);
    if (i < N && ld_group_leader(peers) && s) atomicAdd((unsigned long long *)&Sig[c], (unsigned long long)s);
  }
}
// Batched handles (gid0 non-null) also sum per graph: sigg, sqg, m2g.
// Intra-community weight and (k_rowsum) row sums, rows by windows of up to 32 per
// warp (see window_rows; lanes past a window's rows hold none); rows above
// ROWS_BIG arcs are listed and their chunks summed by the second kernel (launched
// where a row can be that long).  With a warp per row, the longest hub's warp was
// the kernel's time (R-MAT 21: k_rowsum 412 -> 260 us).
constexpr int ROW_UNROLL = 4;

// The rows of a window: lane i's first flat position s, end e, row start minus
// s (ab); rows above ROWS_BIG are listed instead.  Returns the flat length.
__device__ __forceinline__ int window_of(int64_t i, int64_t N, const int64_t *off, const int32_t *deg, int32_t *big,
                                         int32_t *nbig, int &s, int &e, int64_t &ab) {
  int d = i < N ? deg[i] : 0;
  int64_t b = i < N ? off[i] : 0;
  if (d > ROWS_BIG) {
    big[atomicAdd(nbig, 1)] = (int32_t)i;
    d = 0;
  }
  e = ld_warp_incl_i32(d);
  s = e - d;
  ab = b - s;
  return __shfl_sync(LD_FULL, e, 31);
}

__global__ void __launch_bounds__(256) k_sigma_intra(int64_t N, const int64_t *off, const int32_t *deg,
                                                     const int32_t *col, const int32_t *w, const int32_t *C,
                                                     DevCounters *cnt, const int32_t *gid0, int64_t *sigg,
                                                     int32_t *big, int rows) {
  ld_after_previous();
  const int lane = threadIdx.x & 31;
  int64_t warp = ld_gtid() >> 5, nw = ld_gstride() >> 5;
  int64_t acc = 0;
  for (int64_t r = warp * rows; r < N; r += nw * rows) {  // warp-uniform
    int64_t i = lane < rows ? r + lane : N, ab;
    int s, e;
    int total = window_of(i, N, off, deg, big, &cnt->big_count, s, e, ab);
    int32_t c = i < N ? C[i] : -1, g = gid0 && i < N ? gid0[i] : 0;
    int64_t here = 0;
    // the usual window lies in one graph; one across a boundary adds each hit to its row's graph
    int32_t g0 = __shfl_sync(LD_FULL, g, 0);
    bool one = __all_sync(LD_FULL, g == g0 || i >= N);
    for (int x0 = 0; x0 < total; x0 += 32 * ROW_UNROLL) {  // warp-uniform
      int k[ROW_UNROLL];
      int32_t j[ROW_UNROLL], wv[ROW_UNROLL], cj[ROW_UNROLL];
      ld_window_rows<ROW_UNROLL>(s, x0, lane, k);
#pragma unroll
      for (int u = 0; u < ROW_UNROLL; u++) {
        int x = x0 + 32 * u + lane;
        int64_t a = __shfl_sync(LD_FULL, ab, k[u]) + x;
        j[u] = x < total ? col[a] : -1;
        wv[u] = x < total ? w[a] : 0;
      }
#pragma unroll
      for (int u = 0; u < ROW_UNROLL; u++) cj[u] = j[u] >= 0 ? C[j[u]] : -2;
#pragma unroll
      for (int u = 0; u < ROW_UNROLL; u++) {
        int32_t ci = __shfl_sync(LD_FULL, c, k[u]), gi = __shfl_sync(LD_FULL, g, k[u]);
        if (ci != cj[u]) continue;
        here += wv[u];
        if (gid0 && !one) atomicAdd((unsigned long long *)&sigg[gi], (unsigned long long)wv[u]);
      }
    }
    acc += here;
    if (gid0 && one) {
      here = ld_warp_sum_i64(here);
      if (lane == 0 && here) atomicAdd((unsigned long long *)&sigg[g0], (unsigned long long)here);
    }
  }
  acc = ld_warp_sum_i64(acc);
  if (lane == 0 && acc) atomicAdd((unsigned long long *)&cnt->sigma_intra, (unsigned long long)acc);
}

// The same with a warp per row, for long rows (window_rows == 1): few registers,
// so that twice as many loads are in flight as in the windows' form.
__global__ void __launch_bounds__(256) k_sigma_intra_rows(int64_t N, const int64_t *off, const int32_t *deg,
                                                          const int32_t *col, const int32_t *w, const int32_t *C,
                                                          DevCounters *cnt, const int32_t *gid0, int64_t *sigg,
                                                          int32_t *big) {
  ld_after_previous();
  const int lane = threadIdx.x & 31;
  int64_t acc = 0;
  for (int64_t i = ld_gtid() >> 5; i < N; i += ld_gstride() >> 5) {  // warp-uniform
    int32_t c = C[i];
    int64_t b = off[i], d = deg[i], here = 0;
    if (d > ROWS_BIG) {
      if (lane == 0) big[atomicAdd(&cnt->big_count, 1)] = (int32_t)i;
      continue;
    }
    for (int64_t a = lane; a < d; a += 32)
      if (C[col[b + a]] == c) here += w[b + a];
    acc += here;
    if (gid0) {
      here = ld_warp_sum_i64(here);
      if (lane == 0 && here) atomicAdd((unsigned long long *)&sigg[gid0[i]], (unsigned long long)here);
    }
  }
  acc = ld_warp_sum_i64(acc);
  if (lane == 0 && acc) atomicAdd((unsigned long long *)&cnt->sigma_intra, (unsigned long long)acc);
}

__global__ void __launch_bounds__(256) k_sigma_intra_big(const int32_t *big, const int64_t *ch_off, const int64_t *off,
                                                         const int32_t *deg, const int32_t *col, const int32_t *w,
                                                         const int32_t *C, DevCounters *cnt, const int32_t *gid0,
                                                         int64_t *sigg) {
  ld_after_previous();
  const int64_t count = cnt->big_count;
  if (count == 0) return;
  const int64_t nch = ch_off[count];
  int64_t acc = 0;
  for (int64_t t = blockIdx.x; t < nch; t += gridDim.x) {  // block-uniform
    int64_t k = ld_chunk_item(ch_off, count, t);
    int32_t i = big[k], c = C[i];
    int64_t x0 = (t - ch_off[k]) * TABLE_CHUNK, b = off[i] + x0;
    int len = (int)(deg[i] - x0 < TABLE_CHUNK ? deg[i] - x0 : TABLE_CHUNK);
    int64_t here = 0;
#pragma unroll 4
    for (int x = threadIdx.x; x < len; x += 256)
      if (C[col[b + x]] == c) here += w[b + x];
    acc += here;
    if (gid0) {
      here = ld_warp_sum_i64(here);
      if ((threadIdx.x & 31) == 0 && here) atomicAdd((unsigned long long *)&sigg[gid0[i]], (unsigned long long)here);
    }
  }
  acc = ld_warp_sum_i64(acc);
  if ((threadIdx.x & 31) == 0 && acc) atomicAdd((unsigned long long *)&cnt->sigma_intra, (unsigned long long)acc);
}
__global__ void k_sq(int64_t N, const int64_t *Sig, DevCounters *cnt, const int32_t *gid0, unsigned long long *sqg) {
  ld_after_previous();
  i128 acc = 0;
  for (int64_t c0 = (ld_gtid() & ~31ll); c0 < N; c0 += ld_gstride()) {  // warp-uniform trip count
    int64_t c = c0 + (threadIdx.x & 31);
    i128 v = c < N ? (i128)Sig[c] * Sig[c] : 0;
    acc += v;
    if (gid0) ld_graph_add_i128(sqg, c < N && v != 0, c < N ? gid0[c] : 0, v);
  }
  // warp reduce in two halves
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += ld_shfl_xor_i128(acc, o);
  if ((threadIdx.x & 31) == 0) ld_atomic_add_i128(cnt->sq, acc);
}

// K of the rows up to ROWS_BIG arcs; a longer row's K is set to 0 and its
// chunks are added by k_rowsum_big.  Steps inside one row are summed per lane
// and reduced when the row changes; only steps across rows pay for a scan.
constexpr int SUM_UNROLL = 8;
__global__ void __launch_bounds__(256) k_rowsum(int64_t N, const int64_t *off, const int32_t *deg, const int32_t *w,
                                                int64_t *K, DevCounters *cnt, const int32_t *gid0, int64_t *m2g,
                                                int32_t *big, int rows) {
  ld_after_previous();
  __shared__ unsigned long long bsum;
  if (threadIdx.x == 0) bsum = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  int64_t warp = ld_gtid() >> 5, nw = ld_gstride() >> 5;
  int64_t tot = 0;
  for (int64_t r = warp * rows; r < N; r += nw * rows) {  // warp-uniform
    int64_t i = lane < rows ? r + lane : N, ab, kw = 0, lacc = 0;
    int s, e, cur = 0;
    int total = window_of(i, N, off, deg, big, &cnt->big_count, s, e, ab);
    for (int x0 = 0; x0 < total; x0 += 32 * SUM_UNROLL) {  // warp-uniform
      int k[SUM_UNROLL];
      int32_t wv[SUM_UNROLL];
      bool inside = ld_window_rows<SUM_UNROLL>(s, x0, lane, k);
#pragma unroll
      for (int u = 0; u < SUM_UNROLL; u++) {
        int x = x0 + 32 * u + lane;
        int64_t a = __shfl_sync(LD_FULL, ab, k[u]) + x;
        wv[u] = x < total ? w[a] : 0;
      }
      int kc = __shfl_sync(LD_FULL, k[0], 0);
      if (!inside || kc != cur) {  // warp-uniform: the row summed so far is complete
        lacc = ld_warp_sum_i64(lacc);
        if (lane == cur) kw += lacc;
        lacc = 0;
        cur = kc;
      }
#pragma unroll
      for (int u = 0; u < SUM_UNROLL; u++) {
        if (inside) lacc += wv[u];
        else kw += ld_window_part(s, e, x0 + 32 * u, wv[u]);
      }
    }
    lacc = ld_warp_sum_i64(lacc);
    if (lane == cur) kw += lacc;
    if (i < N) {
      K[i] = kw;
      tot += kw;
    }
    if (gid0) ld_graph_add_i64(m2g, i < N, i < N ? gid0[i] : 0, kw);
  }
  tot = ld_warp_sum_i64(tot);
  if (lane == 0 && tot) atomicAdd(&bsum, (unsigned long long)tot);
  __syncthreads();
  if (threadIdx.x == 0 && bsum) atomicAdd((unsigned long long *)&cnt->m2, bsum);
}

__global__ void __launch_bounds__(256) k_rowsum_rows(int64_t N, const int64_t *off, const int32_t *deg,
                                                     const int32_t *w, int64_t *K, DevCounters *cnt,
                                                     const int32_t *gid0, int64_t *m2g, int32_t *big) {
  ld_after_previous();
  const int lane = threadIdx.x & 31;
  int64_t tot = 0;
  for (int64_t i = ld_gtid() >> 5; i < N; i += ld_gstride() >> 5) {  // warp-uniform
    int64_t b = off[i], d = deg[i], acc = 0;
    if (d > ROWS_BIG) {
      if (lane == 0) {
        big[atomicAdd(&cnt->big_count, 1)] = (int32_t)i;
        K[i] = 0;
      }
      continue;
    }
    for (int64_t a = lane; a < d; a += 32) acc += w[b + a];
    acc = ld_warp_sum_i64(acc);
    if (lane == 0) K[i] = acc;
    if (lane == 0 && gid0 && acc) atomicAdd((unsigned long long *)&m2g[gid0[i]], (unsigned long long)acc);
    tot += acc;
  }
  if (lane == 0 && tot) atomicAdd((unsigned long long *)&cnt->m2, (unsigned long long)tot);
}

__global__ void __launch_bounds__(256) k_rowsum_big(const int32_t *big, const int64_t *ch_off, const int64_t *off,
                                                    const int32_t *deg, const int32_t *w, int64_t *K, DevCounters *cnt,
                                                    const int32_t *gid0, int64_t *m2g) {
  ld_after_previous();
  const int64_t count = cnt->big_count;
  if (count == 0) return;
  const int64_t nch = ch_off[count];
  for (int64_t t = blockIdx.x; t < nch; t += gridDim.x) {  // block-uniform
    int64_t k = ld_chunk_item(ch_off, count, t);
    int32_t i = big[k];
    int64_t x0 = (t - ch_off[k]) * TABLE_CHUNK, b = off[i] + x0;
    int len = (int)(deg[i] - x0 < TABLE_CHUNK ? deg[i] - x0 : TABLE_CHUNK);
    int64_t acc = 0;
#pragma unroll 4
    for (int x = threadIdx.x; x < len; x += 256) acc += w[b + x];
    acc = ld_warp_sum_i64(acc);
    if ((threadIdx.x & 31) == 0 && acc) {
      atomicAdd((unsigned long long *)&K[i], (unsigned long long)acc);
      atomicAdd((unsigned long long *)&cnt->m2, (unsigned long long)acc);
      if (gid0) atomicAdd((unsigned long long *)&m2g[gid0[i]], (unsigned long long)acc);
    }
  }
}

}  // namespace

// Scratch (each array used by nobody else between the last lookup and the
// next call): 4-byte cand, dev, choice, flagged, rank, free ids; 8-byte match,
// best.
static void track_narrow(leiden_handle *h, const int32_t *Cnew, const int32_t *root, int64_t nroot) {
  cudaStream_t s = h->stream;
  int64_t N = h->n;
  int gN = grid_for(N, TB);
  int32_t *cand = h->mtarget, *choice = h->movers, *flagged = h->prop, *rank = h->rep, *freel = h->parent;
  uint32_t *dev = (uint32_t *)h->ibuf0, *bits = h->unproc;
  unsigned long long *match = (unsigned long long *)h->lbuf0, *best = (unsigned long long *)h->lbuf1;
  int2 *tiles = (int2 *)h->lbuf2, *granks = (int2 *)h->lbuf3;
  const uint8_t *used = h->G > 1 ? h->dE : nullptr;
  DevCounters *cnt = h->dcnt;
  ld_note_launch(), launch_after(k_tn_cand, grid_for(N, TB, h->sm_count * 4), TB, s, N, h->C, Cnew, cand, dev, match,
                                 cnt);
  ld_note_launch(), launch_after(k_tn_deviants, gN, TB, s, N, h->C, Cnew, h->K, cand, dev);
  ld_note_launch(), launch_after(k_tn_majority, gN, TB, s, N, h->csize0, cand, h->Sig, dev, choice, match, bits,
                                 flagged, best, cnt);
  ld_note_launch(), launch_after(k_tn_insert, gN, TB, s, N, h->C, Cnew, h->K, h->Sig, bits, best, h->tr_cap, h->tr_keys,
                                 h->tr_vals, h->tr_list, cnt);
  ld_note_launch(), launch_after(k_tn_best, h->sm_count * 2, TB, s, cnt, h->tr_list, h->tr_keys, h->tr_vals, best);
  ld_note_launch(), launch_after(k_tn_match, h->sm_count * 2, TB, s, cnt, flagged, best, choice, match);
  const int64_t span = (int64_t)TR_STEP * TR_TILES_MAX;
  int tile = TR_STEP * (int)std::max<int64_t>(1, (N + span - 1) / span);
  int nt = (int)((N + tile - 1) / tile);
  ld_note_launch(), launch_after(k_tn_tiles, nt, TB, s, N, tile, used, root, nroot, match, h->csize0, tiles, cnt);
  ld_note_launch(), launch_after(k_tn_lists, nt, TB, s, N, tile, used, root, nroot, match, h->csize0, tiles, rank,
                                 freel, h->gid0, h->d_voff, granks);
  ld_note_launch(), launch_after(k_tn_relabel, gN, TB, s, N, Cnew, match, rank, freel, choice, h->K, h->C, h->Sig,
                                 h->csize0, h->dSig, h->gid0, granks);
}

// C^{t-1} = h->C, final top-level membership = Cnew  ->  h->C, h->Sig, h->dSig.
// The new ids: the roots of the last level (c < nroot, root[c] == c); of a
// batched handle the ids flagged in h->dE.
void track_communities(leiden_handle *h, const int32_t *Cnew, const int32_t *root, int64_t nroot) {
  if (!wide_sums(h)) { track_narrow(h, Cnew, root, nroot); return; }
  cudaStream_t s = h->stream;
  if (h->G == 1) count_communities(h, nroot, nullptr);
  int64_t N = h->n;
  int gN = grid_for(N, TB);
  long long *bw = (long long *)h->lbuf0, *ow = (long long *)h->lbuf1;
  int32_t *bc = h->ibuf0, *ob = h->ibuf1, *used = h->ibuf2;
  int32_t *cand = h->mtarget, *flag = h->movers;
  int64_t *dev = h->Sp;
  ld_note_launch(), launch_after(k_tr_init, gN, TB, s, N, bw, bc, ow, ob, cand, used, dev);
  cudaMemsetAsync(&h->dcnt->tr_occ, 0, sizeof(int32_t), s);
  ld_note_launch(), launch_after(k_trc_cand, gN, TB, s, N, h->C, Cnew, cand);
  ld_note_launch(), launch_after(k_trc_deviants, gN, TB, s, N, h->C, Cnew, h->K, cand, dev);
  ld_note_launch(), launch_after(k_trc_majority, gN, TB, s, N, cand, h->Sig, dev, bw, bc, flag);
  int32_t *occ = &h->dcnt->tr_occ;
  ld_note_launch(), launch_after(k_trc_insert, gN, TB, s, N, h->C, Cnew, h->K, flag, bc, h->tr_cap, h->tr_keys,
                                 h->tr_vals, h->tr_list, occ);
  ld_note_launch(), launch_after(k_trc_best_w, h->sm_count * 8, TB, s, occ, h->tr_list, h->tr_keys, h->tr_vals, bw);
  ld_note_launch(), launch_after(k_trc_best_c, h->sm_count * 8, TB, s, occ, h->tr_list, h->tr_keys, h->tr_vals, bw, bc);
  ld_note_launch(), launch_after(k_tr_best_old_w, gN, TB, s, N, bc, bw, ow);
  ld_note_launch(), launch_after(k_tr_best_old_b, gN, TB, s, N, bc, bw, ow, ob);
  ld_note_launch(), launch_after(k_tr_new_used, gN, TB, s, N, Cnew, used);
  int32_t *unmatched = h->rep, *freef = h->prop;
  ld_note_launch(), launch_after(k_tr_flags, gN, TB, s, N, used, ob, bc, unmatched, freef);
  int64_t *urank = h->lbuf2, *frank = h->lbuf3;
  exclusive_scan_i32_to_i64(unmatched, urank, N, h->scan_tmp, s);
  exclusive_scan_i32_to_i64(freef, frank, N, h->scan_tmp, s);
  int32_t *flist = h->parent, *map = h->CB;
  ld_note_launch(), launch_after(k_tr_free_list, gN, TB, s, N, freef, frank, flist);
  uint8_t *matched = h->dE;
  cudaMemsetAsync(matched, 0, (size_t)N, s);
  ld_note_launch(), launch_after(k_tr_map, gN, TB, s, N, used, ob, urank, frank, flist, map, matched, h->gid0,
                                 h->d_voff);
  ld_note_launch(), launch_after(k_tr_relabel, gN, TB, s, N, Cnew, map, h->K, h->C, h->Sig, h->csize0);
  ld_note_launch(), launch_after(k_tr_dsig, gN, TB, s, N, matched, h->dSig);
}

// sigma (intra arcs) and sum Sigma_c^2 of membership C on G^t.
void modularity_terms(leiden_handle *h, const int32_t *C) {
  cudaStream_t s = h->stream;
  int64_t N = h->n;
  int64_t *Sig = h->lbuf0;
  cudaMemsetAsync(Sig, 0, (size_t)N * sizeof(int64_t), s);
  cudaMemsetAsync(&h->dcnt->sigma_intra, 0, sizeof(int64_t), s);
  cudaMemsetAsync(&h->dcnt->sq[0], 0, 2 * sizeof(unsigned long long), s);
  ld_note_launch(), launch_after(k_sig_of, grid_for(N, TB), TB, s, N, C, h->K, Sig);
  if (h->gid0) {
    cudaMemsetAsync(h->gc.sigma, 0, (size_t)h->G * sizeof(int64_t), s);
    cudaMemsetAsync(h->gc.sq, 0, (size_t)h->G * 2 * sizeof(unsigned long long), s);
  }
  int32_t *big = h->ibuf0;
  const bool some_big = h->g_maxdeg > ROWS_BIG;
  if (some_big) cudaMemsetAsync(&h->dcnt->big_count, 0, sizeof(int32_t), s);
  const int rows = window_rows(h);
  if (rows == 1)
    ld_note_launch(), launch_after(k_sigma_intra_rows, window_grid(N, 1), TB, s, N, h->g_off, h->g_deg, h->g_col,
                                   h->g_w, C, h->dcnt, h->gid0, h->gc.sigma, big);
  else
    ld_note_launch(), launch_after(k_sigma_intra, window_grid(N, rows), TB, s, N, h->g_off, h->g_deg, h->g_col, h->g_w,
                                   C, h->dcnt, h->gid0, h->gc.sigma, big, rows);
  if (some_big) {
    launch_table_plan(big, &h->dcnt->big_count, h->g_deg, nullptr, 1, h->lbuf2, h->lbuf3, s);
    ld_note_launch(), launch_after(k_sigma_intra_big, h->sm_count * 8, TB, s, big, h->lbuf3, h->g_off, h->g_deg,
                                   h->g_col, h->g_w, C, h->dcnt, h->gid0, h->gc.sigma);
  }
  ld_note_launch(), launch_after(k_sq, grid_for(N, TB), TB, s, N, Sig, h->dcnt, h->gid0, h->gc.sq);
}

// Sigma = per-community sums of K for membership h->C.
void recompute_sigma(leiden_handle *h) {
  cudaStream_t s = h->stream;
  cudaMemsetAsync(h->Sig, 0, (size_t)h->n * sizeof(int64_t), s);
  ld_note_launch(), launch_after(k_sig_of, grid_for(h->n, TB), TB, s, h->n, h->C, h->K, h->Sig);
}

// K = row sums of G^t and 2m.
void recompute_weights(leiden_handle *h) {
  cudaStream_t s = h->stream;
  cudaMemsetAsync(&h->dcnt->m2, 0, sizeof(int64_t), s);
  if (h->gid0) cudaMemsetAsync(h->gc.m2, 0, (size_t)h->G * sizeof(int64_t), s);
  int32_t *big = h->ibuf0;
  const bool some_big = h->g_maxdeg > ROWS_BIG;
  if (some_big) cudaMemsetAsync(&h->dcnt->big_count, 0, sizeof(int32_t), s);
  const int rows = window_rows(h);
  if (rows == 1)
    ld_note_launch(), launch_after(k_rowsum_rows, window_grid(h->n, 1), TB, s, h->n, h->g_off, h->g_deg, h->g_w, h->K,
                                   h->dcnt, h->gid0, h->gc.m2, big);
  else
    ld_note_launch(), launch_after(k_rowsum, window_grid(h->n, rows), TB, s, h->n, h->g_off, h->g_deg, h->g_w, h->K,
                                   h->dcnt, h->gid0, h->gc.m2, big, rows);
  if (some_big) {
    launch_table_plan(big, &h->dcnt->big_count, h->g_deg, nullptr, 1, h->lbuf2, h->lbuf3, s);
    ld_note_launch(), launch_after(k_rowsum_big, h->sm_count * 8, TB, s, big, h->lbuf3, h->g_off, h->g_deg, h->g_w,
                                   h->K, h->dcnt, h->gid0, h->gc.m2);
  }
}

LD_CHECK_WORD_READER(check_word_track)
