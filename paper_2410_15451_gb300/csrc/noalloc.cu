// Modularity of a membership on a caller-owned device CSR, without any
// device allocation: the per-community totals and the reduction counters
// live in one file-scope __device__ array of fixed size.
#include <mutex>
#include <string>

#include "internal.h"

namespace {

// Largest vertex count the entry point accepts: the scratch holds one int64
// community total per vertex id (32 MiB) plus NOALLOC_COUNTERS int64 words.
constexpr int64_t NOALLOC_MAX_VERTICES = (int64_t)1 << 22;
constexpr int64_t NOALLOC_COUNTERS = 6;
constexpr int64_t NOALLOC_WORDS = NOALLOC_MAX_VERTICES + NOALLOC_COUNTERS;

// Every GPU that loads the library holds this array until the process exits.
static __device__ __align__(256) int64_t g_noalloc_scratch[NOALLOC_WORDS];

// Host code must not pass g_noalloc_scratch to a kernel: on the host that
// name is a stand-in symbol, not a device address.  The device address is
// looked up once per device (with that device current) and cached here.
constexpr int MAX_DEVICES = 64;
int64_t *g_scratch_ptr[MAX_DEVICES] = {};
std::mutex g_scratch_mu;

// counters after the per-vertex totals
enum { C_M2 = 0, C_SIGMA = 1, C_SQ_LO = 2, C_SQ_HI = 3, C_BAD = 4, C_BADCOL = 5 };

__global__ void k_na_clear(int64_t n, int64_t *scr) {
  for (int64_t i = ld_gtid(); i < n; i += ld_gstride()) scr[i] = 0;
  if (ld_gtid() < NOALLOC_COUNTERS) scr[NOALLOC_MAX_VERTICES + ld_gtid()] = 0;
}

// K_i (row sum) into Sigma[C_i]; intra-community weight; 2m.  The CSR is flat,
// so every warp takes the same number of arcs, [f0, f1) of all of them, finds
// the row of its first one (a 32-way search over the offsets, once a warp)
// and walks the rows of its range 32 at a time: a hub is spread over as many
// warps as it has spans, where a warp per row left a 200k-arc hub to one.
// Bound by the C[col] gathers (one line each); a warp adds a community's
// total once per 32 rows.  R-MAT 22 (128M arcs):
// 3854 -> 478 us, 270 G gathers/s; four arcs per lane in flight instead of
// eight: 504 us.
// A membership id outside [0, n) sets the C_BAD word and the vertex is
// skipped; a column outside [0, n) sets C_BADCOL (and is not read through).
// Either one turns the call into LEIDEN_ERR_ARG.
constexpr int NA_UNROLL = 8;
constexpr int64_t NA_SPAN_MIN = 256;

// The last of the rows [r, r + cnt) with off[row] <= F, by a 32-way search of the
// whole warp (off[r] <= F).
__device__ __forceinline__ int64_t na_row_of(const int64_t *off, int64_t r, int64_t cnt, int64_t F) {
  const int lane = threadIdx.x & 31;
  while (cnt > 1) {  // warp-uniform
    int64_t step = (cnt + 31) >> 5, q = r + lane * step;
    bool le = q < r + cnt && off[q] <= F;
    uint32_t m = __ballot_sync(LD_FULL, le);
    int k = m ? 31 - __clz(m) : 0;
    r += k * step;
    cnt = cnt - k * step < step ? cnt - k * step : step;
  }
  return r;
}

// The window before the next row that has arcs, after one without (rows [r, r +
// 32), all arcs before flat position F are done): a run of unused ids costs the
// warp whose span lies across it one search instead of a step per 32 of them
// (1.6M arcs with 10^6 unused ids in the middle: 16.1 ms -> 44 us, as without
// them).
__device__ __forceinline__ int64_t na_skip_empty(const int64_t *off, int64_t r, int64_t n, int64_t F) {
  return r + 64 < n ? na_row_of(off, r + 32, n - r - 32, F) - 32 : r;
}

template <bool UNIT>
__global__ void __launch_bounds__(256) k_na_rows(int64_t n, const int64_t *off, const int32_t *col, const int32_t *w,
                                                 const int32_t *C, int64_t *scr) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ld_gtid() >> 5, nw = ld_gstride() >> 5;
  const int64_t a0 = off[0], total = off[n] - a0;
  int64_t span = ((total + nw - 1) / nw + 31) & ~31ll;
  if (span < NA_SPAN_MIN) span = NA_SPAN_MIN;
  int64_t m2 = 0, intra = 0;
  // a span is walked in pieces of at most 2^30 arcs, so that positions fit 32 bits
  for (int64_t p0 = warp * span, pe = p0 + span < total ? p0 + span : total; p0 < pe; p0 += (int64_t)1 << 30) {
    const int64_t F0 = a0 + p0;
    const int len = (int)(pe - p0 < ((int64_t)1 << 30) ? pe - p0 : (int64_t)1 << 30);
    for (int64_t r = na_row_of(off, 0, n, F0); r < n; r += 32) {  // warp-uniform
      int64_t i = r + lane;
      int64_t o0 = i < n ? off[i] - F0 : len, o1 = i < n ? off[i + 1] - F0 : len;
      int s = o0 < 0 ? 0 : o0 > len ? len : (int)o0, e = o1 < s ? s : o1 > len ? len : (int)o1;
      int ws = __shfl_sync(LD_FULL, s, 0), we = __shfl_sync(LD_FULL, e, 31);
      if (ws >= len) break;
      // (where this stands decides how the compiler orders the loads below: R-MAT
      // 22 with weights 743 us here and 768 at the end of the body, without 549
      // and 512)
      if (!UNIT && ws >= we) {
        r = na_skip_empty(off, r, n, F0 + ws);
        continue;
      }
      int32_t c = -1;
      if (e > s) {
        c = C[i];
        if (c < 0 || c >= n) {
          atomicExch((unsigned long long *)&scr[NOALLOC_MAX_VERTICES + C_BAD], 1ull);
          c = -1;
        }
      }
      int64_t kw = UNIT ? e - s : 0;  // K of the rows' parts in this window
      for (int x0 = ws; x0 < we; x0 += 32 * NA_UNROLL) {  // warp-uniform
        int k[NA_UNROLL];
        int32_t j[NA_UNROLL], wv[NA_UNROLL], cj[NA_UNROLL];
#pragma unroll
        for (int u = 0; u < NA_UNROLL; u++) {
          int x = x0 + 32 * u + lane;
          j[u] = x < we ? col[F0 + x] : 0;
          wv[u] = x < we ? (UNIT ? 1 : w[F0 + x]) : 0;
        }
#pragma unroll
        for (int u = 0; u < NA_UNROLL; u++) {
          bool in = j[u] >= 0 && j[u] < n;
          if (!in) atomicExch((unsigned long long *)&scr[NOALLOC_MAX_VERTICES + C_BADCOL], 1ull);
          cj[u] = in ? C[j[u]] : -2;
        }
        ld_window_rows<NA_UNROLL>(s, x0, lane, k);
#pragma unroll
        for (int u = 0; u < NA_UNROLL; u++) {
          int32_t ci = __shfl_sync(LD_FULL, c, k[u]);
          if (ci == cj[u]) intra += wv[u];
          if (!UNIT) kw += ld_window_part(s, e, x0 + 32 * u, wv[u]);
        }
      }
      // added once per community of the window
      m2 += kw;
      uint32_t peers = __match_any_sync(LD_FULL, c >= 0 ? c : -2 - lane);
      if (__any_sync(LD_FULL, __popc(peers) > 1)) kw = ld_group_sum_i64(peers, kw);
      if (c >= 0 && ld_group_leader(peers)) atomicAdd((unsigned long long *)&scr[c], (unsigned long long)kw);
      if (UNIT && ws >= we) r = na_skip_empty(off, r, n, F0 + ws);
    }
  }
  intra = ld_warp_sum_i64(intra);
  m2 = ld_warp_sum_i64(m2);
  if (lane == 0) {
    if (m2) atomicAdd((unsigned long long *)&scr[NOALLOC_MAX_VERTICES + C_M2], (unsigned long long)m2);
    if (intra) atomicAdd((unsigned long long *)&scr[NOALLOC_MAX_VERTICES + C_SIGMA], (unsigned long long)intra);
  }
}

// Sum of Sigma_c^2; a vertex without arcs has its membership id checked here.
__global__ void k_na_sq(int64_t n, const int32_t *C, int64_t *scr) {
  i128 acc = 0;
  for (int64_t c = ld_gtid(); c < n; c += ld_gstride()) {
    acc += (i128)scr[c] * scr[c];
    if (C[c] < 0 || C[c] >= n) atomicExch((unsigned long long *)&scr[NOALLOC_MAX_VERTICES + C_BAD], 1ull);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += ld_shfl_xor_i128(acc, o);
  if ((threadIdx.x & 31) == 0) ld_atomic_add_i128((unsigned long long *)&scr[NOALLOC_MAX_VERTICES + C_SQ_LO], acc);
}

}  // namespace


extern "C" leiden_status leiden_modularity_noalloc(int64_t n, const int64_t *d_offsets, const int32_t *d_cols,
                                                   const int32_t *d_weights, const int32_t *d_membership,
                                                   void *cuda_stream, double *q_out) {
  if (!q_out || n < 1 || !d_offsets || !d_cols || !d_membership) {
    set_handle_free_error("leiden_modularity_noalloc: null pointer or n < 1");
    return LEIDEN_ERR_ARG;
  }
  if (n > NOALLOC_MAX_VERTICES) {
    set_handle_free_error("leiden_modularity_noalloc: n exceeds the fixed scratch of 4194304 vertices");
    return LEIDEN_ERR_ARG;
  }
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) {
    set_handle_free_error(std::string("leiden_modularity_noalloc: cudaGetDevice: ") + cudaGetErrorString(e));
    return LEIDEN_ERR_CUDA;
  }
  if (dev < 0 || dev >= MAX_DEVICES) {
    set_handle_free_error("leiden_modularity_noalloc: device ordinal " + std::to_string(dev) +
                          " is beyond the 64 devices whose scratch address is cached");
    return LEIDEN_ERR_CUDA;
  }
  int64_t *scr = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_scratch_mu);
    if (!g_scratch_ptr[dev]) {
      void *p = nullptr;
      e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
      if (e != cudaSuccess || !p) {
        set_handle_free_error(std::string("leiden_modularity_noalloc: cudaGetSymbolAddress: ") + cudaGetErrorString(e));
        return LEIDEN_ERR_CUDA;
      }
      g_scratch_ptr[dev] = (int64_t *)p;
    }
    scr = g_scratch_ptr[dev];
  }
  cudaStream_t s = (cudaStream_t)cuda_stream;
  int sms = 152;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  ld_note_launch(), k_na_clear<<<grid_for(n, 256), 256, 0, s>>>(n, scr);
  if (d_weights)
    ld_note_launch(), k_na_rows<false><<<sms * 8, 256, 0, s>>>(n, d_offsets, d_cols, d_weights, d_membership, scr);
  else
    ld_note_launch(), k_na_rows<true><<<sms * 8, 256, 0, s>>>(n, d_offsets, d_cols, nullptr, d_membership, scr);
  ld_note_launch(), k_na_sq<<<grid_for(n, 256), 256, 0, s>>>(n, d_membership, scr);
  int64_t cnt[NOALLOC_COUNTERS] = {};
  e = cudaMemcpyAsync(cnt, scr + NOALLOC_MAX_VERTICES, sizeof(cnt), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) {
    set_handle_free_error(std::string("leiden_modularity_noalloc: ") + cudaGetErrorString(e));
    return LEIDEN_ERR_CUDA;
  }
  if (cnt[C_BAD]) {
    set_handle_free_error("leiden_modularity_noalloc: membership id outside [0, n)");
    return LEIDEN_ERR_ARG;
  }
  if (cnt[C_BADCOL]) {
    set_handle_free_error("leiden_modularity_noalloc: column id outside [0, n)");
    return LEIDEN_ERR_ARG;
  }
  int64_t m2 = cnt[C_M2];
  if (m2 == 0) {
    *q_out = 0.0;
    return LEIDEN_OK;
  }
  i128 sq = (i128)(((u128)(uint64_t)cnt[C_SQ_HI] << 64) | (u128)(uint64_t)cnt[C_SQ_LO]);
  i128 num = (i128)m2 * cnt[C_SIGMA] - sq;
  *q_out = i128_to_double(num) / ((double)m2 * (double)m2);
  return LEIDEN_OK;
}

