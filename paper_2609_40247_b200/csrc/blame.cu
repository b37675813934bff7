// ta_blame_gaps: why was a device stream idle, and which host calls did the idle
// time overlap.  A gap counts against the host when the work that ended it was
// submitted only after the stream had gone idle (the late-dispatch test of Sec. 6.2);
// idle time is charged to the operators that were running meanwhile (Sec. 9.1).
//
// Input: the long-gap list of ta_stream_gaps (ordered by lane, then time) and the
// launch of every device record (ta_correlate_launches).
//   k_blame_classify  per long gap: TAIL / NO_LAUNCH / SUBMISSION (the launch of the
//                     record that ends the gap started at or after the gap began) /
//                     QUEUED, folded per warp into per-window counts and lengths;
//   a scan            running total of the gap lengths along the list;
//   k_blame_lanes     the list range of every lane (binary search);
//   k_blame_ops       per OP record: for each device stream of its process the total
//                     long-gap length before a time t is (running total at the last
//                     gap that starts before t) + min(t - its start, its length); the
//                     operator is charged C(ts_end) - C(ts_start), summed over streams.
// The gap list is small (it stays in L2), the OP pass reads 18 B per host record.
#include <climits>
#include <cstring>
#include <vector>

#include "scan.cuh"
#include "ta_internal.cuh"

#define BL_THREADS 256
#define BL_TILE (BL_THREADS * 4)
#define BL_TILE_FEW BL_THREADS  // tiles of windows that have up to BL_FEW of them
#define BL_FEW 1024
#define BL_LANES 64
#define BL_GAPS 768    // gaps staged on chip: 18 KB, five CTAs per SM

struct BlameArgs {
  int64_t n, n_valid, m;  // m = long gaps
  int n_lanes, W;
  const ta_long_gap *list;
  const int32_t *launch_of;
  const int64_t *ts, *te;
  const int16_t *kind;
  const int32_t *lane_off, *lane_window, *lane_slot, *lane_dom_end, *lane_dom_next;
  const int16_t *lane_domain;
  int32_t *g_class, *g_launch;
  u64 *win_count, *win_ns;  // [W][4]
  u64 *pre;                 // exclusive running total of gap_len along the list
  int32_t *lane_first;      // [n_lanes + 1] first list entry of every lane
  int64_t *op_gap_ns;
  const int32_t *status;
};

__global__ void __launch_bounds__(256) k_blame_classify(BlameArgs a) {
  TA_PDL();
  if (ta_failed(a.status)) return;
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31;
  int cls = -1, w = -1;
  u64 len = 0;
  if (k < a.m) {
    const ta_long_gap g = a.list[k];
    int32_t l = -1;
    if (g.next_event < 0) cls = TA_BLAME_TAIL;
    else {
      l = a.launch_of[g.next_event];
      cls = l < 0 ? TA_BLAME_NO_LAUNCH : (a.ts[l] >= g.gap_start ? TA_BLAME_SUBMISSION : TA_BLAME_QUEUED);
    }
    a.g_class[k] = cls;
    a.g_launch[k] = l;
    w = a.lane_window[g.lane];
    len = (u64)g.gap_len;
  }
  // per class and warp: one pair of atomics when the warp sits in one window
  const u32 act = __ballot_sync(0xffffffffu, cls >= 0);
  if (!act) return;
  const int w0 = __shfl_sync(0xffffffffu, w, __ffs(act) - 1);
  if (__all_sync(0xffffffffu, cls < 0 || w == w0)) {
#pragma unroll
    for (int c = 0; c < 4; c++) {
      const u32 mine = __ballot_sync(0xffffffffu, cls == c);
      const u64 t = warp_reduce(cls == c ? len : 0ull, OpAdd());
      if (lane == 0 && mine) {
        atomicAdd(&a.win_count[(size_t)w0 * 4 + c], (u64)__popc(mine));
        atomicAdd(&a.win_ns[(size_t)w0 * 4 + c], t);
      }
    }
  } else if (cls >= 0) {
    atomicAdd(&a.win_count[(size_t)w * 4 + cls], 1ull);
    atomicAdd(&a.win_ns[(size_t)w * 4 + cls], len);
  }
}

struct GapLenIn {
  const ta_long_gap *list;
  __device__ u64 operator()(int64_t k) const { return (u64)list[k].gap_len; }
};
struct GapLenOut {
  u64 *pre;
  __device__ void operator()(int64_t k, u64 excl, u64) const { pre[k] = excl; }
};

// lane_first[l] = number of list entries whose lane is < l
__global__ void __launch_bounds__(256) k_blame_lanes(BlameArgs a) {
  TA_PDL();
  if (ta_failed(a.status)) return;
  const int l = blockIdx.x * blockDim.x + threadIdx.x;
  if (l > a.n_lanes) return;
  int64_t lo = 0, hi = a.m;
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if (a.list[mid].lane < l) lo = mid + 1;
    else hi = mid;
  }
  a.lane_first[l] = (int32_t)lo;
}

// Long gaps by index, in the list or in a part of it staged on chip.
struct GapList {
  const ta_long_gap *list;
  const u64 *before;  // total length in front of an entry
  __device__ __forceinline__ i64 start(int64_t i) const { return list[i].gap_start; }
  __device__ __forceinline__ i64 len(int64_t i) const { return list[i].gap_len; }
  __device__ __forceinline__ u64 pre(int64_t i) const { return before[i]; }
};
struct GapStage {
  const i64 *starts, *lens;
  const u64 *before;
  __device__ __forceinline__ i64 start(int64_t i) const { return starts[i]; }
  __device__ __forceinline__ i64 len(int64_t i) const { return lens[i]; }
  __device__ __forceinline__ u64 pre(int64_t i) const { return before[i]; }
};
// number of gaps of the range [first, last) that start before time t
template <class Gaps>
__device__ __forceinline__ int64_t gaps_started_before(const Gaps &g, int64_t first, int64_t last, i64 t) {
  int64_t lo = first, hi = last;
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if (g.start(mid) < t) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}
// the same by a warp, 32 gaps at a time
template <class Gaps>
__device__ __forceinline__ int64_t warp_gaps_started_before(const Gaps &g, int64_t first, int64_t last, i64 t) {
  const int lane = threadIdx.x & 31;
  int64_t lo = first, hi = last;
  while (lo < hi) {
    const int64_t step = (hi - lo + 31) >> 5, i = lo + lane * step;
    const int c = __popc(__ballot_sync(0xffffffffu, i < hi && g.start(i) < t));
    if (c == 0) break;
    hi = min(hi, lo + c * step);
    lo += (c - 1) * step + 1;
  }
  return lo;
}
// total long-gap length of the range that lies before time t, given i = gaps_started_before(t)
template <class Gaps>
__device__ __forceinline__ i64 gap_time_before(const Gaps &g, int64_t first, int64_t i, i64 t) {
  if (i == first) return 0;
  const int64_t k = i - 1;
  const i64 part = t - g.start(k), len = g.len(k);
  return (i64)(g.pre(k) - g.pre(first)) + (part < len ? part : len);
}
// length of [s, e) that lies inside the gaps of the range
template <class Gaps>
__device__ __forceinline__ i64 gap_time_within(const Gaps &g, int64_t first, int64_t last, i64 s, i64 e) {
  const int64_t ie = gaps_started_before(g, first, last, e);
  if (ie == first) return 0;  // every gap starts at or after e
  const i64 start = g.start(ie - 1);
  if (start < s && start + g.len(ie - 1) <= s) return 0;  // the last gap before e ends before s
  const int64_t is = start < s ? ie : gaps_started_before(g, first, ie, s);
  return gap_time_before(g, first, ie, e) - gap_time_before(g, first, is, s);
}

// One tile of 1024 (256) positions per CTA.  An operator's charge is two binary searches in each of its
// process's streams, a chain of some thirty dependent reads per stream; the operators of the tile are
// listed first and the (operator, stream) pairs are dealt out over the threads, so that no lane idles
// beside a launch record and no thread walks eight streams one after the other (one thread per eight
// records: 120 us for a prefill window of 250 k records, 195 us for 8 M decode records).  The gaps
// that can matter to the tile are few, as a rule, and are searched on chip.
// A window of few tiles leaves SMs idle and waits for a tile's rounds of pairs, ten of them in a prefill
// window of 250 k records: a quarter of the tile takes 51 us to 25 there (half: 33).  Where there are tiles
// enough the searches that a tile makes once count instead (8 M records 72 us, 88 by halves, 143 by
// quarters); the line is where a call's last CTA still brings its results back.
template <int TILE>
__device__ __forceinline__ void blame_ops(const BlameArgs &a) {
  __shared__ int s_lane0, s_n, s_most;
  __shared__ u64 s_sum[TILE];
  __shared__ uint16_t s_op[TILE];
  __shared__ int32_t s_dlo[TILE];
  __shared__ uint16_t s_dn[TILE];
  __shared__ int s_d0;                       // first device lane of the tile's operators, -1: there are several processes
  __shared__ i64 s_from, s_to;               // earliest start, latest end among them
  __shared__ int32_t s_lo[BL_LANES], s_hi[BL_LANES];  // per stream: the gaps that can matter to them
  __shared__ int32_t s_at[BL_LANES + 1];              // and where they are staged
  __shared__ i64 s_start[BL_GAPS], s_len[BL_GAPS];
  __shared__ u64 s_pre[BL_GAPS];
  if (ta_failed(a.status)) return;
  const int tid = threadIdx.x;
  const int64_t tile_start = (int64_t)blockIdx.x * TILE;
  if (tile_start >= a.n_valid) return;
  if (tid < 32) {
    const int l = tile_lane_search(a.lane_off, a.n_lanes, tile_start);
    if (tid == 0) { s_lane0 = l; s_n = 0; s_most = 0; s_d0 = -2; s_from = INT64_MAX; s_to = INT64_MIN; }
  }
  __syncthreads();
  const int l0 = s_lane0;
  const int64_t tile_end = min(tile_start + TILE, a.n_valid);
  if (span_outside_domain(a.lane_domain, a.lane_dom_end, l0, tile_end, 0)) return;
  int l = l0, cur = -1, dlo = 0, dn = 0;
  i64 from = INT64_MAX, to = INT64_MIN;
  int64_t next_off = a.lane_off[l + 1];
  constexpr int PER = TILE / BL_THREADS;
  bool op[PER];
#pragma unroll
  for (int k = 0; k < PER; k++) {
    const int64_t p = tile_start + k * BL_THREADS + tid;
    op[k] = p < tile_end && a.kind[p] == TA_KIND_OP;
  }
  i64 ps[PER], pe[PER];
#pragma unroll
  for (int k = 0; k < PER; k++) {
    const int64_t p = tile_start + k * BL_THREADS + tid;
    ps[k] = op[k] ? (i64)a.ts[p] : INT64_MAX;
    pe[k] = op[k] ? (i64)a.te[p] : INT64_MIN;
  }
#pragma unroll
  for (int k = 0; k < PER; k++) {
    const int x = k * BL_THREADS + tid;
    const int64_t p = tile_start + x;
    if (op[k]) {
      while (p >= next_off) { l++; next_off = a.lane_off[l + 1]; }
      if (l != cur) {  // device lanes of the record's (window, process)
        cur = l;
        dlo = a.lane_dom_next[l];
        int dhi = dlo;
        const int slot = a.lane_slot[l];
        // slots do not descend: the run of device lanes is this process's if its last lane is (one
        // lane after the other: 8 M records 82 us)
        const int run_end = dlo < a.n_lanes ? a.lane_dom_next[dlo] : dlo;
        if (run_end > dlo && a.lane_slot[run_end - 1] == slot) dhi = run_end;
        else
          while (dhi < run_end && a.lane_slot[dhi] == slot) dhi++;
        dn = dhi - dlo;
      }
    }
    // the warp's operators take their places with one add
    const bool take = op[k] && dn > 0;
    const u32 m = __ballot_sync(0xffffffffu, take);
    if (m == 0) continue;
    int base = 0;
    if ((tid & 31) == 0) base = atomicAdd(&s_n, __popc(m));
    const int i = __shfl_sync(0xffffffffu, base, 0) + __popc(m & ((1u << (tid & 31)) - 1u));
    if (!take) continue;
    s_op[i] = (uint16_t)x;
    s_dlo[i] = dlo;
    s_dn[i] = (uint16_t)dn;
    s_sum[i] = 0;
    if (dn > s_most) atomicMax(&s_most, dn);
    if (s_d0 != dlo && atomicCAS(&s_d0, -2, dlo) != -2 && s_d0 != dlo) s_d0 = -1;
    from = min(from, ps[k]);
    to = max(to, pe[k]);
  }
  from = (i64)(~warp_reduce(~((u64)from ^ (1ull << 63)), OpMax()) ^ (1ull << 63));
  to = (i64)(warp_reduce((u64)to ^ (1ull << 63), OpMax()) ^ (1ull << 63));
  if ((tid & 31) == 0 && from <= to) { atomicMin(&s_from, from); atomicMax(&s_to, to); }
  __syncthreads();
  const int ops = s_n, most = s_most;
  // Operators of one tile lie close together in time: with one search per stream for all of them, each
  // has to look among a few gaps only.
  const bool one = s_d0 >= 0 && most <= BL_LANES;
  const GapList list{a.list, a.pre};
  if (one)
    for (int d = tid >> 5; d < most; d += BL_THREADS / 32) {  // a warp per stream
      const int64_t first = a.lane_first[s_d0 + d], last = a.lane_first[s_d0 + d + 1];
      const int64_t lo = warp_gaps_started_before(list, first, last, s_from);
      const int64_t hi = warp_gaps_started_before(list, lo, last, s_to);
      if ((tid & 31) == 0) {
        s_lo[d] = (int32_t)(lo > first ? lo - 1 : first);
        s_hi[d] = (int32_t)hi;
      }
    }
  if (one) __syncthreads();
  bool staged = false;
  if (one) {
    if (tid == 0) {
      int at = 0;
      for (int d = 0; d < most; d++) {
        s_at[d] = at;
        at += s_hi[d] - s_lo[d];
      }
      s_at[most] = at;
    }
    __syncthreads();
    staged = s_at[most] <= BL_GAPS;
    if (staged) {
      for (int d = tid >> 5; d < most; d += BL_THREADS / 32)
        for (int k = tid & 31; k < s_hi[d] - s_lo[d]; k += 32) {
          const int64_t g = s_lo[d] + k;
          s_start[s_at[d] + k] = list.start(g);
          s_len[s_at[d] + k] = list.len(g);
          s_pre[s_at[d] + k] = list.pre(g);
        }
      __syncthreads();
    }
  }
  const GapStage stage{s_start, s_len, s_pre};
  for (int q = tid; q < ops * most; q += BL_THREADS) {
    const int i = q / most, d = q - i * most;  // (a tile nearly always lies in one process: all pairs exist)
    if (d >= s_dn[i]) continue;
    const int64_t p = tile_start + s_op[i];
    i64 t = 0;
    if (staged) {
      if (s_at[d] < s_at[d + 1]) t = gap_time_within(stage, s_at[d], s_at[d + 1], a.ts[p], a.te[p]);
    } else {
      const int64_t first = one ? s_lo[d] : a.lane_first[s_dlo[i] + d], last = one ? s_hi[d] : a.lane_first[s_dlo[i] + d + 1];
      if (first < last) t = gap_time_within(list, first, last, a.ts[p], a.te[p]);
    }
    if (t) atomicAdd(&s_sum[i], (u64)t);
  }
  __syncthreads();
  for (int i = tid; i < ops; i += BL_THREADS)
    if (s_sum[i]) a.op_gap_ns[tile_start + s_op[i]] = (i64)s_sum[i];
}
template <int TILE, bool TAIL>
__global__ void __launch_bounds__(BL_THREADS) k_blame_ops(BlameArgs a, Tail tail) {
  TA_PDL();
  blame_ops<TILE>(a);
  if (TAIL) run_tail(tail);
}

ta_status ta_run_blame(ta_window *h, const ta_gap_result *gaps, ta_blame_result *out,
                       ta_blame_summary *out_summary) {
  cudaStream_t st = h->stream;
  memset(out, 0, sizeof(*out));
  const int W = h->W;
  const int64_t n = h->n, nn = n > 0 ? n : 1, m = gaps->n_long_gaps, mm = m > 0 ? m : 1;
  const int L = h->sorted.n_lanes;
  for (int w = 0; w < W && out_summary; w++) memset(&out_summary[w], 0, sizeof(ta_blame_summary));

  size_t kb = Carver::pad((size_t)nn * 8) + 2 * Carver::pad((size_t)mm * 4) + 256;
  void *keep = ta_dalloc(h, kb);
  if (!keep) return TA_ERR_OOM;
  Carver ck(keep);
  int64_t *op_gap = ck.take<int64_t>(nn);
  int32_t *g_class = ck.take<int32_t>(mm), *g_launch = ck.take<int32_t>(mm);
  TA_CHECK_CUDA(h, cudaMemsetAsync(op_gap, 0, (size_t)nn * 8, st));
  out->n_long_gaps = m;
  out->g_class = g_class; out->g_launch = g_launch; out->op_gap_ns = op_gap;
  h->d_op_gap_ns = op_gap;
  if (m == 0 || h->n_valid == 0) return TA_OK;

  size_t tb = 2 * Carver::pad((size_t)W * 4 * 8) + Carver::pad((size_t)mm * 8) +
              Carver::pad((size_t)(L + 2) * 4) + scan_temp_bytes(m) + 256;
  void *tmpb = ta_dalloc(h, tb);
  if (!tmpb) return TA_ERR_OOM;
  Carver ct(tmpb);
  BlameArgs a;
  memset(&a, 0, sizeof(a));
  a.win_count = ct.take<u64>((size_t)W * 4);
  a.win_ns = ct.take<u64>((size_t)W * 4);
  TA_CHECK_CUDA(h, cudaMemsetAsync(tmpb, 0, ct.off, st));
  a.pre = ct.take<u64>(mm);
  a.lane_first = ct.take<int32_t>(L + 2);
  void *scan_mem = ct.base + ct.off;
  a.n = n; a.n_valid = h->n_valid; a.m = m; a.n_lanes = L; a.W = W;
  a.list = gaps->long_gaps; a.launch_of = h->join.launch_of;
  a.ts = h->sorted.ts_start; a.te = h->sorted.ts_end; a.kind = h->sorted.kind;
  a.lane_off = h->sorted.lane_off; a.lane_window = h->sorted.lane_window; a.lane_slot = h->d_lane_slot;
  a.lane_dom_end = h->d_lane_dom_end; a.lane_dom_next = h->d_lane_dom_next;
  a.lane_domain = h->sorted.lane_domain;
  a.g_class = g_class; a.g_launch = g_launch; a.op_gap_ns = op_gap; a.status = h->d_status;

  ta_launch(k_blame_classify, (unsigned)((m + 255) / 256), 256, 0, st, a);
  ScanTemp s1;
  TA_TRY(scan_temp_init(h, scan_mem, m, &s1));
  GapLenIn gi{a.list};
  GapLenOut go{a.pre};
  TA_TRY((launch_scan<OpAdd, GapLenIn, GapLenOut>(h, m, gi, go, OpAdd(), s1)));
  ta_launch(k_blame_lanes, (unsigned)((L + 1 + 255) / 256), 256, 0, st, a);
  const bool few = h->n_valid <= (int64_t)BL_TILE_FEW * BL_FEW;
  const int tile = few ? BL_TILE_FEW : BL_TILE;
  const int64_t tiles = (h->n_valid + tile - 1) / tile;
  std::vector<u64> hc((size_t)W * 4), hn((size_t)W * 4);
  int32_t words[ST_WORDS];
  TA_TRY(ta_queue_d2h(h, hc.data(), a.win_count, (size_t)W * 32));
  TA_TRY(ta_queue_d2h(h, hn.data(), a.win_ns, (size_t)W * 32));
  TA_TRY(ta_queue_d2h(h, words, h->d_status, sizeof(words)));
  const Tail tail = ta_tail(h, tiles);
  ta_launch(few ? (tail.m ? k_blame_ops<BL_TILE_FEW, true> : k_blame_ops<BL_TILE_FEW, false>)
                : (tail.m ? k_blame_ops<BL_TILE, true> : k_blame_ops<BL_TILE, false>),
            (unsigned)tiles, BL_THREADS, 0, st, a, tail);
  TA_CHECK_CUDA(h, cudaGetLastError());
  TA_TRY(ta_sync_fetch(h));
  ta_dfree(h, tmpb);
  if (words[ST_ERR]) return (ta_status)words[ST_ERR];
  for (int w = 0; w < W && out_summary; w++)
    for (int c = 0; c < 4; c++) {
      out_summary[w].count[c] = (int64_t)hc[(size_t)w * 4 + c];
      out_summary[w].ns[c] = (int64_t)hn[(size_t)w * 4 + c];
    }
  return TA_OK;
}
