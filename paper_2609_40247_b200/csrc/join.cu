// ta_correlate_launches: every device record is joined to the host call that
// submitted it through the correlation id both carry (Sec. 5.2; Fig. "Key
// performance observations" (a)).  Key =
// (window, pid, corr_id); the smallest sorted position among equal LAUNCH keys
// wins.
//
// Two paths, same results:
//   direct   when the correlation ids of each (window, pid) span a compact
//            range (they count up per process in real traces): a table of
//            sorted positions indexed by corr_id - min, filled with atomicMin.
//            Launches and kernels are time-ordered, so the table is touched
//            nearly sequentially.
//   general  any 64-bit ids: launches and probes are compacted, stably sorted
//            by (slot, corr_id) with the pair sorter, and each probe takes the
//            head of its run if that head is a LAUNCH.
// HBM-bound: streams kind/corr/ts columns, writes three outputs per record.
#include <climits>
#include <cstring>
#include <vector>

#include "scan.cuh"
#include "ta_internal.cuh"

#define JN_THREADS 512
#define JN_ITEMS 4
#define JN_TILE (JN_THREADS * JN_ITEMS)
// entry of the direct table: complement of the smallest position, 0 = empty

struct JoinArgs {
  int64_t n, n_valid;
  int n_lanes;
  const int16_t *kind;
  const int64_t *corr, *ts, *te;
  const int32_t *lane_off, *lane_slot, *lane_window, *lane_dom_end;
  const int16_t *lane_domain;
  // per slot (window * n_pids + pid rank)
  i64 *slot_min, *slot_max;       // corr range of LAUNCH records
  const i64 *slot_base;           // direct path: table offset of the slot, -1 = no launches
  u32 *table;                     // direct path
  const int32_t *found;           // general path: winner launch per launch/probe position
  int32_t *launch_of, *kol;
  int64_t *latency, *qdelay;
  ta_join_summary *sum;           // device, per window
  const int32_t *status;
};

__device__ __forceinline__ u64 bias64(i64 v) { return (u64)v ^ (1ull << 63); }
__host__ __device__ __forceinline__ i64 unbias64(u64 v) { return (i64)(v ^ (1ull << 63)); }

// ---- direct path: fill the table -------------------------------------------
__global__ void __launch_bounds__(JN_THREADS) k_join_build(JoinArgs a) {
  TA_PDL();
  __shared__ int s_lane0;
  if (ta_failed(a.status)) return;
  const int tid = threadIdx.x;
  const int64_t tile_start = (int64_t)blockIdx.x * JN_TILE;
  if (tile_start >= a.n_valid) return;
  if (tid < 32) {
    const int l = tile_lane_search(a.lane_off, a.n_lanes, tile_start);
    if (tid == 0) s_lane0 = l;
  }
  __syncthreads();
  const int l0 = s_lane0;
  // launches live in host lanes: a tile of device lanes has none
  if (span_outside_domain(a.lane_domain, a.lane_dom_end, l0, min(tile_start + JN_TILE, a.n_valid), 0)) return;
  const int64_t p0 = tile_start + (int64_t)tid * JN_ITEMS;
  int16_t kd[JN_ITEMS];
  i64 c[JN_ITEMS];
  loadn_i16<JN_ITEMS>(a.kind, p0, a.n, 9, kd);
  loadn_i64<JN_ITEMS>(a.corr, p0, a.n, c);
  int l = l0;
  int64_t next_off = a.lane_off[l + 1];
  int slot = a.lane_slot[l];
#pragma unroll
  for (int j = 0; j < JN_ITEMS; j++) {
    const int64_t p = p0 + j;
    if (p < a.n_valid && kd[j] == TA_KIND_LAUNCH) {
      while (p >= next_off) { l++; next_off = a.lane_off[l + 1]; slot = a.lane_slot[l]; }
      const i64 idx = a.slot_base[slot] + (c[j] - a.slot_min[slot]);
      atomicMax(&a.table[idx], ~(u32)p);
    }
  }
}

// ---- pass 2: probes ----------------------------------------------------------
// 256 threads x JP_ITEMS consecutive positions; every output column is written once.
#define JP_THREADS 256
#ifndef JP_MINB
#define JP_MINB 3
#endif
#ifndef JP_ITEMS
#define JP_ITEMS 8
#endif
#define JP_TILE (JP_THREADS * JP_ITEMS)

// adds a group of probes to the row of their window
__device__ __forceinline__ void join_emit(ta_join_summary *sm, const u64 *t) {
  if (t[0] == 0) return;
  atomicAdd((u64 *)&sm->n_probe, t[0]);
  if (t[1] == 0) return;
  atomicAdd((u64 *)&sm->n_matched, t[1]);
  atomicAdd((u64 *)&sm->sum_latency, t[2]);
  atomicAdd((u64 *)&sm->sum_queue, t[3]);
  // (codes with 0 as "none"; the host turns them into times)
  atomicMax((u64 *)&sm->max_latency, t[4]);
  atomicMax((u64 *)&sm->min_latency, t[5]);
  atomicMax((i64 *)&sm->max_queue, (i64)t[6]);
}

template <bool DIRECT>
__global__ void __launch_bounds__(JP_THREADS, JP_MINB) k_join_probe(JoinArgs a) {
  TA_PDL();
  __shared__ u64 red[7][JP_THREADS / 32];
  __shared__ int s_lane0, s_lane1;
  if (ta_failed(a.status)) return;
  const int tid = threadIdx.x, lane = tid & 31;
  const int64_t tile_start = (int64_t)blockIdx.x * JP_TILE;
  constexpr int IT = JP_ITEMS;
  const int64_t p0 = tile_start + (int64_t)tid * IT;
  if (tid == 0) { s_lane0 = -1; s_lane1 = -1; }
  __syncthreads();
  if (tid < 32 && tile_start < a.n_valid && a.n_lanes > 0) {
    int l = tile_lane_search(a.lane_off, a.n_lanes, tile_start);
    if (lane == 0) s_lane0 = l;
  }
  __syncthreads();
  const int l0 = s_lane0;
  // A tile of host lanes holds no probe: nothing to read, the three outputs are -1 / 0 / 0.
  if (l0 >= 0 && span_outside_domain(a.lane_domain, a.lane_dom_end, l0, min(tile_start + JP_TILE, a.n_valid), 1)) {
    int32_t lo0[IT];
    i64 z[IT];
#pragma unroll
    for (int j = 0; j < IT; j++) { lo0[j] = -1; z[j] = 0; }
    storen_i32<IT>(a.launch_of, p0, a.n, lo0);
    storen_i64<IT>(a.latency, p0, a.n, z);
    storen_i64<IT>(a.qdelay, p0, a.n, z);
    return;
  }
  // kinds, correlation ids and start times are requested together: one round of memory
  // latency less than loading the ids only where the kinds ask for them
  int16_t kd[IT];
  i64 c[IT], s[IT];
  loadn_i16<IT>(a.kind, p0, a.n, 0, kd);
  loadn_i64<IT>(a.corr, p0, a.n, c);
  loadn_i64<IT>(a.ts, p0, a.n, s);
  unsigned pm = 0;  // probes among the thread's records
#pragma unroll
  for (int j = 0; j < IT; j++)
    if (p0 + j < a.n_valid && (kd[j] == TA_KIND_KERNEL || kd[j] == TA_KIND_MEMCPY)) pm |= 1u << j;
  int32_t lo[IT];
  int wn[IT];  // window of the probe
  {
    int l = l0;
    int64_t next_off = l >= 0 ? (int64_t)a.lane_off[l + 1] : LLONG_MAX;
    int slot = l >= 0 ? a.lane_slot[l] : 0;
    int win = l >= 0 ? a.lane_window[l] : 0;
#pragma unroll
    for (int j = 0; j < IT; j++) {
      lo[j] = -1;
      wn[j] = -1;
      if (pm & (1u << j)) {
        const int64_t p = p0 + j;
        if (p >= next_off) {
          do { l++; next_off = a.lane_off[l + 1]; } while (p >= next_off);
          slot = a.lane_slot[l];
          win = a.lane_window[l];
        }
        wn[j] = win;
        if (DIRECT) {
          const i64 base = a.slot_base[slot];
          if (base >= 0 && c[j] >= a.slot_min[slot] && c[j] <= a.slot_max[slot]) {
            const u32 v = a.table[base + (c[j] - a.slot_min[slot])];
            lo[j] = v == 0 ? -1 : (int32_t)~v;
          }
        } else {
          lo[j] = a.found[p];
        }
      }
    }
    const int64_t plast = min(tile_start + JP_TILE, a.n_valid) - 1;
    if (plast >= p0 && plast < p0 + IT) {
      while (plast >= next_off) { l++; next_off = a.lane_off[l + 1]; }
      s_lane1 = l;
    }
  }
  // launch times of the matched probes (independent gathers, issued together)
  i64 ls[IT], le[IT];
#pragma unroll
  for (int j = 0; j < IT; j++) {
    ls[j] = le[j] = 0;
    if (lo[j] >= 0) { ls[j] = a.ts[lo[j]]; le[j] = a.te[lo[j]]; }
  }
  i64 lat[IT], q[IT];
  // probes, matches, latencies and delays summed; largest latency, largest complement, largest delay
  u64 acc[7] = {0, 0, 0, 0, 0, 0, 0};
  int wm = -1;
#pragma unroll
  for (int j = 0; j < IT; j++) {
    lat[j] = q[j] = 0;
    if (!(pm & (1u << j))) continue;
    const bool matched = lo[j] >= 0;
    if (matched) {
      lat[j] = s[j] - ls[j];
      const i64 d = s[j] - le[j];
      q[j] = d > 0 ? d : 0;
      atomicAdd(&a.kol[lo[j]], 1);
    }
    if (wm < 0) wm = wn[j];
    if (wn[j] == wm) {
      acc[0]++;
      if (matched) {
        acc[1]++;
        acc[2] += (u64)lat[j];
        acc[3] += (u64)q[j];
        acc[4] = max(acc[4], bias64(lat[j]));
        acc[5] = max(acc[5], ~bias64(lat[j]));
        acc[6] = max(acc[6], (u64)q[j]);
      }
    } else {  // a thread that straddles a window boundary
      const u64 one[7] = {1, matched ? 1ull : 0ull, (u64)lat[j], (u64)q[j], bias64(lat[j]), ~bias64(lat[j]), (u64)q[j]};
      join_emit(&a.sum[wn[j]], one);
    }
  }
  storen_i32<IT>(a.launch_of, p0, a.n, lo);
  storen_i64<IT>(a.latency, p0, a.n, lat);
  storen_i64<IT>(a.qdelay, p0, a.n, q);
  __syncthreads();
  if (l0 < 0) return;
  fold_by_window<4, 3, JP_THREADS / 32>(acc, wm, a.lane_window[l0], a.lane_window[s_lane1], red,
                                        [&](int w, const u64 *t) { join_emit(&a.sum[w], t); });
}

// ---- pass 3: launch statistics (duplicates, orphans) ---------------------------
#define JS_TILE (JP_THREADS * 8)
// adds a group of launches to the row of their window
__device__ __forceinline__ void launch_emit(ta_join_summary *sm, const u64 *t) {
  if (t[0]) atomicAdd((u64 *)&sm->n_launch, t[0]);
  if (t[1]) atomicAdd((u64 *)&sm->n_dup_launch, t[1]);
  if (t[2]) atomicAdd((u64 *)&sm->n_orphan_launch, t[2]);
}

template <bool DIRECT>
__device__ __forceinline__ void join_launch_stats(const JoinArgs &a) {
  __shared__ u64 red[3][JP_THREADS / 32];
  __shared__ int s_lane0, s_lane1;
  if (ta_failed(a.status)) return;
  const int tid = threadIdx.x, lane = tid & 31;
  const int64_t tile_start = (int64_t)blockIdx.x * JS_TILE;
  const int64_t p0 = tile_start + (int64_t)tid * 8;
  if (tid == 0) { s_lane0 = -1; s_lane1 = -1; }
  __syncthreads();
  if (tid < 32 && tile_start < a.n_valid && a.n_lanes > 0) {
    int l = tile_lane_search(a.lane_off, a.n_lanes, tile_start);
    if (lane == 0) s_lane0 = l;
  }
  __syncthreads();
  const int l0 = s_lane0;
  // launches live in host lanes: a tile of device lanes has none
  if (l0 < 0 || span_outside_domain(a.lane_domain, a.lane_dom_end, l0, min(tile_start + JS_TILE, a.n_valid), 0))
    return;
  // kinds, correlation ids and kernel counts of the thread's records together, then the table
  // entries of its launches together: two rounds of memory latency
  int16_t kd[8];
  i64 cr[8];
  int32_t nk[8];
  load8_i16(a.kind, p0, a.n, 0, kd);
  load8_i64(a.corr, p0, a.n, cr);
  if (p0 + 8 <= a.n) {
    const int4 x = *reinterpret_cast<const int4 *>(a.kol + p0), y = *reinterpret_cast<const int4 *>(a.kol + p0 + 4);
    nk[0] = x.x; nk[1] = x.y; nk[2] = x.z; nk[3] = x.w; nk[4] = y.x; nk[5] = y.y; nk[6] = y.z; nk[7] = y.w;
  } else {
#pragma unroll
    for (int j = 0; j < 8; j++) nk[j] = p0 + j < a.n ? a.kol[p0 + j] : 0;
  }
  unsigned lmask = 0;
#pragma unroll
  for (int j = 0; j < 8; j++)
    if (p0 + j < a.n_valid && kd[j] == TA_KIND_LAUNCH) lmask |= 1u << j;
  u64 acc[3] = {0, 0, 0};  // launches, duplicates, orphans of the thread's first window
  int wm = -1;
  {
    int l = l0;
    int64_t next_off = (int64_t)a.lane_off[l + 1];
    int wn[8];
    int32_t win[8];
#pragma unroll
    for (int j = 0; j < 8; j++) {
      wn[j] = -1;
      win[j] = -1;
      if (!(lmask & (1u << j))) continue;
      const int64_t p = p0 + j;
      while (p >= next_off) { l++; next_off = a.lane_off[l + 1]; }
      wn[j] = a.lane_window[l];
      if (DIRECT) {
        const int slot = a.lane_slot[l];
        const i64 base = a.slot_base[slot];
        if (base >= 0 && cr[j] >= a.slot_min[slot] && cr[j] <= a.slot_max[slot]) {
          const u32 v = a.table[base + (cr[j] - a.slot_min[slot])];
          win[j] = v == 0 ? -1 : (int32_t)~v;
        }
      } else {
        win[j] = a.found[p];
      }
    }
#pragma unroll
    for (int j = 0; j < 8; j++) {
      if (!(lmask & (1u << j))) continue;
      const bool dup = win[j] != (int32_t)(p0 + j);
      const bool orphan = !dup && nk[j] == 0;
      if (wm < 0) wm = wn[j];
      if (wn[j] == wm) {
        acc[0]++;
        acc[1] += dup;
        acc[2] += orphan;
      } else {
        const u64 one[3] = {1, dup, orphan};
        launch_emit(&a.sum[wn[j]], one);
      }
    }
    const int64_t plast = min(tile_start + JS_TILE, a.n_valid) - 1;
    if (plast >= p0 && plast < p0 + 8) {
      while (plast >= next_off) { l++; next_off = a.lane_off[l + 1]; }
      s_lane1 = l;
    }
  }
  __syncthreads();
  fold_by_window<3, 0, JP_THREADS / 32>(acc, wm, a.lane_window[l0], a.lane_window[s_lane1], red,
                                        [&](int w, const u64 *t) { launch_emit(&a.sum[w], t); });
}

template <bool DIRECT>
__global__ void __launch_bounds__(JP_THREADS) k_join_launch_stats(JoinArgs a, Tail tail) {
  TA_PDL();
  join_launch_stats<DIRECT>(a);
  run_tail(tail);
}

// ---- general path helpers -----------------------------------------------------
__global__ void __launch_bounds__(256) k_join_key_corr(const u32 *pos, int64_t m, const int64_t *corr,
                                                       u64 *out, const int32_t *status) {
  TA_PDL();
  if (ta_failed(status)) return;
  int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j < m) out[j] = bias64(corr[pos[j]]);
}
__global__ void __launch_bounds__(256) k_join_key_slot(const u32 *pos, int64_t m,
                                                       const int32_t *lane_off, int n_lanes,
                                                       const int32_t *lane_slot, u64 *out,
                                                       const int32_t *status) {
  TA_PDL();
  if (ta_failed(status)) return;
  int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j < m) out[j] = (u64)lane_slot[lane_of_pos(lane_off, n_lanes, pos[j])];
}
struct JoinHeadIn {
  const u64 *slot_key;
  const u32 *pos;
  const int64_t *corr;
  __device__ u64 operator()(int64_t j) const {
    bool head = j == 0 || slot_key[j] != slot_key[j - 1] || corr[pos[j]] != corr[pos[j - 1]];
    return head ? (u64)(j + 1) : 0ull;
  }
};
struct JoinHeadOut {
  const u32 *pos;
  const int16_t *kind;
  int32_t *found;
  __device__ void operator()(int64_t j, u64 excl, u64 v) const {
    u64 hd = (excl > v ? excl : v) - 1;  // index of the head of j's run
    u32 hp = pos[hd];
    found[pos[j]] = kind[hp] == TA_KIND_LAUNCH ? (int32_t)hp : -1;
  }
};

static int bit_length64(uint64_t v) {
  int b = 0;
  while (v) { b++; v >>= 1; }
  return b;
}

ta_status ta_run_correlate(ta_window *h, ta_join_summary *out_summary) {
  const int64_t n = h->n;
  const int W = h->W;
  const int n_slots = W * (h->n_pids > 0 ? h->n_pids : 1);
  cudaStream_t st = h->stream;
  const int64_t nn = n > 0 ? n : 1;
  size_t keep = Carver::pad(nn * 4) + 2 * Carver::pad(nn * 8) + 256;
  void *kb = ta_dalloc(h, keep);
  if (!kb) return TA_ERR_OOM;
  Carver ck(kb);
  int32_t *launch_of = ck.take<int32_t>(nn);
  int64_t *latency = ck.take<int64_t>(nn), *qdelay = ck.take<int64_t>(nn);
  ta_status zs;
  void *zb = ta_zalloc(h, Carver::pad(nn * 4) + Carver::pad((size_t)W * sizeof(ta_join_summary)), &zs);
  if (!zb) return zs;
  Carver cz(zb);
  int32_t *kol = cz.take<int32_t>(nn);
  ta_join_summary *d_sum = cz.take<ta_join_summary>(W);
  std::vector<ta_join_summary> hs(W);
  const std::vector<int64_t> &hmin = h->h_slot_min, &hmax = h->h_slot_max;

  JoinArgs a;
  memset(&a, 0, sizeof(a));
  a.n = n; a.n_valid = h->n_valid; a.n_lanes = h->sorted.n_lanes;
  a.kind = h->sorted.kind; a.corr = h->sorted.corr_id; a.ts = h->sorted.ts_start; a.te = h->sorted.ts_end;
  a.lane_off = h->sorted.lane_off; a.lane_slot = h->d_lane_slot; a.lane_window = h->sorted.lane_window;
  a.lane_domain = h->sorted.lane_domain; a.lane_dom_end = h->d_lane_dom_end;
  a.slot_min = h->d_slot_min; a.slot_max = h->d_slot_max; a.slot_base = h->d_slot_base;  // filled by the sort
  a.launch_of = launch_of; a.kol = kol; a.latency = latency; a.qdelay = qdelay; a.sum = d_sum;
  a.status = h->d_status;
  const unsigned grid = (unsigned)((n + JN_TILE - 1) / JN_TILE);
  const unsigned grid8 = (unsigned)((n + JS_TILE - 1) / JS_TILE);
  const unsigned grid_probe = (unsigned)((n + JP_TILE - 1) / JP_TILE);
  void *tmp_alloc = nullptr;
  bool direct = true;
  int32_t words[ST_WORDS];
  const bool small = W * sizeof(ta_join_summary) <= 4096;  // (more is copied once the kernels are queued)
  TA_TRY(ta_queue_d2h(h, words, h->d_status, sizeof(words)));
  if (small) TA_TRY(ta_queue_d2h(h, hs.data(), d_sum, W * sizeof(ta_join_summary)));
  if (n > 0) {
    // table size if every slot is addressed directly
    unsigned __int128 total = 0;
    for (int s = 0; s < n_slots; s++)
      if (hmin[s] <= hmax[s]) total += (unsigned __int128)((uint64_t)hmax[s] - (uint64_t)hmin[s]) + 1;
    const uint64_t limit = (uint64_t)4 * (uint64_t)n + 65536;
    direct = total <= limit;
    if (direct) {
      uint64_t M = (uint64_t)total;
      tmp_alloc = ta_zalloc(h, (size_t)(M > 0 ? M : 1) * 4, &zs);
      if (!tmp_alloc) return zs;
      a.table = (u32 *)tmp_alloc;
      ta_launch(k_join_build, grid, JN_THREADS, 0, st, a);
      ta_launch(k_join_probe<true>, grid_probe, JP_THREADS, 0, st, a);
      ta_launch(k_join_launch_stats<true>, grid8, JP_THREADS, 0, st, a, ta_tail(h, grid8));
    } else {
      // general path: compact, sort by (slot, corr) with sorted position as the stable tie-break
      size_t tb = Carver::pad(nn * 4) * 3 + Carver::pad(nn * 8) * 3 + scan_temp_bytes(n) * 2 +
                  ta_sort_temp_bytes(n) + 512;
      tmp_alloc = ta_dalloc(h, tb);
      if (!tmp_alloc) return TA_ERR_OOM;
      Carver ct(tmp_alloc);
      u32 *pos = ct.take<u32>(nn), *pos_s = ct.take<u32>(nn);
      int32_t *found = ct.take<int32_t>(nn);
      u64 *k_in = ct.take<u64>(nn), *k_s = ct.take<u64>(nn), *k_f = ct.take<u64>(nn);
      void *scan_mem1 = ct.base + ct.off; ct.off += scan_temp_bytes(n);
      void *scan_mem2 = ct.base + ct.off; ct.off += scan_temp_bytes(n);
      void *sort_tmp = ct.base + ct.off;
      ScanTemp t1;
      TA_TRY(scan_temp_init(h, scan_mem1, n, &t1));
      TA_TRY(launch_compact_kind(h, a.kind, h->n_valid,
                                 (1u << TA_KIND_LAUNCH) | (1u << TA_KIND_KERNEL) | (1u << TA_KIND_MEMCPY),
                                 pos, t1));
      u64 m64 = 0;
      TA_TRY(ta_queue_d2h(h, &m64, t1.total, 8));
      TA_TRY(ta_sync_fetch(h));
      TA_TRY(ta_queue_d2h(h, words, h->d_status, sizeof(words)));
      if (small) TA_TRY(ta_queue_d2h(h, hs.data(), d_sum, W * sizeof(ta_join_summary)));
      const int64_t m = (int64_t)m64;
      TA_CHECK_CUDA(h, cudaMemsetAsync(found, 0xFF, nn * 4, st));
      if (m > 0) {
        const int gb = (int)((m + 255) / 256);
        u32 *vscr = (u32 *)found;  // found is not needed before the sorts are done
        ta_launch(k_join_key_corr, gb, 256, 0, st, pos, m, a.corr, k_in, h->d_status);
        TA_TRY(ta_radix_sort_pairs(h, k_in, pos, k_s, vscr, k_f, pos_s, m, ta_make_plan(0, 64), nullptr,
                                   sort_tmp));
        ta_launch(k_join_key_slot, gb, 256, 0, st, pos_s, m, a.lane_off, a.n_lanes, a.lane_slot, k_in, h->d_status);
        int sb = bit_length64((uint64_t)(n_slots > 1 ? n_slots - 1 : 1));
        TA_TRY(ta_radix_sort_pairs(h, k_in, pos_s, k_s, vscr, k_f, pos, m, ta_make_plan(0, sb), nullptr,
                                   sort_tmp));
        TA_CHECK_CUDA(h, cudaMemsetAsync(found, 0xFF, nn * 4, st));
        ScanTemp t2;
        TA_TRY(scan_temp_init(h, scan_mem2, m, &t2));
        JoinHeadIn hin{k_f, pos, a.corr};
        JoinHeadOut hout{pos, a.kind, found};
        TA_TRY((launch_scan<OpMax, JoinHeadIn, JoinHeadOut>(h, m, hin, hout, OpMax(), t2)));
      }
      a.found = found;
      ta_launch(k_join_probe<false>, grid_probe, JP_THREADS, 0, st, a);
      ta_launch(k_join_launch_stats<false>, grid8, JP_THREADS, 0, st, a, ta_tail(h, grid8));
    }
    TA_CHECK_CUDA(h, cudaGetLastError());
  }
  if (!small) TA_TRY(ta_queue_d2h(h, hs.data(), d_sum, W * sizeof(ta_join_summary)));
  TA_TRY(ta_sync_fetch(h));
  if (tmp_alloc) ta_dfree(h, tmp_alloc);
  if (words[ST_ERR]) return (ta_status)words[ST_ERR];
  for (int w = 0; w < W; w++) {
    ta_join_summary &s = hs[w];
    s.n_unmatched = s.n_probe - s.n_matched;
    s.max_latency = s.n_matched ? unbias64((u64)s.max_latency) : 0;
    s.min_latency = s.n_matched ? unbias64(~(u64)s.min_latency) : 0;
    if (out_summary) out_summary[w] = s;
  }
  h->join.launch_of = launch_of;
  h->join.launch_latency = latency;
  h->join.queue_delay = qdelay;
  h->join.kernels_of_launch = kol;
  if (n == 0) {
    // nothing was launched: outputs are single dummy entries
  }
  return TA_OK;
}
