// What depends on the lanes of a window alone: the table of its lanes, and the order in which the gather
// takes its tiles.  Of one window both follow from the records counted per triple while it was loaded, and
// are made beside the first radix pass; else the gather notes where lanes begin.
#pragma once
#include "records.cuh"
#include "ta_internal.cuh"

// One CTA: compacts the non-empty lane codes into the lane table (code order is
// canonical order).  For few codes; k_scan with functors does the same for many.
// COUNTS: from the records per triple of the only window.
template <bool COUNTS>
__device__ __forceinline__ void lane_table(const LaneTable &t, const int32_t *status, u64 *tmp) {
  __shared__ u64 base;
  if (ta_failed(status)) {  // no lanes: every later call then finds nothing to index
    if (threadIdx.x == 0) { t.n_lanes_out[0] = 0; t.n_lanes_out[1] = 0; t.n_lanes_out[2] = 0; }
    return;
  }
  if (threadIdx.x == 0) { base = 0; t.n_lanes_out[2] = 0; }
  __syncthreads();
  // lanes in front << 32 | records in front
  for (int64_t c0 = 0; c0 < t.n_codes; c0 += blockDim.x) {
    const int64_t c = c0 + threadIdx.x;
    u32 cnt = 0;
    int32_t st = -1;
    if (c < t.n_codes) {
      if (COUNTS) cnt = t.tt->rank_cnt[c];
      else st = t.lane_start[c] - 1;
    }
    const bool some = COUNTS ? cnt > 0 : st >= 0;
    u64 total;
    const u64 ex = base + block_scan_exclusive<OpAdd>(some ? 1ull << 32 | cnt : 0ull, OpAdd(), tmp, &total);
    if (some) {
      if (COUNTS) st = (int32_t)(u32)ex;
      const int64_t l = (int64_t)(ex >> 32);
      if (l < t.cap) {
        const int w = COUNTS ? 0 : (int)(c >> t.tbits), r = COUNTS ? (int)c : (int)(c & ((1ll << t.tbits) - 1));
        const u64 code = t.tt->sorted_code[r];
        t.lane_window[l] = w;
        t.lane_pid[l] = code_pid(code);
        t.lane_stream[l] = code_stream(code);
        t.lane_domain[l] = code_domain(code);
        t.lane_off[l] = st;
        t.lane_slot[l] = w * t.n_pids + t.tt->pid_rank[r];
      }
    }
    __syncthreads();
    if (threadIdx.x == 0) base += total;
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    base >>= 32;
    const int64_t L = (int64_t)base;
    if (L < t.cap + 1) t.lane_off[L] = (int32_t)t.n_valid;
    *t.n_lanes_out = (int32_t)L;
  }
  __syncthreads();
  // per lane: the first later lane of the other domain, and the position where it begins (host
  // and device lanes alternate per (window, pid), so the runs are a few lanes long - but a batch
  // of device-only windows is one long run, hence a scan and no walk).  Going backwards over
  // the lanes, the nearest boundary at or behind lane l is a running maximum of
  // L - (index of the lane behind a boundary); chunks of blockDim.x lanes, carried in `base`.
  const int64_t L = (int64_t)base < t.cap ? (int64_t)base : t.cap;
  __syncthreads();  // every thread has read the lane count before `base` is reused
  if (threadIdx.x == 0) base = 0;
  __syncthreads();
  for (int64_t r0 = 0; r0 < L; r0 += blockDim.x) {
    const int64_t r = r0 + threadIdx.x;  // reversed lane index
    const int64_t l = L - 1 - r;
    u64 v = 0;
    if (r < L && l + 1 < L && t.lane_domain[l + 1] != t.lane_domain[l]) v = (u64)(L - (l + 1));
    u64 total;
    const u64 ex = block_scan_exclusive<OpMax>(v, OpMax(), tmp, &total);
    if (r < L) {
      u64 best = ex > v ? ex : v;
      best = best > base ? best : base;
      const int64_t m = best ? L - (int64_t)best : L;
      t.lane_dom_end[l] = m < L ? t.lane_off[m] : (int32_t)t.n_valid;
      t.lane_dom_next[l] = (int32_t)m;  // index of the first later lane of the other domain (L if none)
      if (t.lane_domain[l] == 1 && (l == 0 || t.lane_domain[l - 1] != 1)) atomicMax(&t.n_lanes_out[2], (int32_t)(m - l));
    }
    __syncthreads();
    if (threadIdx.x == 0) base = base > total ? base : total;
    __syncthreads();
  }
  // per device lane: how many device records sit in earlier lanes (their index once the device
  // records are taken out in order); t.n_lanes_out[1] = the number of device records
  if (threadIdx.x == 0) base = 0;
  __syncthreads();
  for (int64_t l0 = 0; l0 < L; l0 += blockDim.x) {
    const int64_t l = l0 + threadIdx.x;
    u64 sz = 0;
    if (l < L && t.lane_domain[l] == 1) sz = (u64)((l + 1 < L ? t.lane_off[l + 1] : (int32_t)t.n_valid) - t.lane_off[l]);
    u64 total;
    const u64 ex = block_scan_exclusive<OpAdd>(sz, OpAdd(), tmp, &total);
    if (l < L) t.lane_dev_base[l] = (int32_t)(base + ex);
    __syncthreads();
    if (threadIdx.x == 0) base += total;
    __syncthreads();
  }
  if (threadIdx.x == 0) t.n_lanes_out[1] = (int32_t)base;
}

// The order in which the gather takes its tiles.  Records of the lanes of one process arrive mixed, so
// lanes taken one after the other read the same sectors of the input again, long after they have
// left L2.  Here every lane is cut into as many parts as there are rounds, and a round takes
// the same part of all lanes: what arrived together is read together.  One CTA per round.
__device__ __forceinline__ void gather_order(const u32 *rank_cnt, int n_triples, u32 n_valid, u32 n_tiles,
                                             u32 round, u32 rounds, u32 *order, u64 *tmp) {
  const int tid = threadIdx.x;
  const u64 s = round;
  // lane l holds positions [off, off + count) and the tiles that begin there; lane n_triples: the
  // dropped records behind them.  Tiles of earlier rounds first, then the place inside the round.
  u64 sum = 0, before = 0;
  for (int pass = 0; pass < 2; pass++) {
    u64 off0 = 0, at0 = before;
    for (int l0 = 0; l0 <= n_triples; l0 += (int)blockDim.x) {
      const int l = l0 + tid;
      const u64 cnt = l < n_triples ? rank_cnt[l] : 0;
      u64 total;
      const u64 off = off0 + block_scan_exclusive<OpAdd>(cnt, OpAdd(), tmp, &total);
      off0 += total;
      const u64 first = l < n_triples ? min((off + 255) >> 8, (u64)n_tiles) : min(((u64)n_valid + 255) >> 8, (u64)n_tiles);
      const u64 end = l < n_triples ? min((off + cnt + 255) >> 8, (u64)n_tiles) : (u64)n_tiles;
      const u64 mine = l <= n_triples && end > first ? end - first : 0;
      const u64 b = mine * s / rounds, e = mine * (s + 1) / rounds;
      if (pass == 0) {
        sum += b;
      } else {
        u64 at = at0 + block_scan_exclusive<OpAdd>(e - b, OpAdd(), tmp, &total);
        at0 += total;
        for (u64 t = b; t < e && at < n_tiles; t++) order[at++] = (u32)(first + t);
      }
    }
    if (pass == 0) {
      block_scan_exclusive<OpAdd>(sum, OpAdd(), tmp, &before);
    }
  }
}

__device__ __forceinline__ void timeline_aside(const TimelineAside &a, u32 part, const int32_t *status, u64 *tmp) {
  if (part == 0) lane_table<true>(a.lanes, status, tmp);
  else gather_order(a.lanes.tt->rank_cnt, a.n_triples, (u32)a.lanes.n_valid, a.n_tiles, part - 1, a.rounds, a.order, tmp);
}
