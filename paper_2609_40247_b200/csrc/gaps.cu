// ta_stream_gaps: per device lane, the running maximum of the clipped end times
// (an exclusive max-scan in canonical order) gives the gap before every record,
// the busy union, idle time, a log2 gap histogram and the list of long gaps.
// Idle time of a stream = what none of its activity records covers (Sec. 9.1).
//
// One pass over the sorted ts_start / ts_end columns, k_gaps_rows, where every lane ends its
// records in ascending order; a chained scan, k_gaps, where some lane does not.  The scan is
// made lane-aware without segment flags: the scanned value is (lane + 1) << 40 |
// (clipped end - window start), which grows from lane to lane, so a prefix
// that belongs to an earlier lane is recognised by its upper bits.  Long gaps
// are rare: they are appended to a list with an atomic cursor, each sets the bit of its
// place in the order (two per record: the gap in front of it, the tail gap behind it) in
// a bitmap, and a scan over the bitmap's words tells every entry its rank.
// HBM-bound: 16 B read + 8 B written per device record.
#include <climits>

#include "scan.cuh"
#include "ta_internal.cuh"

#define GP_THREADS 256
#define GP_ITEMS 8
#define GP_MINB 4
#define GP_TILE (GP_THREADS * GP_ITEMS)
#define GR_MINB 5
#define GR_ROWS 12
// lanes of a tile whose statistics are folded on chip: in a batch of many windows a lane is a
// thousand records or so and a tile meets several (a batch of 512 windows of 65 k records: 395 us
// with two lanes folded and the rest by global atomics per record)
#define GP_LANES 8
#define GP_LOW ((1ull << 40) - 1)

struct GapArgs {
  int64_t n, n_valid;
  int n_lanes;
  const int64_t *ts, *te;
  const int16_t *kind;
  const int32_t *lane_off, *lane_window;
  const int16_t *lane_domain;
  const int32_t *lane_dom_end, *lane_dom_next;
  const int64_t *t0, *t1;
  i64 min_gap;
  int list_only;  // second run: only (re)write the long-gap list
  u32 *not_ascending;  // set by k_gaps_rows when some lane does not end its records in ascending order
  int64_t *gap_before;
  ta_lane_gaps *lane_gaps;
  u32 *lane_hist, *win_hist;
  ta_long_gap *list;  // unordered
  u32 *list_key;      // 2 * position for the gap in front of a record, + 1 for the tail gap behind it
  u64 *bits;          // bit `list_key` of every entry
  i64 list_cap;
  u64 *st_max;
  u32 *counter;
  int32_t *status;
  u64 *n_long;        // append cursor
};


// entry `o` of the long-gap list; key: its place in the order
__device__ __forceinline__ void gap_append(const GapArgs &a, i64 o, const ta_long_gap &g, u32 key) {
  if (o < a.list_cap) {
    a.list[o] = g;
    a.list_key[o] = key;
  }
  atomicOr(&a.bits[key >> 6], 1ull << (key & 63u));
}

__device__ __forceinline__ void gaps_tile(const GapArgs &a) {
  __shared__ u64 tmp[33];
  __shared__ u64 red[4][GP_THREADS / 32];
  __shared__ u64 s_excl_max;
  __shared__ u32 s_hist[GP_LANES][TA_NBINS];  // the tile's first lanes; further lanes go straight to global
  __shared__ int s_tile, s_lane0, s_lane1, s_fail;
  const int tid = threadIdx.x;
  if (tid == 0) {
    s_tile = (int)atomicAdd(a.counter, 1u);
    s_lane1 = -1;
    s_fail = ta_failed(a.status) ? 1 : 0;
  }
  for (int i = tid; i < GP_LANES * TA_NBINS; i += GP_THREADS) (&s_hist[0][0])[i] = 0;
  __syncthreads();
  if (s_fail) return;
  const int tile = s_tile;
  const int64_t tile_start = (int64_t)tile * GP_TILE;
  const int64_t p0 = tile_start + (int64_t)tid * GP_ITEMS;
  if (tid < 32) {
    int l = -1;
    if (tile_start < a.n_valid && a.n_lanes > 0) l = tile_lane_search(a.lane_off, a.n_lanes, tile_start);
    if (tid == 0) s_lane0 = l;
  }
  __syncthreads();
  const int l0 = s_lane0;
  const bool full = p0 + GP_ITEMS <= a.n;
  if (l0 >= 0 && span_outside_domain(a.lane_domain, a.lane_dom_end, l0,
                                     min(tile_start + GP_TILE, a.n_valid), 1)) {
    // host lanes only: no gaps here, and no later device lane can use anything scanned so far
    if (tid == 0) st_relaxed(&a.st_max[tile], td_pack(TD_PREFIX, 0));
    if (a.list_only) return;
    if (full) {
      longlong2 *pg = reinterpret_cast<longlong2 *>(a.gap_before + p0);
#pragma unroll
      for (int j = 0; j < GP_ITEMS / 2; j++) pg[j] = make_longlong2(0, 0);
    } else {
      for (int j = 0; j < GP_ITEMS; j++)
        if (p0 + j < a.n) a.gap_before[p0 + j] = 0;
    }
    return;
  }
  // kinds, start and end times of the thread's records, all requested together (the tile holds a
  // device lane, so nearly every record needs its times anyway)
  int16_t kd[GP_ITEMS];
  loadn_i16<GP_ITEMS>(a.kind, p0, a.n, 0, kd);
  i64 s[GP_ITEMS], ce[GP_ITEMS];  // ce: ts_end, clipped below
#pragma unroll
  for (int j = 0; j < GP_ITEMS; j++) s[j] = ce[j] = 0;
  if (full) {
    const longlong2 *ps = reinterpret_cast<const longlong2 *>(a.ts + p0);
    const longlong2 *pe = reinterpret_cast<const longlong2 *>(a.te + p0);
#pragma unroll
    for (int j = 0; j < GP_ITEMS / 2; j++) {
      longlong2 x = ps[j], y = pe[j];
      s[2 * j] = x.x; s[2 * j + 1] = x.y;
      ce[2 * j] = y.x; ce[2 * j + 1] = y.y;
    }
  } else {
#pragma unroll
    for (int j = 0; j < GP_ITEMS; j++)
      if (p0 + j < a.n) { s[j] = a.ts[p0 + j]; ce[j] = a.te[p0 + j]; }
  }
#pragma unroll
  for (int j = 0; j < GP_ITEMS; j++)
    if (p0 + j >= a.n_valid) kd[j] = 0;
  // lanes of the items: walk forward from the tile's first lane
  int ln[GP_ITEMS];
  u64 run = 0;
  unsigned lastmask = 0, firstmask = 0;  // items that end / begin their lane
  {
    int l = l0;
    int64_t next_off = l >= 0 ? (int64_t)a.lane_off[l + 1] : LLONG_MAX;
    int64_t cur_off = l >= 0 ? (int64_t)a.lane_off[l] : 0;
    i64 w0 = 0, w1 = 0;
    int wl = -1;
#pragma unroll
    for (int j = 0; j < GP_ITEMS; j++) {
      const int64_t p = p0 + j;
      ln[j] = -1;
      if (kd[j] >= 3) {
        while (p >= next_off) { l++; cur_off = next_off; next_off = a.lane_off[l + 1]; }
        if (wl != l) { int w = a.lane_window[l]; w0 = a.t0[w]; w1 = a.t1[w]; wl = l; }
        ln[j] = l;
        if (p + 1 == next_off) lastmask |= 1u << j;
        if (p == cur_off) firstmask |= 1u << j;
        ce[j] = ce[j] < w1 ? ce[j] : w1;
        u64 v = ((u64)(l + 1) << 40) | (u64)(ce[j] - w0);
        run = run > v ? run : v;
      }
    }
    const int64_t plast = min(tile_start + GP_TILE, a.n_valid) - 1;
    if (plast >= p0 && plast < p0 + GP_ITEMS) {  // this thread owns the tile's last kept record
      while (plast >= next_off) { l++; next_off = a.lane_off[l + 1]; }
      s_lane1 = l;
    }
  }
  u64 tile_max;
  u64 thread_excl = block_scan_exclusive<OpMax>(run, OpMax(), tmp, &tile_max);
  if (tid < 32) {
    bool failed;
    u64 ex = tile_lookback<OpMax>(a.st_max, tile, tile_max, OpMax(), a.status, &failed);
    if (tid == 0) { s_excl_max = ex; s_fail = failed ? 1 : 0; }
  }
  __syncthreads();
  if (s_fail) return;
  u64 pre = s_excl_max > thread_excl ? s_excl_max : thread_excl;

  // gaps; statistics of the thread's first lane stay in registers, anything else is rare
  i64 gap[GP_ITEMS];
  u64 sb = 0, si = 0, ng = 0, mg = 0;
  int lm = -1;
  {
    i64 w0 = 0, w1 = 0;
    int wl = -1;
#pragma unroll
    for (int j = 0; j < GP_ITEMS; j++) {
      gap[j] = 0;
      const int l = ln[j];
      i64 Pi = 0, g = 0, bz = 0, tl = 0;
      bool last = false, lg = false, lt = false;
      if (l >= 0) {
        if (wl != l) { int w = a.lane_window[l]; w0 = a.t0[w]; w1 = a.t1[w]; wl = l; }
        Pi = ((pre >> 40) == (u64)(l + 1)) ? w0 + (i64)(pre & GP_LOW) : w0;
        g = s[j] > Pi ? s[j] - Pi : 0;
        const i64 from = s[j] > Pi ? s[j] : Pi;
        bz = ce[j] > from ? ce[j] - from : 0;
        last = (lastmask >> j) & 1u;
        if (last) tl = w1 - (Pi > ce[j] ? Pi : ce[j]);
        gap[j] = g;
        pre = max(pre, ((u64)(l + 1) << 40) | (u64)(ce[j] - w0));
        lg = g > 0 && g >= a.min_gap;
        lt = last && tl > 0 && tl >= a.min_gap;
      }
      // long-gap list: the warp reserves its entries with one add on the cursor (the order of
      // the list does not matter, it is sorted afterwards)
      if (__any_sync(0xffffffffu, lg || lt)) {  // rare: one vote decides for the warp
        const u32 m_g = __ballot_sync(0xffffffffu, lg), m_t = __ballot_sync(0xffffffffu, lt);
        {
          const int wlane = threadIdx.x & 31;
          const u32 below = (1u << wlane) - 1u;
          u64 base = 0;
          if (wlane == 0) base = atomicAdd(a.n_long, (u64)(__popc(m_g) + __popc(m_t)));
          base = __shfl_sync(0xffffffffu, base, 0);
          if (lg) gap_append(a, (i64)base + __popc(m_g & below), ta_long_gap{l, (int32_t)(p0 + j), Pi, g}, (u32)(p0 + j) << 1);
          if (lt)
            gap_append(a, (i64)base + __popc(m_g) + __popc(m_t & below), ta_long_gap{l, -1, w1 - tl, tl},
                       (u32)(p0 + j) << 1 | 1u);
        }
      }
      if (l < 0) continue;
      if (a.list_only) continue;
      if (lm < 0) lm = l;
      const int li = l - l0;
      if (l == lm && li < GP_LANES) {
        sb += (u64)bz;
        si += (u64)(g + tl);
        if (g > 0) { ng++; mg = max(mg, (u64)g); atomicAdd(&s_hist[li][log2_bin(g)], 1u); }
        if (tl > 0) { ng++; mg = max(mg, (u64)tl); atomicAdd(&s_hist[li][log2_bin(tl)], 1u); }
      } else {  // a thread that straddles a lane boundary, or a lane too many in the tile
        ta_lane_gaps *gl = &a.lane_gaps[l];
        const int w = a.lane_window[l];
        if (bz) atomicAdd((u64 *)&gl->busy, (u64)bz);
        if (g + tl) atomicAdd((u64 *)&gl->idle, (u64)(g + tl));
        if (g > 0) {
          atomicAdd((u64 *)&gl->n_gaps, 1ull);
          atomicMax((i64 *)&gl->max_gap, g);
          atomicAdd(&a.lane_hist[(size_t)l * TA_NBINS + log2_bin(g)], 1u);
          atomicAdd(&a.win_hist[(size_t)w * TA_NBINS + log2_bin(g)], 1u);
        }
        if (tl > 0) {
          atomicAdd((u64 *)&gl->n_gaps, 1ull);
          atomicMax((i64 *)&gl->max_gap, tl);
          atomicAdd(&a.lane_hist[(size_t)l * TA_NBINS + log2_bin(tl)], 1u);
          atomicAdd(&a.win_hist[(size_t)w * TA_NBINS + log2_bin(tl)], 1u);
        }
      }
      if (last) {
        a.lane_gaps[l].last_end = w1 - tl;
        a.lane_gaps[l].n_events = (i64)a.lane_off[l + 1] - (i64)a.lane_off[l];
      }
      if ((firstmask >> j) & 1u) a.lane_gaps[l].first_start = s[j];
    }
  }
  if (a.list_only) return;
  if (full) {
    longlong2 *pg = reinterpret_cast<longlong2 *>(a.gap_before + p0);
#pragma unroll
    for (int j = 0; j < GP_ITEMS / 2; j++) pg[j] = make_longlong2(gap[2 * j], gap[2 * j + 1]);
  } else {
#pragma unroll
    for (int j = 0; j < GP_ITEMS; j++)
      if (p0 + j < a.n) a.gap_before[p0 + j] = gap[j];
  }
  // fold the register statistics of the tile's first lanes
  const int l1 = s_lane1;
  for (int li = 0; li < GP_LANES; li++) {
    const int l = l0 + li;
    if (l0 < 0 || l > l1) break;
    if (a.lane_domain[l] != 1) continue;  // uniform over the CTA
    const bool mine = lm == l;
    u64 r0 = warp_reduce(mine ? sb : 0, OpAdd());
    u64 r1 = warp_reduce(mine ? si : 0, OpAdd());
    u64 r2 = warp_reduce(mine ? ng : 0, OpAdd());
    u64 r3 = warp_reduce(mine ? mg : 0, OpMax());
    __syncthreads();
    if ((tid & 31) == 0) { red[0][tid >> 5] = r0; red[1][tid >> 5] = r1; red[2][tid >> 5] = r2; red[3][tid >> 5] = r3; }
    __syncthreads();
    if (tid < 4) {
      u64 t = 0;
      for (int w = 0; w < GP_THREADS / 32; w++) t = tid == 3 ? max(t, red[3][w]) : t + red[tid][w];
      if (t) {
        ta_lane_gaps *gl = &a.lane_gaps[l];
        if (tid == 0) atomicAdd((u64 *)&gl->busy, t);
        else if (tid == 1) atomicAdd((u64 *)&gl->idle, t);
        else if (tid == 2) atomicAdd((u64 *)&gl->n_gaps, t);
        else atomicMax((i64 *)&gl->max_gap, (i64)t);
      }
    }
    if (tid < TA_NBINS && s_hist[li][tid]) {
      atomicAdd(&a.lane_hist[(size_t)l * TA_NBINS + tid], s_hist[li][tid]);
      atomicAdd(&a.win_hist[(size_t)a.lane_window[l] * TA_NBINS + tid], s_hist[li][tid]);
    }
  }
}

__global__ void __launch_bounds__(GP_THREADS, GP_MINB) k_gaps(GapArgs a, Tail tail) {
  TA_PDL();
  gaps_tile(a);
  run_tail(tail);
}

// The same for streams that end their records in ascending order, as in-order streams do: the running
// maximum in front of a record is the clipped end of its neighbour, no scan and no tile waits for
// another.  Checked on the way; one record that ends before the one in front of it sends the call
// through k_gaps.
// A warp takes `rows` x 32 consecutive positions, 32 records of ONE lane at a time: lane, window and
// bounds are then the same for the whole warp and the neighbour's end is a shuffle away (a thread
// with eight consecutive records, each with its own lane walk, took 270 warp instructions per 32
// records and bound the kernel: 480 us for 66.8 M records).  Statistics of the CTA's first GR_LANES
// lanes are folded on chip.
// Long gaps are collected on chip and take their places in the list with one add per CTA: in a window of
// stalls every row has some (a fifth of the records of a prefill window), and an add per row on the one
// cursor, at about a nanosecond each, was all the kernel did (16.8 M prefill records 165 us, 85 now).
#define GR_LANES 4
#define GR_LIST 512
__device__ __forceinline__ void gaps_rows(const GapArgs &a, int rows) {
  __shared__ ta_long_gap s_list[GR_LIST];
  __shared__ u32 s_key[GR_LIST];
  __shared__ u32 s_n;
  __shared__ u64 s_base;
  __shared__ u64 s_sum[GR_LANES][3];  // busy, idle, gaps
  __shared__ i64 s_max[GR_LANES];
  __shared__ u32 s_hist[GR_LANES][TA_NBINS];
  __shared__ int s_lane0;
  if (ta_failed(a.status)) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int i = tid; i < GR_LANES * TA_NBINS; i += GP_THREADS) (&s_hist[0][0])[i] = 0;
  if (tid < GR_LANES * 3) (&s_sum[0][0])[tid] = 0;
  if (tid < GR_LANES) s_max[tid] = 0;
  if (tid == 0) s_n = 0;
  const int64_t span = (int64_t)rows * 32;
  const int64_t begin = ((int64_t)blockIdx.x * (GP_THREADS / 32) + warp) * span;
  const int64_t end = min(begin + span, a.n), vend = min(end, a.n_valid);
  int l = begin < vend ? tile_lane_search(a.lane_off, a.n_lanes, begin) : 0;
  if (tid == 0) s_lane0 = l;
  __syncthreads();
  const int l0 = s_lane0;
  int64_t pos = begin;
  while (pos < vend) {
    if (a.lane_domain[l] != 1) {  // host lanes: no gaps
      const int64_t stop = min((int64_t)a.lane_dom_end[l], vend);
      for (int64_t p = pos + lane; p < stop; p += 32) a.gap_before[p] = 0;
      pos = stop;
      l = a.lane_dom_next[l];
      continue;
    }
    const int64_t off = a.lane_off[l], lane_end = a.lane_off[l + 1], seg_end = min(lane_end, vend);
    const int w = a.lane_window[l];
    const i64 w0 = a.t0[w], w1 = a.t1[w];
    const int li = l - l0;
    u32 *hist = li < GR_LANES ? s_hist[li] : nullptr;
    i64 s = 0, e = 0;
    if (pos + lane < seg_end) { s = a.ts[pos + lane]; e = a.te[pos + lane]; }
    i64 carry = pos > off ? min((i64)a.te[pos - 1], w1) : w0;  // P of the row's first record
    u64 sb = 0, si = 0;
    i64 mg = 0;
    u32 ng = 0;
    for (; pos < seg_end; pos += 32) {
      const int64_t p = pos + lane;
      const bool in = p < seg_end;
      const i64 ce = min(e, w1), cs = s;
      if (p + 32 < seg_end) { s = a.ts[p + 32]; e = a.te[p + 32]; }  // the next row's, while this one is worked on
      i64 P = __shfl_up_sync(0xffffffffu, ce, 1);
      if (lane == 0) P = carry;
      carry = __shfl_sync(0xffffffffu, ce, 31);
      const i64 g = in && cs > P ? cs - P : 0;
      bool lt = false;
      i64 tl = 0;
      if (in) {
        if (p > off && ce < P) *a.not_ascending = 1u;
        const i64 from = cs > P ? cs : P;
        sb += (u64)(ce > from ? ce - from : 0);
        si += (u64)g;
        if (g > 0) {
          ng++;
          mg = max(mg, g);
          if (hist) {
            atomicAdd(&hist[log2_bin(g)], 1u);
          } else {
            atomicAdd(&a.lane_hist[(size_t)l * TA_NBINS + log2_bin(g)], 1u);
            atomicAdd(&a.win_hist[(size_t)w * TA_NBINS + log2_bin(g)], 1u);
          }
        }
        a.gap_before[p] = g;
        if (p == off) a.lane_gaps[l].first_start = cs;
        if (p + 1 == lane_end) {
          tl = w1 - max(P, ce);
          if (tl > 0) {
            ng++;
            mg = max(mg, tl);
            si += (u64)tl;
            if (hist) {
              atomicAdd(&hist[log2_bin(tl)], 1u);
            } else {
              atomicAdd(&a.lane_hist[(size_t)l * TA_NBINS + log2_bin(tl)], 1u);
              atomicAdd(&a.win_hist[(size_t)w * TA_NBINS + log2_bin(tl)], 1u);
            }
            lt = tl >= a.min_gap;
          }
          a.lane_gaps[l].last_end = w1 - tl;
          a.lane_gaps[l].n_events = lane_end - off;
        }
      }
      // long-gap list (put in order afterwards): what finds no room on chip takes its place in memory
      // with an add per row
      const bool lg = g > 0 && g >= a.min_gap;
      if (__any_sync(0xffffffffu, lg || lt)) {
        const u32 m_g = __ballot_sync(0xffffffffu, lg), m_t = __ballot_sync(0xffffffffu, lt);
        const u32 below = (1u << lane) - 1u, n_g = (u32)__popc(m_g), cnt = n_g + (u32)__popc(m_t);
        u32 at = 0;
        if (lane == 0) at = atomicAdd(&s_n, cnt);
        at = __shfl_sync(0xffffffffu, at, 0);
        const u32 room = at < GR_LIST ? min(cnt, GR_LIST - at) : 0u;
        u64 base = 0;
        if (room < cnt) {
          if (lane == 0) base = atomicAdd(a.n_long, (u64)(cnt - room));
          base = __shfl_sync(0xffffffffu, base, 0);
        }
        auto put = [&](u32 k, const ta_long_gap &x, u32 key) {
          if (k < room) { s_list[at + k] = x; s_key[at + k] = key; }
          else gap_append(a, (i64)(base + (k - room)), x, key);
        };
        if (lg) put((u32)__popc(m_g & below), ta_long_gap{l, (int32_t)p, P, g}, (u32)p << 1);
        if (lt) put(n_g + (u32)__popc(m_t & below), ta_long_gap{l, -1, w1 - tl, tl}, (u32)p << 1 | 1u);
      }
    }
    pos = seg_end;
    // the lane's share of this warp
    sb = warp_reduce(sb, OpAdd());
    si = warp_reduce(si, OpAdd());
    ng = __reduce_add_sync(0xffffffffu, ng);
    mg = (i64)warp_reduce((u64)mg, OpMax());
    if (lane == 0) {
      if (hist) {
        if (sb) atomicAdd(&s_sum[li][0], sb);
        if (si) atomicAdd(&s_sum[li][1], si);
        if (ng) atomicAdd(&s_sum[li][2], (u64)ng);
        if (mg > s_max[li]) atomicMax(&s_max[li], mg);
      } else {
        ta_lane_gaps *gl = &a.lane_gaps[l];
        if (sb) atomicAdd((u64 *)&gl->busy, sb);
        if (si) atomicAdd((u64 *)&gl->idle, si);
        if (ng) atomicAdd((u64 *)&gl->n_gaps, (u64)ng);
        if (mg) atomicMax((i64 *)&gl->max_gap, mg);
      }
    }
    if (lane_end <= vend) l++;
  }
  for (int64_t p = max(begin, vend) + lane; p < end; p += 32) a.gap_before[p] = 0;  // dropped records
  __syncthreads();
  const u32 listed = min(s_n, (u32)GR_LIST);
  if (listed) {  // the same in every thread
    if (tid == 0) s_base = atomicAdd(a.n_long, (u64)listed);
    __syncthreads();
    for (u32 i = tid; i < listed; i += GP_THREADS) gap_append(a, (i64)(s_base + i), s_list[i], s_key[i]);
  }
  for (int i = tid; i < GR_LANES * (TA_NBINS + 4); i += GP_THREADS) {
    const int li = i / (TA_NBINS + 4), k = i - li * (TA_NBINS + 4), ll = l0 + li;
    if (ll >= a.n_lanes) continue;
    ta_lane_gaps *gl = &a.lane_gaps[ll];
    if (k < TA_NBINS) {
      const u32 c = s_hist[li][k];
      if (c) {
        atomicAdd(&a.lane_hist[(size_t)ll * TA_NBINS + k], c);
        atomicAdd(&a.win_hist[(size_t)a.lane_window[ll] * TA_NBINS + k], c);
      }
    } else if (k < TA_NBINS + 3) {
      const u64 v = s_sum[li][k - TA_NBINS];
      if (v) atomicAdd(k == TA_NBINS ? (u64 *)&gl->busy : k == TA_NBINS + 1 ? (u64 *)&gl->idle : (u64 *)&gl->n_gaps, v);
    } else if (s_max[li]) {
      atomicMax((i64 *)&gl->max_gap, s_max[li]);
    }
  }
}
template <bool TAIL>
__global__ void __launch_bounds__(GP_THREADS, GR_MINB) k_gaps_rows(GapArgs a, int rows, Tail tail) {
  TA_PDL();
  gaps_rows(a, rows);
  if (TAIL) run_tail(tail);
}

struct GapBitsIn {
  const u64 *bits;
  __device__ u64 operator()(int64_t i) const { return (u64)__popcll(bits[i]); }
};
struct GapBitsOut {
  u32 *rank;
  __device__ void operator()(int64_t i, u64 excl, u64) const { rank[i] = (u32)excl; }
};
// every entry to its place
__global__ void __launch_bounds__(256) k_gap_list_order(const ta_long_gap *src, const u32 *key, const u64 *bits,
                                                        const u32 *rank, int64_t m, ta_long_gap *dst,
                                                        const int32_t *status) {
  TA_PDL();
  if (ta_failed(status)) return;
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m) return;
  const u32 k = key[i];
  dst[rank[k >> 6] + __popcll(bits[k >> 6] & ((1ull << (k & 63u)) - 1ull))] = src[i];
}

// Both steps in one CTA for a short bitmap and list: what a launch costs more than the work.
#define GL_THREADS 1024
#define GL_WORDS 8192    // words of the bitmap (262 k records)
#define GL_ENTRIES 8192
__global__ void __launch_bounds__(GL_THREADS) k_gap_list_one(const ta_long_gap *src, const u32 *key, const u64 *bits,
                                                             int n_bits, int m, ta_long_gap *dst, const int32_t *status) {
  TA_PDL();
  __shared__ u64 tmp[33];
  __shared__ u32 rank[GL_WORDS];
  if (ta_failed(status)) return;
  constexpr int PER = GL_WORDS / GL_THREADS;
  const int w0 = threadIdx.x * PER;
  u32 c[PER], mine = 0;
#pragma unroll
  for (int k = 0; k < PER; k++) {
    c[k] = w0 + k < n_bits ? (u32)__popcll(bits[w0 + k]) : 0u;
    mine += c[k];
  }
  u64 total;
  u32 r = (u32)block_scan_exclusive<OpAdd>((u64)mine, OpAdd(), tmp, &total);
#pragma unroll
  for (int k = 0; k < PER; k++) {
    rank[w0 + k] = r;
    r += c[k];
  }
  __syncthreads();
#pragma unroll 2
  for (int i = threadIdx.x; i < m; i += GL_THREADS) {
    const u32 k = key[i];
    dst[rank[k >> 6] + __popcll(bits[k >> 6] & ((1ull << (k & 63u)) - 1ull))] = src[i];
  }
}

ta_status ta_run_gaps(ta_window *h, int64_t min_gap, ta_gap_result *out) {
  const int64_t n = h->n;
  const int L = h->sorted.n_lanes;
  const int W = h->W;
  cudaStream_t st = h->stream;
  if (L >= (1 << 22) - 1) return TA_ERR_TOO_LARGE;
  const int64_t tiles = (n + GP_TILE - 1) / GP_TILE;
  int64_t cap = n / 8 > 65536 ? n / 8 : 65536;  // first guess; a longer list is rebuilt below
  const size_t bytes = Carver::pad((size_t)(L + 1) * sizeof(ta_lane_gaps)) +
                       Carver::pad((size_t)(L + 1) * TA_NBINS * 4) + Carver::pad((size_t)W * TA_NBINS * 4);
  // temporary: look-back state, scalars, the bitmap of the list's order, its scan
  const int64_t n_bits = (n + 31) / 32;
  const size_t tmp_bytes = Carver::pad((size_t)(tiles + 1) * 8) + Carver::pad(64) + Carver::pad((size_t)n_bits * 8) +
                           scan_temp_bytes(n_bits) + Carver::pad((size_t)n_bits * 4) + 512;
  int64_t *gap_before = (int64_t *)ta_dalloc(h, (size_t)(n > 0 ? n : 1) * 8);
  if (!gap_before) return TA_ERR_OOM;
  ta_status zs;
  void *b = ta_zalloc(h, bytes, &zs);
  if (!b) return zs;
  Carver c(b);
  ta_lane_gaps *lane_gaps = c.take<ta_lane_gaps>(L + 1);
  u32 *lane_hist = c.take<u32>((size_t)(L + 1) * TA_NBINS);
  u32 *win_hist = c.take<u32>((size_t)W * TA_NBINS);
  void *tb = ta_zpool(h, tmp_bytes);
  const bool pooled = tb != nullptr;
  if (!tb) tb = ta_dalloc(h, tmp_bytes);
  if (!tb) return TA_ERR_OOM;
  Carver ct(tb);
  u64 *st_max = ct.take<u64>(tiles + 1);
  u64 *scal = ct.take<u64>(8);  // [0] list cursor, [1] tile counter, [2] not ascending
  const size_t state_bytes = ct.off;
  u64 *bits = ct.take<u64>(n_bits);
  ScanTemp scan;
  ct.off += scan_temp_carve(ct.base + ct.off, n_bits, &scan);
  const size_t tmp_zero = ct.off;
  u32 *rank = ct.take<u32>(n_bits);
  if (!pooled) TA_CHECK_CUDA(h, cudaMemsetAsync(tb, 0, tmp_zero, st));
  // unordered list + keys (temporary)
  void *lt = ta_dalloc(h, Carver::pad((size_t)cap * sizeof(ta_long_gap)) + Carver::pad((size_t)cap * 4) + 256);
  if (!lt) return TA_ERR_OOM;
  Carver cl(lt);
  ta_long_gap *ulist = cl.take<ta_long_gap>(cap);
  u32 *ukeys = cl.take<u32>(cap);

  GapArgs a;
  a.n = n; a.n_valid = h->n_valid; a.n_lanes = L;
  a.ts = h->sorted.ts_start; a.te = h->sorted.ts_end; a.kind = h->sorted.kind;
  a.lane_off = h->sorted.lane_off; a.lane_window = h->sorted.lane_window;
  a.lane_domain = h->sorted.lane_domain; a.lane_dom_end = h->d_lane_dom_end; a.lane_dom_next = h->d_lane_dom_next; a.t0 = h->d_t0; a.t1 = h->d_t1;
  a.min_gap = min_gap; a.list_only = 0;
  a.gap_before = gap_before; a.lane_gaps = lane_gaps; a.lane_hist = lane_hist; a.win_hist = win_hist;
  a.list = ulist; a.list_key = ukeys; a.list_cap = cap; a.st_max = st_max; a.bits = bits;
  a.counter = (u32 *)(scal + 1); a.status = h->d_status; a.n_long = scal;
  a.not_ascending = (u32 *)(scal + 2);
  u64 n_long = 0;
  int32_t words[ST_WORDS];
  // first without the scan (every lane is taken to end its records in ascending order, which the
  // kernel checks); if a lane does not, once more with the chained maximum scan
  for (int scan = 0; scan < 2; scan++) {
    u64 three[3] = {0, 0, 0};
    TA_TRY(ta_queue_d2h(h, three, scal, 24));
    TA_TRY(ta_queue_d2h(h, words, h->d_status, sizeof(words)));
    if (tiles > 0 && scan) {
      ta_launch(k_gaps, (unsigned)tiles, GP_THREADS, 0, st, a, ta_tail(h, tiles));
    } else if (tiles > 0) {
      // rows per warp: 12 (66.8 M records: 292 us; 32: 383, 8: 319), fewer while that would leave SMs
      // without work
      int64_t rows = n / 32 / (148 * 16);
      rows = rows < 4 ? 4 : rows > GR_ROWS ? GR_ROWS : rows;
      const int64_t per_cta = rows * GP_THREADS, grid = (n + per_cta - 1) / per_cta;
      const Tail tail = ta_tail(h, grid);
      ta_launch(tail.m ? k_gaps_rows<true> : k_gaps_rows<false>, (unsigned)grid, GP_THREADS, 0, st, a, (int)rows, tail);
    }
    TA_CHECK_CUDA(h, cudaGetLastError());
    TA_TRY(ta_sync_fetch(h));
    if (words[ST_ERR]) return (ta_status)words[ST_ERR];
    n_long = three[0];
    if (scan || !(u32)three[2]) break;
    TA_CHECK_CUDA(h, cudaMemsetAsync(b, 0, bytes, st));
    TA_CHECK_CUDA(h, cudaMemsetAsync(tb, 0, tmp_zero, st));
  }
  if ((int64_t)n_long > cap) {
    // rare: a tiny min_gap made the list longer than the first guess; rebuild it
    ta_dfree(h, lt);
    cap = (int64_t)n_long;
    lt = ta_dalloc(h, Carver::pad((size_t)cap * sizeof(ta_long_gap)) + Carver::pad((size_t)cap * 4) + 256);
    if (!lt) return TA_ERR_OOM;
    Carver cl2(lt);
    ulist = cl2.take<ta_long_gap>(cap);
    ukeys = cl2.take<u32>(cap);
    TA_CHECK_CUDA(h, cudaMemsetAsync(tb, 0, state_bytes, st));
    a.list = ulist; a.list_key = ukeys; a.list_cap = cap; a.list_only = 1;
    ta_launch(k_gaps, (unsigned)tiles, GP_THREADS, 0, st, a, ta_tail(h, tiles));
    TA_CHECK_CUDA(h, cudaGetLastError());
    TA_TRY(ta_read_status(h, words));
    if (words[ST_ERR]) return (ta_status)words[ST_ERR];
  }
  // order the list by (lane, position; tail last)
  ta_long_gap *list = nullptr;
  const int64_t m = (int64_t)n_long;
  if (m > 0) {
    list = (ta_long_gap *)ta_dalloc(h, (size_t)m * sizeof(ta_long_gap));
    if (!list) return TA_ERR_OOM;
    if (n_bits <= GL_WORDS && m <= GL_ENTRIES) {
      ta_launch(k_gap_list_one, 1, GL_THREADS, 0, st, ulist, ukeys, bits, (int)n_bits, (int)m, list, h->d_status);
    } else {
      GapBitsIn bi{bits};
      GapBitsOut bo{rank};
      TA_TRY((launch_scan<OpAdd, GapBitsIn, GapBitsOut>(h, n_bits, bi, bo, OpAdd(), scan)));
      ta_launch(k_gap_list_order, (unsigned)((m + 255) / 256), 256, 0, st, ulist, ukeys, bits, rank, m, list, h->d_status);
    }
    TA_CHECK_CUDA(h, cudaGetLastError());
    // both kernels are still queued: their temporaries go back after the handle's next
    // wait (the list itself is used in stream order like every other result)
    ta_dfree_later(h, tb);
    ta_dfree_later(h, lt);
    tb = lt = nullptr;
  }
  if (tb) ta_dfree(h, tb);
  if (lt) ta_dfree(h, lt);
  out->gap_before = gap_before;
  out->lane_gaps = lane_gaps;
  out->lane_hist = lane_hist;
  out->win_hist = win_hist;
  out->long_gaps = list;
  out->n_long_gaps = m;
  return TA_OK;
}
