// ta_correlate_launches: every device record is joined to the host call that
// submitted it through the correlation id both carry (Sec. 5.2; Fig. "Key
// performance observations" (a)).  Key =
// (window, pid, corr_id); the smallest sorted position among equal LAUNCH keys
// wins.
//
// One table of sorted positions, two ways to address it:
//   direct   when the correlation ids of each (window, pid) span a compact
//            range (they count up per process in real traces): the entry of
//            corr_id - min.  Launches and kernels are time-ordered, so the
//            table is touched nearly sequentially.
//   hashed   any 64-bit ids: open addressing, twice as many entries as launches.
//            An entry holds nothing but a position; whether it is the wanted key
//            is read off the corr_id column and off the range of positions its
//            (window, pid) occupies.
// Equal keys share an entry and an atomic maximum over complements leaves the smallest
// position.  HBM-bound: streams kind/corr/ts columns, writes three outputs per record.
#include <climits>
#include <cstring>
#include <vector>

#include "scan.cuh"
#include "ta_internal.cuh"

#define JN_THREADS 512
#define JN_ITEMS 4
#define JN_TILE (JN_THREADS * JN_ITEMS)

struct JoinArgs {
  int64_t n, n_valid;
  int n_lanes;
  const int16_t *kind;
  const int64_t *corr, *ts, *te;
  const int32_t *lane_off, *lane_slot, *lane_window, *lane_dom_end, *lane_dom_next;
  const int16_t *lane_domain;
  // per slot (window * n_pids + pid rank)
  i64 *slot_min, *slot_max;       // corr range of LAUNCH records
  const i64 *slot_base;           // direct: table offset of the slot, -1 = no launches
  const int32_t *slot_pos;        // hashed: first position of the slot (n_slots + 1 entries)
  u32 table_size;                 // hashed: entries
  u32 *table;                     // complement of the smallest position, 0 = empty
  int32_t *launch_of, *kol;
  int32_t *kernel_of;             // per launch with exactly one kernel: its position
  u32 *multi;                     // set when a launch has more than one
  int64_t *latency, *qdelay;
  ta_join_summary *sum;           // device, per window
  const int32_t *status;
};

__device__ __forceinline__ u64 bias64(i64 v) { return (u64)v ^ (1ull << 63); }
__host__ __device__ __forceinline__ i64 unbias64(u64 v) { return (i64)(v ^ (1ull << 63)); }

// ---- hashed addressing -------------------------------------------------------
__device__ __forceinline__ u32 join_hash(const JoinArgs &a, int slot, i64 c) {
  // multiplicative hashing (the golden ratio in 64 bits), twice so that low bits reach the top word
  u64 x = ((u64)c ^ ((u64)(u32)slot << 40)) * 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 32)) * 0x9E3779B97F4A7C15ull;
  return __umulhi((u32)(x >> 32), a.table_size);
}
__device__ __forceinline__ bool join_same(const JoinArgs &a, u32 pos, int slot, i64 c) {
  return a.corr[pos] == c && (i64)pos >= a.slot_pos[slot] && (i64)pos < a.slot_pos[slot + 1];
}
// entry of the key or the empty entry that ends its chain, from entry i on; v = what it holds.  Half
// of the table is empty, so the walk ends (bounded by the table all the same).
__device__ __forceinline__ u32 join_find(const JoinArgs &a, u32 i, u32 v, int slot, i64 c) {
  for (u32 step = 0; v != 0 && !join_same(a, ~v, slot, c) && step < a.table_size; step++) {
    i = i + 1 == a.table_size ? 0 : i + 1;
    v = a.table[i];
  }
  return v;
}
// first position of every slot
__global__ void __launch_bounds__(256) k_join_slot_pos(const int32_t *lane_off, const int32_t *lane_slot, int n_lanes,
                                                       int n_slots, int32_t *slot_pos, const int32_t *status) {
  TA_PDL();
  if (ta_failed(status)) return;
  const int l = blockIdx.x * blockDim.x + threadIdx.x;
  if (l > n_lanes) return;
  const int lo = l == 0 ? 0 : lane_slot[l - 1] + 1, hi = l == n_lanes ? n_slots : lane_slot[l];
  for (int s = lo; s <= hi; s++) slot_pos[s] = lane_off[l];  // lane_off[n_lanes] = records
}

// ---- fill the table -------------------------------------------------------------
template <bool DIRECT>
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
      if (DIRECT) {
        const i64 idx = a.slot_base[slot] + (c[j] - a.slot_min[slot]);
        atomicMax(&a.table[idx], ~(u32)p);
      } else {
        u32 i = join_hash(a, slot, c[j]);
        for (u32 step = 0; step < a.table_size; step++) {
          const u32 old = atomicCAS(&a.table[i], 0u, ~(u32)p);
          if (old == 0) break;
          if (join_same(a, ~old, slot, c[j])) {
            atomicMax(&a.table[i], ~(u32)p);
            break;
          }
          i = i + 1 == a.table_size ? 0 : i + 1;
        }
      }
    }
  }
}

// ---- pass 2: probes ----------------------------------------------------------
// A warp takes so many rows of 32 records, every row of ONE lane: window, process and table range are
// the same for the whole row, and no warp waits for another.  The kernel waits on its gathers, a
// chain of three (columns, table, launch times), so a warp works on JP_ROWS rows at a time and has the
// columns of the next JP_ROWS on their way meanwhile.  (A CTA per 1024 records, lanes walked by every
// thread, two block barriers at the start: 1035 us of 66.8 M records, half of it in those waits.)
#define JP_THREADS 256
#ifndef JP_MINB
#define JP_MINB 3
#endif
#ifndef JP_ROWS
#define JP_ROWS 3
#endif

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

struct ProbeRow {
  i64 c, s;
  bool probe;
};
__device__ __forceinline__ void probe_row(const JoinArgs &a, u32 q, u32 end, ProbeRow &x) {
  x.probe = false;
  x.c = x.s = 0;
  if (q < end) {
    // all three requested together: one round of memory latency less than loading the ids only where the kinds ask for them
    const int kd = a.kind[q];
    x.c = a.corr[q];
    x.s = a.ts[q];
    x.probe = kd == TA_KIND_KERNEL || kd == TA_KIND_MEMCPY;
  }
}

template <bool DIRECT>
__global__ void __launch_bounds__(JP_THREADS, JP_MINB) k_join_probe(JoinArgs a, int rows) {
  TA_PDL();
  __shared__ u64 red[7][JP_THREADS / 32];
  __shared__ int red_w[JP_THREADS / 32];
  if (ta_failed(a.status)) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const u32 n = (u32)a.n, nv = (u32)a.n_valid;
  const u64 first = ((u64)blockIdx.x * (JP_THREADS / 32) + warp) * (u32)rows * 32;
  const u32 begin = (u32)min(first, (u64)n), end = (u32)min(first + (u32)rows * 32, (u64)n), vend = min(end, nv);
  // probes and matches; latencies and delays summed; largest latency, largest complement, largest delay
  u32 n_probe = 0, n_match = 0;
  u64 acc[5] = {0, 0, 0, 0, 0};
  int cur = -1;  // window they are of
  auto fold = [&](u64 *t) {
    t[0] = __reduce_add_sync(0xffffffffu, n_probe);
    t[1] = __reduce_add_sync(0xffffffffu, n_match);
    t[2] = warp_reduce(acc[0], OpAdd());
    t[3] = warp_reduce(acc[1], OpAdd());
#pragma unroll
    for (int k = 4; k < 7; k++) t[k] = warp_reduce(acc[k - 2], OpMax());
  };
  int l = begin < vend ? tile_lane_search(a.lane_off, a.n_lanes, begin) : 0;
  for (u32 p = begin; p < vend;) {
    if (a.lane_domain[l] != 1) {  // host lanes hold no probe: the three outputs are -1 / 0 / 0
      const u32 e = min((u32)a.lane_dom_end[l], vend);
      for (u32 q = p + lane; q < e; q += 32) {
        a.launch_of[q] = -1;
        a.latency[q] = 0;
        a.qdelay[q] = 0;
      }
      p = e;
      if (p >= vend) break;
      l = a.lane_dom_next[l];
    }
    const u32 lane_end = (u32)a.lane_off[l + 1], e = min(lane_end, vend);
    const int slot = a.lane_slot[l], win = a.lane_window[l];
    if (win != cur) {
      if (cur >= 0) {
        u64 t[7];
        fold(t);
        if (lane == 0) join_emit(&a.sum[cur], t);
        n_probe = n_match = 0;
#pragma unroll
        for (int k = 0; k < 5; k++) acc[k] = 0;
      }
      cur = win;
    }
    const i64 base = DIRECT ? a.slot_base[slot] : 0;
    // direct: ids of the slot; hashed: positions of the slot
    const i64 lo_id = DIRECT ? a.slot_min[slot] : a.slot_pos[slot], hi_id = DIRECT ? (base >= 0 ? a.slot_max[slot] : INT64_MIN) : a.slot_pos[slot + 1];
    ProbeRow x[JP_ROWS];
#pragma unroll
    for (int r = 0; r < JP_ROWS; r++) probe_row(a, p + 32 * r + lane, e, x[r]);
    for (u32 q0 = p + lane;; q0 += 32 * JP_ROWS) {
      u32 v[JP_ROWS], at[JP_ROWS];  // what the table holds, 0 = nothing
#pragma unroll
      for (int r = 0; r < JP_ROWS; r++) {
        v[r] = at[r] = 0;
        if (DIRECT) {
          if (x[r].probe && x[r].c >= lo_id && x[r].c <= hi_id) v[r] = a.table[base + (x[r].c - lo_id)];
        } else if (x[r].probe) {
          at[r] = join_hash(a, slot, x[r].c);
          v[r] = a.table[at[r]];
        }
      }
      ProbeRow nx[JP_ROWS];
      const u32 q1 = q0 + 32 * JP_ROWS;
#pragma unroll
      for (int r = 0; r < JP_ROWS; r++) probe_row(a, q1 + 32 * r, e, nx[r]);
      if (!DIRECT) {  // the ids the first entries name, then the chains
        i64 cq[JP_ROWS];
#pragma unroll
        for (int r = 0; r < JP_ROWS; r++) cq[r] = v[r] ? a.corr[~v[r]] : 0;
#pragma unroll
        for (int r = 0; r < JP_ROWS; r++)
          if (v[r] && (cq[r] != x[r].c || (i64)~v[r] < lo_id || (i64)~v[r] >= hi_id))
            v[r] = join_find(a, at[r], v[r], slot, x[r].c);
      }
      // launch times of the matched probes (independent gathers, issued together)
      i64 ls[JP_ROWS], le[JP_ROWS];
#pragma unroll
      for (int r = 0; r < JP_ROWS; r++) {
        ls[r] = le[r] = 0;
        if (v[r]) { ls[r] = a.ts[~v[r]]; le[r] = a.te[~v[r]]; }
      }
#pragma unroll
      for (int r = 0; r < JP_ROWS; r++) {
        const u32 q = q0 + 32 * r;
        if (q < e) {
          i64 lat = 0, delay = 0;
          if (v[r]) {
            lat = x[r].s - ls[r];
            delay = max(x[r].s - le[r], (i64)0);
            atomicAdd(&a.kol[~v[r]], 1);
            a.kernel_of[~v[r]] = (int32_t)q;
            n_match++;
            acc[0] += (u64)lat;
            acc[1] += (u64)delay;
            acc[2] = max(acc[2], bias64(lat));
            acc[3] = max(acc[3], ~bias64(lat));
            acc[4] = max(acc[4], (u64)delay);
          }
          n_probe += x[r].probe;
          a.launch_of[q] = v[r] ? (int32_t)~v[r] : -1;
          a.latency[q] = lat;
          a.qdelay[q] = delay;
        }
        x[r] = nx[r];
      }
      if (q1 - lane >= e) break;
    }
    p = e;
    if (lane_end == e) l++;
  }
  for (u32 q = max(begin, vend) + lane; q < end; q += 32) {  // dropped records
    a.launch_of[q] = -1;
    a.latency[q] = 0;
    a.qdelay[q] = 0;
  }
  u64 t[7] = {0, 0, 0, 0, 0, 0, 0};
  if (cur >= 0) fold(t);
  if (lane == 0) {
    red_w[warp] = cur;
#pragma unroll
    for (int k = 0; k < 7; k++) red[k][warp] = t[k];
  }
  __syncthreads();
  if (warp > 0) return;
  const int w = lane < JP_THREADS / 32 ? red_w[lane] : -1;
  const u32 has = __ballot_sync(0xffffffffu, w >= 0);
  if (has == 0) return;
#pragma unroll
  for (int k = 0; k < 7; k++) t[k] = w >= 0 ? red[k][lane] : 0;
  const int w0 = __shfl_sync(0xffffffffu, w, __ffs(has) - 1);
  if (__all_sync(0xffffffffu, w < 0 || w == w0)) {
#pragma unroll
    for (int k = 0; k < 4; k++) t[k] = warp_reduce(t[k], OpAdd());
#pragma unroll
    for (int k = 4; k < 7; k++) t[k] = warp_reduce(t[k], OpMax());
    if (lane == 0) join_emit(&a.sum[w0], t);
  } else if (w >= 0) {
    join_emit(&a.sum[w], t);
  }
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
      const int slot = a.lane_slot[l];
      u32 v = 0;
      if (DIRECT) {
        const i64 base = a.slot_base[slot];
        if (base >= 0 && cr[j] >= a.slot_min[slot] && cr[j] <= a.slot_max[slot])
          v = a.table[base + (cr[j] - a.slot_min[slot])];
      } else {
        const u32 i = join_hash(a, slot, cr[j]);
        v = join_find(a, i, a.table[i], slot, cr[j]);
      }
      win[j] = v == 0 ? -1 : (int32_t)~v;
    }
#pragma unroll
    for (int j = 0; j < 8; j++) {
      if (!(lmask & (1u << j))) continue;
      const bool dup = win[j] != (int32_t)(p0 + j);
      const bool orphan = !dup && nk[j] == 0;
      if (nk[j] > 1) *a.multi = 1u;
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

ta_status ta_run_correlate(ta_window *h, ta_join_summary *out_summary) {
  const int64_t n = h->n;
  const int W = h->W;
  const int n_slots = W * (h->n_pids > 0 ? h->n_pids : 1);
  cudaStream_t st = h->stream;
  const int64_t nn = n > 0 ? n : 1;
  size_t keep = 2 * Carver::pad(nn * 4) + 2 * Carver::pad(nn * 8) + 256;
  void *kb = ta_dalloc(h, keep);
  if (!kb) return TA_ERR_OOM;
  Carver ck(kb);
  int32_t *launch_of = ck.take<int32_t>(nn);
  h->d_kernel_of = ck.take<int32_t>(nn);
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
  a.lane_domain = h->sorted.lane_domain; a.lane_dom_end = h->d_lane_dom_end; a.lane_dom_next = h->d_lane_dom_next;
  a.slot_min = h->d_slot_min; a.slot_max = h->d_slot_max; a.slot_base = h->d_slot_base;  // filled by the sort
  a.launch_of = launch_of; a.kol = kol; a.kernel_of = h->d_kernel_of; a.multi = (u32 *)&h->d_status[ST_MULTI]; a.latency = latency; a.qdelay = qdelay; a.sum = d_sum;
  a.status = h->d_status;
  const unsigned grid = (unsigned)((n + JN_TILE - 1) / JN_TILE);
  const unsigned grid8 = (unsigned)((n + JS_TILE - 1) / JS_TILE);
  // Rows per warp: 12, fewer where that would be less than a round of the 148 * 24 warps on the chip
  // (1.2 M records: 101 us with 12, 90 with 8), 24 where it leaves twenty rounds and more (66.8 M: 730 us
  // with 12, 690 with 24; 16.8 M: 182 with 12, 233 with 32, whose last warps run long).
  int64_t rows = n / 32 / (148 * 32);
  rows = rows < JP_ROWS ? JP_ROWS : rows > 12 ? 12 : rows / JP_ROWS * JP_ROWS;
  if (n > (int64_t)20 * 148 * 24 * 24 * 32) rows = 24;
  const unsigned grid_probe = (unsigned)((n + rows * JP_THREADS - 1) / (rows * JP_THREADS));
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
    // entries of the table: the span of all ids, or twice the launches
    const uint64_t M = direct ? (uint64_t)total : 2 * (uint64_t)h->n_launch + 1;
    if (!direct) {
      const size_t sb = Carver::pad((size_t)(n_slots + 1) * 4);
      void *sp = ta_dalloc(h, sb);
      if (!sp) return TA_ERR_OOM;
      a.slot_pos = (int32_t *)sp;
      a.table_size = (u32)M;
      ta_launch(k_join_slot_pos, (unsigned)((a.n_lanes + 256) / 256), 256, 0, st, a.lane_off, a.lane_slot, a.n_lanes,
                n_slots, (int32_t *)sp, h->d_status);
    }
    tmp_alloc = ta_zalloc(h, (size_t)(M > 0 ? M : 1) * 4, &zs);
    if (!tmp_alloc) return zs;
    a.table = (u32 *)tmp_alloc;
    if (direct) {
      ta_launch(k_join_build<true>, grid, JN_THREADS, 0, st, a);
      ta_launch(k_join_probe<true>, grid_probe, JP_THREADS, 0, st, a, (int)rows);
      ta_launch(k_join_launch_stats<true>, grid8, JP_THREADS, 0, st, a, ta_tail(h, grid8));
    } else {
      ta_launch(k_join_build<false>, grid, JN_THREADS, 0, st, a);
      ta_launch(k_join_probe<false>, grid_probe, JP_THREADS, 0, st, a, (int)rows);
      ta_launch(k_join_launch_stats<false>, grid8, JP_THREADS, 0, st, a, ta_tail(h, grid8));
    }
    TA_CHECK_CUDA(h, cudaGetLastError());
  }
  if (!small) TA_TRY(ta_queue_d2h(h, hs.data(), d_sum, W * sizeof(ta_join_summary)));
  TA_TRY(ta_sync_fetch(h));
  if (tmp_alloc) ta_dfree(h, tmp_alloc);
  if (a.slot_pos) ta_dfree(h, (void *)a.slot_pos);
  if (words[ST_ERR]) return (ta_status)words[ST_ERR];
  for (int w = 0; w < W; w++) {
    ta_join_summary &s = hs[w];
    s.n_unmatched = s.n_probe - s.n_matched;
    s.max_latency = s.n_matched ? unbias64((u64)s.max_latency) : 0;
    s.min_latency = s.n_matched ? unbias64(~(u64)s.min_latency) : 0;
    if (out_summary) out_summary[w] = s;
  }
  h->multi_launch = words[ST_MULTI];
  h->join.launch_of = launch_of;
  h->join.launch_latency = latency;
  h->join.queue_delay = qdelay;
  h->join.kernels_of_launch = kol;
  if (n == 0) {
    // nothing was launched: outputs are single dummy entries
  }
  return TA_OK;
}
