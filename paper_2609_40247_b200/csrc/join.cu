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
//   hashed   any 64-bit ids: open addressing, two to four times as many entries as launches.
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
  // multiplicative hashing (the golden ratio in 64 bits), twice so that low bits reach the top word; the
  // slot enters with all 64 bits: shifted to the upper ones it met ids that carry a number there, and
  // 64 processes with a rank or a thread in bits 40 and up shared every chain (8 M records 7.57 ms instead
  // of 0.51)
  u64 x = ((u64)c + (u64)(u32)slot * 0xD6E8FEB86659FD93ull) * 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 32)) * 0x9E3779B97F4A7C15ull;
  return __umulhi((u32)(x >> 32), a.table_size);
}
__device__ __forceinline__ bool join_same(const JoinArgs &a, u32 pos, int slot, i64 c) {
  return a.corr[pos] == c && (i64)pos >= a.slot_pos[slot] && (i64)pos < a.slot_pos[slot + 1];
}
// entry of the key or the empty entry that ends its chain, from entry i on; v = what it holds.  Half
// of the table at least is empty, so the walk ends (bounded by the table all the same).
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

#define JN_THREADS 256
#define JN_WARPS (JN_THREADS / 32)
#define JN_COUNT_APART (24 << 20)  // records from which launches with kernels are counted by a pass of their own

// The span of records a warp works on: so many rows of 32.
struct JoinSpan {
  u32 begin, end, vend;  // vend: end of the kept records in it
};
__device__ __forceinline__ JoinSpan join_span(const JoinArgs &a, int rows) {
  const u64 first = ((u64)blockIdx.x * JN_WARPS + (threadIdx.x >> 5)) * (u32)rows * 32;
  JoinSpan x;
  x.begin = (u32)min(first, (u64)a.n);
  x.end = (u32)min(first + (u32)rows * 32, (u64)a.n);
  x.vend = min(x.end, (u32)a.n_valid);
  return x;
}
// Adds the figures of a CTA's warps (t: the same in every lane of a warp; cur: their window, -1 = none)
// to the rows of their windows.  Called by all threads.
template <int NS, int NM, class Emit>
__device__ __forceinline__ void join_fold(u64 (&t)[NS + NM], int cur, Emit emit) {
  __shared__ u64 red[NS + NM][JN_WARPS];
  __shared__ int red_w[JN_WARPS];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) {
    red_w[warp] = cur;
#pragma unroll
    for (int k = 0; k < NS + NM; k++) red[k][warp] = t[k];
  }
  __syncthreads();
  if (warp > 0) return;
  const int w = lane < JN_WARPS ? red_w[lane] : -1;
  const u32 has = __ballot_sync(0xffffffffu, w >= 0);
  if (has == 0) return;
#pragma unroll
  for (int k = 0; k < NS + NM; k++) t[k] = w >= 0 ? red[k][lane] : 0;
  const int w0 = __shfl_sync(0xffffffffu, w, __ffs(has) - 1);
  if (__all_sync(0xffffffffu, w < 0 || w == w0)) {
#pragma unroll
    for (int k = 0; k < NS; k++) t[k] = warp_reduce(t[k], OpAdd());
#pragma unroll
    for (int k = NS; k < NS + NM; k++) t[k] = warp_reduce(t[k], OpMax());
    if (lane == 0) emit(w0, t);
  } else if (w >= 0) {
    emit(w, t);
  }
}

// ---- fill the table -------------------------------------------------------------
// A warp takes rows of 32 records of one host lane, JB_ROWS at a time, with the kinds and ids of the
// next JB_ROWS on their way.  What an entry held before tells a first launch of its id from a repeated
// one, so that launches, duplicates and ids are counted here and no later pass has to look them up.
#define JB_ROWS 2
// adds a group of launches to the row of their window; k_join_probe takes the ids with a kernel off the orphans again
__device__ __forceinline__ void launch_emit(ta_join_summary *sm, const u64 *t) {
  if (t[0] == 0) return;
  atomicAdd((u64 *)&sm->n_launch, t[0]);
  if (t[1]) atomicAdd((u64 *)&sm->n_dup_launch, t[1]);
  atomicAdd((u64 *)&sm->n_orphan_launch, t[0] - t[1]);
}
struct LaunchRow {
  i64 c;
  bool launch;
};
__device__ __forceinline__ void launch_row(const JoinArgs &a, u32 q, u32 end, LaunchRow &x) {
  x.launch = false;
  x.c = 0;
  if (q < end) {
    x.launch = a.kind[q] == TA_KIND_LAUNCH;
    x.c = a.corr[q];
  }
}
template <bool DIRECT>
__global__ void __launch_bounds__(JN_THREADS) k_join_build(JoinArgs a, int rows) {
  TA_PDL();
  if (ta_failed(a.status)) return;
  const int lane = threadIdx.x & 31;
  const JoinSpan sp = join_span(a, rows);
  u32 n_launch = 0, n_dup = 0;
  int cur = -1;  // window they are of
  int l = sp.begin < sp.vend ? tile_lane_search(a.lane_off, a.n_lanes, sp.begin) : 0;
  for (u32 p = sp.begin; p < sp.vend;) {
    if (a.lane_domain[l] != 0) {  // launches live in host lanes
      p = min((u32)a.lane_dom_end[l], sp.vend);
      if (p >= sp.vend) break;
      l = a.lane_dom_next[l];
    }
    const u32 lane_end = (u32)a.lane_off[l + 1], e = min(lane_end, sp.vend);
    const int slot = a.lane_slot[l], win = a.lane_window[l];
    if (win != cur) {
      if (cur >= 0) {
        const u64 t[2] = {__reduce_add_sync(0xffffffffu, n_launch), __reduce_add_sync(0xffffffffu, n_dup)};
        if (lane == 0) launch_emit(&a.sum[cur], t);
        n_launch = n_dup = 0;
      }
      cur = win;
    }
    const i64 base = DIRECT ? a.slot_base[slot] - a.slot_min[slot] : 0;
    LaunchRow x[JB_ROWS];
#pragma unroll
    for (int r = 0; r < JB_ROWS; r++) launch_row(a, p + 32 * r + lane, e, x[r]);
    for (u32 q0 = p + lane;; q0 += 32 * JB_ROWS) {
      LaunchRow nx[JB_ROWS];
      const u32 q1 = q0 + 32 * JB_ROWS;
#pragma unroll
      for (int r = 0; r < JB_ROWS; r++) launch_row(a, q1 + 32 * r, e, nx[r]);
      u32 old[JB_ROWS], at[JB_ROWS];
#pragma unroll
      for (int r = 0; r < JB_ROWS; r++) {
        const u32 q = q0 + 32 * r;
        old[r] = at[r] = 0;
        if (!x[r].launch) continue;
        if (DIRECT) {
          old[r] = atomicMax(&a.table[base + x[r].c], ~q);
        } else {  // (the first entries of all rows together)
          at[r] = join_hash(a, slot, x[r].c);
          old[r] = atomicCAS(&a.table[at[r]], 0u, ~q);
        }
      }
      if (!DIRECT) {
        i64 cq[JB_ROWS];
#pragma unroll
        for (int r = 0; r < JB_ROWS; r++) cq[r] = old[r] ? a.corr[~old[r]] : 0;
#pragma unroll
        for (int r = 0; r < JB_ROWS; r++) {
          const u32 q = q0 + 32 * r;
          bool same = cq[r] == x[r].c;
          for (u32 step = 0; old[r] && step < a.table_size; step++) {
            if (same && (i64)~old[r] >= a.slot_pos[slot] && (i64)~old[r] < a.slot_pos[slot + 1]) {
              atomicMax(&a.table[at[r]], ~q);
              break;
            }
            at[r] = at[r] + 1 == a.table_size ? 0 : at[r] + 1;
            old[r] = atomicCAS(&a.table[at[r]], 0u, ~q);
            same = old[r] && a.corr[~old[r]] == x[r].c;
          }
        }
      }
#pragma unroll
      for (int r = 0; r < JB_ROWS; r++) {
        n_launch += x[r].launch;
        n_dup += old[r] != 0;
        x[r] = nx[r];
      }
      if (q1 - lane >= e) break;
    }
    p = e;
    if (lane_end == e) l++;
  }
  u64 t[2] = {__reduce_add_sync(0xffffffffu, n_launch), __reduce_add_sync(0xffffffffu, n_dup)};
  join_fold<2, 0>(t, cur, [&](int w, const u64 *v) { launch_emit(&a.sum[w], v); });
}

// ---- pass 2: probes ----------------------------------------------------------
// A warp takes so many rows of 32 records, every row of ONE lane: window, process and table range are
// the same for the whole row, and no warp waits for another.  The kernel waits on its gathers, a
// chain of three (columns, table, launch times), so a warp works on JP_ROWS rows at a time and has the
// columns of the next JP_ROWS on their way meanwhile.  (A CTA per 1024 records, lanes walked by every
// thread, two block barriers at the start: 1035 us of 66.8 M records, half of it in those waits.)
#define JP_MINB 3
#define JP_ROWS 3

// adds a group of probes to the row of their window
__device__ __forceinline__ void join_emit(ta_join_summary *sm, const u64 *t) {
  if (t[0] == 0) return;
  atomicAdd((u64 *)&sm->n_probe, t[0]);
  if (t[1] == 0) return;
  atomicAdd((u64 *)&sm->n_matched, t[1]);
  atomicAdd((u64 *)&sm->sum_latency, t[2]);
  atomicAdd((u64 *)&sm->sum_queue, t[3]);
  // (codes with 0 as "none"; the host turns them into times)
  atomicMax((u64 *)&sm->max_latency, t[5]);
  atomicMax((u64 *)&sm->min_latency, t[6]);
  atomicMax((u64 *)&sm->max_queue, t[7]);
  if (t[4]) atomicAdd((u64 *)&sm->n_orphan_launch, 0ull - t[4]);
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

template <bool DIRECT, bool COUNT>
__device__ __forceinline__ void join_probe(const JoinArgs &a, int rows) {
  if (ta_failed(a.status)) return;
  const int lane = threadIdx.x & 31;
  const JoinSpan sp = join_span(a, rows);
  const u32 begin = sp.begin, end = sp.end, vend = sp.vend;
  // probes, matches, launches met for the first time; latencies and delays summed; largest latency, largest complement, largest delay
  u32 n_probe = 0, n_match = 0, n_first = 0;
  bool multi = false;
  u64 acc[5] = {0, 0, 0, 0, 0};
  int cur = -1;  // window they are of
  int had[JP_ROWS];  // kernels a matched launch had before this warp's last rows; -1 = none matched
#pragma unroll
  for (int r = 0; r < JP_ROWS; r++) had[r] = -1;
  auto count_had = [&]() {
#pragma unroll
    for (int r = 0; r < JP_ROWS; r++) {
      n_first += had[r] == 0;
      multi |= had[r] > 0;
      had[r] = -1;
    }
  };
  auto fold = [&](u64 *t) {
    count_had();
    t[0] = __reduce_add_sync(0xffffffffu, n_probe);
    t[1] = __reduce_add_sync(0xffffffffu, n_match);
    t[2] = warp_reduce(acc[0], OpAdd());
    t[3] = warp_reduce(acc[1], OpAdd());
    t[4] = __reduce_add_sync(0xffffffffu, n_first);
#pragma unroll
    for (int k = 5; k < 8; k++) t[k] = warp_reduce(acc[k - 3], OpMax());
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
        u64 t[8];
        fold(t);
        if (lane == 0) join_emit(&a.sum[cur], t);
        n_probe = n_match = n_first = 0;
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
      count_had();  // (asked for a round of rows ago: nothing waits here)
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
            if (COUNT) had[r] = atomicAdd(&a.kol[~v[r]], 1);
            else atomicAdd(&a.kol[~v[r]], 1);
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
  u64 t[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  if (cur >= 0) fold(t);
  if (multi) *a.multi = 1u;
  join_fold<5, 3>(t, cur, [&](int w, const u64 *v) { join_emit(&a.sum[w], v); });
}

// COUNT: the launches met for the first time are counted on the way (the old value of an atomic: half as
// many bytes again cross the chip); else k_join_counted does it.
template <bool DIRECT, bool COUNT, bool TAIL>
__global__ void __launch_bounds__(JN_THREADS, JP_MINB) k_join_probe(JoinArgs a, int rows, Tail tail) {
  TA_PDL();
  join_probe<DIRECT, COUNT>(a, rows);
  if (TAIL) run_tail(tail);
}

// Launches with a kernel, and whether some have several, from the column of counts.
__device__ __forceinline__ void join_counted(const JoinArgs &a, int rows) {
  if (ta_failed(a.status)) return;
  const int lane = threadIdx.x & 31;
  const JoinSpan sp = join_span(a, rows);
  u32 n_first = 0;
  bool multi = false;
  int cur = -1;
  int l = sp.begin < sp.vend ? tile_lane_search(a.lane_off, a.n_lanes, sp.begin) : 0;
  for (u32 p = sp.begin; p < sp.vend;) {
    if (a.lane_domain[l] != 0) {
      p = min((u32)a.lane_dom_end[l], sp.vend);
      if (p >= sp.vend) break;
      l = a.lane_dom_next[l];
    }
    const u32 lane_end = (u32)a.lane_off[l + 1], e = min(lane_end, sp.vend);
    const int win = a.lane_window[l];
    if (win != cur) {
      if (cur >= 0) {
        const u32 t = __reduce_add_sync(0xffffffffu, n_first);
        if (lane == 0 && t) atomicAdd((u64 *)&a.sum[cur].n_orphan_launch, 0ull - t);
        n_first = 0;
      }
      cur = win;
    }
#pragma unroll 4
    for (u32 q = p + lane; q < e; q += 32) {
      const int k = a.kol[q];
      n_first += k > 0;
      multi |= k > 1;
    }
    p = e;
    if (lane_end == e) l++;
  }
  if (multi) *a.multi = 1u;
  u64 t[1] = {__reduce_add_sync(0xffffffffu, n_first)};
  join_fold<1, 0>(t, cur, [&](int w, const u64 *v) {
    if (v[0]) atomicAdd((u64 *)&a.sum[w].n_orphan_launch, 0ull - v[0]);
  });
}
__global__ void __launch_bounds__(JN_THREADS) k_join_counted(JoinArgs a, int rows, Tail tail) {
  TA_PDL();
  join_counted(a, rows);
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
  // Rows per warp: 12, fewer where that would be less than a round of the 148 * 24 warps on the chip
  // (1.2 M records: 101 us with 12, 90 with 8), 24 where it leaves twenty rounds and more.  The call with 12
  // and with 24 rows: experts, 20 M records 315 and 345 us, 36 M 512 and 545, 52 M 761 and 811, 60 M 922 and
  // 914, 66.8 M 40 less; prefill 20 M 366 and 330, 52 M 1163 and 984, 60 M 1359 and 1197.  The line lies where
  // neither loses.
  int64_t rows = n / 32 / (148 * 32);
  rows = rows < JP_ROWS ? JP_ROWS : rows > 12 ? 12 : rows / JP_ROWS * JP_ROWS;
  if (n > (int64_t)20 * 148 * 24 * 24 * 32) rows = 24;
  const unsigned grid = (unsigned)((n + rows * JN_THREADS - 1) / (rows * JN_THREADS));
  int64_t brows = n / 32 / (148 * 64);  // (of k_join_build, the same way)
  brows = brows < JB_ROWS ? JB_ROWS : brows > 16 ? 16 : brows / JB_ROWS * JB_ROWS;
  const unsigned bgrid = (unsigned)((n + brows * JN_THREADS - 1) / (brows * JN_THREADS));
  void *tmp_alloc = nullptr;
  bool direct = true;
  int32_t words[ST_WORDS];
  TA_TRY(ta_queue_d2h(h, words, h->d_status, sizeof(words)));
  TA_TRY(ta_queue_d2h(h, hs.data(), d_sum, W * sizeof(ta_join_summary)));
  if (n > 0) {
    // table size if every slot is addressed directly
    unsigned __int128 total = 0;
    for (int s = 0; s < n_slots; s++)
      if (hmin[s] <= hmax[s]) total += (unsigned __int128)((uint64_t)hmax[s] - (uint64_t)hmin[s]) + 1;
    const uint64_t limit = (uint64_t)4 * (uint64_t)n + 65536;
    direct = total <= limit;
    // entries of the table: the span of all ids, or twice the launches and more
    // (four times while the table stays in the caches: shorter chains, and they are what the inserts wait for)
    const uint64_t M = direct ? (uint64_t)total : (h->n_launch < (1 << 21) ? 4 : 2) * (uint64_t)h->n_launch + 1;
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
    ta_launch(direct ? k_join_build<true> : k_join_build<false>, bgrid, JN_THREADS, 0, st, a, (int)brows);
    // A pass more against the returns of the atomics, which cost nothing while the columns they go to
    // stay in the caches: 16.8 M records 198 us against 190 + 13, 512 windows of 52 k records 352 against
    // 279 + 15, 66.8 M 733 against 660 + 41.
    if (n < JN_COUNT_APART) {
      const Tail tail = ta_tail(h, grid);
      auto probe = direct ? (tail.m ? k_join_probe<true, true, true> : k_join_probe<true, true, false>)
                          : (tail.m ? k_join_probe<false, true, true> : k_join_probe<false, true, false>);
      ta_launch(probe, grid, JN_THREADS, 0, st, a, (int)rows, tail);
    } else {
      ta_launch(direct ? k_join_probe<true, false, false> : k_join_probe<false, false, false>, grid, JN_THREADS, 0, st, a, (int)rows,
                Tail());
      const unsigned cgrid = (unsigned)((n + 32 * JN_THREADS - 1) / (32 * JN_THREADS));
      ta_launch(k_join_counted, cgrid, JN_THREADS, 0, st, a, 32, ta_tail(h, cgrid));
    }
    TA_CHECK_CUDA(h, cudaGetLastError());
  }
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
  return TA_OK;
}
