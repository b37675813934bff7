// ta_aggregate_ops: per (window, pid, name_id) count / sum / min / max and a log2
// histogram of a value column (own duration, T_op of operators with kernels, or the
// idle time charged to an operator by the gap blame).
// Per-symbol counts and duration statistics are what Sec. 8.1 compares.
//
// Symbol popularity is heavy-tailed (a few names carry most records), so global
// atomics alone would serialise on the hot rows.  Each CTA takes up to 8192
// consecutive sorted positions (one process, mostly; CTAs whose lanes cannot
// hold a selected kind return at once) and folds its records into a
// shared-memory hash table first, which is flushed to global rows with one atomic
// per field.  A cell = (window, pid rank, symbol rank); three ways to give cells rows:
//   dense   few cells: one row per cell, a scan compacts the non-empty ones in key order;
//   marked  many cells (a batch of windows), few of them occupied: a first pass over kinds
//           and symbols sets one bit per occupied cell, a scan over the words of the bitmap
//           numbers the occupied cells in key order, and the records are folded straight
//           into the result rows;
//   sorted  more distinct symbols than the symbol table holds, or more cells than a bitmap:
//           group by sorting, at the end of this file.
// Symbol rank = name_id - min name when the ids are close together; symbol ids spread wide
// (hashes) are ranked through a table of the distinct ones, built once per window.
// HBM-bound on the column reads: 2 B (kind) for every record, 24 B more for the
// selected ones.
#include <climits>
#include <cstring>
#include <vector>

#include "records.cuh"
#include "scan.cuh"
#include "ta_internal.cuh"

#define AG_THREADS 256
#define AG_ITEMS 4
#define AG_STEP (AG_THREADS * AG_ITEMS)
// Slots of a CTA's table: 512 (a CTA of 8192 records of a window with 4096 symbols meets some 700, and what
// finds no slot goes to memory by itself), 256 where a window has no more cells than that.
#define AG_SLOTS_LOG2 9
#define AG_SLOTS_FEW_LOG2 8
#define AG_PROBES 8
// bins a slot holds, 64 ns to 17 ms; the counts of others share a table
#define AG_BIN0 6
#define AG_BINS 18
#define AG_ODD_LOG2 9
// slots of values from 2^32 ns on (four seconds): there are few of them, but of few symbols
#define AG_WIDE_LOG2 5
#define AG_ITEM (8 * AG_STEP)    // positions per CTA at most
static_assert(AG_ITEM < (1 << 15), "a CTA's bins are 16 bits wide, the limbs of its sums 17 bits in a word");

struct AggArgs {
  int64_t n_valid;
  int n_lanes;
  const int16_t *kind;
  const int32_t *name;
  const int64_t *ts, *te;
  const int32_t *lane_off, *lane_slot;
  const int32_t *op_n;
  const int64_t *op_first, *op_last;
  const int64_t *op_gap;  // value_sel 2
  const uint8_t *on_path; // value_sel 3
  uint32_t kind_mask;
  int value_sel;
  int64_t min_name, R;
  const int16_t *lane_domain;
  const int32_t *lane_dom_end;
  int want_domain;  // 0 / 1: the selected kinds all live in lanes of this domain; -1: both
  int64_t chunk;    // positions per CTA, a multiple of AG_STEP
  unsigned n_items, spread, per;
  const u64 *names;        // symbol table when the ids are spread wide, else null
  const u32 *name_rank;
  // rows (all zero-initialised; min is kept as the complement of the biased value)
  u64 *d_cnt, *d_sum, *d_minc, *d_maxb;
  u32 *d_hist;
  // marked cells: row of cell g = rank[g / 32] + set bits of bits[g / 32] below g; null: row = cell
  u32 *bits;
  const u32 *rank;
  int32_t *status;
};

// ---- symbol table: the distinct symbol ids of the window, open addressing ------------------
#define NT_SLOTS (1u << 18)
#define NT_MAX (1u << 17)
#define NT_PROBES 512
#define NT_EMPTY 0ull  // entries are biased ids + 1
__device__ __forceinline__ u32 name_hash(u32 b) {
  u32 h = b * 0x9E3779B1u;
  h ^= h >> 15;
  h *= 0x2C1B3C6Du;
  return (h ^ (h >> 13)) & (NT_SLOTS - 1);
}
__global__ void __launch_bounds__(256) k_name_set(const int32_t *name, int64_t n_valid, u64 *names, u64 *n_names,
                                                  u64 *list, int32_t *status) {
  TA_PDL();
  __shared__ u64 cache[2048];  // ids this CTA has seen already (direct mapped, one word each)
  if (ta_failed(status)) return;
  for (int i = threadIdx.x; i < 2048; i += 256) cache[i] = NT_EMPTY;
  __syncthreads();
  for (int64_t p0 = ((int64_t)blockIdx.x * 256 + threadIdx.x) * 4; p0 < n_valid; p0 += (int64_t)gridDim.x * 1024) {
    int32_t nm[4];
    const int cnt = (int)min((int64_t)4, n_valid - p0);
    if (cnt == 4) {
      const int4 q = *reinterpret_cast<const int4 *>(name + p0);
      nm[0] = q.x; nm[1] = q.y; nm[2] = q.z; nm[3] = q.w;
    } else {
      for (int j = 0; j < 4; j++) nm[j] = j < cnt ? name[p0 + j] : 0;
    }
#pragma unroll
    for (int j = 0; j < 4; j++) {
      if (j >= cnt) break;
      const u64 e = (u64)((u32)nm[j] ^ 0x80000000u) + 1;
      u32 slot = name_hash((u32)(e - 1));
      if (cache[slot & 2047] == e) continue;
      cache[slot & 2047] = e;
      for (u32 probe = 0;; probe++) {
        u64 cur = ld_relaxed(&names[slot]);
        if (cur == NT_EMPTY || probe == NT_PROBES) {
          // too many symbols (a table half full has no run of NT_PROBES): the caller groups by sorting
          if (probe == NT_PROBES) atomicAdd(n_names, (u64)NT_MAX + 1);
          if (ld_relaxed(n_names) > NT_MAX) return;
          cur = atomicCAS(&names[slot], NT_EMPTY, e);
          if (cur == NT_EMPTY) {
            const u64 at = atomicAdd(n_names, 1ull);
            if (at < NT_MAX) list[at] = (e - 1) << 32 | slot;
            break;
          }
        }
        if (cur == e) break;
        slot = (slot + 1) & (NT_SLOTS - 1);
      }
    }
  }
}
__global__ void __launch_bounds__(256) k_name_rank(const u64 *sorted, int64_t D, u32 *name_rank, int32_t *name_of,
                                                   const int32_t *status) {
  TA_PDL();
  if (ta_failed(status)) return;
  const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (i >= D) return;
  const u64 x = sorted[i];
  name_rank[(u32)x & (NT_SLOTS - 1)] = (u32)i;
  name_of[i] = (int32_t)((u32)(x >> 32) ^ 0x80000000u);
}
template <bool TABLE>
__device__ __forceinline__ int64_t name_rank_of(const AggArgs &a, int32_t nm) {
  if (!TABLE) return (int64_t)nm - a.min_name;
  const u64 e = (u64)((u32)nm ^ 0x80000000u) + 1;
  u32 slot = name_hash((u32)(e - 1));
  // every id of the window is in the table: a bounded probe all the same
  for (u32 probe = 0; probe < NT_SLOTS && a.names[slot] != e; probe++) slot = (slot + 1) & (NT_SLOTS - 1);
  return (int64_t)a.name_rank[slot];
}
__device__ __forceinline__ int64_t row_of(const AggArgs &a, int64_t g) {
  if (!a.rank) return g;
  return (int64_t)a.rank[g >> 5] + __popc(a.bits[g >> 5] & ((1u << (g & 31)) - 1u));
}

// Values below 2^32 ns, so that everything is native 32-bit shared-memory atomics: 64-bit extremes are
// compare-and-swap loops, and with their 16 bytes and all 40 bins a slot was twice as large.  What a CTA holds
// is paid for by the cache: the two tables of 66.8 M records take 576 us, with bins from 1 ns on (38 KB a CTA) 646.
// Bins and values that a slot has no room for are added up on chip all the same, in tables of their own: in
// memory the records of no length or of a second meet at the rows of their symbols (a call on 8 M of 4 / 200
// symbols, all of no length: 2570 / 1480 us, 93 / 189 so; one in twenty of 100 ms: 217 / 187 and 99 / 172).
template <int LOG2>
struct AggSmem {
  static constexpr int SLOTS = 1 << LOG2, ODD = 1 << AG_ODD_LOG2, WIDE = 1 << AG_WIDE_LOG2;
  int32_t key[SLOTS];
  u32 sum[2][SLOTS];  // limbs of 17 and 15 bits: one atomic for a value below 131 us; the count is the sum of the bins
  u32 minc[SLOTS];    // complement of the smallest
  u32 max[SLOTS];
  uint16_t hist[SLOTS][AG_BINS];
  u32 odd[ODD];       // (slot << 6 | bin) + 1 << 16 | count; slots from SLOTS on are wide ones
  int32_t wide_key[WIDE];
  u32 wide_sum[3][WIDE];  // limbs of 17 and 17 bits and the rest, modulo 2^32
  u64 wide_minc[WIDE], wide_maxb[WIDE];
};
static_assert(((1 << AG_SLOTS_LOG2) + (1 << AG_WIDE_LOG2)) << 6 < 1 << 16 && AG_ITEM < 1 << 16, "a slot and a bin in 16 bits, a count in 16");

__device__ __forceinline__ void agg_global_add(const AggArgs &a, int64_t g, u64 cnt, u64 sum, u64 minc,
                                               u64 maxb) {
  // none of the results is used: the adds go out without the thread waiting for them
  atomicAdd(&a.d_cnt[g], cnt);
  atomicAdd(&a.d_sum[g], sum);
  atomicMax(&a.d_minc[g], minc);
  atomicMax(&a.d_maxb[g], maxb);
}

template <int LOG2>
__device__ __forceinline__ void agg_clear(AggSmem<LOG2> &s) {
  for (int i = threadIdx.x; i < s.SLOTS; i += AG_THREADS) {
    s.key[i] = -1;
    s.sum[0][i] = s.sum[1][i] = 0;
    s.minc[i] = 0;
    s.max[i] = 0;
  }
  u32 *hw = reinterpret_cast<u32 *>(&s.hist[0][0]);
  for (int i = threadIdx.x; i < s.SLOTS * AG_BINS / 2; i += AG_THREADS) hw[i] = 0;
  for (int i = threadIdx.x; i < s.ODD; i += AG_THREADS) s.odd[i] = 0;
  for (int i = threadIdx.x; i < s.WIDE; i += AG_THREADS) {
    s.wide_key[i] = -1;
    s.wide_sum[0][i] = s.wide_sum[1][i] = s.wide_sum[2][i] = 0;
    s.wide_minc[i] = s.wide_maxb[i] = 0;
  }
}

// the slot of cell g, claimed if it has none; -1: no room near
template <int LOG2>
__device__ __forceinline__ int agg_slot(int32_t *key, int32_t g) {
  int slot = (int)((u32)g * 2654435761u >> (32 - LOG2));
  for (int probe = 0; probe < AG_PROBES; probe++) {
    const int32_t cur = key[slot];
    if (cur == g) return slot;
    if (cur == -1) {
      const int32_t old = atomicCAS(&key[slot], -1, g);
      if (old == -1 || old == g) return slot;
    }
    slot = (slot + 1) & ((1 << LOG2) - 1);
  }
  return -1;
}

// What agg_chunk leaves: the bin of a value whose slot (at) does not hold it, and wide values (of cell at).
template <int LOG2>
__device__ __forceinline__ void agg_rest(const AggArgs &a, AggSmem<LOG2> &s, int32_t at, i64 v) {
  const int bin = log2_bin(v);
  int slot = at;
  if (v >> 32) {
    const u64 vb = (u64)v ^ (1ull << 63);
    slot = v > 0 ? agg_slot<AG_WIDE_LOG2>(s.wide_key, at) : -1;
    if (slot < 0) {
      const int64_t row = row_of(a, at);
      atomicAdd(&a.d_cnt[row], 1ull);
      atomicAdd(&a.d_sum[row], (u64)v);
      if (~vb > __ldcg(&a.d_minc[row])) atomicMax(&a.d_minc[row], ~vb);
      if (vb > __ldcg(&a.d_maxb[row])) atomicMax(&a.d_maxb[row], vb);
      atomicAdd(&a.d_hist[(size_t)row * TA_NBINS + bin], 1u);
      return;
    }
    atomicAdd(&s.wide_sum[0][slot], (u32)v & 0x1FFFFu);
    atomicAdd(&s.wide_sum[1][slot], (u32)(v >> 17) & 0x1FFFFu);
    atomicAdd(&s.wide_sum[2][slot], (u32)(v >> 34));
    if (~vb > s.wide_minc[slot]) atomicMax(&s.wide_minc[slot], ~vb);
    if (vb > s.wide_maxb[slot]) atomicMax(&s.wide_maxb[slot], vb);
    slot += s.SLOTS;
  }
  const u32 key = (u32)(slot << 6 | bin) + 1;
  int o = (int)(key * 2654435761u >> (32 - AG_ODD_LOG2));
  for (int probe = 0; probe < AG_PROBES; probe++) {
    u32 cur = s.odd[o];
    if (cur == 0) cur = atomicCAS(&s.odd[o], 0u, key << 16);
    if (cur == 0 || cur >> 16 == key) {
      atomicAdd(&s.odd[o], 1u);
      return;
    }
    o = (o + 1) & (s.ODD - 1);
  }
  const int64_t row = row_of(a, slot < s.SLOTS ? s.key[slot] : s.wide_key[slot - s.SLOTS]);
  atomicAdd(&a.d_cnt[row], 1ull);
  atomicAdd(&a.d_hist[(size_t)row * TA_NBINS + bin], 1u);
}

template <int LOG2>
__device__ __forceinline__ void agg_flush(const AggArgs &a, AggSmem<LOG2> &s) {
  __syncthreads();
  for (int i = threadIdx.x; i < s.SLOTS; i += AG_THREADS) {
    int32_t k = s.key[i];
    if (k >= 0) {
      k = (int32_t)row_of(a, k);
      s.key[i] = k;
      const u32 *hw = reinterpret_cast<const u32 *>(&s.hist[i][0]);
      u32 cnt = 0;
#pragma unroll
      for (int b = 0; b < AG_BINS / 2; b++) cnt += (hw[b] & 0xFFFFu) + (hw[b] >> 16);
      agg_global_add(a, k, cnt, (u64)s.sum[0][i] + ((u64)s.sum[1][i] << 17), ~((u64)(u32)~s.minc[i] ^ (1ull << 63)),
                     (u64)s.max[i] ^ (1ull << 63));
    }
  }
  for (int i = threadIdx.x; i < s.WIDE; i += AG_THREADS)
    if (s.wide_key[i] >= 0) {
      const int32_t k = (int32_t)row_of(a, s.wide_key[i]);
      s.wide_key[i] = k;
      agg_global_add(a, k, 0, (u64)s.wide_sum[0][i] + ((u64)s.wide_sum[1][i] << 17) + ((u64)s.wide_sum[2][i] << 34),
                     s.wide_minc[i], s.wide_maxb[i]);
    }
  __syncthreads();
  for (int i = threadIdx.x; i < s.ODD; i += AG_THREADS)
    if (s.odd[i]) {
      const u32 sb = (s.odd[i] >> 16) - 1, sl = sb >> 6, c = s.odd[i] & 0xFFFFu;
      const int32_t row = sl < s.SLOTS ? s.key[sl] : s.wide_key[sl - s.SLOTS];
      atomicAdd(&a.d_cnt[row], (u64)c);
      atomicAdd(&a.d_hist[(size_t)row * TA_NBINS + (sb & 63u)], c);
    }
  // histogram bins: one thread per (slot, bin).  Not unrolled: fetching the longer code costs a window of
  // 60 k records 1.5 us a call (24.5 and 23.7 us against 26.1 and 25.7), and saves 16.8 M two of 135
#pragma unroll 1
  for (int i = threadIdx.x; i < s.SLOTS * AG_BINS; i += AG_THREADS) {
    const int sl = i / AG_BINS, b = i - sl * AG_BINS;
    const u32 c = s.hist[sl][b];
    if (c) atomicAdd(&a.d_hist[(size_t)s.key[sl] * TA_NBINS + AG_BIN0 + b], c);
  }
}

// Which of the thread's four records are selected, their values and symbols (a caller that makes no
// use of the values pays for no load of them).
__device__ __forceinline__ void agg_select(const AggArgs &a, int64_t p0, int64_t end, bool (&sel)[AG_ITEMS],
                                           i64 (&v)[AG_ITEMS], int32_t (&nm)[AG_ITEMS]) {
  // all loads of the thread's four records are issued before any of them is used; for the
  // plain duration the times and names are requested with the kinds, not after them (the
  // step holds lanes of the wanted domain, so most records are selected anyway)
  int16_t kd[AG_ITEMS];
  i64 pre_v[AG_ITEMS];
  int32_t pre_nm[AG_ITEMS];
#pragma unroll
  for (int j = 0; j < AG_ITEMS; j++) { pre_v[j] = 0; pre_nm[j] = 0; }
  if (p0 + AG_ITEMS <= end) {
    uint2 q = *reinterpret_cast<const uint2 *>(a.kind + p0);
    if (a.value_sel == 0) {
      const longlong2 *ps = reinterpret_cast<const longlong2 *>(a.ts + p0);
      const longlong2 *pe = reinterpret_cast<const longlong2 *>(a.te + p0);
      const int4 nq = *reinterpret_cast<const int4 *>(a.name + p0);
#pragma unroll
      for (int h2 = 0; h2 < AG_ITEMS / 2; h2++) {
        const longlong2 x = ps[h2], y = pe[h2];
        pre_v[2 * h2] = y.x - x.x;
        pre_v[2 * h2 + 1] = y.y - x.y;
      }
      pre_nm[0] = nq.x; pre_nm[1] = nq.y; pre_nm[2] = nq.z; pre_nm[3] = nq.w;
    } else if (a.value_sel == 1) {  // the kernel counts with the kinds (pre_nm holds them)
      const int4 cq = *reinterpret_cast<const int4 *>(a.op_n + p0);
      pre_nm[0] = cq.x; pre_nm[1] = cq.y; pre_nm[2] = cq.z; pre_nm[3] = cq.w;
    }
    const int16_t *hq = reinterpret_cast<const int16_t *>(&q);
#pragma unroll
    for (int j = 0; j < AG_ITEMS; j++) kd[j] = hq[j];
  } else {
#pragma unroll
    for (int j = 0; j < AG_ITEMS; j++) {
      kd[j] = p0 + j < end ? a.kind[p0 + j] : (int16_t)-1;
      if (a.value_sel == 0 && p0 + j < end) { pre_v[j] = a.te[p0 + j] - a.ts[p0 + j]; pre_nm[j] = a.name[p0 + j]; }
      if (a.value_sel == 1 && p0 + j < end) pre_nm[j] = a.op_n[p0 + j];
    }
  }
#pragma unroll
  for (int j = 0; j < AG_ITEMS; j++) {
    sel[j] = kd[j] >= 0 && ((a.kind_mask >> kd[j]) & 1u);
    v[j] = 0;
    nm[j] = 0;
  }
  if (a.value_sel == 0) {
#pragma unroll
    for (int j = 0; j < AG_ITEMS; j++)
      if (sel[j]) { v[j] = pre_v[j]; nm[j] = pre_nm[j]; }
  } else if (a.value_sel == 1) {
#pragma unroll
    for (int j = 0; j < AG_ITEMS; j++)
      if (sel[j]) sel[j] = pre_nm[j] > 0;
#pragma unroll
    for (int j = 0; j < AG_ITEMS; j++)
      if (sel[j]) { v[j] = a.op_last[p0 + j] - a.op_first[p0 + j]; nm[j] = a.name[p0 + j]; }
  } else if (a.value_sel == 2) {
#pragma unroll
    for (int j = 0; j < AG_ITEMS; j++)
      if (sel[j]) { v[j] = a.op_gap[p0 + j]; sel[j] = v[j] > 0; }
#pragma unroll
    for (int j = 0; j < AG_ITEMS; j++)
      if (sel[j]) nm[j] = a.name[p0 + j];
  } else {
#pragma unroll
    for (int j = 0; j < AG_ITEMS; j++)
      if (sel[j]) sel[j] = a.on_path[p0 + j] != 0;
#pragma unroll
    for (int j = 0; j < AG_ITEMS; j++)
      if (sel[j]) { v[j] = a.te[p0 + j] - a.ts[p0 + j]; nm[j] = a.name[p0 + j]; }
  }
}

// sets the bit of every cell that holds a selected record
template <bool TABLE>
__global__ void __launch_bounds__(AG_THREADS) k_agg_mark(AggArgs a) {
  TA_PDL();
  if (ta_failed(a.status)) return;
  LaneWalker lw(a.lane_off, a.n_lanes, a.n_valid, a.n_valid);
  const int64_t begin = (int64_t)blockIdx.x * a.chunk, end = min(begin + a.chunk, a.n_valid);
  if (begin >= end) return;
  int bl = lane_of_pos(a.lane_off, a.n_lanes, begin);
  for (int64_t base = begin; base < end; base += AG_STEP) {
    while (bl + 1 < a.n_lanes && (int64_t)a.lane_off[bl + 1] <= base) bl++;
    if (a.want_domain >= 0 &&
        span_outside_domain(a.lane_domain, a.lane_dom_end, bl, min(base + AG_STEP, end), a.want_domain))
      continue;
    lw.lane = bl;
    const int64_t p0 = base + (int64_t)threadIdx.x * AG_ITEMS;
    bool sel[AG_ITEMS];
    i64 v[AG_ITEMS];
    int32_t nm[AG_ITEMS];
    agg_select(a, p0, end, sel, v, nm);
#pragma unroll
    for (int j = 0; j < AG_ITEMS; j++) {
      if (!sel[j]) continue;
      const int64_t g = (int64_t)a.lane_slot[lw.at(p0 + j)] * a.R + name_rank_of<TABLE>(a, nm[j]);
      // a stale word only costs a second atomic: popular cells are set once and then read from L1
      if (!((a.bits[g >> 5] >> (g & 31)) & 1u)) atomicOr(&a.bits[g >> 5], 1u << (g & 31));
    }
  }
}

template <bool TABLE, int LOG2>
__device__ __forceinline__ void agg_chunk(const AggArgs &a) {
  __shared__ AggSmem<LOG2> s;
  if (ta_failed(a.status)) return;
  LaneWalker lw(a.lane_off, a.n_lanes, a.n_valid, a.n_valid);
  {
    // CTA b -> chunk (b mod G) * S + b / G: CTAs that run together work far apart in the
    // timeline (different processes), so their flushes rarely meet on the same global rows;
    // chunks whose lanes cannot hold a selected kind return at once and make room
    const unsigned item = (blockIdx.x % a.spread) * a.per + blockIdx.x / a.spread;
    if (item >= a.n_items) return;
    const int64_t begin = (int64_t)item * a.chunk;
    const int64_t end = min(begin + a.chunk, a.n_valid);
    int bl = lane_of_pos(a.lane_off, a.n_lanes, begin);  // lane of `base`, the same in every thread
    if (a.want_domain >= 0 &&
        span_outside_domain(a.lane_domain, a.lane_dom_end, bl, end, a.want_domain))
      return;
    agg_clear(s);
    __syncthreads();
    for (int64_t base = begin; base < end; base += AG_STEP) {
      while (bl + 1 < a.n_lanes && (int64_t)a.lane_off[bl + 1] <= base) bl++;
      if (a.want_domain >= 0 && span_outside_domain(a.lane_domain, a.lane_dom_end, bl,
                                                    min(base + AG_STEP, end), a.want_domain))
        continue;
      lw.lane = bl;
      const int64_t p0 = base + (int64_t)threadIdx.x * AG_ITEMS;
      bool sel[AG_ITEMS];
      i64 v[AG_ITEMS];
      int32_t nm[AG_ITEMS];
      agg_select(a, p0, end, sel, v, nm);
      u32 rest = 0;
#pragma unroll
      for (int j = 0; j < AG_ITEMS; j++) {
        if (!sel[j]) continue;
        const int lane = lw.at(p0 + j);
        const int32_t g = nm[j] = (int32_t)((int64_t)a.lane_slot[lane] * a.R + name_rank_of<TABLE>(a, nm[j]));
        if ((u64)v[j] >> 32) {
          rest |= 1u << j;
          continue;
        }
        const int slot = agg_slot<LOG2>(s.key, g), bin = log2_bin(v[j]);
        if (slot < 0) {
          const int64_t row = row_of(a, g);
          const u64 vb = (u64)v[j] ^ (1ull << 63);
          agg_global_add(a, row, 1, (u64)v[j], ~vb, vb);
          atomicAdd(&a.d_hist[(size_t)row * TA_NBINS + bin], 1u);
          continue;
        }
        // values are durations (>= 0), fewer than 2^15 adds per CTA: 2^15 x 2^17 fits a word
        const u32 uv = (u32)v[j];
        atomicAdd(&s.sum[0][slot], uv & 0x1FFFFu);
        if (uv >> 17) atomicAdd(&s.sum[1][slot], uv >> 17);
        // an atomic only where the value would move the extreme (rare once a slot has seen a few records)
        if (~uv > s.minc[slot]) atomicMax(&s.minc[slot], ~uv);
        if (uv > s.max[slot]) atomicMax(&s.max[slot], uv);
        const u32 b = (u32)(bin - AG_BIN0);
        if (b < AG_BINS) {  // 16-bit bins packed two per word
          u32 *hw = reinterpret_cast<u32 *>(&s.hist[slot][0]) + (b >> 1);
          atomicAdd(hw, (b & 1) ? 0x10000u : 1u);
        } else {
          rest |= 1u << j;
          nm[j] = slot;
        }
      }
#pragma unroll 1
      for (; rest; rest &= rest - 1) {
        const int j = __ffs((int)rest) - 1;
        i64 vj = v[0];
        int32_t at = nm[0];
#pragma unroll
        for (int k = 1; k < AG_ITEMS; k++)
          if (j == k) { vj = v[k]; at = nm[k]; }
        agg_rest(a, s, at, vj);
      }
    }
  }
  agg_flush(a, s);
}

struct AggRowOut {
  const u64 *cnt, *sum, *minc, *maxb;
  const u32 *hist;
  const TripleTable *tt;
  int n_pids;
  int64_t R, min_name;
  const int32_t *name_of;  // symbol of a rank, null: rank + min_name
  int32_t *g_window, *g_pid, *g_name;
  int64_t *g_count, *g_sum, *g_min, *g_max;
  u32 *g_hist;
};

// Dense cells: compaction of the non-empty ones in cell (= key) order, chained over the CTAs.  The histograms (160 of a row's 200 bytes) are copied by the CTA together, 16 bytes per
// thread, rows side by side: one thread per row copying its own took 36 us for the 4096 cells of a
// prefill window, most of it waiting.
#define AC_THREADS 256
// Cells per CTA: 64 while a window has a few thousand; 256 beyond 4096, where all CTAs look back at once and
// the length of the chain is what counts (62 k cells: 20 us with 977 CTAs).
template <int AC_CELLS>
__global__ void __launch_bounds__(AC_THREADS) k_agg_rows(int64_t G, AggRowOut o, u64 *state, u64 *total,
                                                         u32 *ticket, int32_t *status, Tail tail) {
  TA_PDL();
  __shared__ u64 tmp[33];
  __shared__ u64 s_excl;
  __shared__ u32 s_cell[AC_CELLS];
  __shared__ int s_fail, s_tile;
  const int tid = threadIdx.x;
  if (tid == 0) s_tile = (int)atomicAdd(ticket, 1u);
  __syncthreads();
  const int tile = s_tile;
  const int64_t g = tid < AC_CELLS ? (int64_t)tile * AC_CELLS + tid : G;
  const bool failed = ta_failed(status);
  // everything a row takes is asked for before the CTAs in front are looked back at
  const bool in = !failed && g < G;
  const u64 c = in ? o.cnt[g] : 0, sum = in ? o.sum[g] : 0, minc = in ? o.minc[g] : 0, maxb = in ? o.maxb[g] : 0;
  const int64_t slot = in ? g / o.R : 0, r = in ? g - slot * o.R : 0;
  const int32_t pid = in ? o.tt->pid_value[slot % o.n_pids] : 0;
  const int32_t name = in && o.name_of ? o.name_of[r] : (int32_t)(o.min_name + r);
  u64 rows;
  const u64 ex = block_scan_exclusive<OpAdd>(c ? 1ull : 0ull, OpAdd(), tmp, &rows);
  if (tid < 32) {
    bool gave_up = false;
    const u64 e = failed ? 0 : tile_lookback<OpAdd>(state, tile, rows, OpAdd(), status, &gave_up);
    if (tid == 0) {
      s_excl = e;
      s_fail = failed || gave_up;
      if (!s_fail && tile == (int)gridDim.x - 1) *total = e + rows;
    }
  }
  if (c) s_cell[ex] = (u32)tid;
  __syncthreads();
  if (!s_fail) {
    const u64 first = s_excl;
    if (c) {
      const u64 row = first + ex;
      o.g_window[row] = (int32_t)(slot / o.n_pids);
      o.g_pid[row] = pid;
      o.g_name[row] = name;
      o.g_count[row] = (int64_t)c;
      o.g_sum[row] = (int64_t)sum;
      o.g_min[row] = (int64_t)((~minc) ^ (1ull << 63));
      o.g_max[row] = (int64_t)(maxb ^ (1ull << 63));
    }
    const uint4 *src = reinterpret_cast<const uint4 *>(o.hist) + (size_t)tile * AC_CELLS * (TA_NBINS / 4);
    uint4 *dst = reinterpret_cast<uint4 *>(o.g_hist) + first * (TA_NBINS / 4);
    const int words = (int)rows * (TA_NBINS / 4);
    constexpr int BATCH = 5;
    for (int i0 = tid; i0 < words; i0 += AC_THREADS * BATCH) {
      uint4 v[BATCH];
#pragma unroll
      for (int k = 0; k < BATCH; k++) {
        const int i = i0 + k * AC_THREADS, row = i / (TA_NBINS / 4);
        if (i < words) v[k] = src[s_cell[row] * (TA_NBINS / 4) + (i - row * (TA_NBINS / 4))];
      }
#pragma unroll
      for (int k = 0; k < BATCH; k++)
        if (i0 + k * AC_THREADS < words) dst[i0 + k * AC_THREADS] = v[k];
    }
  }
  run_tail(tail);
}

// The same for a few cells, by the last CTA of k_agg.
#define AG_ROWS_HERE AG_THREADS
static_assert(AG_ROWS_HERE <= 1 << AG_SLOTS_FEW_LOG2, "a slot for every cell");
__device__ __forceinline__ void agg_rows_here(int G, const AggRowOut &o, u64 *total) {
  __shared__ u64 tmp[33];
  __shared__ u32 s_cell[AG_ROWS_HERE];
  const int g = threadIdx.x;
  // everything a row takes is asked for together (one field after the other, each is a round trip to L2)
  const bool in = g < G;
  const u64 c = in ? __ldcg(&o.cnt[g]) : 0, sum = in ? __ldcg(&o.sum[g]) : 0, minc = in ? __ldcg(&o.minc[g]) : 0,
            maxb = in ? __ldcg(&o.maxb[g]) : 0;
  const int slot = in ? g / (int)o.R : 0, r = in ? g - slot * (int)o.R : 0;
  const int32_t pid = in ? o.tt->pid_value[slot % o.n_pids] : 0;
  const int32_t name = in && o.name_of ? o.name_of[r] : (int32_t)(o.min_name + r);
  u64 rows;
  const u64 row = block_scan_exclusive<OpAdd>(c ? 1ull : 0ull, OpAdd(), tmp, &rows);
  if (c) {
    s_cell[row] = (u32)g;
    o.g_window[row] = slot / o.n_pids;
    o.g_pid[row] = pid;
    o.g_name[row] = name;
    o.g_count[row] = (int64_t)c;
    o.g_sum[row] = (int64_t)sum;
    o.g_min[row] = (int64_t)((~minc) ^ (1ull << 63));
    o.g_max[row] = (int64_t)(maxb ^ (1ull << 63));
  }
  if (g == 0) {
    *total = rows;
    __threadfence();
  }
  __syncthreads();
  const uint4 *src = reinterpret_cast<const uint4 *>(o.hist);
  uint4 *dst = reinterpret_cast<uint4 *>(o.g_hist);
  const int words = (int)rows * (TA_NBINS / 4);
  constexpr int BATCH = 5;
  for (int i0 = g; i0 < words; i0 += AG_THREADS * BATCH) {
    uint4 v[BATCH];
#pragma unroll
    for (int k = 0; k < BATCH; k++) {
      const int i = i0 + k * AG_THREADS, q = i / (TA_NBINS / 4);
      if (i < words) v[k] = __ldcg(src + s_cell[q] * (TA_NBINS / 4) + (i - q * (TA_NBINS / 4)));
    }
#pragma unroll
    for (int k = 0; k < BATCH; k++)
      if (i0 + k * AG_THREADS < words) dst[i0 + k * AG_THREADS] = v[k];
  }
}

// rows_here: cells whose rows the last CTA compacts, 0 = none (k_agg_rows does, or there is nothing to compact)
template <bool TABLE, bool TAIL>
__global__ void __launch_bounds__(AG_THREADS, 6) k_agg(AggArgs a, int rows_here, AggRowOut o, u64 *total, Tail tail) {
  TA_PDL();
  agg_chunk<TABLE, TAIL ? AG_SLOTS_FEW_LOG2 : AG_SLOTS_LOG2>(a);
  if (TAIL) run_tail(tail, [&] {
    if (rows_here && !ta_failed(a.status)) agg_rows_here(rows_here, o, total);
  });
}

// ---- marked cells: numbering, and what is left to write of a row -----------------------------
struct AggBitsIn {
  const u32 *bits;
  __device__ u64 operator()(int64_t i) const { return (u64)__popc(bits[i]); }
};
struct AggBitsOut {
  u32 *rank;
  __device__ void operator()(int64_t i, u64 excl, u64) const { rank[i] = (u32)excl; }
};
// key and extremes of the rows (the extremes were accumulated in order-preserving codes with 0 as
// "nothing yet"): a warp takes 32 words of the bitmap, whose rows follow one another, and writes them side
// by side (a thread per word, each with its own rows: 65 and 44 us of the two tables of 512 windows of 65 k
// records, 38 and 26 now)
__global__ void __launch_bounds__(256) k_agg_marked_rows(const u32 *bits, const u32 *rank, int64_t words,
                                                         AggRowOut o, const int32_t *status) {
  TA_PDL();
  if (ta_failed(status)) return;
  const int lane = threadIdx.x & 31;
  const int64_t w0 = ((int64_t)blockIdx.x * 256 + threadIdx.x) - lane;
  const u32 m = w0 + lane < words ? bits[w0 + lane] : 0;
  const u32 mine = (u32)__popc(m), upto = (u32)warp_scan_inclusive((u64)mine, OpAdd()), before = upto - mine;
  const u32 total = __shfl_sync(0xffffffffu, upto, 31);
  if (total == 0) return;
  const u32 first = rank[w0];  // rows in front of the warp's
  for (u32 t0 = 0; t0 < total; t0 += 32) {
    const u32 t = min(t0 + lane, total - 1);
    // the word the row is of: the last whose first row is not behind it (of several, the one with rows)
    int at = 0;
#pragma unroll
    for (int step = 16; step > 0; step >>= 1)
      if (__shfl_sync(0xffffffffu, before, at + step) <= t) at += step;
    u32 word = __shfl_sync(0xffffffffu, m, at), k = t - __shfl_sync(0xffffffffu, before, at);
    int bit = 0;  // its set bit number k
#pragma unroll
    for (int half = 16; half > 0; half >>= 1) {
      const u32 low = (u32)__popc(word & ((1u << half) - 1u));
      if (k >= low) { k -= low; word >>= half; bit += half; }
      else word &= (1u << half) - 1u;
    }
    if (t0 + lane >= total) continue;
    const int64_t row = (int64_t)first + t, g = (w0 + at) * 32 + bit;
    const int64_t slot = g / o.R, r = g - slot * o.R;
    const i64 lo = o.g_min[row], hi = o.g_max[row];
    o.g_window[row] = (int32_t)(slot / o.n_pids);
    o.g_pid[row] = o.tt->pid_value[slot % o.n_pids];
    o.g_name[row] = o.name_of ? o.name_of[r] : (int32_t)(o.min_name + r);
    o.g_min[row] = (int64_t)((~(u64)lo) ^ (1ull << 63));
    o.g_max[row] = (int64_t)((u64)hi ^ (1ull << 63));
  }
}

// ---- too many symbols or cells: aggregate by sorting ---------------
// The selected records are compacted to (key, position) pairs with key = (window, pid) slot
// << 32 | name_id (order-preserving code), sorted with the pair sorter, cut into groups where
// the key changes, and reduced with atomics on the group rows - one per run of equal keys
// inside a thread's eight consecutive elements, so a popular symbol costs an eighth of its
// records in atomics.  Rows come out in key order, as from the dense path.
struct AggSortCtx {
  int64_t n_valid;
  int n_lanes, n_pids;
  uint32_t kind_mask;
  int value_sel;
  const int16_t *kind;
  const int32_t *name;
  const int64_t *ts, *te;
  const int32_t *op_n;
  const int64_t *op_first, *op_last, *op_gap;
  const uint8_t *on_path;
  const int32_t *lane_off, *lane_slot;
  const TripleTable *tt;
  const int32_t *status;
};
__device__ __forceinline__ bool agg_selected(const AggSortCtx &c, int64_t p, i64 *v) {
  const int k = c.kind[p];
  if (k < 0 || k > 5 || !((c.kind_mask >> k) & 1u)) return false;
  if (c.value_sel == 0) { *v = c.te[p] - c.ts[p]; return true; }
  if (c.value_sel == 1) {
    if (c.op_n[p] <= 0) return false;
    *v = c.op_last[p] - c.op_first[p];
    return true;
  }
  if (c.value_sel == 2) {
    *v = c.op_gap[p];
    return *v > 0;
  }
  if (!c.on_path[p]) return false;
  *v = c.te[p] - c.ts[p];
  return true;
}
struct AggSelIn {
  AggSortCtx c;
  __device__ u64 operator()(int64_t p) const {
    i64 v;
    return agg_selected(c, p, &v) ? 1ull : 0ull;
  }
};
struct AggSelOut {
  AggSortCtx c;
  u64 *keys;
  u32 *pos;
  __device__ void operator()(int64_t p, u64 excl, u64 v) const {
    if (!v) return;
    const int lane = lane_of_pos(c.lane_off, c.n_lanes, p);
    keys[excl] = ((u64)c.lane_slot[lane] << 32) | (u64)((u32)c.name[p] ^ 0x80000000u);
    pos[excl] = (u32)p;
  }
};
struct AggHeadIn {
  const u64 *ks;
  __device__ u64 operator()(int64_t j) const { return (j == 0 || ks[j] != ks[j - 1]) ? 1ull : 0ull; }
};
struct AggHeadOut {
  int32_t *gid;     // per sorted element
  int32_t *gstart;  // per group
  __device__ void operator()(int64_t j, u64 excl, u64 v) const {
    const int32_t g = (int32_t)(excl + v) - 1;
    gid[j] = g;
    if (v) gstart[g] = (int32_t)j;
  }
};
struct AggSortedOut {
  int32_t *g_window, *g_pid, *g_name;
  int64_t *g_count, *g_sum, *g_min, *g_max;
  u32 *g_hist;
};
__global__ void __launch_bounds__(256) k_agg_sorted_rows(AggSortCtx c, const u64 *ks, const int32_t *gstart,
                                                        int64_t ng, AggSortedOut o) {
  TA_PDL();
  if (ta_failed(c.status)) return;
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= ng) return;
  const u64 key = ks[gstart[g]];
  const int64_t slot = (int64_t)(key >> 32);
  o.g_window[g] = (int32_t)(slot / c.n_pids);
  o.g_pid[g] = c.tt->pid_value[slot % c.n_pids];
  o.g_name[g] = (int32_t)((u32)key ^ 0x80000000u);
  o.g_min[g] = INT64_MAX;
  o.g_max[g] = INT64_MIN;
}
__global__ void __launch_bounds__(256) k_agg_sorted_reduce(AggSortCtx c, const u32 *pos, const int32_t *gid,
                                                          int64_t m, AggSortedOut o) {
  TA_PDL();
  if (ta_failed(c.status)) return;
  const int64_t j0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * 8;
  if (j0 >= m) return;
  int32_t cur = -1;
  u64 cnt = 0, sum = 0;
  i64 mn = INT64_MAX, mx = INT64_MIN;
  for (int k = 0; k < 8 && j0 + k < m; k++) {
    const int32_t g = gid[j0 + k];
    i64 v = 0;
    agg_selected(c, pos[j0 + k], &v);
    if (g != cur) {
      if (cur >= 0) {
        atomicAdd((u64 *)&o.g_count[cur], cnt);
        atomicAdd((u64 *)&o.g_sum[cur], sum);
        atomicMin((i64 *)&o.g_min[cur], mn);
        atomicMax((i64 *)&o.g_max[cur], mx);
      }
      cur = g; cnt = 0; sum = 0; mn = INT64_MAX; mx = INT64_MIN;
    }
    cnt++;
    sum += (u64)v;
    mn = v < mn ? v : mn;
    mx = v > mx ? v : mx;
    atomicAdd(&o.g_hist[(size_t)g * TA_NBINS + log2_bin(v)], 1u);
  }
  if (cur >= 0) {
    atomicAdd((u64 *)&o.g_count[cur], cnt);
    atomicAdd((u64 *)&o.g_sum[cur], sum);
    atomicMin((i64 *)&o.g_min[cur], mn);
    atomicMax((i64 *)&o.g_max[cur], mx);
  }
}

static ta_status ta_run_aggregate_sorted(ta_window *h, uint32_t kind_mask, int value_sel,
                                         ta_agg_result *out) {
  cudaStream_t st = h->stream;
  const int n_pids = h->n_pids > 0 ? h->n_pids : 1;
  const int64_t nv = h->n_valid;
  AggSortCtx c;
  memset(&c, 0, sizeof(c));
  c.n_valid = nv; c.n_lanes = h->sorted.n_lanes; c.n_pids = n_pids;
  c.kind_mask = kind_mask & 63u; c.value_sel = value_sel;
  c.kind = h->sorted.kind; c.name = h->sorted.name_id; c.ts = h->sorted.ts_start; c.te = h->sorted.ts_end;
  c.op_n = h->attr.op_n_kernels; c.op_first = h->attr.op_first_start; c.op_last = h->attr.op_last_end;
  c.op_gap = h->d_op_gap_ns; c.on_path = h->d_on_path; c.lane_off = h->sorted.lane_off; c.lane_slot = h->d_lane_slot;
  c.tt = h->d_triples; c.status = h->d_status;

  // 1. selection
  size_t t1b = Carver::pad((size_t)nv * 8) + Carver::pad((size_t)nv * 4) + scan_temp_bytes(nv) + 256;
  void *t1 = ta_dalloc(h, t1b);
  if (!t1) return TA_ERR_OOM;
  Carver c1(t1);
  u64 *k_in = c1.take<u64>(nv);
  u32 *v_in = c1.take<u32>(nv);
  ScanTemp s1;
  TA_TRY(scan_temp_init(h, c1.base + c1.off, nv, &s1));
  AggSelIn si{c};
  AggSelOut so{c, k_in, v_in};
  TA_TRY((launch_scan<OpAdd, AggSelIn, AggSelOut>(h, nv, si, so, OpAdd(), s1)));
  u64 m64 = 0;
  int32_t words[ST_WORDS];
  TA_TRY(ta_queue_d2h(h, &m64, s1.total, 8));
  TA_TRY(ta_read_status(h, words));
  if (words[ST_ERR]) return (ta_status)words[ST_ERR];  // (nothing was selected then)
  const int64_t m = (int64_t)m64;
  if (m == 0) { ta_dfree(h, t1); return TA_OK; }

  // 2. sort, 3. groups
  int slot_bits = 1;
  while (slot_bits < 31 && ((int64_t)h->W * n_pids - 1) >> slot_bits) slot_bits++;
  size_t t2b = 2 * Carver::pad((size_t)m * 8) + 2 * Carver::pad((size_t)m * 4) + 2 * Carver::pad((size_t)(m + 1) * 4) +
               ta_sort_temp_bytes(m) + scan_temp_bytes(m) + 256;
  void *t2 = ta_dalloc(h, t2b);
  if (!t2) return TA_ERR_OOM;
  Carver c2(t2);
  u64 *k_scr = c2.take<u64>(m), *ks = c2.take<u64>(m);
  u32 *v_scr = c2.take<u32>(m), *vs = c2.take<u32>(m);
  int32_t *gid = c2.take<int32_t>(m + 1), *gstart = c2.take<int32_t>(m + 1);
  void *sort_tmp = c2.base + c2.off; c2.off += ta_sort_temp_bytes(m);
  void *scan2 = c2.base + c2.off;
  TA_TRY(ta_radix_sort_pairs(h, k_in, v_in, k_scr, v_scr, ks, vs, m, ta_make_plan(0, 32 + slot_bits), nullptr,
                             sort_tmp));
  ScanTemp s2;
  TA_TRY(scan_temp_init(h, scan2, m, &s2));
  AggHeadIn hi{ks};
  AggHeadOut ho{gid, gstart};
  TA_TRY((launch_scan<OpAdd, AggHeadIn, AggHeadOut>(h, m, hi, ho, OpAdd(), s2)));
  u64 ng64 = 0;
  TA_TRY(ta_queue_d2h(h, &ng64, s2.total, 8));
  TA_TRY(ta_sync_fetch(h));
  const int64_t ng = (int64_t)ng64;

  // 4. rows
  size_t ob = 3 * Carver::pad((size_t)ng * 4) + 4 * Carver::pad((size_t)ng * 8) +
              Carver::pad((size_t)ng * TA_NBINS * 4) + 256;
  void *outb = ta_dalloc(h, ob);
  if (!outb) return TA_ERR_OOM;
  TA_CHECK_CUDA(h, cudaMemsetAsync(outb, 0, ob, st));
  Carver co(outb);
  AggSortedOut o;
  o.g_window = co.take<int32_t>(ng); o.g_pid = co.take<int32_t>(ng); o.g_name = co.take<int32_t>(ng);
  o.g_count = co.take<int64_t>(ng); o.g_sum = co.take<int64_t>(ng);
  o.g_min = co.take<int64_t>(ng); o.g_max = co.take<int64_t>(ng);
  o.g_hist = co.take<u32>((size_t)ng * TA_NBINS);
  ta_launch(k_agg_sorted_rows, (unsigned)((ng + 255) / 256), 256, 0, st, c, ks, gstart, ng, o);
  ta_launch(k_agg_sorted_reduce, (unsigned)((m + 2047) / 2048), 256, 0, st, c, vs, gid, m, o);
  TA_CHECK_CUDA(h, cudaGetLastError());
  TA_TRY(ta_read_status(h, words));
  ta_dfree(h, t1);
  ta_dfree(h, t2);
  if (words[ST_ERR]) return (ta_status)words[ST_ERR];
  out->n_groups = ng;
  out->g_window = o.g_window; out->g_pid = o.g_pid; out->g_name = o.g_name;
  out->g_count = o.g_count; out->g_sum = o.g_sum; out->g_min = o.g_min; out->g_max = o.g_max;
  out->g_hist = o.g_hist;
  return TA_OK;
}

// Builds the symbol table of the window (once per handle); h->n_names = number of distinct ids, or
// -1 if there are more than NT_MAX.
static ta_status build_names(ta_window *h) {
  if (h->n_names) return TA_OK;
  cudaStream_t st = h->stream;
  void *tmp = ta_dalloc(h, Carver::pad((size_t)NT_MAX * 8));
  const size_t keep = Carver::pad((size_t)NT_SLOTS * 8) + Carver::pad(64) + Carver::pad((size_t)NT_SLOTS * 4) +
                      Carver::pad((size_t)NT_MAX * 4);
  void *kb = ta_dalloc(h, keep);
  if (!tmp || !kb) return TA_ERR_OOM;
  u64 *list = (u64 *)tmp;
  Carver ck(kb);
  h->d_names = ck.take<u64>(NT_SLOTS);
  u64 *count = ck.take<u64>(8);
  TA_CHECK_CUDA(h, cudaMemsetAsync(kb, 0, ck.off, st));
  h->d_name_rank = ck.take<u32>(NT_SLOTS);
  h->d_name_of = ck.take<int32_t>(NT_MAX);
  const int64_t want = (h->n_valid + 1023) / 1024;
  ta_launch(k_name_set, (unsigned)(want < 148 * 8 ? want : 148 * 8), 256, 0, st, h->sorted.name_id, h->n_valid, h->d_names, count, list, h->d_status);
  TA_CHECK_CUDA(h, cudaGetLastError());
  u64 D = 0;
  TA_TRY(ta_queue_d2h(h, &D, count, 8));
  TA_TRY(ta_sync_fetch(h));
  if (D == 0 || D > NT_MAX) {  // (0: an earlier kernel failed; the caller's status check reports it)
    h->n_names = -1;
  } else {
    void *sb = ta_dalloc(h, 2 * Carver::pad(D * 8) + ta_sort_temp_bytes((int64_t)D) + 256);
    if (!sb) return TA_ERR_OOM;
    Carver cs(sb);
    u64 *scr = cs.take<u64>(D), *sorted = cs.take<u64>(D);
    TA_TRY(ta_radix_sort_keys(h, list, scr, sorted, (int64_t)D, ta_make_plan(32, 64), nullptr, cs.base + cs.off, false));
    ta_launch(k_name_rank, (unsigned)((D + 255) / 256), 256, 0, st, sorted, (int64_t)D, h->d_name_rank, h->d_name_of, h->d_status);
    TA_CHECK_CUDA(h, cudaGetLastError());
    h->n_names = (int64_t)D;
    ta_dfree_later(h, sb);
  }
  ta_dfree_later(h, tmp);
  return TA_OK;
}

ta_status ta_run_aggregate(ta_window *h, uint32_t kind_mask, int value_sel, ta_agg_result *out) {
  cudaStream_t st = h->stream;
  const int n_pids = h->n_pids > 0 ? h->n_pids : 1;
  memset(out, 0, sizeof(*out));
  if (h->n_valid == 0 || (kind_mask & 63u) == 0) return TA_OK;
  const int64_t n_slots = (int64_t)h->W * n_pids;
  int64_t R = h->max_name - h->min_name + 1;  // names are 32-bit: no overflow
  // Ids spread wide (R x slots cells would not fit the dense table): ranks through the symbol table.
  const bool table = R > TA_AGG_DENSE_LIMIT / n_slots;
  if (table) {
    TA_TRY(build_names(h));
    if (h->n_names < 0 || h->n_names > TA_AGG_MARK_LIMIT / n_slots)
      return ta_run_aggregate_sorted(h, kind_mask, value_sel, out);
    R = h->n_names;
  }
  const int64_t G = R * n_slots;

  AggArgs a;
  memset(&a, 0, sizeof(a));
  a.n_valid = h->n_valid; a.n_lanes = h->sorted.n_lanes;
  a.kind = h->sorted.kind; a.name = h->sorted.name_id; a.ts = h->sorted.ts_start; a.te = h->sorted.ts_end;
  a.lane_off = h->sorted.lane_off; a.lane_slot = h->d_lane_slot;
  a.op_n = h->attr.op_n_kernels; a.op_first = h->attr.op_first_start; a.op_last = h->attr.op_last_end;
  a.op_gap = h->d_op_gap_ns; a.on_path = h->d_on_path;
  a.kind_mask = kind_mask & 63u; a.value_sel = value_sel; a.min_name = h->min_name; a.R = R;
  a.names = table ? h->d_names : nullptr; a.name_rank = h->d_name_rank;
  a.lane_domain = h->sorted.lane_domain; a.lane_dom_end = h->d_lane_dom_end; a.status = h->d_status;
  const bool host_kinds = (a.kind_mask & 7u) != 0, dev_kinds = (a.kind_mask & 56u) != 0;
  a.want_domain = host_kinds && dev_kinds ? -1 : (dev_kinds ? 1 : 0);
  // Positions per CTA: long chunks share their flush (up to 256 rows) among more records, but a
  // window of a few million records has to fill the chip first - with 16 K positions throughout, 60 k
  // records ran on four CTAs (37 us a call) and a million on sixty-four (51 us).  Where the kinds live in
  // lanes of one domain, about half of the chunks return at once: twice as many as the chip holds
  // CTAs, at most 8 K positions each (two calls on 16.8 M records 290 -> 222 us, 8 M 227 -> 208).
  a.chunk = (h->n_valid / (148 * (a.want_domain < 0 ? 6 : 12)) + AG_STEP) / AG_STEP * AG_STEP;
  if (a.chunk > AG_ITEM) a.chunk = AG_ITEM;
  a.n_items = (unsigned)((h->n_valid + a.chunk - 1) / a.chunk);
  a.spread = a.n_items < 148u * 6u ? a.n_items : 148u * 6u;
  a.per = (a.n_items + a.spread - 1) / a.spread;
  const int64_t blocks = (int64_t)a.spread * a.per;


  AggRowOut ro;
  memset(&ro, 0, sizeof(ro));
  ro.tt = h->d_triples; ro.n_pids = n_pids; ro.R = R; ro.min_name = h->min_name;
  ro.name_of = table ? h->d_name_of : nullptr;
  u64 ng = 0;
  auto run_agg = [&](int rows_here, u64 *total, Tail tail) {
    auto kernel = table ? (tail.m ? k_agg<true, true> : k_agg<true, false>) : (tail.m ? k_agg<false, true> : k_agg<false, false>);
    ta_launch(kernel, (unsigned)blocks, AG_THREADS, 0, st, a, rows_here, ro, total, tail);
  };
  int32_t status[ST_WORDS];
  void *tmpb = nullptr, *outb = nullptr;
  // the three row tables (window, pid, symbol), the four 64-bit columns and the histograms of `rows` rows
  auto carve_rows = [&](int64_t rows) -> size_t {
    const size_t b = Carver::pad(rows * 8) * 4 + Carver::pad(rows * TA_NBINS * 4) + Carver::pad(rows * 4) * 3 + 256;
    outb = ta_dalloc(h, b);
    if (!outb) return 0;
    Carver c(outb);
    ro.g_count = c.take<int64_t>(rows); ro.g_sum = c.take<int64_t>(rows);
    ro.g_min = c.take<int64_t>(rows); ro.g_max = c.take<int64_t>(rows);
    ro.g_hist = c.take<u32>(rows * TA_NBINS);
    const size_t zero = c.off;  // what has to start at zero when records are folded into the rows directly
    ro.g_window = c.take<int32_t>(rows); ro.g_pid = c.take<int32_t>(rows); ro.g_name = c.take<int32_t>(rows);
    return zero;
  };
  // Dense rows: 192 bytes per cell to clear and a scan over the cells.  Marked cells: one more pass
  // over kinds and symbols (6 bytes per record) and a round trip for the number of rows.  The line
  // is drawn where the dense table's bytes reach those of the extra pass plus what some 20 us
  // (pass, scan, round trip) are worth.  512 windows of 65 k records have 33 M cells, one in
  // twenty of them occupied: 1.85 ms per call dense.
  if (G * 232 <= 8 * h->n_valid + (64ll << 20)) {
    const int cells = G <= 4096 ? 64 : 256;
    const int64_t tiles = (G + cells - 1) / cells;
    size_t tb = 4 * Carver::pad((size_t)G * 8) + Carver::pad((size_t)G * TA_NBINS * 4) + Carver::pad((size_t)(tiles + 2) * 8);
    ta_status zs;
    tmpb = ta_zalloc(h, tb, &zs);
    if (!tmpb) return zs;
    Carver ct(tmpb);
    a.d_cnt = ct.take<u64>(G);
    a.d_sum = ct.take<u64>(G);
    a.d_minc = ct.take<u64>(G);
    a.d_maxb = ct.take<u64>(G);
    a.d_hist = ct.take<u32>((size_t)G * TA_NBINS);
    u64 *state = ct.take<u64>(tiles + 2), *total = state + tiles;
    // the rows are compacted without waiting for their count: it is bounded by cells and records
    carve_rows(G < h->n_valid ? G : h->n_valid);
    if (!outb) return TA_ERR_OOM;
    ro.cnt = a.d_cnt; ro.sum = a.d_sum; ro.minc = a.d_minc; ro.maxb = a.d_maxb; ro.hist = a.d_hist;
    TA_TRY(ta_queue_d2h(h, &ng, total, 8));
    TA_TRY(ta_queue_d2h(h, status, h->d_status, sizeof(status)));
    Tail here;
    if (G <= AG_ROWS_HERE) here = ta_tail(h, blocks);
    run_agg(here.m ? (int)G : 0, total, here);
    if (here.m == 0) ta_launch(cells == 64 ? k_agg_rows<64> : k_agg_rows<256>, (unsigned)tiles, AC_THREADS, 0, st, G, ro, state, total, (u32 *)(total + 1),
              h->d_status, ta_tail(h, tiles));
  } else {
    const int64_t words = (G + 31) / 32;
    ScanTemp t;
    tmpb = ta_dalloc(h, 2 * Carver::pad((size_t)words * 4) + scan_temp_bytes(words) + 256);
    if (!tmpb) return TA_ERR_OOM;
    Carver ct(tmpb);
    a.bits = ct.take<u32>(words);
    ct.off += scan_temp_carve(ct.base + ct.off, words, &t);
    TA_CHECK_CUDA(h, cudaMemsetAsync(tmpb, 0, ct.off, st));
    u32 *rank = ct.take<u32>(words);
    if (table) ta_launch(k_agg_mark<true>, a.n_items, AG_THREADS, 0, st, a);
    else ta_launch(k_agg_mark<false>, a.n_items, AG_THREADS, 0, st, a);
    AggBitsIn bi{a.bits};
    AggBitsOut bo{rank};
    TA_TRY((launch_scan<OpAdd, AggBitsIn, AggBitsOut>(h, words, bi, bo, OpAdd(), t)));
    TA_TRY(ta_queue_d2h(h, &ng, t.total, 8));
    TA_TRY(ta_sync_fetch(h));
    if (ng > 0) {
      const size_t zero = carve_rows((int64_t)ng);
      if (!outb) return TA_ERR_OOM;
      TA_CHECK_CUDA(h, cudaMemsetAsync(outb, 0, zero, st));
      a.rank = rank;
      a.d_cnt = (u64 *)ro.g_count; a.d_sum = (u64 *)ro.g_sum; a.d_minc = (u64 *)ro.g_min; a.d_maxb = (u64 *)ro.g_max;
      a.d_hist = ro.g_hist;
      run_agg(0, nullptr, Tail());
      ta_launch(k_agg_marked_rows, (unsigned)((words + 255) / 256), 256, 0, st, a.bits, rank, words, ro, h->d_status);
    }
    TA_TRY(ta_queue_d2h(h, status, h->d_status, sizeof(status)));
  }
  TA_CHECK_CUDA(h, cudaGetLastError());
  TA_TRY(ta_sync_fetch(h));
  ta_dfree(h, tmpb);
  if (status[ST_ERR]) return (ta_status)status[ST_ERR];
  out->n_groups = (int64_t)ng;
  if (ng == 0) return TA_OK;
  out->g_window = ro.g_window; out->g_pid = ro.g_pid; out->g_name = ro.g_name;
  out->g_count = ro.g_count; out->g_sum = ro.g_sum; out->g_min = ro.g_min; out->g_max = ro.g_max;
  out->g_hist = ro.g_hist;
  return TA_OK;
}
