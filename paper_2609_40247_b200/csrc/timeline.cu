// ta_sort_timeline: canonical order of the timeline.
//
// Packed keys (the usual case): the key carries the record's index in its low bits and the
// start time at a coarser resolution, so four keys-only radix passes settle the order down
// to (lane, coarse time); k_gather, which brings every 40-byte record into registers once to
// write the eight sorted columns, ranks the members of a run of equal coarse keys by
// (ts_start, -ts_end, input index) on the way, and records the lane boundaries and the
// correlation-id range of every (window, pid) for the join.
// Fallback (a run longer than TA_TIE_RUN_MAX, or keys that do not fit): stable radix sort of
// (key, input index) pairs at full time resolution; runs of equal keys are reordered by
// ts_end descending in place (k_fix_ties), and if even such a run is too long the sort is
// redone with the duration as a least-significant key.
// Dropped records (the tail) are ordered by the full tuple with a chain of stable sorts.
#include <climits>

#include "lanes.cuh"
#include "records.cuh"
#include "scan.cuh"
#include "ta_internal.cuh"

// ---- pair path: equal-key runs -------------------------------------------
__global__ void __launch_bounds__(256) k_fix_ties(const u64 *keys, u32 *perm, int64_t n_valid,
                                                  const ta_event *ev, int32_t *status) {
  TA_PDL();
  if (ta_failed(status)) return;
  int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n_valid || p + 1 >= n_valid) return;
  u64 k = keys[p];
  if (keys[p + 1] != k) return;
  if (p > 0 && keys[p - 1] == k) return;
  int len = 2;
  while (p + len < n_valid && len <= TA_TIE_RUN_MAX && keys[p + len] == k) len++;
  if (len > TA_TIE_RUN_MAX) {
    status[ST_LONG_RUN] = 1;
    return;
  }
  u32 idx[TA_TIE_RUN_MAX];
  i64 end[TA_TIE_RUN_MAX];
  for (int i = 0; i < len; i++) {
    idx[i] = perm[p + i];
    end[i] = reinterpret_cast<const i64 *>(ev)[(int64_t)idx[i] * 5 + 1];
  }
  for (int i = 1; i < len; i++) {  // stable insertion sort, ts_end descending
    u32 xi = idx[i];
    i64 xe = end[i];
    int j = i - 1;
    while (j >= 0 && end[j] < xe) {
      idx[j + 1] = idx[j];
      end[j + 1] = end[j];
      j--;
    }
    idx[j + 1] = xi;
    end[j + 1] = xe;
  }
  for (int i = 0; i < len; i++) perm[p + i] = idx[i];
}

// ---- fallback: duration as a least-significant key ------------------------
__global__ void __launch_bounds__(256) k_duration_key(const ta_event *ev, int64_t n, const u64 *keys,
                                                      u64 dropped_bit, i64 max_dur, u64 *out) {
  TA_PDL();
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  if (keys[i] & dropped_bit) { out[i] = 0; return; }
  const i64 *p = reinterpret_cast<const i64 *>(ev) + i * 5;
  out[i] = (u64)(max_dur - (p[1] - p[0]));  // longer first
}
__global__ void __launch_bounds__(256) k_gather_u64(const u64 *src, const u32 *idx, int64_t n, u64 *dst,
                                                    const int32_t *status) {
  TA_PDL();
  if (ta_failed(status)) return;
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) dst[i] = src[idx[i]];
}

// ---- step 3: full-tuple keys for the dropped tail -------------------------
// stage 0: ~ts_end, 1: ts_start, 2: (pid, domain, stream), 3: window
__global__ void __launch_bounds__(256) k_tail_key(const ta_event *ev, const u32 *idx, int64_t m,
                                                  int stage, const int64_t *off, int W, u64 *out,
                                                  const int32_t *status) {
  TA_PDL();
  if (ta_failed(status)) return;
  int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= m) return;
  Rec r = load_rec(ev, idx[j]);
  u64 k;
  if (stage == 0) k = ~((u64)r.ts_end ^ (1ull << 63));
  else if (stage == 1) k = (u64)r.ts_start ^ (1ull << 63);
  else if (stage == 2) k = triple_code(r.pid, r.kind, r.stream);
  else k = (u64)window_of(off, W, idx[j]);
  out[j] = k;
}

// A tail of up to TL_COUNT records (a few per thousand of an ordinary window) is ranked by counting,
// every record against every other, instead of the chain of stable sorts (27 radix passes, some
// 200 us for a few thousand records; a comparison is six instructions, so 4096 records take 3 us
// and 16 K about what the chain does).
#define TL_COUNT 16384
struct TailKey {
  u64 where;  // window, then (pid, domain, stream)
  u64 lane;
  u64 ts, ne;
  u32 idx;
};
__device__ __forceinline__ TailKey tail_key(const ta_event *ev, u32 idx, const int64_t *off, int W) {
  const Rec r = load_rec(ev, idx);
  TailKey k;
  k.where = (u64)window_of(off, W, idx);
  k.lane = triple_code(r.pid, r.kind, r.stream);
  k.ts = (u64)r.ts_start ^ (1ull << 63);
  k.ne = ~((u64)r.ts_end ^ (1ull << 63));
  k.idx = idx;
  return k;
}
__device__ __forceinline__ bool tail_less(const TailKey &a, const TailKey &b) {
  if (a.where != b.where) return a.where < b.where;
  if (a.lane != b.lane) return a.lane < b.lane;
  if (a.ts != b.ts) return a.ts < b.ts;
  if (a.ne != b.ne) return a.ne < b.ne;
  return a.idx < b.idx;
}
// CTA (bi, bj): counts for the 256 records of block bi those of block bj in front of them
__global__ void __launch_bounds__(256) k_tail_count(const ta_event *ev, const u32 *idx, int m, int blocks,
                                                    const int64_t *off, int W, u32 *rank, const int32_t *status) {
  TA_PDL();
  __shared__ TailKey other[256];
  if (ta_failed(status)) return;
  const int bi = blockIdx.x / blocks, bj = blockIdx.x - bi * blocks;
  const int i = bi * 256 + threadIdx.x, j = bj * 256 + threadIdx.x;
  if (j < m) other[threadIdx.x] = tail_key(ev, idx[j], off, W);
  __syncthreads();
  if (i >= m) return;
  const TailKey mine = tail_key(ev, idx[i], off, W);
  const int cnt = min(256, m - bj * 256);
  u32 before = 0;
  for (int q = 0; q < cnt; q++) before += tail_less(other[q], mine);
  if (before) atomicAdd(&rank[i], before);
}
__global__ void __launch_bounds__(256) k_tail_place(const u32 *idx, const u32 *rank, int m, u32 *out,
                                                    const int32_t *status) {
  TA_PDL();
  if (ta_failed(status)) return;
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i < m) out[rank[i]] = idx[i];
}

// ---- step 4: gather records into sorted columns + lane heads ---------------
// Tiles of a round of the gather's order (a wave of CTAs; 148 to 4736 are within 1 %), and records per
// process from which the order is made: below some 100 MB the records of a process stay in L2 from its
// first lane to its last, and in lane order the writes lie closer together (prefill, 4 processes, the kernel
// without and with the order: 8 M records 174 and 174 us, 16.8 M 425 and 398; experts, 16 processes, 8 M 154
// and 158, 66.8 M 1388 and 1258).
#define GO_ROUND 1184
#define GO_MIN 2500000
struct GatherArgs {
  const u32 *order;   // tiles in the order they are taken, null: as they lie
  const ta_event *ev;
  u32 *perm;          // pairs: input; packed keys: written here for the kept records
  const u64 *keys;
  int64_t n, n_valid;
  int sbits;          // key bits below the lane code (time bits kept [+ index bits])
  int packed, ibits, wshift, wbits;
  int cshift;         // packed keys: bits below the cell, which the passes did not sort
  u32 xmask;          // those of them above the index
  const int64_t *off;
  // corr_id range of the LAUNCH records per (window, pid) slot, for the join
  const TripleTable *tt;
  int tbits, n_pids;
  u64 *slot_code;     // [slot] largest biased id, [n_slots + slot] largest complement of one; 0 = none
  int64_t n_slots;
  i64 *ts_start, *ts_end, *corr;
  int32_t *pid, *name, *seq;
  int16_t *stream, *kind;
  int32_t *lane_start;  // per lane code: first position + 1, 0 = empty
  int32_t *status;
};
template <bool ONE>  // one window: its records begin at 0
__device__ __forceinline__ u32 gather_index(u64 k, const GatherArgs &a) {
  const u32 i = (u32)(k & ((1ull << a.ibits) - 1));
  if (ONE) return i;
  const int w = a.wbits ? (int)((k >> a.wshift) & ((1ull << a.wbits) - 1)) : 0;
  return (u32)a.off[w] + i;
}

// eight CTAs per SM (32 registers): the kernel lives on occupancy, 42 or 51 registers measured slower.
// It is bound by instruction issue as much as by its scattered reads, so the members of a run of
// equal coarse keys are counted by bit operations on one vote (loops over neighbouring keys, with a
// fifth of the records in runs, made every warp diverge: 410 instructions per warp), and no warp
// waits for the others at the end.
#define GT_MINB 8
template <bool PACKED, bool ONE>
__device__ __forceinline__ void gather_tile(const GatherArgs &a) {
  __shared__ int s_slot[8];
  __shared__ u64 s_mx[8], s_mn[8];
  __shared__ u32 s_done;
  const bool failed = ta_failed(a.status);  // the sort gave up: the keys name no records
  if (threadIdx.x == 0) s_done = 0;
  __syncthreads();
  if (failed) return;
  // positions fit 32 bits (n < 2^31): 32-bit indices keep the address arithmetic of the nine
  // column stores and of the neighbour reads short
  const u32 p = (a.order ? a.order[blockIdx.x] : blockIdx.x) * 256u + threadIdx.x;
  const u32 n = (u32)a.n, nv = (u32)a.n_valid;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const u64 k = p < nv ? a.keys[p] : 0;
  u64 kprev = __shfl_up_sync(0xffffffffu, k, 1);
  if (lane == 0 && p > 0 && p < nv) kprev = a.keys[p - 1];
  const u64 knext = PACKED && lane == 31 && p + 1 < nv ? a.keys[p + 1] : 0;
  const bool head = !ONE && p < nv && (p == 0 || (kprev >> a.sbits) != (k >> a.sbits));  // of its lane
  u32 idx = 0;
  if (p < n) idx = PACKED && p < nv ? gather_index<ONE>(k, a) : a.perm[p];
  Rec r;
  if (p < n) r = load_rec(a.ev, idx);
  u32 dst = p;  // where the record goes: p, or its place inside a run of equal cells
  if (PACKED) {
    // packed keys order the records down to a coarse time only: members of a run of equal
    // (lane, coarse time) sit in no particular order (the first radix pass is not stable) and
    // are ranked here by (ts_start, -ts_end, input index): of one window by the time bits the passes left
    // alone, and by the records where those are the same
    constexpr bool FINE = ONE;
    const u64 hk = k >> a.cshift;
    const u32 eq = __ballot_sync(0xffffffffu, p < nv && p > 0 && (kprev >> a.cshift) == hk);
    const bool next = __any_sync(0xffffffffu, lane == 31 && p + 1 < nv && (knext >> a.cshift) == hk);
    if (eq || next) {
      const u32 fine = FINE ? (u32)(k >> a.ibits) & a.xmask : 0u;
      // equal cells in front of the record and behind it, as far as the warp reaches
      int before = __clz((int)~(eq << (31 - lane)));
      int after = lane < 31 ? __ffs((int)~(eq >> (lane + 1))) - 1 : 0;
      // a run that meets the warp's edge goes on in memory
      const bool open = p < nv && (before == lane + 1 || (lane + after == 31 && next));
      int rank = 0;
      const int rounds = __reduce_max_sync(0xffffffffu, open ? 0 : before);
      // every member is compared with the one d places in front of it, and what it
      // learns holds the other way round for that one
      for (int d = 1; d <= rounds; d++) {
        const bool me = !open && before >= d;
        const u32 m = __ballot_sync(0xffffffffu, me);
        bool first;
        if (FINE) {
          const u32 of = __shfl_up_sync(0xffffffffu, fine, d);
          first = of < fine;
          if (__any_sync(0xffffffffu, me && of == fine)) {
            const i64 os = __shfl_up_sync(0xffffffffu, r.ts_start, d);
            const i64 oe = __shfl_up_sync(0xffffffffu, r.ts_end, d);
            const u32 oi = __shfl_up_sync(0xffffffffu, idx, d);
            first = first || (of == fine && (os < r.ts_start || (os == r.ts_start && (oe > r.ts_end || (oe == r.ts_end && oi < idx)))));
          }
        } else {
          const i64 os = __shfl_up_sync(0xffffffffu, r.ts_start, d);
          first = os < r.ts_start;
          if (__any_sync(0xffffffffu, me && os == r.ts_start)) {
            const i64 oe = __shfl_up_sync(0xffffffffu, r.ts_end, d);
            const u32 oi = __shfl_up_sync(0xffffffffu, idx, d);
            first = first || (os == r.ts_start && (oe > r.ts_end || (oe == r.ts_end && oi < idx)));
          }
        }
        const u32 b = __ballot_sync(0xffffffffu, me && first);
        rank += (me && first ? 1 : 0) + (int)(((m & ~b) >> d) >> lane & 1u);
      }
      if (open) {
        if (before == lane + 1)
          while (before <= TA_TIE_RUN_MAX && p > (u32)before && (a.keys[p - before - 1] >> a.cshift) == hk) before++;
        if (lane + after == 31)
          while (after <= TA_TIE_RUN_MAX && p + after + 1 < nv && (a.keys[p + after + 1] >> a.cshift) == hk) after++;
        if (before + after + 1 > TA_TIE_RUN_MAX) {
          a.status[ST_LONG_RUN] = 1;  // the caller starts over with full-resolution keys
          before = after = 0;
        }
        for (int q = -before; q <= after; q++) {
          if (q == 0) continue;
          const u64 ok = a.keys[p + q];
          const u32 of = FINE ? (u32)(ok >> a.ibits) & a.xmask : 0u;
          if (of != fine) {
            rank += of < fine ? 1 : 0;
            continue;
          }
          const u32 oi = gather_index<ONE>(ok, a);
          const i64 *o = reinterpret_cast<const i64 *>(a.ev) + (u64)oi * 5;
          const i64 os = o[0], oe = o[1];
          const bool first = os < r.ts_start || (os == r.ts_start && (oe > r.ts_end || (oe == r.ts_end && oi < idx)));
          rank += first ? 1 : 0;
        }
      }
      if (p < nv) dst = p - before + rank;
    }
  }
  int slot = -1;
  u64 mx = 0, mn_inv = 0;
  if (p < n) {
    if (PACKED && p < nv) a.perm[dst] = idx;
    a.ts_start[dst] = r.ts_start;
    a.ts_end[dst] = r.ts_end;
    a.corr[dst] = r.corr;
    a.pid[dst] = r.pid;
    a.name[dst] = r.name;
    a.seq[dst] = r.seq;
    a.stream[dst] = r.stream;
    a.kind[dst] = r.kind;
    if (p < nv) {
      const u64 code = k >> a.sbits;
      if (head) a.lane_start[code] = (int32_t)p + 1;
      if (r.kind == TA_KIND_LAUNCH) {
        slot = (int)(code >> a.tbits) * a.n_pids + a.tt->pid_rank[code & ((1ull << a.tbits) - 1)];
        mx = (u64)r.corr ^ (1ull << 63);
        mn_inv = ~mx;
      }
    }
  }
  // fold the range per CTA (a CTA almost always sits inside one lane); the last warp to get here
  // adds the CTA's share
  const u32 has = __ballot_sync(0xffffffffu, slot >= 0);
  int wslot = -1;
  if (has) {
    wslot = __shfl_sync(0xffffffffu, slot, __ffs(has) - 1);
    if (__all_sync(0xffffffffu, slot < 0 || slot == wslot)) {
      mx = warp_reduce(mx, OpMax());
      mn_inv = warp_reduce(mn_inv, OpMax());
    } else {  // mixed warp (lane boundary): every thread for itself
      if (slot >= 0) {
        atomicMax(&a.slot_code[slot], mx);
        atomicMax(&a.slot_code[a.n_slots + slot], mn_inv);
      }
      wslot = -1;
    }
  }
  if (lane == 0) {
    s_slot[warp] = wslot; s_mx[warp] = mx; s_mn[warp] = mn_inv;
    __threadfence_block();
    if (atomicAdd(&s_done, 1u) == 7u) {
      __threadfence_block();
      int cur = -1;
      u64 cmx = 0, cmn = 0;
      for (int w = 0; w <= 8; w++) {
        const int sl = w < 8 ? ((volatile int *)s_slot)[w] : -2;
        if (sl == -1) continue;
        if (sl != cur) {
          if (cur >= 0) {
            if (cmx > a.slot_code[cur]) atomicMax(&a.slot_code[cur], cmx);
            if (cmn > a.slot_code[a.n_slots + cur]) atomicMax(&a.slot_code[a.n_slots + cur], cmn);
          }
          cur = sl;
          cmx = 0;
          cmn = 0;
        }
        if (w < 8) { cmx = max(cmx, ((volatile u64 *)s_mx)[w]); cmn = max(cmn, ((volatile u64 *)s_mn)[w]); }
      }
    }
  }
}

// One CTA: the correlation-id range of every slot in plain numbers, and where each range begins
// when all are laid end to end (the join's direct table; meaningless, and not used, when the ranges
// add up to more than such a table may hold).
struct SlotRanges {
  const u64 *code;
  int64_t n_slots;
  i64 *slot_min, *slot_max, *slot_base;
};
__device__ __forceinline__ void slot_ranges(const SlotRanges &a, u64 *tmp) {
  u64 base = 0;
  for (int64_t s0 = 0; s0 < a.n_slots; s0 += blockDim.x) {
    const int64_t s = s0 + threadIdx.x;
    u64 size = 0;
    if (s < a.n_slots) {
      const u64 mx = __ldcg(&a.code[s]), mn_inv = __ldcg(&a.code[a.n_slots + s]);
      const bool any = mx != 0 || mn_inv != 0;
      a.slot_max[s] = any ? (i64)(mx ^ (1ull << 63)) : INT64_MIN;
      a.slot_min[s] = any ? (i64)((~mn_inv) ^ (1ull << 63)) : INT64_MAX;
      if (any) size = min(mx - ~mn_inv, (1ull << 38) - 1) + 1;
    }
    u64 total;
    const u64 ex = block_scan_exclusive<OpAdd>(size, OpAdd(), tmp, &total);
    if (s < a.n_slots) a.slot_base[s] = size ? (i64)(base + ex) : -1;
    base += total;
  }
}
// Of one window whose lane table is there already the ranges are all that is left behind the gather: up to
// the grids that carry a tail its last CTA makes them.
template <bool PACKED, bool ONE, bool TAIL>
__global__ void __launch_bounds__(256, GT_MINB) k_gather(GatherArgs a, SlotRanges ranges, Tail tail) {
  TA_PDL();
  gather_tile<PACKED, ONE>(a);
  __shared__ u64 tmp[TAIL ? 33 : 1];
  if (TAIL) run_tail(tail, [&] {
    if (!ta_failed(a.status)) slot_ranges(ranges, tmp);
  });
}
__global__ void __launch_bounds__(1024) k_slot_ranges(SlotRanges a, const int32_t *status, Tail tail) {
  TA_PDL();
  __shared__ u64 tmp[33];
  if (!ta_failed(status)) slot_ranges(a, tmp);
  run_tail(tail);
}

__global__ void __launch_bounds__(1024) k_lane_table(LaneTable t, const int32_t *status, SlotRanges ranges, Tail tail) {
  TA_PDL();
  __shared__ u64 tmp[33];
  lane_table<false>(t, status, tmp);
  if (!ta_failed(status)) slot_ranges(ranges, tmp);
  run_tail(tail);
}

// The same for many codes (a batch of 512 windows has 65 k of them, and one CTA was bound by the
// scattered writes it has to make alone: 165 us): three scans over as many CTAs as it takes.
struct LaneRows : LaneTable {
  const u64 *n_lanes;  // total of the first scan
  int64_t bound;       // lanes <= bound
};
struct LaneCodeIn {
  LaneRows t;
  __device__ u64 operator()(int64_t c) const { return t.lane_start[c] > 0 ? 1ull : 0ull; }
};
struct LaneCodeOut {
  LaneRows t;
  __device__ void operator()(int64_t c, u64 l, u64 v) const {
    if (!v || (int64_t)l >= t.bound) return;
    const int w = (int)(c >> t.tbits), r = (int)(c & ((1ll << t.tbits) - 1));
    const u64 code = t.tt->sorted_code[r];
    t.lane_window[l] = w;
    t.lane_pid[l] = code_pid(code);
    t.lane_stream[l] = code_stream(code);
    t.lane_domain[l] = code_domain(code);
    t.lane_off[l] = t.lane_start[c] - 1;
    t.lane_slot[l] = w * t.n_pids + t.tt->pid_rank[r];
  }
};
struct LaneDomIn {  // element r = lane L - 1 - r
  LaneRows t;
  __device__ u64 operator()(int64_t r) const {
    const int64_t L = (int64_t)*t.n_lanes, l = L - 1 - r;
    return l >= 0 && l + 1 < L && t.lane_domain[l + 1] != t.lane_domain[l] ? (u64)(L - (l + 1)) : 0ull;
  }
};
struct LaneDomOut {
  LaneRows t;
  __device__ void operator()(int64_t r, u64 excl, u64 v) const {
    const int64_t L = (int64_t)*t.n_lanes, l = L - 1 - r;
    if (r == 0) {
      t.lane_off[L] = (int32_t)t.n_valid;
      t.n_lanes_out[0] = (int32_t)L;
    }
    if (l < 0) return;
    const u64 best = excl > v ? excl : v;
    const int64_t m = best ? L - (int64_t)best : L;
    t.lane_dom_end[l] = m < L ? t.lane_off[m] : (int32_t)t.n_valid;
    t.lane_dom_next[l] = (int32_t)m;
    if (t.lane_domain[l] == 1 && (l == 0 || t.lane_domain[l - 1] != 1)) atomicMax(&t.n_lanes_out[2], (int32_t)(m - l));
  }
};
struct LaneDevIn {
  LaneRows t;
  __device__ u64 operator()(int64_t l) const {
    const int64_t L = (int64_t)*t.n_lanes;
    if (l >= L || t.lane_domain[l] != 1) return 0;
    return (u64)((l + 1 < L ? t.lane_off[l + 1] : (int32_t)t.n_valid) - t.lane_off[l]);
  }
};
struct LaneDevOut {
  LaneRows t;
  __device__ void operator()(int64_t l, u64 excl, u64 v) const {
    if (l < (int64_t)*t.n_lanes) t.lane_dev_base[l] = (int32_t)excl;
    if (l == t.bound - 1) t.n_lanes_out[1] = (int32_t)(excl + v);
  }
};
// codes up to which one CTA makes the table
#define LT_ONE_CTA 4096

// ---- packed keys: index of the record a key stands for -------------------------
struct PackInfo {
  int ibits, wshift, wbits;
  const int64_t *off;
};
__device__ __forceinline__ u32 packed_index(u64 k, const PackInfo &pi) {
  const int w = pi.wbits ? (int)((k >> pi.wshift) & ((1ull << pi.wbits) - 1)) : 0;
  return (u32)(pi.off[w] + (int64_t)(k & ((1ull << pi.ibits) - 1)));
}
__global__ void __launch_bounds__(256) k_unpack_tail(const u64 *keys, int64_t n_valid, int64_t n,
                                                     PackInfo pi, u32 *perm, const int32_t *status) {
  TA_PDL();
  if (ta_failed(status)) return;
  int64_t p = n_valid + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p < n) perm[p] = packed_index(keys[p], pi);
}

static inline int nblk(int64_t n, int t) { return (int)((n + t - 1) / t); }

ta_status ta_run_sort_timeline(ta_window *h) {
  const int64_t n = h->n;
  cudaStream_t st = h->stream;
  const int64_t n_codes = (int64_t)h->W << h->tbits;  // lane code = window << tbits | triple rank
  const int64_t lane_cap = (n_codes < n ? n_codes : n) + 1;  // lanes <= min(codes, records)
  const int64_t n_slots = (int64_t)h->W * (h->n_pids > 0 ? h->n_pids : 1);

  // result buffers (kept until ta_free)
  size_t keep = Carver::pad(n * 4) + 3 * Carver::pad(n * 8) + 3 * Carver::pad(n * 4) +
                2 * Carver::pad(n * 2) + 6 * Carver::pad(lane_cap * 4) + 2 * Carver::pad(lane_cap * 2) +
                Carver::pad((lane_cap + 1) * 4) + Carver::pad((size_t)n_slots * 24) + 512;
  void *kb = ta_dalloc(h, keep);
  if (!kb) return TA_ERR_OOM;
  Carver ck(kb);
  u32 *perm = ck.take<u32>(n);
  i64 *c_ts = ck.take<i64>(n), *c_te = ck.take<i64>(n), *c_corr = ck.take<i64>(n);
  int32_t *c_pid = ck.take<int32_t>(n), *c_name = ck.take<int32_t>(n), *c_seq = ck.take<int32_t>(n);
  int16_t *c_stream = ck.take<int16_t>(n), *c_kind = ck.take<int16_t>(n);
  int32_t *lane_window = ck.take<int32_t>(lane_cap), *lane_pid = ck.take<int32_t>(lane_cap);
  int32_t *lane_slot = ck.take<int32_t>(lane_cap);
  int16_t *lane_stream = ck.take<int16_t>(lane_cap), *lane_domain = ck.take<int16_t>(lane_cap);
  int32_t *lane_off = ck.take<int32_t>(lane_cap + 1);
  int32_t *lane_dom_end = ck.take<int32_t>(lane_cap);
  int32_t *lane_dev_base = ck.take<int32_t>(lane_cap);
  int32_t *lane_dom_next = ck.take<int32_t>(lane_cap);
  int32_t *n_lanes_dev = ck.take<int32_t>(3);  // [0] lanes, [1] device records, [2] device lanes of a process at most
  h->d_slot_min = ck.take<i64>(3 * n_slots);
  h->d_slot_max = h->d_slot_min + n_slots;
  h->d_slot_base = h->d_slot_max + n_slots;

  // temporaries (released at the end of the call)
  const u32 tiles = (u32)((n + 255) / 256);
  const bool by_round = h->packed && h->fast_keys && h->W == 1 && n / (h->n_pids > 0 ? h->n_pids : 1) >= GO_MIN;
  size_t tmp_bytes = 2 * Carver::pad(n * 8) + Carver::pad(n * 4) + Carver::pad(by_round ? (size_t)tiles * 4 : 0) + ta_sort_temp_bytes(n) +
                     2 * scan_temp_bytes(lane_cap) + scan_temp_bytes(n_codes) + 512;
  void *tb = ta_dalloc(h, tmp_bytes);
  if (!tb) return TA_ERR_OOM;
  Carver ct(tb);
  u64 *kscr = ct.take<u64>(n), *skeys = ct.take<u64>(n);
  u32 *vscr = ct.take<u32>(n);
  u32 *order = ct.take<u32>(by_round ? tiles : 0);
  ta_status zs;
  // cleared: first positions per lane code, correlation-id ranges per slot
  const size_t zero_bytes = Carver::pad((size_t)n_codes * 4) + Carver::pad((size_t)n_slots * 16);
  void *zb = ta_zalloc(h, zero_bytes, &zs);
  if (!zb) return zs;
  Carver cz(zb);
  int32_t *lane_start = cz.take<int32_t>(n_codes);
  u64 *slot_code = cz.take<u64>(2 * n_slots);
  void *sort_tmp = ct.base + ct.off;

  // of one window the lanes follow from the counts of the load, beside the first pass
  const bool lanes_early = h->W == 1 && h->packed && h->fast_keys && n > 0;
  const LaneTable lanes{lane_start, n_codes, h->tbits, h->n_pids > 0 ? h->n_pids : 1, h->d_triples, h->n_valid, lane_cap,
                        lane_window, lane_pid, lane_stream, lane_domain, lane_off, lane_slot,
                        lane_dom_end, lane_dom_next, lane_dev_base, n_lanes_dev};
  const SlotRanges ranges{slot_code, n_slots, h->d_slot_min, h->d_slot_max, h->d_slot_base};
  bool tailed = false;  // the gather did the ranges and brings the results
  int32_t n_lanes_host[3] = {0, 0, 0};
  // Packed keys settle the order down to a coarse time; the gather ranks the members of a run
  // of equal coarse keys itself.  A run too long for that is reported at the end, and the
  // second attempt sorts (key, index) pairs at full time resolution.
  for (int attempt = 0; attempt < 2; attempt++) {
    int32_t words[ST_WORDS];
    h->h_slot_min.resize((size_t)n_slots);
    h->h_slot_max.resize((size_t)n_slots);
    auto fetch = [&]() -> ta_status {
      TA_TRY(ta_queue_d2h(h, n_lanes_host, n_lanes_dev, 3 * sizeof(int32_t)));
      TA_TRY(ta_queue_d2h(h, words, h->d_status, sizeof(words)));
      TA_TRY(ta_queue_d2h(h, h->h_slot_min.data(), h->d_slot_min, n_slots * 8));
      return ta_queue_d2h(h, h->h_slot_max.data(), h->d_slot_max, n_slots * 8);
    };
    if (attempt) TA_CHECK_CUDA(h, cudaMemsetAsync(zb, 0, zero_bytes, st));
    if (n > 0) {
      if (h->packed) {
        // keys carry the index: 8-byte elements, fewer bytes per pass
        PackInfo pi{h->ibits, h->ibits + h->tbits + (h->sbits - h->dshift), h->wbits, h->d_off};
        PrekeyInfo pre{h->d_off, h->W, h->d_triples->rank_of_slot, h->tbits, h->wbits,
                       h->sbits - h->dshift, h->dshift, h->ibits, TimelineAside()};
        if (lanes_early) {
          TimelineAside &x = pre.aside;
          x.lanes = lanes;
          x.lanes.n_codes = x.n_triples = h->n_triples;
          x.n_tiles = tiles;
          x.rounds = by_round ? (tiles + GO_ROUND - 1) / GO_ROUND : 0;
          x.order = order;
          x.parts = 1 + x.rounds;
        }
        TA_TRY(ta_radix_sort_keys(h, h->d_keys, kscr, skeys, n, h->plan, h->d_hist, sort_tmp, true,
                                  h->fast_keys ? &pre : nullptr, h->fast_keys && h->W == 1 ? h->d_bin_offset : nullptr));
        if (n > h->n_valid)
          ta_launch(k_unpack_tail, nblk(n - h->n_valid, 256), 256, 0, st, skeys, h->n_valid, n, pi, perm, h->d_status);
      }
      if (!h->packed) {
        // step 1: (key, input index) pairs; the last pass writes (skeys, perm)
        TA_TRY(ta_radix_sort_pairs(h, h->d_keys, nullptr, kscr, vscr, skeys, perm, n, h->plan,
                                   h->d_hist, sort_tmp));
        // step 2: equal-key runs
        if (h->n_valid > 1)
          ta_launch(k_fix_ties, nblk(h->n_valid, 256), 256, 0, st, skeys, perm, h->n_valid, h->events, h->d_status);
        TA_TRY(ta_read_status(h, words));
        if (words[ST_ERR]) return (ta_status)words[ST_ERR];
        if (words[ST_LONG_RUN]) {
          TA_CHECK_CUDA(h, cudaMemsetAsync(h->d_status + ST_LONG_RUN, 0, sizeof(int32_t), st));
          // redo with the duration as a least-significant key: first a stable sort by
          // (max_dur - duration), then the timeline key on top of that order
          void *xb = ta_dalloc(h, Carver::pad(n * 8) + Carver::pad(n * 4));
          if (!xb) return TA_ERR_OOM;
          Carver cx(xb);
          u64 *dkeys = cx.take<u64>(n);
          u32 *dorder = cx.take<u32>(n);
          const u64 dropped_bit = h->has_dropped ? 1ull << (h->sbits + h->tbits + h->wbits) : 0ull;
          ta_launch(k_duration_key, nblk(n, 256), 256, 0, st, h->events, n, h->d_keys, dropped_bit, h->max_dur, dkeys);
          int dbits = 1;
          while (dbits < 63 && (h->max_dur >> dbits) != 0) dbits++;
          SortPlan dplan = ta_make_plan(0, dbits);
          TA_TRY(ta_radix_sort_pairs(h, dkeys, nullptr, kscr, vscr, skeys, dorder, n, dplan, nullptr,
                                     sort_tmp));
          ta_launch(k_gather_u64, nblk(n, 256), 256, 0, st, h->d_keys, dorder, n, dkeys, h->d_status);
          TA_TRY(ta_radix_sort_pairs(h, dkeys, dorder, kscr, vscr, skeys, perm, n, h->plan, nullptr,
                                     sort_tmp));
          TA_TRY(ta_sync_fetch(h));
          ta_dfree(h, xb);
        }
      }
      // step 3: dropped tail, chain of stable sorts over the full tuple (least
      // significant field first); perm[n_valid..n) holds the tail in input order
      const int64_t m = n - h->n_valid;
      if (m > 1 && m <= TL_COUNT) {
        const size_t rb = Carver::pad((size_t)m * 4);
        u32 *rank = (u32 *)ta_zalloc(h, rb, &zs);
        if (!rank) return zs;
        u32 *order = vscr;  // (free once the records are sorted)
        TA_CHECK_CUDA(h, cudaMemcpyAsync(order, perm + h->n_valid, (size_t)m * 4, cudaMemcpyDeviceToDevice, st));
        const int blocks = (int)((m + 255) / 256);
        ta_launch(k_tail_count, blocks * blocks, 256, 0, st, h->events, order, (int)m, blocks, h->d_off, h->W, rank,
                  h->d_status);
        ta_launch(k_tail_place, blocks, 256, 0, st, order, rank, (int)m, perm + h->n_valid, h->d_status);
        ta_dfree_later(h, rank);
      } else if (m > 1) {
        void *xb = ta_dalloc(h, 2 * Carver::pad(m * 8) + Carver::pad(m * 4));
        if (!xb) return TA_ERR_OOM;
        Carver cx(xb);
        u64 *tk = cx.take<u64>(m), *tk2 = cx.take<u64>(m);
        u32 *alt = cx.take<u32>(m);
        u32 *cur = perm + h->n_valid, *nxt = alt;
        // packed keys: the first radix pass does not keep equal keys in input order, and all
        // dropped records of a window share one key, so the tail is put in input order first
        for (int stage = h->packed ? -1 : 0; stage < 4; stage++) {
          if (stage == 3 && h->W == 1) break;
          ta_launch(k_tail_key, nblk(m, 256), 256, 0, st, h->events, cur, m, stage, h->d_off, h->W, tk, h->d_status);
          int bits = stage == 2 ? 49 : stage == 3 ? (h->wbits > 0 ? h->wbits : 1) : stage < 0 ? 32 : 64;
          SortPlan tp = ta_make_plan(0, bits);
          TA_TRY(ta_radix_sort_pairs(h, tk, cur, kscr, vscr, tk2, nxt, m, tp, nullptr, sort_tmp));
          u32 *t = cur; cur = nxt; nxt = t;
        }
        if (cur != perm + h->n_valid)
          TA_CHECK_CUDA(h, cudaMemcpyAsync(perm + h->n_valid, cur, m * sizeof(u32),
                                           cudaMemcpyDeviceToDevice, st));
        TA_TRY(ta_sync_fetch(h));
        ta_dfree(h, xb);
      }
      // step 4
      GatherArgs g;
      g.order = h->packed && by_round ? order : nullptr;
      g.ev = h->events; g.perm = perm; g.keys = skeys; g.n = n; g.n_valid = h->n_valid;
      g.packed = h->packed; g.ibits = h->ibits; g.wbits = h->wbits; g.off = h->d_off;
      g.cshift = h->ibits + h->xbits; g.xmask = (u32)((1ull << h->xbits) - 1);
      g.wshift = h->ibits + h->tbits + (h->sbits - h->dshift);
      g.sbits = h->packed ? h->ibits + (h->sbits - h->dshift) : h->sbits;
      g.ts_start = c_ts; g.ts_end = c_te; g.corr = c_corr; g.pid = c_pid; g.name = c_name; g.seq = c_seq;
      g.stream = c_stream; g.kind = c_kind; g.lane_start = lane_start;
      g.tt = h->d_triples; g.tbits = h->tbits; g.n_pids = h->n_pids > 0 ? h->n_pids : 1;
      g.slot_code = slot_code; g.n_slots = n_slots; g.status = h->d_status;
      TA_TRY(fetch());
      const unsigned grid = (unsigned)nblk(n, 256);
      Tail tail;
      if (lanes_early && h->packed && grid <= 1024) tail = ta_tail(h, grid);
      tailed = tail.m > 0;
      auto gather = !h->packed ? k_gather<false, false, false>
                    : !lanes_early ? k_gather<true, false, false>
                    : tailed ? k_gather<true, true, true> : k_gather<true, true, false>;
      ta_launch(gather, grid, 256, 0, st, g, ranges, tail);
    } else {
      TA_TRY(fetch());
    }
    if (tailed) {
    } else if (lanes_early) {
      ta_launch(k_slot_ranges, 1, n_slots <= 256 ? 256 : 1024, 0, st, ranges, h->d_status, ta_tail(h, 1));
    } else if (n_codes <= LT_ONE_CTA || n == 0) {
      // (few codes: fewer warps to wait for at each of its barriers)
      ta_launch(k_lane_table, 1, n_codes <= 256 && n_slots <= 256 ? 256 : 1024, 0, st, lanes, h->d_status, ranges, ta_tail(h, 1));
    } else {
      LaneRows t{lanes, nullptr, lane_cap - 1};
      Carver cs(sort_tmp);  // the sort is done with its temporaries by the time the scans run
      ScanTemp s1, s2, s3;
      cs.off += scan_temp_carve(cs.base + cs.off, n_codes, &s1);
      cs.off += scan_temp_carve(cs.base + cs.off, t.bound, &s2);
      cs.off += scan_temp_carve(cs.base + cs.off, t.bound, &s3);
      TA_CHECK_CUDA(h, cudaMemsetAsync(sort_tmp, 0, cs.off, st));
      t.n_lanes = s1.total;
      TA_CHECK_CUDA(h, cudaMemsetAsync(n_lanes_dev, 0, 12, st));
      TA_TRY((launch_scan<OpAdd, LaneCodeIn, LaneCodeOut>(h, n_codes, LaneCodeIn{t}, LaneCodeOut{t}, OpAdd(), s1)));
      TA_TRY((launch_scan<OpMax, LaneDomIn, LaneDomOut>(h, t.bound, LaneDomIn{t}, LaneDomOut{t}, OpMax(), s2)));
      TA_TRY((launch_scan<OpAdd, LaneDevIn, LaneDevOut>(h, t.bound, LaneDevIn{t}, LaneDevOut{t}, OpAdd(), s3)));
      ta_launch(k_slot_ranges, 1, 1024, 0, st, ranges, h->d_status, ta_tail(h, 1));
    }
    TA_CHECK_CUDA(h, cudaGetLastError());
    TA_TRY(ta_sync_fetch(h));
    if (words[ST_ERR]) return (ta_status)words[ST_ERR];
    if (!words[ST_LONG_RUN]) break;
    if (!h->packed) return TA_ERR_OVERFLOW;  // cannot happen: the pair path resolves long runs itself
    TA_CHECK_CUDA(h, cudaMemsetAsync(h->d_status + ST_LONG_RUN, 0, sizeof(int32_t), st));
    TA_TRY(ta_launch_load(h, false));
  }
  ta_dfree(h, tb);
  ta_dfree(h, zb);
  ta_dfree(h, h->d_keys);
  h->d_keys = nullptr;

  const int32_t n_lanes = n_lanes_host[0];
  h->n_device = n_lanes_host[1];
  h->max_dev_lanes = n_lanes_host[2];
  ta_sort_result &r = h->sorted;
  r.n = n; r.n_valid = h->n_valid; r.n_lanes = n_lanes; r.n_windows = h->W;
  r.perm = (const int32_t *)perm;
  r.ts_start = (const int64_t *)c_ts; r.ts_end = (const int64_t *)c_te;
  r.corr_id = (const int64_t *)c_corr;
  r.pid = c_pid; r.name_id = c_name; r.seq = c_seq; r.stream = c_stream; r.kind = c_kind;
  r.lane_window = lane_window; r.lane_pid = lane_pid; r.lane_stream = lane_stream;
  r.lane_domain = lane_domain; r.lane_off = lane_off;
  h->d_lane_slot = lane_slot;
  h->d_lane_dom_end = lane_dom_end;
  h->d_lane_dev_base = lane_dev_base;
  h->d_lane_dom_next = lane_dom_next;
  return TA_OK;
}
