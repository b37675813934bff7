// ta_device_overlap: per (window, process), over ALL device streams, the time the
// device was busy, the time covered by computation (KERNEL) and by communication /
// IO (MEMCPY, COLL), how much of the communication was hidden under computation and
// how much stayed exposed, all as measures of unions of intervals (Sec. 6.1, "Execution
// progress and state"; Fig. "Overlap and exposed work").
//
// The measure of a union of intervals taken in start order is
//   sum_i max(0, e_i - max(s_i, P_i)),   P_i = max of the ends seen before i,
// the same recurrence as the per-stream gap scan, so the step is: bring the device
// records of every process out of their stream lanes into one order by ts_start and run ONE
// chained max-scan with three channels (all records, computation, communication).  The lanes of a process
// are in that order already, so the records of a few lanes are merged (k_ov_merge); those of
// many are sorted by (window, process, ts_start) - keys that carry the record's index in their low
// bits when (process slot, time, index) fit 64 bits, (key, index) pairs otherwise.  The measure of the intersection follows
// from the three unions: |A n B| = |A| + |B| - |A u B|.  Scanned values are tagged with
// the (window, process) slot in their upper bits, as in the gap scan, so a prefix that
// belongs to an earlier process is recognised and ignored.
// Merging reads 18 B and writes 16 B per device record; the sort moves 8 B + 8 B (keys) or 12 B + 12 B
// (pairs) per device record and pass, and the scan then gathers.
#include <climits>
#include <cstring>

#include "scan.cuh"
#include "ta_internal.cuh"

#define OV_THREADS 256
#define OV_ITEMS 8
#define OV_TILE (OV_THREADS * OV_ITEMS)
#define OV_LOW ((1ull << 40) - 1)

struct OvKeyArgs {
  int64_t n, n_valid;
  int n_lanes;
  const int64_t *ts;
  const int32_t *lane_off, *lane_slot, *lane_window, *lane_dom_end, *lane_dev_base;
  const int16_t *lane_domain;
  const int64_t *t0;
  int tsbits, idxbits;
  u64 *keys;  // [device record index] ((slot << tsbits) | (ts_start - t0)) << idxbits | index
  u32 *pos;   // [device record index] sorted position
  const int32_t *status;
};

// one tile of 2048 sorted positions per CTA; tiles that hold host lanes only leave at once
__global__ void __launch_bounds__(OV_THREADS) k_ov_keys(OvKeyArgs a) {
  TA_PDL();
  __shared__ int s_lane0;
  if (ta_failed(a.status)) return;
  const int tid = threadIdx.x;
  const int64_t tile_start = (int64_t)blockIdx.x * OV_TILE;
  if (tile_start >= a.n_valid) return;
  if (tid < 32) {
    const int l = tile_lane_search(a.lane_off, a.n_lanes, tile_start);
    if (tid == 0) s_lane0 = l;
  }
  __syncthreads();
  const int l0 = s_lane0;
  const int64_t tile_end = min(tile_start + OV_TILE, a.n_valid);
  if (span_outside_domain(a.lane_domain, a.lane_dom_end, l0, tile_end, 1)) return;
  const int64_t p0 = tile_start + (int64_t)tid * OV_ITEMS;
  if (p0 >= tile_end) return;
  i64 s[OV_ITEMS];
  load8_i64(a.ts, p0, a.n, s);
  int l = l0;
  int64_t cur_off = a.lane_off[l], next_off = a.lane_off[l + 1];
  bool dev = a.lane_domain[l] == 1;
  int slot = a.lane_slot[l];
  i64 w0 = a.t0[a.lane_window[l]];
  int64_t cbase = a.lane_dev_base[l];
#pragma unroll
  for (int j = 0; j < OV_ITEMS; j++) {
    const int64_t p = p0 + j;
    if (p >= tile_end) break;
    while (p >= next_off) {
      l++;
      cur_off = next_off;
      next_off = a.lane_off[l + 1];
      dev = a.lane_domain[l] == 1;
      slot = a.lane_slot[l];
      w0 = a.t0[a.lane_window[l]];
      cbase = a.lane_dev_base[l];
    }
    if (!dev) continue;
    const int64_t c = cbase + (p - cur_off);
    a.keys[c] = ((((u64)slot << a.tsbits) | (u64)(s[j] - w0)) << a.idxbits) |
                (a.idxbits ? (u64)c : 0ull);
    a.pos[c] = (u32)p;
  }
}

// ---- merging the lanes of a process -------------------------------------------------------
// A process is cut in front of its first record, and every lane of it behind every OM_STEP records (lanes at
// different ones of them, so that lanes in step are cut at different times).  Where a cut falls in the other lanes is
// searched, and the number of cuts in front of it is its place among the cuts of the process: between
// neighbouring cuts there is at most OM_STEP records of each lane, whatever the lanes look like - a stream of
// 300 copies beside one of 2 M kernels, streams that work in turns, lanes of one record.  A CTA merges the
// records between two cuts on chip.
// (Warps that took rows of 32 records of one lane, with cursors they moved through the others: 300 records
// beside 2 M took 11.6 ms, because one warp went through all of them; 100 us so, and 226 by sorting.)
// A record is searched in every other lane, so many lanes are sorted.  A call on even lanes of 4 M records
// together, merged and sorted: 2 lanes 177 and 336 us, 8 264 and 340, 12 328 and 334, 14 368 and 335; of
// 250 k: 2 lanes 55 and 97, 12 88 and 95, 16 98 and 96.
#define OM_LANES 12    // device lanes of a process at most
#define OM_STEP 256
#define OM_CUTS_FEW 8192  // places for cuts that cost a small window no more than its launches
#define OM_THREADS 256
#define OM_GRID (148 * 32)  // CTAs that merge where most places are empty (short lanes)
struct OvMergeArgs {
  int64_t m;
  int n_lanes, n_cuts;  // places for cuts; not all are taken
  int width;            // of a row of `cut`: device lanes of a process at most, and one
  const int64_t *ts, *te;
  const int16_t *kind;
  const int32_t *lane_off, *lane_slot, *lane_window, *lane_dev_base;
  const int16_t *lane_domain;
  const int64_t *t0, *t1;
  u32 *lanes;    // per place: (first lane of the process + 1) << 5 | its lanes, 0 = no cut
  int32_t *cut;  // per place: device records in front of the cut, then where the lanes of the process go on
  ulonglong2 *out;  // per device record in order: (ts_start - t0) << 1 | not a kernel; slot << 40 | clipped end - t0
  const int32_t *status;
};
// First place of the cuts of lane l: a lane of c records has at most c / OM_STEP + 1, the process's own among
// those of its first lane.
__device__ __forceinline__ int ov_cut_base(const OvMergeArgs &a, int l) { return a.lane_dev_base[l] / OM_STEP + l; }
// Cuts in front of record c of a lane whose cuts are `phase` records early.
__device__ __forceinline__ int ov_cuts_before(int c, int phase) { return c + phase > 0 ? (c + phase - 1) / OM_STEP : 0; }

// A warp per cut.  It searches all lanes at the same time: of k lanes, 32 / k threads each, so many probes a round.
__global__ void __launch_bounds__(OM_THREADS) k_ov_cuts(OvMergeArgs a) {
  TA_PDL();
  if (ta_failed(a.status)) return;
  const int lane = threadIdx.x & 31, q = (int)(blockIdx.x * (OM_THREADS / 32) + (threadIdx.x >> 5));
  if (q >= a.n_cuts) return;
  int l = 0;
  for (int hi = a.n_lanes; hi - l > 1;) {
    const int step = (hi - l + 31) >> 5, at = l + lane * step;
    const u32 b = __ballot_sync(0xffffffffu, at < hi && ov_cut_base(a, at) <= q);
    l += (31 - __clz((int)b)) * step;  // (the first lane begins at 0: thread 0 always qualifies)
    hi = min(hi, l + step);
  }
  if (a.lane_domain[l] != 1) return;
  // the process's device lanes [f, f + k): neighbours of l
  const int around = l - (OM_LANES - 1) + lane;  // threads 0 .. 2 * OM_LANES - 2
  const bool same = lane < 2 * OM_LANES - 1 && around >= 0 && around < a.n_lanes && a.lane_slot[around] == a.lane_slot[l] &&
                    a.lane_domain[around] == 1;
  const u32 mask = __ballot_sync(0xffffffffu, same);
  const int f = l - (OM_LANES - 1) + (__ffs((int)mask) - 1), k = __popc(mask);
  if (k > a.width - 1) return;
  const int own = l - f, s = q - ov_cut_base(a, l) + (own > 0);  // cut s of its lane; s = 0: of the process
  const int p = s ? s * OM_STEP - own * OM_STEP / k : 0;
  const int off = a.lane_off[l];
  if (p >= a.lane_off[l + 1] - off) return;
  const i64 x = a.ts[off + p];
  int probes = 32;
  while (probes * k > 32) probes >>= 1;
  const int j = lane / probes, t = lane & (probes - 1);
  const bool in = j < k && t == 0;
  int lo = 0, hi = 0, joff = 0;
  if (j < k) {
    joff = a.lane_off[f + j];
    if (j == own) lo = hi = p;
    else if (s) hi = a.lane_off[f + j + 1] - joff;
  }
  // records of lane f + j in front of the cut; of records that begin together those of the lanes in front come first
  while (__any_sync(0xffffffffu, lo < hi)) {
    const int w = (hi - lo + probes) / (probes + 1), at = lo + (t + 1) * w - 1;
    bool front = false;
    if (lo < hi && at < hi) {
      const i64 v = a.ts[joff + at];
      front = v < x || (v == x && j < own);
    }
    const u32 all = __ballot_sync(0xffffffffu, front);
    const int n = __popc((all >> (j * probes)) & (0xffffffffu >> (32 - probes)));
    if (lo < hi) {
      lo += n * w;
      if (n < probes) hi = min(hi, lo + w - 1);
    }
  }
  const u32 place = __reduce_add_sync(0xffffffffu, in && s ? (u32)ov_cuts_before(lo, j * OM_STEP / k) : 0u) + (s > 0) + (u32)ov_cut_base(a, f);
  const u32 front = __reduce_add_sync(0xffffffffu, in ? (u32)lo : 0u);
  if (place >= (u32)a.n_cuts) return;
  int32_t *row = a.cut + (int64_t)place * a.width;
  if (lane == 0) {
    a.lanes[place] = (u32)(f + 1) << 5 | (u32)k;
    row[0] = a.lane_dev_base[f] + (int32_t)front;
  }
  if (in) row[1 + j] = joff + lo;
}

__global__ void __launch_bounds__(OM_THREADS) k_ov_merge(OvMergeArgs a) {
  TA_PDL();
  extern __shared__ u64 ov_key[];  // ts_start - t0 of the records between the cuts, lane by lane
  __shared__ int s_from[OM_LANES], s_pre[OM_LANES + 1];
  if (ta_failed(a.status)) return;
  const int tid = (int)threadIdx.x;
  for (int i = (int)blockIdx.x; i < a.n_cuts; i += (int)gridDim.x) {
    const u32 lanes = a.lanes[i], next = i + 1 < a.n_cuts ? a.lanes[i + 1] : 0u;
    if (!lanes) continue;
    const int f = (int)(lanes >> 5) - 1, k = (int)(lanes & 31u);
    const int32_t *row = a.cut + (int64_t)i * a.width;
    __syncthreads();  // the round before is done with the shared arrays
    if (tid < 32) {
      int from = 0, n = 0;
      if (tid < k) {
        from = row[1 + tid];
        n = (next == lanes ? row[a.width + 1 + tid] : a.lane_off[f + tid + 1]) - from;
        n = min(max(n, 0), OM_STEP);
      }
      const int upto = (int)warp_scan_inclusive((u64)n, OpAdd());
      if (tid < k) {
        s_from[tid] = from;
        s_pre[tid + 1] = upto;
      }
      if (tid == 0) s_pre[0] = 0;
    }
    const int slot = a.lane_slot[f], w = a.lane_window[f];
    const i64 w0 = a.t0[w], w1 = a.t1[w];
    const int first = row[0];
    __syncthreads();
    const int total = s_pre[k];
    auto lane_of = [&](int e) {
      int j = 0;
      while (e >= s_pre[j + 1]) j++;
      return j;
    };
    for (int e = tid; e < total; e += OM_THREADS) {
      const int j = lane_of(e);
      ov_key[e] = (u64)(a.ts[s_from[j] + e - s_pre[j]] - w0);
    }
    __syncthreads();
    for (int e = tid; e < total; e += OM_THREADS) {
      const int own = lane_of(e), p = s_from[own] + e - s_pre[own];
      const i64 te = a.te[p], end = te < w1 ? te : w1;
      const int kd = a.kind[p];
      const u64 x = ov_key[e];
      int rank = e - s_pre[own];
      for (int j = 0; j < k; j++) {
        if (j == own) continue;
        int lo = s_pre[j], hi = s_pre[j + 1];
        const int at = lo;
        const u64 y = x + (j < own ? 1 : 0);
        while (lo < hi) {
          const int mid = (lo + hi) >> 1;
          if (ov_key[mid] < y) lo = mid + 1;
          else hi = mid;
        }
        rank += lo - at;
      }
      if ((u64)(first + rank) < (u64)a.m)
        a.out[first + rank] = make_ulonglong2(x << 1 | (kd != TA_KIND_KERNEL), (u64)slot << 40 | (u64)(end - w0));
    }
  }
}

struct OvScanArgs {
  int64_t m;          // device records
  const ulonglong2 *merged;
  const u64 *keys;    // sorted
  const u32 *pos;     // sorted position: of element i (pairs), or of device record index c (packed keys)
  int idxbits;        // packed keys: low bits hold the device record index; 0 = pairs
  const int64_t *te;
  const int16_t *kind;
  const int64_t *t0, *t1;
  int tsbits, n_pids;
  u64 *st[3];         // tile descriptors of the three channels
  u32 *counter;
  u64 *acc;           // [slot][4]: records, busy, compute, communication
  int32_t *status;
};

template <bool MERGED>
__global__ void __launch_bounds__(OV_THREADS, 3) k_ov_scan(OvScanArgs a) {
  TA_PDL();
  __shared__ u64 tmp[3][33];
  __shared__ u64 s_excl[3];
  __shared__ int s_tile, s_fail;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) {
    s_tile = (int)atomicAdd(a.counter, 1u);
    s_fail = ta_failed(a.status) ? 1 : 0;
  }
  __syncthreads();
  if (s_fail) return;  // the sort gave up: the keys name no records
  const int tile = s_tile;
  const int64_t i0 = (int64_t)tile * OV_TILE + (int64_t)tid * OV_ITEMS;
  u64 val[OV_ITEMS];   // (slot + 1) << 40 | clipped end - window start
  i64 srel[OV_ITEMS];  // ts_start - window start
  int slot_of[OV_ITEMS];
  int ch_of[OV_ITEMS]; // 1 computation, 2 communication
  u64 run[3] = {0, 0, 0};
  if constexpr (MERGED) {
    ulonglong2 x[OV_ITEMS];
#pragma unroll
    for (int j = 0; j < OV_ITEMS; j++) x[j] = i0 + j < a.m ? a.merged[i0 + j] : make_ulonglong2(0, ~0ull);
#pragma unroll
    for (int j = 0; j < OV_ITEMS; j++) {
      const bool in = i0 + j < a.m;
      slot_of[j] = in ? (int)(x[j].y >> 40) : -1;
      srel[j] = (i64)(x[j].x >> 1);
      ch_of[j] = 1 + (int)(x[j].x & 1u);
      val[j] = in ? x[j].y + (1ull << 40) : 0;
    }
  } else {
    // keys and positions of the thread's eight records, then the gathers, all issued together
    u64 key[OV_ITEMS];
    u32 pp[OV_ITEMS];
    i64 en[OV_ITEMS];
    int16_t kd[OV_ITEMS];
#pragma unroll
    for (int j = 0; j < OV_ITEMS; j++) {
      const bool in = i0 + j < a.m;
      key[j] = in ? a.keys[i0 + j] : ~0ull;
      if (a.idxbits) {
        pp[j] = in ? a.pos[key[j] & ((1ull << a.idxbits) - 1)] : 0u;
        key[j] >>= a.idxbits;
      } else {
        pp[j] = in ? a.pos[i0 + j] : 0u;
      }
    }
#pragma unroll
    for (int j = 0; j < OV_ITEMS; j++) {
      const bool in = i0 + j < a.m;
      en[j] = in ? a.te[pp[j]] : 0;
      kd[j] = in ? a.kind[pp[j]] : (int16_t)-1;
    }
    const u64 tsmask = (1ull << a.tsbits) - 1;
    int wl = -1;
    i64 w0 = 0, w1 = 0;
#pragma unroll
    for (int j = 0; j < OV_ITEMS; j++) {
      val[j] = 0;
      srel[j] = 0;
      slot_of[j] = -1;
      ch_of[j] = kd[j] == TA_KIND_KERNEL ? 1 : 2;
      if (kd[j] < 0) continue;
      const int slot = (int)(key[j] >> a.tsbits);
      const int w = slot / a.n_pids;
      if (w != wl) { w0 = a.t0[w]; w1 = a.t1[w]; wl = w; }
      const i64 ce = (en[j] < w1 ? en[j] : w1) - w0;
      slot_of[j] = slot;
      srel[j] = (i64)(key[j] & tsmask);
      val[j] = ((u64)(slot + 1) << 40) | (u64)ce;
    }
  }
#pragma unroll
  for (int j = 0; j < OV_ITEMS; j++) {
    run[0] = max(run[0], val[j]);
    if (ch_of[j] == 1) run[1] = max(run[1], val[j]);
    else run[2] = max(run[2], val[j]);
  }
  u64 pre[3];
#pragma unroll
  for (int ch = 0; ch < 3; ch++) {
    u64 total;
    pre[ch] = block_scan_exclusive<OpMax>(run[ch], OpMax(), tmp[ch], &total);
    if (warp == ch) {  // three warps look back at the same time, one channel each
      bool failed;
      const u64 ex = tile_lookback<OpMax>(a.st[ch], tile, total, OpMax(), a.status, &failed);
      if (lane == 0) s_excl[ch] = ex;
      if (lane == 0 && failed) s_fail = 1;
    }
  }
  __syncthreads();
  if (s_fail) return;
#pragma unroll
  for (int ch = 0; ch < 3; ch++) pre[ch] = max(pre[ch], s_excl[ch]);

  // coverage added by each record; sums of the thread's first slot stay in registers
  u64 sum[4] = {0, 0, 0, 0};
  int first = -1;
#pragma unroll
  for (int j = 0; j < OV_ITEMS; j++) {
    const int slot = slot_of[j];
    if (slot < 0) continue;
    const i64 ce = (i64)(val[j] & OV_LOW);
    const int ch = ch_of[j];
    u64 add[4] = {1, 0, 0, 0};
#pragma unroll
    for (int c = 0; c < 3; c++) {
      if (c != 0 && c != ch) continue;
      const i64 P = ((pre[c] >> 40) == (u64)(slot + 1)) ? (i64)(pre[c] & OV_LOW) : 0;
      const i64 from = srel[j] > P ? srel[j] : P;
      add[1 + c] = ce > from ? (u64)(ce - from) : 0ull;
      pre[c] = max(pre[c], val[j]);
    }
    if (first < 0) first = slot;
    if (slot == first) {
#pragma unroll
      for (int c = 0; c < 4; c++) sum[c] += add[c];
    } else {  // the thread straddles two processes
#pragma unroll
      for (int c = 0; c < 4; c++)
        if (add[c]) atomicAdd(&a.acc[(size_t)slot * 4 + c], add[c]);
    }
  }
  // fold per warp when the warp sits inside one process (almost always)
  const u32 has = __ballot_sync(0xffffffffu, first >= 0);
  if (!has) return;
  const int wfirst = __shfl_sync(0xffffffffu, first, __ffs(has) - 1);
  if (__all_sync(0xffffffffu, first < 0 || first == wfirst)) {
#pragma unroll
    for (int c = 0; c < 4; c++) {
      const u64 t = warp_reduce(sum[c], OpAdd());
      if (lane == 0 && t) atomicAdd(&a.acc[(size_t)wfirst * 4 + c], t);
    }
  } else if (first >= 0) {
#pragma unroll
    for (int c = 0; c < 4; c++)
      if (sum[c]) atomicAdd(&a.acc[(size_t)first * 4 + c], sum[c]);
  }
}

// compaction of the (window, process) slots that have device records, in slot order
struct OvRowIn {
  const u64 *acc;
  __device__ u64 operator()(int64_t s) const { return acc[(size_t)s * 4] ? 1ull : 0ull; }
};
struct OvRowOut {
  const u64 *acc;
  const TripleTable *tt;
  const int64_t *t0, *t1;
  int n_pids;
  int32_t *d_window, *d_pid;
  int64_t *d_n_events, *d_busy, *d_idle, *d_compute, *d_comm, *d_overlap, *d_exposed;
  __device__ void operator()(int64_t s, u64 row, u64 v) const {
    if (!v) return;
    const int w = (int)(s / n_pids);
    const i64 all = (i64)acc[(size_t)s * 4 + 1], comp = (i64)acc[(size_t)s * 4 + 2],
              comm = (i64)acc[(size_t)s * 4 + 3];
    d_window[row] = w;
    d_pid[row] = tt->pid_value[s % n_pids];
    d_n_events[row] = (i64)acc[(size_t)s * 4];
    d_busy[row] = all;
    d_idle[row] = (t1[w] - t0[w]) - all;
    d_compute[row] = comp;
    d_comm[row] = comm;
    d_overlap[row] = comp + comm - all;
    d_exposed[row] = all - comp;
  }
};

ta_status ta_run_overlap(ta_window *h, ta_overlap_result *out) {
  cudaStream_t st = h->stream;
  memset(out, 0, sizeof(*out));
  const int n_pids = h->n_pids > 0 ? h->n_pids : 1;
  const int64_t n_slots = (int64_t)h->W * n_pids;
  const int64_t m = h->n_device;
  if (m <= 0 || h->n_valid <= 0) return TA_OK;
  int64_t max_span = 1;
  for (int w = 0; w < h->W; w++) max_span = h->h_t1[w] - h->h_t0[w] > max_span ? h->h_t1[w] - h->h_t0[w] : max_span;
  const int tsbits = ta_bit_len((uint64_t)max_span);
  const int slot_bits = ta_bit_len((uint64_t)(n_slots - 1));
  if (tsbits > 40 || tsbits + slot_bits > 63 || n_slots >= (1ll << 22)) return TA_ERR_TOO_LARGE;
  // when (slot, time, index) fit one 64-bit word the index travels inside the key and the
  // passes move keys only (8 B + 8 B per record instead of 12 B + 12 B)
  int idxbits = ta_bit_len((uint64_t)(m - 1));
  if (idxbits < 1) idxbits = 1;
  if (tsbits + slot_bits + idxbits > 64) idxbits = 0;

  // results (kept): at most one row per slot
  size_t kb = 2 * Carver::pad((size_t)n_slots * 4) + 7 * Carver::pad((size_t)n_slots * 8) + 256;
  void *keep = ta_dalloc(h, kb);
  if (!keep) return TA_ERR_OOM;
  Carver ck(keep);
  OvRowOut ro;
  ro.d_window = ck.take<int32_t>(n_slots); ro.d_pid = ck.take<int32_t>(n_slots);
  ro.d_n_events = ck.take<int64_t>(n_slots); ro.d_busy = ck.take<int64_t>(n_slots);
  ro.d_idle = ck.take<int64_t>(n_slots); ro.d_compute = ck.take<int64_t>(n_slots);
  ro.d_comm = ck.take<int64_t>(n_slots); ro.d_overlap = ck.take<int64_t>(n_slots);
  ro.d_exposed = ck.take<int64_t>(n_slots);

  const int64_t tiles = (m + OV_TILE - 1) / OV_TILE;
  // Short lanes have places for cuts that nothing is between, and a table of them that is larger than what
  // sorting takes: 2.9 M records in lanes of 120 196 us merged and 312 sorted, 1 M in lanes of eight 325 and 186.
  const int width = h->max_dev_lanes + 1;
  const int64_t n_cuts = m / OM_STEP + (int64_t)h->sorted.n_lanes + 1;
  const bool merge = h->max_dev_lanes <= OM_LANES && n_cuts <= (m / 32 > OM_CUTS_FEW ? m / 32 : OM_CUTS_FEW) &&
                     n_cuts * (width + 1) * 4 <= 16 * m + (64 << 10);
  size_t tb = merge ? Carver::pad((size_t)m * 16) + Carver::pad((size_t)n_cuts * width * 4)
                    : 3 * Carver::pad((size_t)m * 8) + 3 * Carver::pad((size_t)m * 4) + ta_sort_temp_bytes(m);
  tb += scan_temp_bytes(n_slots) + 512;
  void *tmpb = ta_dalloc(h, tb);
  if (!tmpb) return TA_ERR_OOM;
  Carver ct(tmpb);
  ta_status zs;
  void *zb = ta_zalloc(h, 3 * Carver::pad((size_t)tiles * 8) + Carver::pad(64) + Carver::pad((size_t)n_slots * 32) +
                              (merge ? Carver::pad((size_t)n_cuts * 4) : 0), &zs);
  if (!zb) return zs;
  Carver cz(zb);
  OvScanArgs sa;
  memset(&sa, 0, sizeof(sa));
  for (int c = 0; c < 3; c++) sa.st[c] = cz.take<u64>(tiles);
  sa.counter = (u32 *)cz.take<u64>(8);
  sa.acc = cz.take<u64>(n_slots * 4);
  if (merge) {
    OvMergeArgs ma;
    ma.m = m; ma.n_lanes = h->sorted.n_lanes; ma.n_cuts = (int)n_cuts; ma.width = width;
    ma.ts = h->sorted.ts_start; ma.te = h->sorted.ts_end; ma.kind = h->sorted.kind;
    ma.lane_off = h->sorted.lane_off; ma.lane_slot = h->d_lane_slot; ma.lane_window = h->sorted.lane_window;
    ma.lane_dev_base = h->d_lane_dev_base; ma.lane_domain = h->sorted.lane_domain; ma.t0 = h->d_t0; ma.t1 = h->d_t1;
    ma.out = ct.take<ulonglong2>(m); ma.cut = ct.take<int32_t>(n_cuts * width); ma.lanes = cz.take<u32>(n_cuts);
    ma.status = h->d_status;
    sa.merged = ma.out;
    const size_t smem = (size_t)h->max_dev_lanes * OM_STEP * sizeof(u64);
    static_assert(OM_LANES * OM_STEP * sizeof(u64) <= 40u << 10 && 2 * OM_LANES - 1 <= 32, "within what a kernel has without being asked");
    ta_launch(k_ov_cuts, (unsigned)((n_cuts + OM_THREADS / 32 - 1) / (OM_THREADS / 32)), OM_THREADS, 0, st, ma);
    // (a CTA per place else: 12 even lanes of 4 M records 328 us, by that grid 350)
    const bool empty = h->sorted.n_lanes > m / OM_STEP && n_cuts > OM_GRID;
    ta_launch(k_ov_merge, (unsigned)(empty ? OM_GRID : n_cuts), OM_THREADS, smem, st, ma);
  } else {
    u64 *k_in = ct.take<u64>(m), *k_scr = ct.take<u64>(m), *k_fin = ct.take<u64>(m);
    u32 *v_in = ct.take<u32>(m), *v_scr = ct.take<u32>(m), *v_fin = ct.take<u32>(m);
    void *sort_tmp = ct.base + ct.off; ct.off += ta_sort_temp_bytes(m);
    OvKeyArgs ka;
    ka.n = h->n; ka.n_valid = h->n_valid; ka.n_lanes = h->sorted.n_lanes;
    ka.ts = h->sorted.ts_start;
    ka.lane_off = h->sorted.lane_off; ka.lane_slot = h->d_lane_slot; ka.lane_window = h->sorted.lane_window;
    ka.lane_dom_end = h->d_lane_dom_end; ka.lane_dev_base = h->d_lane_dev_base;
    ka.lane_domain = h->sorted.lane_domain; ka.t0 = h->d_t0; ka.tsbits = tsbits; ka.idxbits = idxbits;
    ka.keys = k_in; ka.pos = v_in; ka.status = h->d_status;
    const int64_t key_tiles = (h->n_valid + OV_TILE - 1) / OV_TILE;
    ta_launch(k_ov_keys, (unsigned)key_tiles, OV_THREADS, 0, st, ka);
    TA_CHECK_CUDA(h, cudaGetLastError());
    if (idxbits) {
      TA_TRY(ta_radix_sort_keys(h, k_in, k_scr, k_fin, m,
                                ta_make_plan(idxbits, idxbits + tsbits + slot_bits), nullptr, sort_tmp,
                                true));  // coverage sums do not depend on the order of equal starts
      sa.pos = v_in;
    } else {
      TA_TRY(ta_radix_sort_pairs(h, k_in, v_in, k_scr, v_scr, k_fin, v_fin, m,
                                 ta_make_plan(0, tsbits + slot_bits), nullptr, sort_tmp));
      sa.pos = v_fin;
    }
    sa.keys = k_fin;
  }
  void *scan_mem = ct.base + ct.off;
  sa.m = m; sa.idxbits = idxbits;
  sa.te = h->sorted.ts_end; sa.kind = h->sorted.kind; sa.t0 = h->d_t0; sa.t1 = h->d_t1;
  sa.tsbits = tsbits; sa.n_pids = n_pids; sa.status = h->d_status;
  ta_launch(merge ? k_ov_scan<true> : k_ov_scan<false>, (unsigned)tiles, OV_THREADS, 0, st, sa);
  TA_CHECK_CUDA(h, cudaGetLastError());

  ro.acc = sa.acc; ro.tt = h->d_triples; ro.t0 = h->d_t0; ro.t1 = h->d_t1; ro.n_pids = n_pids;
  ScanTemp s3;
  TA_TRY(scan_temp_init(h, scan_mem, n_slots, &s3));
  OvRowIn ri{sa.acc};
  u64 rows = 0;
  int32_t words[ST_WORDS];
  TA_TRY(ta_queue_d2h(h, &rows, s3.total, 8));
  TA_TRY(ta_queue_d2h(h, words, h->d_status, sizeof(words)));
  TA_TRY((launch_scan<OpAdd, OvRowIn, OvRowOut>(h, n_slots, ri, ro, OpAdd(), s3, true)));
  TA_TRY(ta_sync_fetch(h));
  ta_dfree(h, tmpb);
  ta_dfree(h, zb);
  if (words[ST_ERR]) return (ta_status)words[ST_ERR];
  out->n_rows = (int64_t)rows;
  out->d_window = ro.d_window; out->d_pid = ro.d_pid; out->d_n_events = ro.d_n_events;
  out->d_busy = ro.d_busy; out->d_idle = ro.d_idle; out->d_compute = ro.d_compute;
  out->d_comm = ro.d_comm; out->d_overlap = ro.d_overlap; out->d_exposed = ro.d_exposed;
  return TA_OK;
}
