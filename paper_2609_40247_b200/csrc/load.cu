// ta_load_window kernels: validity (a record belongs to the window in which it
// starts, Sec. 5.2), discovery and dense ranking of the (pid, domain, stream) triples
// that name a lane, and the 64-bit sort key together with the digit histograms
// of every radix pass.
//   k_plan          one CTA samples the records and decides how many time bits the packed
//                   sort key keeps (before anything is known about the lanes);
//   k_discover_staged  one pass over the 40-byte records, tiles of them brought to shared memory
//                   by bulk asynchronous copies (two tiles in flight per CTA): defect counters,
//                   the triple and communicator sets, value ranges, and one 64-bit word per
//                   record (dropped flag | triple slot | ts_start - t0); it also takes the
//                   digit histograms of the radix passes over the time bits and counts the
//                   records of every triple, so that the first radix pass can build the keys
//                   itself and no separate key pass is needed;
//   k_top_hist_*    digit histograms of the passes over the (window, lane) bits of several windows,
//                   from the records counted per window and triple, or from the words when there
//                   are too many windows for that (of one window: k_rank);
//   k_rank_*        one CTA each: sort and rank the few triples / communicator ids;
//   k_load_pre      turns those words into keys in place - [dropped][window][triple
//                   rank][(ts_start - t0) >> dshift]{[index in window]} - and takes the
//                   histograms; k_load does the same from the records when the sort
//                   falls back to full-resolution (key, index) pairs.
// The records are streamed once here and gathered once by the sort.
#include "ta_internal.cuh"
#include "records.cuh"

#define TRIPLE_EMPTY (~0ull)  // in the per-CTA caches and the sampling table

__device__ __forceinline__ i64 warp_max_i64(i64 v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = max(v, (i64)__shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// The discovery pass leaves one 64-bit word per record with all the sort needs - bit 63 for a dropped
// record, else the triple's slot in the hash table (13 bits) and ts_start - t0 (40 bits) - so that
// the 40-byte records are read once.
#define PRE_DROPPED (1ull << 63)
#define PRE_TS_BITS 40

// ---- planning: how many time bits the packed key keeps -----------------------------------
// The sort settles the order down to cells of 2^d ns; records of one lane that share a cell
// are ranked afterwards, which stays cheap while cells rarely hold more than one record.  One
// CTA samples up to 4096 records spread over the input, estimates the size of the largest
// lane and keeps the smallest number of whole radix passes over time bits for which the
// expected occupancy of a cell (largest lane x cell / span) stays at or below 1/4.  Any answer
// is correct (long runs fall back to full resolution); the estimate only steers the cost.
// misc[6] <- time bits kept, misc[7] <- estimated size of the largest lane.
#define PL_THREADS 1024
#define PL_PER_THREAD 4
#define PL_SLOTS 2048
// Before that it writes down what the other kernels of the call expect in memory: the bounds of the
// windows when they came as arguments (a copy costs more than the kernel), and where the value
// ranges start.
struct PlanWindows {
  int64_t v[3 * TA_PLAN_WINDOWS + 1];  // off, t0, t1 as they lie in memory
  int n;                               // 0: the bounds were copied
};
// What the handle has to find cleared is cleared by the other CTAs meanwhile (a fill in front of the
// plan was one operation more in a row, and the plan waited for it to end).
struct PlanClear {
  uint4 *p;
  int64_t n;  // of 16 bytes each
};
__global__ void __launch_bounds__(PL_THREADS) k_plan(const ta_event *ev, int64_t n, int64_t *off,
                                                     const int64_t *t0, const int64_t *t1, int W,
                                                     int sbits, int64_t max_span, int64_t max_win,
                                                     int64_t *misc, PlanWindows pw, PlanClear clear) {
  TA_PDL();
  if (blockIdx.x > 0) {
    const int64_t step = (int64_t)(gridDim.x - 1) * PL_THREADS;
#pragma unroll 4
    for (int64_t i = (int64_t)(blockIdx.x - 1) * PL_THREADS + threadIdx.x; i < clear.n; i += step)
      clear.p[i] = make_uint4(0, 0, 0, 0);
    return;
  }
  if (threadIdx.x < pw.n) off[threadIdx.x] = pw.v[threadIdx.x];
  if (threadIdx.x < 16) {  // [0] / [1] smallest / largest name, [3] / [4] sequence number, the rest 0
    const int k = threadIdx.x;
    misc[k] = k == 0 || k == 3 ? INT64_MAX : k == 1 || k == 4 ? INT64_MIN : 0;
  }
  __shared__ u64 code[PL_SLOTS];
  __shared__ u32 cnt[PL_SLOTS];
  __shared__ u32 s_max;
  for (int i = threadIdx.x; i < PL_SLOTS; i += PL_THREADS) { code[i] = TRIPLE_EMPTY; cnt[i] = 0; }
  if (threadIdx.x == 0) s_max = 0;
  __syncthreads();
  const int64_t S = n < (int64_t)PL_THREADS * PL_PER_THREAD ? n : (int64_t)PL_THREADS * PL_PER_THREAD;
  // the thread's samples together, then the table (one sample after the other was a chain of four
  // cold reads, window searches in between)
  u64 mine[PL_PER_THREAD];
#pragma unroll
  for (int j = 0; j < PL_PER_THREAD; j++) {
    const int64_t k = (int64_t)j * PL_THREADS + threadIdx.x;
    mine[j] = TRIPLE_EMPTY;
    if (k >= S) continue;
    const int64_t i = k * (n / S);  // S <= n: evenly spread, in range
    const Rec r = load_rec(ev, i);
    const int w = window_of(off, W, i);
    // lanes are per window: the window is part of the sampled code
    if (!defect_of(r, t0[w], t1[w]))
      mine[j] = triple_code(r.pid, r.kind, r.stream) ^ ((u64)w * 0x9E3779B97F4A7C15ull);
  }
  for (int j = 0; j < PL_PER_THREAD; j++) {
    const u64 c = mine[j];
    if (c == TRIPLE_EMPTY) continue;
    u32 slot = hash_code(c) & (PL_SLOTS - 1);
    for (int probe = 0; probe < 16; probe++) {  // a table that fills up only loses samples
      const u64 cur = code[slot];
      if (cur == c) { atomicAdd(&cnt[slot], 1u); break; }
      if (cur == TRIPLE_EMPTY) {
        const u64 old = atomicCAS(&code[slot], TRIPLE_EMPTY, c);
        if (old == TRIPLE_EMPTY || old == c) { atomicAdd(&cnt[slot], 1u); break; }
      }
      slot = (slot + 1) & (PL_SLOTS - 1);
    }
  }
  __syncthreads();
  u32 m = 0;
  for (int i = threadIdx.x; i < PL_SLOTS; i += PL_THREADS) m = max(m, cnt[i]);
  m = (u32)warp_reduce((u64)m, OpMax());
  if ((threadIdx.x & 31) == 0) atomicMax(&s_max, m);
  __syncthreads();
  if (threadIdx.x == 0) {
    // few samples in the fullest lane say little: take at least 32 of them for granted
    const double per_sample = S > 0 ? (double)n / (double)S : 1.0;
    double est = (double)(s_max < 32u ? 32u : s_max) * per_sample;
    if (est > (double)max_win) est = (double)max_win;
    if (est < 1.0) est = 1.0;
    int keep = sbits;
    for (int passes = 1; passes * 8 < sbits; passes++) {
      const int d = sbits - passes * 8;
      if (est * (double)(1ull << d) / (double)max_span <= 0.25) { keep = passes * 8; break; }
    }
    misc[6] = keep;
    misc[7] = (int64_t)est;
  }
}

// ---- discovery with staged tiles -----------------------------------------------------------
#define DS_THREADS 256
#define DS_RPT 2                          // records per thread and tile
#define DS_TILE (DS_THREADS * DS_RPT)     // 512 records = 20480 bytes
#define DS_TILE_BYTES (DS_TILE * 40)
#define DS_CACHE_BITS 9
#define DS_CACHE (1 << DS_CACHE_BITS)
#define DS_PROBES 4
#define DS_WAIT_POLLS (1 << 18)  // a tile arrives within microseconds; each poll may itself wait a little

__device__ __forceinline__ u32 smem_addr(const void *p) { return (u32)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(u64 *bar, u32 count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count));
}
// one tile of whole records from this GPU's memory into shared memory: a 1-D bulk copy (no
// tensor map; the copy goes to this CTA alone) that reports its bytes to the barrier
__device__ __forceinline__ void bulk_load(void *dst, const void *src, u32 bytes, u64 *bar) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
               : "memory");
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_addr(dst)),
      "l"(src), "r"(bytes), "r"(smem_addr(bar))
      : "memory");
}
// bounded wait for the phase with the given parity; false = gave up
__device__ __forceinline__ bool mbar_wait(u64 *bar, u32 parity) {
  for (int polls = 0; polls < DS_WAIT_POLLS; polls++) {
    u32 done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

struct DiscoverArgs {
  const ta_event *ev;
  int64_t n;
  const int64_t *off, *t0, *t1;
  int W;
  TripleTable *tt;
  CommTable *cm;
  ta_load_summary *sum;
  int64_t *misc;
  int32_t *status;
  u64 *prekey;
  u32 *hist;      // [pass][256]: digit histograms of the passes over time bits
  u32 *slot_cnt;  // [window][TA_TRIPLE_SLOTS] kept records per triple slot, or null (too many windows)
  int sbits;
};

struct __align__(128) DiscoverSmem {
  unsigned char buf[2][DS_TILE_BYTES + 16];  // records that begin at an odd eight bytes: copied from the eight before on
  u64 bar[2];
  u64 cache[DS_CACHE];  // (triple code << 13) | slot of the triples this CTA has met; an entry, once taken, stays
  u32 count[DS_CACHE];  // records of that triple, in the window w_cnt, not yet added to the global counters
  u64 ccache[64];
  u32 hist[5][256];
  // ranges and counts of the CTA's warps
  int32_t mn, mx, qmn, qmx;
  u32 n_coll, n_launch;
  i64 md;
  int fail;
};

__global__ void __launch_bounds__(DS_THREADS, 4) k_discover_staged(DiscoverArgs a) {
  TA_PDL();
  extern __shared__ __align__(128) unsigned char ds_raw[];
  DiscoverSmem &s = *reinterpret_cast<DiscoverSmem *>(ds_raw);
  const int tid = threadIdx.x, lane = tid & 31;
  for (int i = tid; i < DS_CACHE; i += DS_THREADS) { s.cache[i] = TRIPLE_EMPTY; s.count[i] = 0; }
  if (tid < 64) s.ccache[tid] = TRIPLE_EMPTY;
  for (int i = tid; i < 5 * 256; i += DS_THREADS) (&s.hist[0][0])[i] = 0;
  if (tid == 0) {
    mbar_init(&s.bar[0], 1);
    mbar_init(&s.bar[1], 1);
    s.fail = 0;
    s.mn = s.qmn = INT32_MAX;
    s.mx = s.qmx = INT32_MIN;
    s.n_coll = s.n_launch = 0;
    s.md = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  // passes over the time bits kept (decided by k_plan): digit p = (ts_rel >> dshift >> sh[p]) & mk[p]
  const int keep = (int)a.misc[6];
  const int dshift = a.sbits - keep;
  const SortPlan tp = ta_plan_bits(0, keep);
  const int n_tp = tp.n_pass <= 5 ? tp.n_pass : 0;  // more than five time passes: no histograms here
  int sh[5];
  u32 mk[5];
#pragma unroll
  for (int p = 0; p < 5; p++) {
    sh[p] = tp.shift[p];
    mk[p] = (1u << tp.bits[p]) - 1u;
  }
  const int64_t n_tiles = (a.n + DS_TILE - 1) / DS_TILE;
  // name and sequence ranges in 32 bits (the fields are int32), folded to 64 at the end
  int32_t mn = INT32_MAX, mx = INT32_MIN, qmn = INT32_MAX, qmx = INT32_MIN;
  i64 md = 0;
  u32 n_coll = 0, n_launch = 0;
  WindowWalker ww(a.off, a.W), wt(a.off, a.W);
  int cw = -1;  // window whose bounds are in registers
  int w_cnt = 0;  // window the CTA's counts are of: that of the tile's first record
  auto flush_counts = [&]() {
    for (int i = tid; i < DS_CACHE; i += DS_THREADS)
      if (s.count[i]) {
        atomicAdd(&a.slot_cnt[w_cnt * TA_TRIPLE_SLOTS + (int)(s.cache[i] & (TA_TRIPLE_SLOTS - 1))], s.count[i]);
        s.count[i] = 0;
      }
  };
  i64 ct0 = 0, ct1 = 0;
  int64_t tile = blockIdx.x;
  auto tile_bytes = [&](int64_t t) -> u32 {
    const int64_t cntr = min((int64_t)DS_TILE, a.n - t * DS_TILE);
    return (u32)(cntr * 40);
  };
  // A bulk copy starts and ends on 16 bytes.  Records at an odd eight bytes (mis = 8) are copied with
  // the eight bytes in front of them and behind them; the first and the last tile, where those are not
  // the caller's, with plain loads, as is a tile whose size is no multiple of 16 bytes (the last).
  const u32 mis = (u32)((uintptr_t)a.ev & 15u);
  auto bulk_tile = [&](int64_t t) -> bool {
    return mis ? t > 0 && t + 1 < n_tiles : (tile_bytes(t) & 15u) == 0;
  };
  auto load_tile = [&](int64_t t, int b) {
    bulk_load(s.buf[b], reinterpret_cast<const unsigned char *>(a.ev) + t * DS_TILE_BYTES - mis,
              tile_bytes(t) + 2 * mis, &s.bar[b]);
  };
  if (tid == 0 && tile < n_tiles && bulk_tile(tile)) load_tile(tile, 0);
  u32 phase[2] = {0, 0};  // copies waited for so far, per buffer
  for (int it = 0; tile < n_tiles; tile += gridDim.x, it++) {
    const int cur = it & 1;
    const int64_t nxt = tile + gridDim.x;
    if (tid == 0 && nxt < n_tiles && bulk_tile(nxt)) load_tile(nxt, cur ^ 1);
    const u32 bytes = tile_bytes(tile);
    const int count = (int)(bytes / 40);
    if (bulk_tile(tile)) {
      // one thread polls the barrier; the others sleep at the block barrier below instead of
      // spending issue slots on polls
      if (tid == 0 && !mbar_wait(&s.bar[cur], cur ? phase[1] & 1u : phase[0] & 1u)) s.fail = 1;
      if (cur) phase[1]++; else phase[0]++;
    } else {
      const u64 *src = reinterpret_cast<const u64 *>(a.ev) + tile * (DS_TILE * 5);
      u64 *dst = reinterpret_cast<u64 *>(s.buf[cur] + mis);
      for (int k = tid; k < count * 5; k += DS_THREADS) dst[k] = __ldg(src + k);
      // a later bulk copy writes the same buffer
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncthreads();
    if (s.fail) {  // the copy never arrived: report, wait for the one behind it (bounded as well) and leave
      if (tid == 0) {
        ta_set_err(a.status, TA_ERR_TIMEOUT);
        if (nxt < n_tiles && bulk_tile(nxt)) mbar_wait(&s.bar[cur ^ 1], cur ? phase[0] & 1u : phase[1] & 1u);
      }
      return;
    }
    if (a.W > 1) {  // the same in every thread; the barrier above is behind the counts of the tile before
      const int w = wt.at(tile * DS_TILE);
      if (w != w_cnt) {
        if (a.slot_cnt) flush_counts();
        w_cnt = w;
        __syncthreads();
      }
    }
#pragma unroll
    for (int j = 0; j < DS_RPT; j++) {
      const int rl = j * DS_THREADS + tid;
      const bool in = rl < count;
      const int64_t i = tile * DS_TILE + rl;
      int slot_mine = -1;  // triple slot of a kept record
      int entry = -1;      // its entry in the CTA's table
      u64 trel = 0;
      if (in) {
        const u64 *q = reinterpret_cast<const u64 *>(s.buf[cur] + mis + (size_t)rl * 40);
        Rec r;
        r.ts_start = (i64)q[0];
        r.ts_end = (i64)q[1];
        r.corr = (i64)q[2];
        const u64 x = q[3], y = q[4];
        r.pid = (int32_t)(u32)x;
        r.name = (int32_t)(u32)(x >> 32);
        r.seq = (int32_t)(u32)y;
        r.stream = (int16_t)(uint16_t)(y >> 32);
        r.kind = (int16_t)(uint16_t)(y >> 48);
        const int w = ww.at(i);
        if (w != cw) { cw = w; ct0 = a.t0[w]; ct1 = a.t1[w]; }
        const int def = defect_of(r, ct0, ct1);
        if (def) {
          int64_t *f = def == 1 ? &a.sum[w].n_bad_kind
                                : def == 2 ? &a.sum[w].n_bad_interval : &a.sum[w].n_out_of_window;
          atomicAdd((u64 *)f, 1ull);
          a.prekey[i] = PRE_DROPPED;
        } else {
          mn = min(mn, r.name);
          mx = max(mx, r.name);
          md = max(md, r.ts_end - r.ts_start);
          n_launch += r.kind == TA_KIND_LAUNCH;
          if (r.kind == TA_KIND_COLL) {  // communicator set and sequence range
            n_coll++;
            qmn = min(qmn, r.seq);
            qmx = max(qmx, r.seq);
            const u64 cc = (u64)r.corr ^ (1ull << 63);
            const u32 ch = (((u32)cc ^ (u32)(cc >> 32)) * 0x9E3779B1u) >> 26;
            if (cc == TRIPLE_EMPTY) ta_set_err(a.status, TA_ERR_INVALID_ARG);  // reserved id
            else if (s.ccache[ch] != cc) {
              u32 slot = hash_code(cc) & (TA_COMM_SLOTS - 1);
              bool ok = false;
              for (int probe = 0; probe < TA_COMM_SLOTS; probe++) {
                const u64 c2 = ld_relaxed(&a.cm->slots[slot]);
                if (c2 == ~cc) { ok = true; break; }
                if (c2 == 0) {
                  const u64 old = atomicCAS(&a.cm->slots[slot], 0ull, ~cc);
                  if (old == 0 || old == ~cc) { ok = true; break; }
                }
                slot = (slot + 1) & (TA_COMM_SLOTS - 1);
              }
              if (!ok) ta_set_err(a.status, TA_ERR_TOO_LARGE);
              s.ccache[ch] = cc;
            }
          }
          const u64 code = triple_code(r.pid, r.kind, r.stream);
          trel = (u64)(r.ts_start - ct0);
          // the CTA's own table first: an entry or an empty one within a few steps
          int at = (int)(((u32)code * 0x9E3779B1u + (u32)(code >> 32) * 0x85EBCA77u) >> (32 - DS_CACHE_BITS));
          u64 hit = s.cache[at];
          for (int probe = 1; probe < DS_PROBES && (hit >> 13) != code && hit != TRIPLE_EMPTY; probe++) {
            at = (at + 1) & (DS_CACHE - 1);
            hit = s.cache[at];
          }
          if ((hit >> 13) == code) {
            slot_mine = (int)(hit & (TA_TRIPLE_SLOTS - 1));
            entry = at;
          } else {
            u32 slot = hash_code(code) & (TA_TRIPLE_SLOTS - 1);
            bool done = false;
            for (int probe = 0; probe < TA_TRIPLE_SLOTS; probe++) {
              const u64 c2 = ld_relaxed(&a.tt->slots[slot]);
              if (c2 == code + 1) { done = true; break; }
              if (c2 == 0) {
                const u64 old = atomicCAS(&a.tt->slots[slot], 0ull, code + 1);
                if (old == 0 || old == code + 1) { done = true; break; }
              }
              slot = (slot + 1) & (TA_TRIPLE_SLOTS - 1);
            }
            if (!done) ta_set_err(a.status, TA_ERR_TOO_LARGE);
            slot_mine = (int)slot;
            const u64 mine = (code << 13) | slot;
            if (hit == TRIPLE_EMPTY) {
              const u64 old = atomicCAS(&s.cache[at], TRIPLE_EMPTY, mine);
              if (old == TRIPLE_EMPTY || old == mine) entry = at;
            }
          }
          if (w != w_cnt) entry = -1;  // counts of another window than the tile's first
          a.prekey[i] = ((u64)slot_mine << PRE_TS_BITS) | trel;
        }
      }
      // digit histograms of the time passes (dropped records count in digit 0 later, from the
      // defect counters).  The upper digits are the same for a whole warp most of the time
      // (neighbouring records are close in time): one vote, one add.
      const u32 kept = __ballot_sync(0xffffffffu, slot_mine >= 0);
      if (kept) {
        const int leader = __ffs(kept) - 1;
        const u64 tk = trel >> dshift;  // (digits are at most 8 bits wide: the first four begin below bit 32)
#pragma unroll
        for (int p = 0; p < 5; p++) {
          if (p >= n_tp) break;
          const u32 d = (p < 4 ? __funnelshift_r((u32)tk, (u32)(tk >> 32), sh[p]) : (u32)(tk >> sh[p])) & mk[p];
          if (p >= 1) {
            const u32 d0 = __shfl_sync(0xffffffffu, d, leader);
            if (__all_sync(0xffffffffu, slot_mine < 0 || d == d0)) {
              if (lane == leader) atomicAdd(&s.hist[p][d0], (u32)__popc(kept));
              continue;
            }
          }
          if (slot_mine >= 0) atomicAdd(&s.hist[p][d], 1u);
        }
        // records per triple: in the CTA's table (neighbouring records mostly share their triple:
        // one add for all of them; input in no order at all takes an add each, on chip - adding
        // to the global counters per distinct triple of a warp took 70 us of 1.2 M shuffled records)
        if (a.slot_cnt) {
          const int e0 = __shfl_sync(0xffffffffu, entry, leader);
          if (__all_sync(0xffffffffu, slot_mine < 0 || entry == e0) && e0 >= 0) {
            if (lane == leader) atomicAdd(&s.count[e0], (u32)__popc(kept));
          } else if (entry >= 0) {
            atomicAdd(&s.count[entry], 1u);
          } else if (slot_mine >= 0) {
            atomicAdd(&a.slot_cnt[cw * TA_TRIPLE_SLOTS + slot_mine], 1u);  // (cw: the record's window)
          }
        }
      }
    }
    __syncthreads();  // every thread is done with buf[cur] before the next copy into it is issued
  }
  if (a.slot_cnt) flush_counts();
  for (int i = tid; i < n_tp * 256; i += DS_THREADS) {
    const u32 c = (&s.hist[0][0])[i];
    if (c) atomicAdd(&a.hist[i], c);
  }
  // ranges and counts: on chip first, one thread's atomics per CTA (from every warp they queued up in
  // one memory sector at the kernel's end)
  mn = __reduce_min_sync(0xffffffffu, mn);
  mx = __reduce_max_sync(0xffffffffu, mx);
  qmn = __reduce_min_sync(0xffffffffu, qmn);
  qmx = __reduce_max_sync(0xffffffffu, qmx);
  n_coll = __reduce_add_sync(0xffffffffu, n_coll);
  n_launch = __reduce_add_sync(0xffffffffu, n_launch);
  md = warp_max_i64(md);
  if (lane == 0) {
    atomicMin(&s.mn, mn);
    atomicMax(&s.mx, mx);
    atomicMin(&s.qmn, qmn);
    atomicMax(&s.qmx, qmx);
    if (n_coll) atomicAdd(&s.n_coll, n_coll);
    if (n_launch) atomicAdd(&s.n_launch, n_launch);
    if (md > 0) atomicMax(&s.md, md);
  }
  __syncthreads();
  if (tid == 0) {
    if (s.n_launch) atomicAdd((u64 *)&a.misc[8], (u64)s.n_launch);
    if (s.n_coll) {
      atomicMin((i64 *)&a.misc[3], (i64)s.qmn);
      atomicMax((i64 *)&a.misc[4], (i64)s.qmx);
      atomicAdd((u64 *)&a.misc[5], (u64)s.n_coll);
    }
    if (s.mn <= s.mx) {
      atomicMin((i64 *)&a.misc[0], (i64)s.mn);
      atomicMax((i64 *)&a.misc[1], (i64)s.mx);
    }
    if (s.md > 0) atomicMax((i64 *)&a.misc[2], s.md);
  }
}

// ---- histograms of the passes over the (dropped, window, triple rank) bits ------------------
// (of a single window they follow from the records counted per triple, in k_rank)
struct TopHistArgs {
  SortPlan plan;        // the whole plan; passes [n_time, n_pass) are the top passes
  int n_time;
  int top_lo;           // key bit where the top bits begin (index bits + time bits kept)
  int tbits, wbits;
  const TripleTable *tt;
  u32 *hist;            // [pass][256]
  const u64 *prekey;
  int64_t n;
  const int64_t *off;
  int W;
};
__device__ __forceinline__ void top_hist_add(const TopHistArgs &a, u32 *hist, u64 c, u32 count) {
  for (int p = a.n_time; p < a.plan.n_pass; p++) {
    const u32 d = (u32)(c >> (a.plan.shift[p] - a.top_lo)) & ((1u << a.plan.bits[p]) - 1u);
    atomicAdd(&hist[p * 256 + d], count);
  }
}
// several windows, counted by window and slot: from the counts
__global__ void __launch_bounds__(256) k_top_hist_counts(TopHistArgs a, const u32 *slot_cnt, const ta_load_summary *sum) {
  TA_PDL();
  __shared__ u32 sh[10 * 256];
  for (int i = threadIdx.x; i < a.plan.n_pass * 256; i += blockDim.x) sh[i] = 0;
  __syncthreads();
  const int64_t cells = (int64_t)a.W * TA_TRIPLE_SLOTS;
  for (int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * 4; i < cells;
       i += (int64_t)gridDim.x * blockDim.x * 4) {
    const uint4 q = *reinterpret_cast<const uint4 *>(slot_cnt + i);
    const u32 c[4] = {q.x, q.y, q.z, q.w};
    const u64 w = (u64)(i / TA_TRIPLE_SLOTS);
#pragma unroll
    for (int j = 0; j < 4; j++)
      if (c[j])
        top_hist_add(a, sh, (w << a.tbits) | (u64)a.tt->rank_of_slot[(int)(i + j) & (TA_TRIPLE_SLOTS - 1)], c[j]);
  }
  for (int w = blockIdx.x * blockDim.x + threadIdx.x; w < a.W; w += gridDim.x * blockDim.x) {
    const u32 nd = (u32)(sum[w].n_bad_kind + sum[w].n_bad_interval + sum[w].n_out_of_window);
    if (!nd) continue;
    top_hist_add(a, sh, (1ull << (a.wbits + a.tbits)) | ((u64)w << a.tbits), nd);
    for (int p = 0; p < a.n_time; p++) atomicAdd(&sh[p * 256], nd);  // time digits 0
  }
  __syncthreads();
  for (int i = threadIdx.x; i < a.plan.n_pass * 256; i += blockDim.x)
    if (sh[i]) atomicAdd(&a.hist[i], sh[i]);
}
// more windows: one pass over the words (8 bytes per record)
__global__ void __launch_bounds__(256) k_top_hist_words(TopHistArgs a) {
  TA_PDL();
  __shared__ u32 sh[10 * 256];
  for (int i = threadIdx.x; i < a.plan.n_pass * 256; i += blockDim.x) sh[i] = 0;
  __syncthreads();
  WindowWalker ww(a.off, a.W);
  const int64_t n_round = ((a.n + 31) / 32) * 32;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_round;
       i += (int64_t)gridDim.x * blockDim.x) {
    const bool in = i < a.n;
    u64 c = 0;
    bool dropped = false;
    if (in) {
      const u64 pk = a.prekey[i];
      const int w = ww.at(i);
      dropped = (pk & PRE_DROPPED) != 0;
      if (dropped) c = (1ull << (a.wbits + a.tbits)) | ((u64)w << a.tbits);
      else c = ((u64)w << a.tbits) |
               (u64)__ldg(&a.tt->rank_of_slot[(u32)(pk >> PRE_TS_BITS) & (TA_TRIPLE_SLOTS - 1)]);
    }
    // neighbouring records mostly share window and lane: one vote, one add per pass
    const u32 act = __ballot_sync(0xffffffffu, in);
    if (!act) continue;
    const int leader = __ffs(act) - 1;
    const u64 c0 = __shfl_sync(0xffffffffu, c, leader);
    const bool same = __all_sync(0xffffffffu, !in || c == c0);
    const u32 nd = __popc(__ballot_sync(0xffffffffu, in && dropped));
    if (same) {
      if ((threadIdx.x & 31) == leader) top_hist_add(a, sh, c0, (u32)__popc(act));
    } else if (in) {
      top_hist_add(a, sh, c, 1u);
    }
    if ((threadIdx.x & 31) == leader && nd)
      for (int p = 0; p < a.n_time; p++) atomicAdd(&sh[p * 256], nd);  // time digits 0
  }
  __syncthreads();
  for (int i = threadIdx.x; i < a.plan.n_pass * 256; i += blockDim.x)
    if (sh[i]) atomicAdd(&a.hist[i], sh[i]);
}

// ascending bitonic sort of buf[0 .. n) in shared memory by the whole CTA; positions up to the next
// power of two are overwritten with all ones
__device__ __forceinline__ void block_sort(u64 *buf, int n) {
  const int tid = threadIdx.x;
  int padded = 32;
  while (padded < n) padded <<= 1;
  for (int i = n + tid; i < padded; i += blockDim.x) buf[i] = ~0ull;
  __syncthreads();
  for (int k = 2; k <= padded; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int i = tid; i < padded; i += blockDim.x) {
        int ixj = i ^ j;
        if (ixj > i) {
          u64 a = buf[i], b = buf[ixj];
          bool up = (i & k) == 0;
          if ((a > b) == up) { buf[i] = b; buf[ixj] = a; }
        }
      }
      __syncthreads();
    }
}

// One CTA: sorts the discovered triples, ranks them and the pids they contain.  A window has tens
// of triples: the occupied slots are packed to the front in any order, as code << 13 | slot, so
// that the sorted entry names its slot; the table is read once and only its occupied slots are
// written (two passes over all slots in block-scan rounds and a serial pid walk took 20 us).
__device__ __forceinline__ int rank_triples(TripleTable *tt, const u32 *slot_cnt, int32_t *status,
                                             u64 *buf /* TA_TRIPLE_SLOTS */) {
  __shared__ u64 tmp[33];
  __shared__ int n_tr;
  const int tid = threadIdx.x;
  if (tid == 0) n_tr = 0;
  __syncthreads();
  for (int s = tid; s < TA_TRIPLE_SLOTS; s += blockDim.x) {
    const u64 v = tt->slots[s];
    if (v) buf[atomicAdd(&n_tr, 1)] = ((v - 1) << 13) | (u64)s;
  }
  __syncthreads();
  block_sort(buf, n_tr);
  int n = n_tr;
  if (n > TA_MAX_TRIPLES) {
    if (tid == 0) ta_set_err(status, TA_ERR_TOO_LARGE);
    n = TA_MAX_TRIPLES;
  }
  int pids = 0;  // pids in front of the round
  for (int i0 = 0; i0 < n; i0 += blockDim.x) {
    const int i = i0 + tid;
    const u64 c = i < n ? buf[i] >> 13 : 0;
    const bool head = i < n && (i == 0 || (buf[i - 1] >> 30) != (c >> 17));
    u64 total;
    const u64 ex = block_scan_exclusive<OpAdd>(head ? 1ull : 0ull, OpAdd(), tmp, &total);
    const int pr = pids + (int)ex + (head ? 1 : 0) - 1;
    if (i < n) {
      tt->sorted_code[i] = c;
      tt->rank_of_slot[(u32)buf[i] & (TA_TRIPLE_SLOTS - 1)] = i;
      tt->pid_rank[i] = pr;
      tt->rank_cnt[i] = slot_cnt[(u32)buf[i] & (TA_TRIPLE_SLOTS - 1)];
      if (head) tt->pid_value[pr] = (int32_t)((u32)(c >> 17) ^ 0x80000000u);
    }
    pids += (int)total;
  }
  if (tid == 0) {
    status[ST_N_TRIPLES] = n;
    status[ST_N_PIDS] = pids;
  }
  return n;
}

// One CTA: sorts and ranks the communicator ids.
__device__ __forceinline__ void rank_comms(CommTable *cm, int32_t *status, u64 *buf /* TA_COMM_SLOTS */) {
  __shared__ int n_c;
  __shared__ u32 slot_of[TA_COMM_SLOTS];
  const int tid = threadIdx.x;
  if (tid == 0) n_c = 0;
  __syncthreads();
  for (int s = tid; s < TA_COMM_SLOTS; s += blockDim.x) {
    const u64 v = cm->slots[s];
    if (v) {
      const int at = atomicAdd(&n_c, 1);
      buf[at] = ~v;
      slot_of[at] = (u32)s;
    }
  }
  __syncthreads();
  int n = n_c;
  if (tid == 0) status[ST_N_COMMS] = n > TA_MAX_COMMS ? TA_MAX_COMMS : n;
  if (n == 0) return;
  block_sort(buf, n);
  if (n > TA_MAX_COMMS && tid == 0) ta_set_err(status, TA_ERR_TOO_LARGE);
  for (int i = tid; i < n && i < TA_MAX_COMMS; i += blockDim.x) cm->sorted_id[i] = buf[i];
  for (int i = tid; i < n; i += blockDim.x) {
    const u64 c = ~cm->slots[slot_of[i]];
    int lo = 0, hi = n - 1;
    while (lo < hi) {
      int mid = (lo + hi) >> 1;
      if (buf[mid] < c) lo = mid + 1;
      else hi = mid;
    }
    cm->rank_of_slot[slot_of[i]] = lo;
  }
}

// Of one window: where the digits of every radix pass begin in its output, the exclusive scan of
// the digit histograms, a warp per pass (a launch of its own in front of the first pass otherwise).  The passes over the
// time bits are counted; those over the (dropped, triple rank) bits follow from the records per triple, and
// dropped records have time digits 0.
struct RankBins {
  const u32 *hist;
  const int64_t *misc;
  const ta_load_summary *sum;  // null: several windows
  u32 *bin_offset;
};
__device__ __forceinline__ void scan_bins(u32 (&v)[8], u32 *out) {
  const int lane = threadIdx.x & 31;
  u32 mine = 0;
#pragma unroll
  for (int k = 0; k < 8; k++) mine += v[k];
  u32 ex = (u32)warp_scan_inclusive((u64)mine, OpAdd()) - mine;
#pragma unroll
  for (int k = 0; k < 8; k++) {
    out[lane * 8 + k] = ex;
    ex += v[k];
  }
}
__device__ __forceinline__ void rank_time_bins(const RankBins &b) {
  const int lane = threadIdx.x & 31, p = threadIdx.x >> 5;
  const SortPlan tp = ta_plan_bits(0, (int)b.misc[6]);
  if (p >= tp.n_pass || tp.n_pass > 5) return;  // (more: the passes are counted anew)
  const u32 dropped = (u32)(b.sum->n_bad_kind + b.sum->n_bad_interval + b.sum->n_out_of_window);
  u32 v[8];
#pragma unroll
  for (int k = 0; k < 8; k++) v[k] = b.hist[p * 256 + lane * 8 + k] + (lane + k == 0 ? dropped : 0u);
  scan_bins(v, b.bin_offset + p * 256);
}
// n triples are ranked, their counts written
__device__ __forceinline__ void rank_top_bins(const RankBins &b, const TripleTable *tt, int n, u32 *sh /* 512 */) {
  const int lane = threadIdx.x & 31, p = threadIdx.x >> 5;
  const int n_time = ta_plan_bits(0, (int)b.misc[6]).n_pass;
  const u32 dropped = (u32)(b.sum->n_bad_kind + b.sum->n_bad_interval + b.sum->n_out_of_window);
  int tbits = 0;
  while (n > 1 && (n - 1) >> tbits) tbits++;
  const int L = tbits + (dropped ? 1 : 0);
  if (L == 0 || n_time > 5) return;
  const SortPlan lp = ta_plan_bits(0, L);  // two passes at most
  for (int i = threadIdx.x; i < 512; i += blockDim.x) sh[i] = 0;
  __syncthreads();
  for (int r = threadIdx.x; r <= n; r += blockDim.x) {
    const u32 code = r < n ? (u32)r : 1u << tbits, c = r < n ? tt->rank_cnt[r] : dropped;
    if (c)
      for (int q = 0; q < lp.n_pass; q++) atomicAdd(&sh[q * 256 + ((code >> lp.shift[q]) & ((1u << lp.bits[q]) - 1u))], c);
  }
  __syncthreads();
  if (p >= lp.n_pass) return;
  u32 v[8];
#pragma unroll
  for (int k = 0; k < 8; k++) v[k] = sh[p * 256 + lane * 8 + k];
  scan_bins(v, b.bin_offset + (n_time + p) * 256);
}

// Both rankings in one launch: CTA 0 the triples, CTA 1 the communicator ids, CTA 2 the time bins (they are
// independent, and single-CTA kernels one after the other cost a launch latency more each).
__global__ void __launch_bounds__(1024) k_rank(TripleTable *tt, CommTable *cm, const u32 *slot_cnt,
                                               int32_t *status, RankBins bins, Tail tail) {
  TA_PDL();
  extern __shared__ u64 rank_buf[];  // TA_TRIPLE_SLOTS
  if (blockIdx.x == 0) {
    const int n = rank_triples(tt, slot_cnt, status, rank_buf);
    __syncthreads();
    if (bins.sum) rank_top_bins(bins, tt, n, reinterpret_cast<u32 *>(rank_buf));
  } else if (blockIdx.x == 1) {
    rank_comms(cm, status, rank_buf);
  } else {
    rank_time_bins(bins);
  }
  run_tail(tail);
}

struct LoadArgs {
  const ta_event *ev;
  int64_t n;
  const int64_t *off, *t0, *t1;
  int W;
  const TripleTable *tt;
  u64 *keys;
  u32 *hist;
  int sbits, tbits, wbits;
  int packed, dshift, ibits;  // packed: key also carries the index inside the window (low ibits)
  SortPlan plan;
  int32_t *status;
};

// Pass 2 over the records: sort key and the digit histograms of all passes.
__global__ void __launch_bounds__(256) k_load(LoadArgs a) {
  TA_PDL();
  __shared__ u32 sh[10 * 256];
  for (int i = threadIdx.x; i < a.plan.n_pass * 256; i += blockDim.x) sh[i] = 0;
  __syncthreads();
  const int tsb = a.sbits - a.dshift;  // time bits kept in the key
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t n_round = ((a.n + 31) / 32) * 32;  // keep warps converged for the votes
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_round; i += stride) {
    bool in = i < a.n;
    u64 key = 0;
    if (in) {
      Rec r = load_rec(a.ev, i);
      int w = window_of(a.off, a.W, i);
      u64 hi;  // [dropped][window][triple rank][time]
      if (defect_of(r, a.t0[w], a.t1[w])) {
        hi = (1ull << (a.wbits + a.tbits + tsb)) | ((u64)w << (a.tbits + tsb));
        if (!a.packed) hi = 1ull << (a.wbits + a.tbits + tsb);
      } else {
        u64 code = triple_code(r.pid, r.kind, r.stream);
        // the discovery pass inserted every triple; a record that is not found was changed
        // behind the library's back (the records are borrowed): bounded probe, error, rank 0
        u32 slot = hash_code(code) & (TA_TRIPLE_SLOTS - 1);
        int probes = 0;
        while (__ldg(&a.tt->slots[slot]) != code + 1 && ++probes < TA_TRIPLE_SLOTS)
          slot = (slot + 1) & (TA_TRIPLE_SLOTS - 1);
        u64 rank = 0;
        if (probes < TA_TRIPLE_SLOTS) rank = (u64)__ldg(&a.tt->rank_of_slot[slot]);
        else ta_set_err(a.status, TA_ERR_OVERFLOW);
        hi = ((u64)w << (a.tbits + tsb)) | (rank << tsb) | ((u64)(r.ts_start - a.t0[w]) >> a.dshift);
      }
      key = a.packed ? (hi << a.ibits) | (u64)(i - a.off[w]) : hi;
      a.keys[i] = key;
    }
    u32 active = __ballot_sync(0xffffffffu, in);
    if (!in) continue;
    const int lane = threadIdx.x & 31;
    const int leader = __ffs(active) - 1;
    for (int p = 0; p < a.plan.n_pass; p++) {
      // high digits are the same across a warp most of the time: one vote, one add
      u32 d = (u32)(key >> a.plan.shift[p]) & ((1u << a.plan.bits[p]) - 1u);
      u32 d0 = __shfl_sync(active, d, leader);
      if (__all_sync(active, d == d0)) {
        if (lane == leader) atomicAdd(&sh[p * 256 + d0], (u32)__popc(active));
      } else {
        atomicAdd(&sh[p * 256 + d], 1u);
      }
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < a.plan.n_pass * 256; i += blockDim.x)
    if (sh[i]) atomicAdd(&a.hist[i], sh[i]);
}

// The same from the words k_discover_staged left in a.keys (rewritten in place): 8 B read + 8 B
// written per record instead of another pass over the 40-byte records.
__global__ void __launch_bounds__(256) k_load_pre(LoadArgs a) {
  TA_PDL();
  __shared__ u32 sh[10 * 256];
  for (int i = threadIdx.x; i < a.plan.n_pass * 256; i += blockDim.x) sh[i] = 0;
  __syncthreads();
  const int tsb = a.sbits - a.dshift;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t n_round = ((a.n + 31) / 32) * 32;
  WindowWalker ww(a.off, a.W);
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_round; i += stride) {
    bool in = i < a.n;
    u64 key = 0;
    if (in) {
      const u64 pk = a.keys[i];
      int w = ww.at(i);
      u64 hi;
      if (pk & PRE_DROPPED) {
        hi = (1ull << (a.wbits + a.tbits + tsb)) | ((u64)w << (a.tbits + tsb));
        if (!a.packed) hi = 1ull << (a.wbits + a.tbits + tsb);
      } else {
        const u32 slot = (u32)(pk >> PRE_TS_BITS) & (TA_TRIPLE_SLOTS - 1);
        const u64 rank = (u64)__ldg(&a.tt->rank_of_slot[slot]);
        hi = ((u64)w << (a.tbits + tsb)) | (rank << tsb) | ((pk & ((1ull << PRE_TS_BITS) - 1)) >> a.dshift);
      }
      key = a.packed ? (hi << a.ibits) | (u64)(i - a.off[w]) : hi;
      a.keys[i] = key;
    }
    u32 active = __ballot_sync(0xffffffffu, in);
    if (!in) continue;
    const int lane = threadIdx.x & 31;
    const int leader = __ffs(active) - 1;
    for (int p = 0; p < a.plan.n_pass; p++) {
      u32 d = (u32)(key >> a.plan.shift[p]) & ((1u << a.plan.bits[p]) - 1u);
      // only the two most significant digits (window, lane, top time bits) are ever the same for
      // a whole warp: the test is not worth its instructions on the others
      if (p >= a.plan.n_pass - 2) {
        u32 d0 = __shfl_sync(active, d, leader);
        if (__all_sync(active, d == d0)) {
          if (lane == leader) atomicAdd(&sh[p * 256 + d0], (u32)__popc(active));
          continue;
        }
      }
      atomicAdd(&sh[p * 256 + d], 1u);
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < a.plan.n_pass * 256; i += blockDim.x)
    if (sh[i]) atomicAdd(&a.hist[i], sh[i]);
}

// ------------------------------------------------------------------ host
static int grid_for(int64_t n, int threads, int per_sm) {
  int64_t g = (n + threads - 1) / threads;
  int64_t cap = 148ll * per_sm;
  return (int)(g < 1 ? 1 : (g > cap ? cap : g));
}

ta_status ta_launch_discover(ta_window *h, void *zero, size_t zero_bytes, int32_t spin) {
  h->tkeep = 0;
  h->fast_keys = 0;
  int64_t max_span = 1, max_win = 1;
  for (int w = 0; w < h->W; w++) {
    max_span = max_span > h->h_t1[w] - h->h_t0[w] ? max_span : h->h_t1[w] - h->h_t0[w];
    max_win = max_win > h->h_off[w + 1] - h->h_off[w] ? max_win : h->h_off[w + 1] - h->h_off[w];
  }
  const int sbits = ta_bit_len((uint64_t)(max_span - 1));
  PlanWindows pw;
  memset(&pw, 0, sizeof(pw));
  if (h->W <= TA_PLAN_WINDOWS) {
    pw.n = 3 * h->W + 1;
    memcpy(pw.v, h->h_off.data(), (size_t)(h->W + 1) * 8);
    memcpy(pw.v + h->W + 1, h->h_t0.data(), (size_t)h->W * 8);
    memcpy(pw.v + 2 * h->W + 1, h->h_t1.data(), (size_t)h->W * 8);
  }
  // (64 KB a CTA and more: 128 MB in a round of two CTAs per SM)
  const PlanClear clear{(uint4 *)zero, (int64_t)(zero_bytes / 16)};
  const int64_t parts = ((int64_t)zero_bytes + (64 << 10) - 1) / (64 << 10);
  ta_launch(k_plan, 1 + (unsigned)(parts < 296 ? parts : 296), PL_THREADS, 0, h->stream, h->events, h->n, h->d_off,
            h->d_t0, h->d_t1, h->W, sbits, max_span, max_win, h->d_misc, pw, clear);
  if (spin > 0)
    TA_CHECK_CUDA(h, cudaMemcpyAsync(h->d_status + ST_SPIN, &spin, sizeof(spin), cudaMemcpyHostToDevice, h->stream));
  if (h->n > 0) {
    // plan the time resolution (above), then the pass over the records, which also takes the histograms of
    // the time passes and counts the records per triple
    DiscoverArgs a;
    a.ev = h->events; a.n = h->n; a.off = h->d_off; a.t0 = h->d_t0; a.t1 = h->d_t1; a.W = h->W;
    a.tt = h->d_triples; a.cm = h->d_comms; a.sum = h->d_load_sum; a.misc = h->d_misc;
    a.status = h->d_status; a.prekey = h->d_keys; a.hist = h->d_hist;
    a.slot_cnt = h->cnt_windows ? h->d_slot_cnt : nullptr;
    a.sbits = sbits;
    TA_CHECK_CUDA(h, cudaFuncSetAttribute(k_discover_staged, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)sizeof(DiscoverSmem)));
    const int64_t tiles = (h->n + DS_TILE - 1) / DS_TILE;
#define DS_CTAS_PER_SM 4
    const int grid = (int)(tiles < 148 * DS_CTAS_PER_SM ? tiles : 148 * DS_CTAS_PER_SM);
    ta_launch(k_discover_staged, grid, DS_THREADS, sizeof(DiscoverSmem), h->stream, a);
    h->tkeep = -1;  // read back with the other results of the pass
    h->prekeys = 1;
  }
  TA_CHECK_CUDA(h, cudaFuncSetAttribute(k_rank, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        TA_TRIPLE_SLOTS * (int)sizeof(u64)));
  const bool one = h->W == 1;
  const RankBins bins{h->d_hist, h->d_misc, one ? h->d_load_sum : nullptr, h->d_bin_offset};
  ta_launch(k_rank, one ? 3 : 2, 1024, TA_TRIPLE_SLOTS * sizeof(u64), h->stream, h->d_triples, h->d_comms, h->d_slot_cnt,
            h->d_status, bins, ta_tail(h, one ? 3 : 2));
  TA_CHECK_CUDA(h, cudaGetLastError());
  return TA_OK;
}

// Chooses the key layout and launches k_load.  allow_packed: try the layout that also
// carries the record's index inside its window in the low bits, so that the sort
// moves 8-byte keys only; it needs (window + triple + time + index) bits to fit 64
// after giving up at most TA_PACK_MAX_DROP low time bits (records that collide in
// the coarser time are put right by the equal-key fix-up).
ta_status ta_launch_load(ta_window *h, bool allow_packed) {
  // key layout: [dropped][window][triple rank][(ts_start - t0) >> dshift]{[index in window]}
  int64_t max_span = 1, max_win = 1;
  for (int w = 0; w < h->W; w++) {
    max_span = max_span > h->h_t1[w] - h->h_t0[w] ? max_span : h->h_t1[w] - h->h_t0[w];
    max_win = max_win > h->h_off[w + 1] - h->h_off[w] ? max_win : h->h_off[w + 1] - h->h_off[w];
  }
  h->sbits = ta_bit_len((uint64_t)(max_span - 1));
  h->tbits = ta_bit_len((uint64_t)(h->n_triples > 0 ? h->n_triples - 1 : 0));
  h->wbits = ta_bit_len((uint64_t)(h->W - 1));
  const int hd = h->has_dropped ? 1 : 0;
  int total = h->sbits + h->tbits + h->wbits + hd;
  if (total > 63) return TA_ERR_TOO_LARGE;
  if (((int64_t)h->W << h->tbits) > (1ll << 24)) return TA_ERR_TOO_LARGE;
  h->ibits = ta_bit_len((uint64_t)(max_win - 1));
  if (h->ibits < 1) h->ibits = 1;
  // A single lane has no bits of its own; what names it is shifted all the same, by 63 at most.
  const int lane_bits = hd + h->wbits + h->tbits, room = 64 - (lane_bits > 0 ? lane_bits : 1) - h->ibits;
  h->fast_keys = 0;
  h->xbits = 0;
  if (allow_packed && h->prekeys && h->tkeep > 0 && h->tkeep <= h->sbits) {
    // The staged discovery pass took the histograms of the passes over the time bits kept, and
    // the lane sizes give those of the passes above them: the first radix pass can build the
    // keys from the discovery words, no key pass is needed.  Passes over time bits and passes
    // over (dropped, window, triple rank) bits never share a digit.
    const int T = h->tkeep, L = lane_bits;
    // What is left of the 64 bits goes to further time bits below those that are sorted: the gather
    // ranks the records of a cell by them, without a look at the records.  Bursts are what gains by it: the
    // gather of 16.8 M prefill records, 82 % of them in cells with others and seven to a cell, takes 393 us
    // and 422 without; of 66.8 M expert records, 22 % and two, 1262 and 1255, and 512 windows of 65 k records
    // lost 490 to 468: windows of a batch go without.
    const int spare = h->W == 1 ? room - T : 0;
    const int X = spare < 0 ? 0 : spare < h->sbits - T ? spare : h->sbits - T;
    const int lo = h->ibits + X;
    const SortPlan tp = ta_plan_bits(lo, lo + T);
    const SortPlan lp = ta_plan_bits(lo + T, lo + T + L);
    const int n_top = L > 0 ? lp.n_pass : 0;
    if (T <= room && tp.n_pass <= 5 && tp.n_pass + n_top <= 10) {
      h->packed = 1;
      h->xbits = X;
      h->dshift = h->sbits - T - X;
      h->plan = tp;
      for (int q = 0; q < n_top; q++) {
        h->plan.shift[tp.n_pass + q] = lp.shift[q];
        h->plan.bits[tp.n_pass + q] = lp.bits[q];
      }
      h->plan.n_pass = tp.n_pass + n_top;
      h->fast_keys = 1;
      if (h->n == 0) return TA_OK;
      if (h->W == 1) return TA_OK;  // k_rank has scanned the histograms
      TopHistArgs a;
      memset(&a, 0, sizeof(a));
      a.plan = h->plan; a.n_time = tp.n_pass; a.top_lo = lo + T;
      a.tbits = h->tbits; a.wbits = h->wbits; a.tt = h->d_triples; a.hist = h->d_hist;
      a.prekey = h->d_keys; a.n = h->n; a.off = h->d_off; a.W = h->W;
      // (512 windows of 65 k records: 211 us from the words)
      if (h->cnt_windows)
        ta_launch(k_top_hist_counts, grid_for((int64_t)h->W * TA_TRIPLE_SLOTS, 1024, 4), 256, 0, h->stream, a,
                  h->d_slot_cnt, h->d_load_sum);
      else ta_launch(k_top_hist_words, grid_for(h->n, 256, 8), 256, 0, h->stream, a);
      TA_CHECK_CUDA(h, cudaGetLastError());
      return TA_OK;  // the words stay in d_keys (h->prekeys stays set): a retry can still use them
    }
  }
  int drop = h->sbits - room;
  if (drop < 0) drop = 0;
  h->packed = allow_packed && drop <= TA_PACK_MAX_DROP && drop < h->sbits;
  if (h->packed) {
    // Coarser time saves whole passes as long as records of one lane rarely share a time
    // bucket (the equal-key fix-up restores the exact order).  Allow a coarsening whose
    // expected bucket occupancy stays below 1/4, assuming lanes up to 4x the average size.
    const double per_lane = 4.0 * (double)(h->n_valid > 0 ? h->n_valid : 1) /
                            ((double)h->W * (double)(h->n_triples > 0 ? h->n_triples : 1));
    int best = drop, best_pass = (total - drop + 7) / 8;
    for (int d = drop + 1; d <= TA_PACK_MAX_DROP && d < h->sbits; d++) {
      if (per_lane * (double)(1ull << d) / (double)max_span > 0.25) break;
      const int np = (total - d + 7) / 8;
      if (np < best_pass) { best = d; best_pass = np; }
    }
    drop = best;
  }
  h->dshift = h->packed ? drop : 0;
  if (h->packed) h->plan = ta_make_plan(h->ibits, h->ibits + total - h->dshift);
  else h->plan = ta_make_plan(0, total);
  if (h->n == 0) return TA_OK;
  TA_CHECK_CUDA(h, cudaMemsetAsync(h->d_hist, 0, 10 * 256 * 4, h->stream));
  LoadArgs a;
  a.ev = h->events; a.n = h->n; a.off = h->d_off; a.t0 = h->d_t0; a.t1 = h->d_t1; a.W = h->W;
  a.tt = h->d_triples; a.keys = h->d_keys; a.hist = h->d_hist;
  a.sbits = h->sbits; a.tbits = h->tbits; a.wbits = h->wbits; a.plan = h->plan;
  a.packed = h->packed; a.dshift = h->dshift; a.ibits = h->ibits; a.status = h->d_status;
  // the words of the discovery pass are there once; a later call (the fall back to full
  // resolution keys) goes back to the records
  if (h->prekeys) ta_launch(k_load_pre, grid_for(h->n, 256, 8), 256, 0, h->stream, a);
  else ta_launch(k_load, grid_for(h->n, 256, 8), 256, 0, h->stream, a);
  h->prekeys = 0;
  TA_CHECK_CUDA(h, cudaGetLastError());
  return TA_OK;
}
