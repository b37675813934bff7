// ta_match_collectives: records of different processes that name the same collective
// are linked, and every rank's wait for the last arrival is measured (cross-process
// links: Sec. 6.1 "Execution progress and state"; ranks held up by a late one: Sec. 9.2).  Group key (window, comm_id, seq).
//
// Sequence numbers count up per communicator, so the keys of a window's groups fill a table well, and a
// collective's members meet in one of its cells:
//
//   1. every COLL record adds itself to its cell (k_coll_cells), which lists it for 3 on the way;
//   2. the cells that hold a group, in order, become rows: arrival range, skew, straggler, flags (k_coll_rows);
//   3. one thread per member: wait, and per-(window, pid) totals folded per CTA before they touch
//      global memory (k_coll_members).
//
// With more than 64 processes, numbers too sparse, or no memory for as many cells, the members are sorted instead:
// compaction in sorted-position order, which is pid-major; stable pair sort by (window | communicator rank |
// seq - min seq), so that the members of a group become adjacent and stay ordered by pid; group heads by
// comparing neighbours, group ids by a scan; one thread per group; then 3.
#include <algorithm>
#include <climits>
#include <vector>

#include "scan.cuh"
#include "ta_internal.cuh"


struct CollCtx {
  int64_t m;
  const u32 *posc;      // compacted index -> sorted position
  const int64_t *corr, *ts, *te;
  const int32_t *seq, *pid;
  const int32_t *lane_off, *lane_slot, *lane_window;
  int n_lanes, n_pids;
  const CommTable *cm;
  int64_t min_seq;
  int qbits, cbits;
};

// lane of position p, walking on from a lane at or in front of it (a few lanes at most as a rule; a full
// search after eight steps)
__device__ __forceinline__ int coll_lane(const CollCtx &c, int lane, u32 p) {
  for (int step = 0; lane + 1 < c.n_lanes && (int64_t)c.lane_off[lane + 1] <= (int64_t)p; step++) {
    if (step == 8) return lane_of_pos(c.lane_off, c.n_lanes, p);
    lane++;
  }
  return lane;
}
// rank of a communicator id; every one was inserted while the records were loaded: a bounded probe all
// the same
__device__ __forceinline__ u64 coll_rank(const CollCtx &c, i64 id, int32_t *status) {
  const u64 cc = (u64)id ^ (1ull << 63);
  u32 s = hash_code(cc) & (TA_COMM_SLOTS - 1);
  int probes = 0;
  while (c.cm->slots[s] != ~cc && ++probes < TA_COMM_SLOTS) s = (s + 1) & (TA_COMM_SLOTS - 1);
  if (probes < TA_COMM_SLOTS) return (u64)c.cm->rank_of_slot[s];
  ta_set_err(status, TA_ERR_OVERFLOW);
  return 0;
}

__global__ void __launch_bounds__(256) k_coll_keys(CollCtx c, u64 *keys, int32_t *slot_of, int32_t *status) {
  TA_PDL();
  __shared__ int s_lane0;
  int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  // the compacted positions ascend: the lane of the CTA's first record is searched once, the
  // others walk on from it.  One thread asks for the error word: another CTA may set it meanwhile (coll_rank).
  if (threadIdx.x == 0) s_lane0 = ta_failed(status) ? -1 : lane_of_pos(c.lane_off, c.n_lanes, c.posc[min(j, c.m - 1)]);
  __syncthreads();
  if (s_lane0 < 0 || j >= c.m) return;
  const u32 p = c.posc[j];
  const int lane = coll_lane(c, s_lane0, p);
  const u64 rank = coll_rank(c, c.corr[p], status), w = (u64)c.lane_window[lane];
  keys[j] = (w << (c.cbits + c.qbits)) | (rank << c.qbits) | (u64)((int64_t)c.seq[p] - c.min_seq);
  slot_of[j] = c.lane_slot[lane];
}

struct CollHeadIn {
  const u64 *ks;
  __device__ u64 operator()(int64_t j) const { return (j == 0 || ks[j] != ks[j - 1]) ? 1ull : 0ull; }
};
struct CollHeadOut {
  const u32 *cs;     // sorted rank -> compacted index
  int32_t *gid_of_c; // per compacted index
  int32_t *gstart;   // per group
  __device__ void operator()(int64_t j, u64 excl, u64 v) const {
    int32_t g = (int32_t)(excl + v) - 1;
    gid_of_c[cs[j]] = g;
    if (v) gstart[g] = (int32_t)j;
  }
};

struct CollGroupArgs {
  CollCtx c;
  int64_t n_groups;          // rows allocated; the number of groups unless n_groups_dev is set
  const u64 *n_groups_dev;   // device: the number of groups (the total of the head scan), or null
  const u64 *ks;
  const u32 *cs;
  const int32_t *gstart;
  const int32_t *slot_of;        // per compacted index
  const int32_t *expected;       // per communicator rank, -1 = not given
  int32_t *g_window, *g_seq, *g_n, *g_strag, *g_flags;
  int64_t *g_comm, *g_min, *g_max, *g_skew, *g_end;
  u64 *r_nstrag;                 // per (window, pid) slot
  const int32_t *status;
};

__global__ void __launch_bounds__(256) k_coll_groups(CollGroupArgs a) {
  TA_PDL();
  if (ta_failed(a.status)) return;
  int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t n_groups = a.n_groups_dev ? (int64_t)*a.n_groups_dev : a.n_groups;
  if (g >= n_groups) return;
  const int64_t b = a.gstart[g], e = g + 1 < n_groups ? (int64_t)a.gstart[g + 1] : a.c.m;
  i64 mn = INT64_MAX, mx = INT64_MIN, me = INT64_MIN;
  int32_t strag = 0, strag_slot = 0, prev_pid = 0;
  int flags = 0;
  // members four at a time: each is reached through two index levels (sorted rank -> compacted
  // index -> sorted position), and one member after the other would make the group a chain of
  // forty-odd dependent loads; the order of the updates stays the members' order
  for (int64_t j0 = b; j0 < e; j0 += 4) {
    u32 ci[4], p[4];
    i64 s[4], en[4];
    int32_t pd[4], sl[4];
#pragma unroll
    for (int k = 0; k < 4; k++) ci[k] = j0 + k < e ? a.cs[j0 + k] : 0u;
#pragma unroll
    for (int k = 0; k < 4; k++) p[k] = j0 + k < e ? a.c.posc[ci[k]] : 0u;
#pragma unroll
    for (int k = 0; k < 4; k++) {
      s[k] = en[k] = 0;
      pd[k] = sl[k] = 0;
      if (j0 + k < e) { s[k] = a.c.ts[p[k]]; en[k] = a.c.te[p[k]]; pd[k] = a.c.pid[p[k]]; sl[k] = a.slot_of[ci[k]]; }
    }
#pragma unroll
    for (int k = 0; k < 4; k++) {
      if (j0 + k >= e) break;
      mn = min(mn, s[k]);
      me = max(me, en[k]);
      if (s[k] > mx || (s[k] == mx && pd[k] < strag)) { mx = s[k]; strag = pd[k]; strag_slot = sl[k]; }
      if (j0 + k > b && pd[k] == prev_pid) flags |= TA_COLL_DUP_PID;
      prev_pid = pd[k];
    }
  }
  const u64 key = a.ks[b];
  const int rank = (int)((key >> a.c.qbits) & ((1ull << a.c.cbits) - 1));
  const int32_t ex = a.expected[rank];
  const int64_t nm = e - b;
  if (ex >= 0) { if (nm != ex) flags |= TA_COLL_INCOMPLETE; }
  else if (nm < 2) flags |= TA_COLL_INCOMPLETE;
  a.g_window[g] = (int32_t)(key >> (a.c.cbits + a.c.qbits));
  a.g_comm[g] = (int64_t)(a.c.cm->sorted_id[rank] ^ (1ull << 63));
  a.g_seq[g] = (int32_t)((int64_t)(key & ((1ull << a.c.qbits) - 1)) + a.c.min_seq);
  a.g_n[g] = (int32_t)nm;
  a.g_min[g] = mn;
  a.g_max[g] = mx;
  a.g_skew[g] = mx - mn;
  a.g_end[g] = me;
  a.g_strag[g] = strag;
  a.g_flags[g] = flags;
  if (flags == 0) atomicAdd(&a.r_nstrag[strag_slot], 1ull);
}

struct CollMemberArgs {
  CollCtx c;
  // sorted groups
  const int32_t *slot_of, *gid_of_c;
  const int64_t *g_max;
  const int32_t *g_flags;
  // cells
  const u32 *cell_of;
  const u64 *rel_of, *done;
  int64_t *wait_ns;
  u64 *r_seen, *r_ncoll, *r_sum, *r_maxw;  // per (window, pid) slot
  const int32_t *status;
};

// ---- groups addressed directly -----------------------------------------------------------
// Sequence numbers count up per communicator, so the groups of a window fill a table of (window,
// communicator rank, seq - min seq) well, and its cells in order are the groups in order: nothing has to be
// sorted.  A member adds itself to its cell by four atomics.  66.8 M records, 5.3 M of them members: up to the
// group rows 650 us with the compaction, the sort, its heads and a walk over every group, 265 now; 4.2 M
// records 74 and 37.
#define CC_MAX_PIDS 64  // a bit per process in a cell
#define CC_REL_BITS 40  // a start relative to its window fits
#define CC_FEW 32       // communicators whose sizes travel as an argument
struct CollCells {
  u64 *late;    // latest start << 12 | complement of the process: the last to arrive, the lowest process of several
  u64 *early;   // complement of the earliest start
  u64 *end;     // latest end
  u64 *who;     // processes seen
  u32 *more;    // members beyond the first of a process
  u64 *done;    // latest start << 1 | the group counts: written over `early`
  int64_t n;    // cells
  int64_t range, per_window;  // sequence numbers; cells of a window
  const int64_t *t0;
  const int32_t *expected;    // per communicator rank, -1 = not given; null: in `few`
  int32_t few[CC_FEW];        // (a copy costs more than the kernel)
};

static_assert(24 + CC_REL_BITS <= 64, "fewer than 2^24 slots");
// A CTA takes 8192 sorted positions: it picks out the COLL records, clears the wait column, and has its threads
// add the records to their cells, one each.  The list it leaves for k_coll_members is in order inside a
// tile; tiles take their places as they come.
#define CT_THREADS 256
#define CT_ITEMS 32
#define CT_TILE (CT_THREADS * CT_ITEMS)
struct CollList {
  u32 *pos, *cell;
  u64 *rel;       // slot << CC_REL_BITS | start relative to the window
  u32 *n;
};
__global__ void __launch_bounds__(CT_THREADS) k_coll_cells(CollCtx c, CollCells x, const int16_t *kind, int64_t n_valid,
                                                           int64_t n, i64 *wait_ns, CollList o, int32_t *status) {
  TA_PDL();
  __shared__ u64 tmp[33];
  __shared__ uint16_t s_pos[CT_TILE];
  __shared__ int s_lane0, s_fail;
  __shared__ u32 s_base;
  const int tid = threadIdx.x;
  // (one thread asks: another CTA may set the word meanwhile, and warps that leave would leave the others
  // without their part of the list)
  if (tid == 0) s_fail = ta_failed(status) ? 1 : 0;
  const int64_t start = (int64_t)blockIdx.x * CT_TILE, p0 = start + (int64_t)tid * CT_ITEMS;
  int16_t kd[CT_ITEMS];
#pragma unroll
  for (int j = 0; j < CT_ITEMS; j += 8) load8_i16(kind, p0 + j, n_valid, -1, kd + j);
#pragma unroll
  for (int k = 0; k < CT_ITEMS / 2; k++) {
    const int64_t z = start + (int64_t)k * (2 * CT_THREADS) + 2 * tid;
    if (z + 2 <= n) *reinterpret_cast<longlong2 *>(wait_ns + z) = make_longlong2(0, 0);
    else if (z < n) wait_ns[z] = 0;
  }
  u32 sel = 0;
#pragma unroll
  for (int j = 0; j < CT_ITEMS; j++) sel |= (kd[j] == TA_KIND_COLL ? 1u : 0u) << j;
  u64 total;
  u32 at = (u32)block_scan_exclusive<OpAdd>((u64)__popc(sel), OpAdd(), tmp, &total);
  const u32 count = (u32)total;
  if (count == 0 || s_fail) return;  // (the scan has met a block barrier)
  for (; sel; sel &= sel - 1) s_pos[at++] = (uint16_t)(tid * CT_ITEMS + __ffs((int)sel) - 1);
  if (tid < 32) {
    const int l = tile_lane_search(c.lane_off, c.n_lanes, start);
    if (tid == 0) {
      s_lane0 = l;
      s_base = atomicAdd(o.n, count);
    }
  }
  __syncthreads();
  const u32 base = s_base;
  int lane = s_lane0;
  for (u32 j = tid; j < count; j += CT_THREADS) {
    const u32 p = (u32)start + s_pos[j];
    const i64 id = c.corr[p], s = c.ts[p], e = c.te[p];
    const int32_t q = c.seq[p];
    lane = coll_lane(c, lane, p);
    const int w = c.lane_window[lane], slot = c.lane_slot[lane], pid = slot - w * c.n_pids;
    const u64 rank = coll_rank(c, id, status);
    const i64 t0 = x.t0[w];
    const u64 rel = (u64)(s - t0);
    const int64_t cell = w * x.per_window + (int64_t)rank * x.range + ((int64_t)q - c.min_seq);
    if (cell < 0 || cell >= x.n || base + j >= (u64)c.m) {  // (a record the load did not see)
      ta_set_err(status, TA_ERR_OVERFLOW);
      return;
    }
    const u64 bit = 1ull << pid, seen = atomicOr(&x.who[cell], bit);
    atomicMax(&x.late[cell], rel << 12 | (u64)(0xFFF - pid));
    atomicMax(&x.early[cell], (1ull << CC_REL_BITS) - 1 - rel);
    atomicMax(&x.end[cell], (u64)e - (u64)t0);
    if (seen & bit) atomicAdd(&x.more[cell], 1u);
    o.pos[base + j] = p;
    o.cell[base + j] = (u32)cell;
    o.rel[base + j] = (u64)slot << CC_REL_BITS | rel;
  }
}

// The cells that hold a group, in order, as rows; a tile of cells per CTA, chained like every scan here.
#define CW_THREADS 512
#define CW_ITEMS 4
#define CW_TILE (CW_THREADS * CW_ITEMS)
static_assert(CW_TILE >= SC_TILE, "the descriptors of a scan over as many elements are enough");
struct CollRows {
  int32_t *g_window, *g_seq, *g_n, *g_strag, *g_flags;
  int64_t *g_comm, *g_min, *g_max, *g_skew, *g_end;
  u64 *r_nstrag;
  const TripleTable *tt;
};
__global__ void __launch_bounds__(CW_THREADS) k_coll_rows(CollCtx c, CollCells x, CollRows o, ScanTemp t, int32_t *status) {
  TA_PDL();
  __shared__ u64 tmp[33];
  __shared__ u64 s_excl;
  __shared__ u32 s_strag[CC_MAX_PIDS];  // last arrivals per process, window of the tile's first cell
  __shared__ int s_tile, s_fail;
  const int tid = threadIdx.x;
  if (tid == 0) {
    s_tile = (int)atomicAdd(t.counter, 1u);
    s_fail = ta_failed(status) ? 1 : 0;
  }
  if (tid < CC_MAX_PIDS) s_strag[tid] = 0;
  __syncthreads();
  if (s_fail) return;
  const int tile = s_tile;
  const int64_t first = (int64_t)tile * CW_TILE, i0 = first + tid * CW_ITEMS;
  u64 who[CW_ITEMS], late[CW_ITEMS], early[CW_ITEMS], end[CW_ITEMS];
  u32 more[CW_ITEMS];
  u32 mine = 0;
#pragma unroll
  for (int k = 0; k < CW_ITEMS; k++) {
    const bool in = i0 + k < x.n;
    who[k] = in ? x.who[i0 + k] : 0;
    late[k] = in ? x.late[i0 + k] : 0;
    early[k] = in ? x.early[i0 + k] : 0;
    end[k] = in ? x.end[i0 + k] : 0;
    more[k] = in ? x.more[i0 + k] : 0;
    mine += who[k] != 0;
  }
  u64 total;
  const u64 ex = block_scan_exclusive<OpAdd>((u64)mine, OpAdd(), tmp, &total);
  if (tid < 32) {
    bool failed;
    const u64 b = tile_lookback<OpAdd>(t.state, tile, total, OpAdd(), status, &failed);
    if (tid == 0) {
      s_excl = b;
      s_fail = failed ? 1 : 0;
      if (!failed && first + CW_TILE >= x.n) *t.total = b + total;
    }
  }
  __syncthreads();
  if (s_fail) return;
  u64 row = s_excl + ex;
  const int w0 = (int)(first / x.per_window);
#pragma unroll
  for (int k = 0; k < CW_ITEMS; k++) {
    if (!who[k]) continue;
    const int64_t cell = i0 + k;
    const int w = (int)(cell / x.per_window);
    const int64_t in_w = cell - w * x.per_window;
    const int rank = (int)(in_w / x.range);
    const int64_t q = in_w - rank * x.range;
    const i64 t0 = x.t0[w];
    const int pid = 0xFFF - (int)(late[k] & 0xFFF);
    const u64 mx = late[k] >> 12, mn = (1ull << CC_REL_BITS) - 1 - early[k];
    const int32_t nm = __popcll(who[k]) + (int32_t)more[k], want = x.expected ? x.expected[rank] : x.few[rank];
    const int flags = (more[k] ? TA_COLL_DUP_PID : 0) | ((want >= 0 ? nm != want : nm < 2) ? TA_COLL_INCOMPLETE : 0);
    o.g_window[row] = w;
    o.g_comm[row] = (int64_t)(c.cm->sorted_id[rank] ^ (1ull << 63));
    o.g_seq[row] = (int32_t)(q + c.min_seq);
    o.g_n[row] = nm;
    o.g_min[row] = t0 + (i64)mn;
    o.g_max[row] = t0 + (i64)mx;
    o.g_skew[row] = (i64)(mx - mn);
    o.g_end[row] = (i64)((u64)t0 + end[k]);
    o.g_strag[row] = o.tt->pid_value[pid];
    o.g_flags[row] = flags;
    x.done[cell] = mx << 1 | (flags == 0);
    row++;
    if (flags == 0) {
      if (w == w0) atomicAdd(&s_strag[pid], 1u);
      else atomicAdd(&o.r_nstrag[(int64_t)w * c.n_pids + pid], 1ull);
    }
  }
  __syncthreads();
  if (tid < c.n_pids && s_strag[tid]) atomicAdd(&o.r_nstrag[(int64_t)w0 * c.n_pids + tid], (u64)s_strag[tid]);
}

struct RankRowIn {
  const u64 *seen;
  __device__ u64 operator()(int64_t s) const { return seen[s] ? 1ull : 0ull; }
};
struct RankRowOut {
  const u64 *ncoll, *sum, *maxw, *nstrag;
  const TripleTable *tt;
  int n_pids;
  int32_t *r_window, *r_pid;
  int64_t *r_n_coll, *r_sum_wait, *r_max_wait, *r_n_straggler;
  __device__ void operator()(int64_t s, u64 row, u64 v) const {
    if (!v) return;
    r_window[row] = (int32_t)(s / n_pids);
    r_pid[row] = tt->pid_value[s % n_pids];
    r_n_coll[row] = (int64_t)ncoll[s];
    r_sum_wait[row] = (int64_t)sum[s];
    r_max_wait[row] = (int64_t)maxw[s];
    r_n_straggler[row] = (int64_t)nstrag[s];
  }
};

// members in compacted (= pid-major) order: a CTA almost always sees one slot
template <bool CELLS>
__device__ __forceinline__ void coll_members(const CollMemberArgs &a) {
  __shared__ int s_same;
  __shared__ u64 red[4][8];
  if (ta_failed(a.status)) return;
  auto slot_at = [&](int64_t i) { return CELLS ? (int)(a.rel_of[i] >> CC_REL_BITS) : a.slot_of[i]; };
  int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool in = j < a.c.m;
  int slot = -1;
  u64 ok = 0, wait = 0;
  if (in) {
    u32 p = a.c.posc[j];
    i64 w;
    bool counts;
    if (CELLS) {
      const u64 d = a.done[a.cell_of[j]];
      w = (i64)(d >> 1) - (i64)(a.rel_of[j] & ((1ull << CC_REL_BITS) - 1));
      counts = d & 1u;
    } else {
      int g = a.gid_of_c[j];
      w = a.g_max[g] - a.c.ts[p];
      counts = a.g_flags[g] == 0;
    }
    a.wait_ns[p] = w;
    slot = slot_at(j);
    if (counts) { ok = 1; wait = (u64)w; }
  }
  if (threadIdx.x == 0) s_same = 1;
  __syncthreads();
  const int block_first = slot_at(min((int64_t)blockIdx.x * blockDim.x, a.c.m - 1));
  if (in && slot != block_first) s_same = 0;
  __syncthreads();
  if (s_same) {
    u64 seen = in ? 1 : 0;
    u64 v0 = warp_reduce(seen, OpAdd()), v1 = warp_reduce(ok, OpAdd()), v2 = warp_reduce(wait, OpAdd()),
        v3 = warp_reduce(wait, OpMax());
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) { red[0][warp] = v0; red[1][warp] = v1; red[2][warp] = v2; red[3][warp] = v3; }
    __syncthreads();
    if (threadIdx.x == 0) {
      u64 t0 = 0, t1 = 0, t2 = 0, t3 = 0;
      for (int w = 0; w < 8; w++) { t0 += red[0][w]; t1 += red[1][w]; t2 += red[2][w]; t3 = max(t3, red[3][w]); }
      atomicAdd(&a.r_seen[block_first], t0);
      if (t1) {
        atomicAdd(&a.r_ncoll[block_first], t1);
        atomicAdd(&a.r_sum[block_first], t2);
        atomicMax(&a.r_maxw[block_first], t3);
      }
    }
    return;
  }
  // a CTA that meets several: its warps, most of which meet one
  const u32 act = __ballot_sync(0xffffffffu, in);
  if (!act) return;
  const int slot0 = __shfl_sync(0xffffffffu, slot, __ffs((int)act) - 1);
  u64 seen = in ? 1 : 0;
  if (__all_sync(0xffffffffu, !in || slot == slot0)) {
    seen = (u64)__popc(act);
    ok = warp_reduce(ok, OpAdd());
    const u64 most = warp_reduce(wait, OpMax());
    wait = warp_reduce(wait, OpAdd());
    if ((threadIdx.x & 31) != 0) return;
    atomicAdd(&a.r_seen[slot0], seen);
    if (ok) {
      atomicAdd(&a.r_ncoll[slot0], ok);
      atomicAdd(&a.r_sum[slot0], wait);
      atomicMax(&a.r_maxw[slot0], most);
    }
  } else if (in) {
    atomicAdd(&a.r_seen[slot], 1ull);
    if (ok) {
      atomicAdd(&a.r_ncoll[slot], 1ull);
      atomicAdd(&a.r_sum[slot], wait);
      atomicMax(&a.r_maxw[slot], wait);
    }
  }
}
// The rows of the few processes there are, as a rule, by the last CTA.
#define CR_HERE 256
__device__ __forceinline__ void coll_rank_rows(const u64 *seen, int n_slots, const RankRowOut &o, u64 *total) {
  __shared__ u64 tmp[33];
  const int s = threadIdx.x;
  const bool in = s < n_slots;
  const u64 some = in && __ldcg(&seen[s]) ? 1 : 0;
  const u64 ncoll = in ? __ldcg(&o.ncoll[s]) : 0, sum = in ? __ldcg(&o.sum[s]) : 0, maxw = in ? __ldcg(&o.maxw[s]) : 0,
            nstrag = in ? __ldcg(&o.nstrag[s]) : 0;
  u64 rows;
  const u64 row = block_scan_exclusive<OpAdd>(some, OpAdd(), tmp, &rows);
  if (some) {
    o.r_window[row] = s / o.n_pids;
    o.r_pid[row] = o.tt->pid_value[s % o.n_pids];
    o.r_n_coll[row] = (int64_t)ncoll;
    o.r_sum_wait[row] = (int64_t)sum;
    o.r_max_wait[row] = (int64_t)maxw;
    o.r_n_straggler[row] = (int64_t)nstrag;
  }
  if (s == 0) {
    *total = rows;
    __threadfence();
  }
  __syncthreads();
}
template <bool CELLS, bool TAIL>
__global__ void __launch_bounds__(256) k_coll_members(CollMemberArgs a, int n_slots, RankRowOut o, u64 *total, Tail tail) {
  TA_PDL();
  coll_members<CELLS>(a);
  if (TAIL) run_tail(tail, [&] {
    if (!ta_failed(a.status)) coll_rank_rows(a.r_seen, n_slots, o, total);
  });
}

ta_status ta_run_collectives(ta_window *h, const ta_comm_size *sizes, int32_t n_comms_given,
                             ta_coll_result *out) {
  const int64_t n = h->n, nn = n > 0 ? n : 1;
  cudaStream_t st = h->stream;
  const int n_pids = h->n_pids > 0 ? h->n_pids : 1;
  const int64_t n_slots = (int64_t)h->W * n_pids;
  memset(out, 0, sizeof(*out));

  // kept: wait_ns; everything else is sized once the counts are known
  int64_t *wait_ns = (int64_t *)ta_dalloc(h, (size_t)nn * 8);
  if (!wait_ns) return TA_ERR_OOM;
  out->wait_ns = wait_ns;
  const int64_t m = h->n_coll;  // kept COLL records, counted while the records were loaded
  if (h->n_valid == 0 || h->n_comms == 0 || m == 0) {
    TA_CHECK_CUDA(h, cudaMemsetAsync(wait_ns, 0, (size_t)nn * 8, st));
    return TA_OK;
  }

  const std::vector<u64> &comm_sorted = h->h_comm_sorted;

  // expected communicator sizes by rank
  std::vector<int32_t> expected(h->n_comms, -1);
  for (int i = 0; i < n_comms_given; i++) {
    u64 b = (u64)sizes[i].comm_id ^ (1ull << 63);
    auto it = std::lower_bound(comm_sorted.begin(), comm_sorted.end(), b);
    if (it != comm_sorted.end() && *it == b) expected[it - comm_sorted.begin()] = sizes[i].n_ranks;
  }

  CollCtx cx;
  cx.m = m; cx.posc = nullptr;
  cx.corr = h->sorted.corr_id; cx.ts = h->sorted.ts_start; cx.te = h->sorted.ts_end;
  cx.seq = h->sorted.seq; cx.pid = h->sorted.pid;
  cx.lane_off = h->sorted.lane_off; cx.lane_slot = h->d_lane_slot; cx.lane_window = h->sorted.lane_window;
  cx.n_lanes = h->sorted.n_lanes; cx.n_pids = n_pids; cx.cm = h->d_comms; cx.min_seq = h->min_seq;
  cx.qbits = ta_bit_len((uint64_t)(h->max_seq - h->min_seq));
  cx.cbits = ta_bit_len((uint64_t)(h->n_comms - 1));
  const int wbits = ta_bit_len((uint64_t)(h->W - 1));
  if (cx.qbits < 1) cx.qbits = 1;
  if (cx.qbits + cx.cbits + wbits > 62) return TA_ERR_TOO_LARGE;

  const int gb = (int)((m + 255) / 256);
  ta_status zs;
  void *zb = ta_zalloc(h, 5 * Carver::pad((size_t)n_slots * 8), &zs);
  if (!zb) return zs;
  Carver cz(zb);
  u64 *r_seen = cz.take<u64>(n_slots), *r_ncoll = cz.take<u64>(n_slots), *r_sum = cz.take<u64>(n_slots);
  u64 *r_maxw = cz.take<u64>(n_slots), *r_nstrag = cz.take<u64>(n_slots);

  // Cells of the direct table.  Up to two per member (and a few thousand): clearing and scanning them
  // costs less than sorting the members.  They are taken from the handle's cleared pool; where it has no room
  // (long windows) the way by cells must not ask for more memory than sorting does, some 108 bytes per member.
  const unsigned __int128 all_cells = (unsigned __int128)h->W * (unsigned)h->n_comms * (uint64_t)(h->max_seq - h->min_seq + 1);
  bool cells = n_pids <= CC_MAX_PIDS && all_cells <= (unsigned __int128)(2 * m + 4096);
  const int64_t nc = cells ? (int64_t)all_cells : 0;
  const size_t cells_zeroed = 4 * Carver::pad((size_t)nc * 8) + Carver::pad((size_t)nc * 4) + Carver::pad(4) + scan_temp_bytes(nc);
  const size_t cells_temp = Carver::pad((size_t)m * 8) + 2 * Carver::pad((size_t)m * 4) + Carver::pad((size_t)h->n_comms * 4) +
                            scan_temp_bytes(n_slots) + 256;
  const size_t sort_list = Carver::pad((size_t)m * 4) + scan_temp_bytes(n) + 256;
  const size_t sort_temp = 3 * Carver::pad((size_t)m * 8) + 4 * Carver::pad((size_t)m * 4) + Carver::pad((size_t)(m + 1) * 4) +
                           Carver::pad((size_t)h->n_comms * 4) + ta_sort_temp_bytes(m) + scan_temp_bytes(m) +
                           scan_temp_bytes(n_slots) + 512;
  auto rows_bytes = [](int64_t ng) { return 5 * Carver::pad((size_t)ng * 4) + 5 * Carver::pad((size_t)ng * 8) + 256; };
  // Sorting: the group tables are sized by the number of groups when that is worth a round trip; while
  // the bound "one group per COLL record" keeps them under 1 GiB they are sized by the bound
  // and the count comes back with the call's one wait.
  const bool bounded = (u64)m * 60 <= (1ull << 30);
  void *t1 = nullptr, *t2, *zc = nullptr;
  if (cells && !(zc = ta_zpool(h, cells_zeroed)))
    cells = cells_zeroed + cells_temp + rows_bytes(nc < m ? nc : m) <= sort_list + sort_temp + (bounded ? rows_bytes(m) : 0);
  u64 ng64 = 0;
  const u64 *ng_dev = nullptr;
  CollMemberArgs ma;
  memset(&ma, 0, sizeof(ma));
  CollGroupArgs ga;
  memset(&ga, 0, sizeof(ga));
  void *scan3;
  auto rows_of = [&](int64_t ng) -> bool {
    void *outb = ta_dalloc(h, rows_bytes(ng));
    if (!outb) return false;
    Carver co(outb);
    ga.g_window = co.take<int32_t>(ng); ga.g_seq = co.take<int32_t>(ng); ga.g_n = co.take<int32_t>(ng);
    ga.g_strag = co.take<int32_t>(ng); ga.g_flags = co.take<int32_t>(ng);
    ga.g_comm = co.take<int64_t>(ng); ga.g_min = co.take<int64_t>(ng); ga.g_max = co.take<int64_t>(ng);
    ga.g_skew = co.take<int64_t>(ng); ga.g_end = co.take<int64_t>(ng);
    return true;
  };
  if (cells) {
    // 1. to 3. members to their cells; 4. the cells that are groups
    if (!rows_of(nc < m ? nc : m)) return TA_ERR_OOM;
    t2 = ta_dalloc(h, cells_temp);
    if (!t2) return TA_ERR_OOM;
    Carver c2(t2);
    CollCells x;
    CollList list;
    list.rel = c2.take<u64>(m);
    list.pos = c2.take<u32>(m); list.cell = c2.take<u32>(m);
    int32_t *d_expected = c2.take<int32_t>(h->n_comms);
    scan3 = c2.base + c2.off;
    if (!zc && !(zc = ta_zalloc(h, cells_zeroed, &zs))) return zs;
    Carver cc(zc);
    x.late = cc.take<u64>(nc); x.early = cc.take<u64>(nc); x.end = cc.take<u64>(nc); x.who = cc.take<u64>(nc);
    x.done = x.early;
    x.more = cc.take<u32>(nc);
    list.n = cc.take<u32>(1);
    ScanTemp s2;
    scan_temp_carve(cc.base + cc.off, nc, &s2);
    x.n = nc; x.range = h->max_seq - h->min_seq + 1; x.per_window = x.range * h->n_comms;
    x.t0 = h->d_t0; x.expected = nullptr;
    if (h->n_comms <= CC_FEW) {
      memcpy(x.few, expected.data(), (size_t)h->n_comms * 4);
    } else {
      x.expected = d_expected;
      TA_CHECK_CUDA(h, cudaMemcpyAsync(d_expected, expected.data(), h->n_comms * 4, cudaMemcpyHostToDevice, st));
    }
    ta_launch(k_coll_cells, (unsigned)((n + CT_TILE - 1) / CT_TILE), CT_THREADS, 0, st, cx, x, h->sorted.kind, h->n_valid, n,
              (i64 *)wait_ns, list, h->d_status);
    const CollRows o{ga.g_window, ga.g_seq, ga.g_n, ga.g_strag, ga.g_flags, ga.g_comm, ga.g_min, ga.g_max, ga.g_skew,
                     ga.g_end, r_nstrag, h->d_triples};
    ta_launch(k_coll_rows, (unsigned)((nc + CW_TILE - 1) / CW_TILE), CW_THREADS, 0, st, cx, x, o, s2, h->d_status);
    ng_dev = s2.total;
    ma.cell_of = list.cell; ma.rel_of = list.rel; ma.done = x.done;
    cx.posc = list.pos;
  } else {
    // 1. compaction
    t1 = ta_dalloc(h, sort_list);
    if (!t1) return TA_ERR_OOM;
    Carver c1(t1);
    u32 *pos_all = c1.take<u32>(m);
    ScanTemp s1;
    TA_TRY(scan_temp_init(h, c1.base + c1.off, n, &s1));
    // the compaction pass clears the wait column on its way (one 0.5 GB memset less on c3)
    TA_TRY(launch_compact_kind(h, h->sorted.kind, h->n_valid, 1u << TA_KIND_COLL, pos_all, s1, reinterpret_cast<i64 *>(wait_ns), nn));
    cx.posc = pos_all;
    // 2. keys + sort; 3. heads
    t2 = ta_dalloc(h, sort_temp);
    if (!t2) return TA_ERR_OOM;
    Carver c2(t2);
    u64 *k_in = c2.take<u64>(m), *k_s = c2.take<u64>(m), *ks = c2.take<u64>(m);
    u32 *v_s = c2.take<u32>(m), *cs = c2.take<u32>(m);
    int32_t *slot_of = c2.take<int32_t>(m), *gid_of_c = c2.take<int32_t>(m);
    int32_t *gstart = c2.take<int32_t>(m + 1);
    int32_t *d_expected = c2.take<int32_t>(h->n_comms);
    void *sort_tmp = c2.base + c2.off; c2.off += ta_sort_temp_bytes(m);
    void *scan2 = c2.base + c2.off; c2.off += scan_temp_bytes(m);
    scan3 = c2.base + c2.off;
    TA_CHECK_CUDA(h, cudaMemcpyAsync(d_expected, expected.data(), h->n_comms * 4, cudaMemcpyHostToDevice, st));

    ta_launch(k_coll_keys, gb, 256, 0, st, cx, k_in, slot_of, h->d_status);
    TA_TRY(ta_radix_sort_pairs(h, k_in, nullptr, k_s, v_s, ks, cs, m,
                               ta_make_plan(0, cx.qbits + cx.cbits + wbits), nullptr, sort_tmp));
    ScanTemp s2;
    TA_TRY(scan_temp_init(h, scan2, m, &s2));
    CollHeadIn hin{ks};
    CollHeadOut hout{cs, gid_of_c, gstart};
    TA_TRY((launch_scan<OpAdd, CollHeadIn, CollHeadOut>(h, m, hin, hout, OpAdd(), s2)));
    if (!bounded) {
      TA_TRY(ta_queue_d2h(h, &ng64, s2.total, 8));
      TA_TRY(ta_sync_fetch(h));
    }
    const int64_t ng = bounded ? m : (int64_t)ng64;  // rows allocated (an upper bound when bounded)

    // 4. groups
    if (!rows_of(ng)) return TA_ERR_OOM;
    ga.c = cx; ga.n_groups = ng; ga.n_groups_dev = bounded ? s2.total : nullptr; ga.ks = ks; ga.cs = cs; ga.gstart = gstart; ga.slot_of = slot_of;
    ga.expected = d_expected;
    ga.r_nstrag = r_nstrag; ga.status = h->d_status;
    ta_launch(k_coll_groups, (unsigned)((ng + 255) / 256), 256, 0, st, ga);
    if (bounded) ng_dev = s2.total;
    ma.gid_of_c = gid_of_c; ma.slot_of = slot_of; ma.g_max = ga.g_max; ma.g_flags = ga.g_flags;
  }

  // 5. members
  ma.c = cx;
  ma.status = h->d_status;
  ma.wait_ns = wait_ns; ma.r_seen = r_seen; ma.r_ncoll = r_ncoll; ma.r_sum = r_sum; ma.r_maxw = r_maxw;

  // rank table: compact the (window, pid) slots that saw a COLL record
  size_t rb = 2 * Carver::pad((size_t)n_slots * 4) + 4 * Carver::pad((size_t)n_slots * 8) + 256;
  void *rankb = ta_dalloc(h, rb);
  if (!rankb) return TA_ERR_OOM;
  Carver cr(rankb);
  RankRowOut ro;
  ro.ncoll = r_ncoll; ro.sum = r_sum; ro.maxw = r_maxw; ro.nstrag = r_nstrag;
  ro.tt = h->d_triples; ro.n_pids = n_pids;
  ro.r_window = cr.take<int32_t>(n_slots); ro.r_pid = cr.take<int32_t>(n_slots);
  ro.r_n_coll = cr.take<int64_t>(n_slots); ro.r_sum_wait = cr.take<int64_t>(n_slots);
  ro.r_max_wait = cr.take<int64_t>(n_slots); ro.r_n_straggler = cr.take<int64_t>(n_slots);
  ScanTemp s3;
  TA_TRY(scan_temp_init(h, scan3, n_slots, &s3));
  RankRowIn ri{r_seen};
  u64 nr64 = 0;
  int32_t words[ST_WORDS];
  TA_TRY(ta_queue_d2h(h, &nr64, s3.total, 8));
  if (ng_dev) TA_TRY(ta_queue_d2h(h, &ng64, ng_dev, 8));
  TA_TRY(ta_queue_d2h(h, words, h->d_status, sizeof(words)));
  Tail tail;
  if (n_slots <= CR_HERE) tail = ta_tail(h, gb);
  auto members = cells ? (tail.m ? k_coll_members<true, true> : k_coll_members<true, false>)
                       : (tail.m ? k_coll_members<false, true> : k_coll_members<false, false>);
  ta_launch(members, gb, 256, 0, st, ma, (int)n_slots, ro, s3.total, tail);
  TA_CHECK_CUDA(h, cudaGetLastError());
  if (tail.m == 0) TA_TRY((launch_scan<OpAdd, RankRowIn, RankRowOut>(h, n_slots, ri, ro, OpAdd(), s3, true)));
  TA_TRY(ta_sync_fetch(h));
  ta_dfree(h, t1);
  ta_dfree(h, t2);
  ta_dfree(h, zb);
  ta_dfree(h, zc);
  if (words[ST_ERR]) return (ta_status)words[ST_ERR];

  out->n_groups = (int64_t)ng64;
  out->n_ranks = (int64_t)nr64;
  out->g_window = ga.g_window; out->g_comm = ga.g_comm; out->g_seq = ga.g_seq; out->g_n_members = ga.g_n;
  out->g_min_start = ga.g_min; out->g_max_start = ga.g_max; out->g_skew = ga.g_skew;
  out->g_max_end = ga.g_end; out->g_straggler_pid = ga.g_strag; out->g_flags = ga.g_flags;
  out->r_window = ro.r_window; out->r_pid = ro.r_pid; out->r_n_coll = ro.r_n_coll;
  out->r_sum_wait = ro.r_sum_wait; out->r_max_wait = ro.r_max_wait; out->r_n_straggler = ro.r_n_straggler;
  return TA_OK;
}
