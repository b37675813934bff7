// ta_attribute_operators: every host record gets the operator range of its own
// thread that contains it (same thread, nested intervals: the linkage of Sec. 9.1);
// device records inherit the operator of their launch; per operator, T_op runs from
// the start of its first kernel to the end of its last (Sec. 6.1).
//
// In canonical order (ts_start ascending, ts_end descending) a properly nested
// host lane has a simple structure: the innermost encloser of record i is the
// nearest earlier OP that is still running when i starts.  Tiles of 128 to 1024 records, no kernel ever waits for another CTA:
//   k_attr_agg     per tile, the stack of OPs that are still undominated at the
//                  tile's end (at most TA_MAX_DEPTH + 1 entries when nesting is
//                  legal);
//   k_attr_fold_*  an exclusive scan of those stacks under the stack monoid (one
//                  stack entry per warp lane; entries that end no later than a
//                  later tile's outermost surviving OP are dropped; a tile whose
//                  last lane starts inside it cuts off what came before), as a
//                  fan-out-32 tree, leaves every tile the stack open at its start;
//   k_attr_resolve parent and level of every record, 32 at a time.  The kernels of every
//                  operator are added up on the way, from the launches inside it,
//                  and all columns of the operator are written once, with the zeros of
//                  all other rows;
//   k_attr_ops     device records inherit the operator of their launch; what a tile owes to
//                  operators of earlier tiles is added to their rows.
// Partial overlap is detected on the way: that nearest running OP must also
// cover i's end.
// HBM-bound by design: 26 B read per host record, 16 B per kernel (nearly sequential), 33 B
// written per record.
#include <climits>
#include <cstring>
#include <vector>

#include "scan.cuh"
#include "ta_internal.cuh"

#define AT_THREADS 256
#define AT_CAP 16
#define AS_MINB 4
#define AT_OPS_MINB 6

struct AttrArgs {
  int64_t n, n_valid;
  int n_lanes;
  int64_t n_tiles;
  const int16_t *kind;
  const int64_t *ts, *te;
  const int32_t *lane_off, *lane_window, *lane_dom_end, *lane_dom_next;
  const int16_t *lane_domain;
  int32_t *parent;
  uint8_t *depth;
  ta_attr_summary *sum;
  // per tile: stack at the tile's end (agg) and stack open at its start (carry)
  int32_t *agg_meta, *carry_cnt;  // agg_meta = count | reset << 8
  i64 *agg_e, *carry_e;           // [tile][AT_CAP]
  int32_t *agg_pos, *carry_pos;
  int32_t *status;
  const int32_t *kol;        // kernels of each launch (from the join)
  const int32_t *kernel_of;  // the kernel of each launch that has exactly one
  const int32_t *launch_of;
  int32_t *op_of, *op_n;
  i64 *op_first, *op_last, *op_ns;
  struct AttrSpill *spill;   // what tiles owe to operators of earlier tiles
  u32 *n_spill;
  unsigned spill_blocks;     // k_attr_ops: so many CTAs in front work through that list
  int fold_here;             // k_attr_resolve folds the stacks in front of a tile itself: tiles ...
  const int32_t *group_meta; // ... and, of more than 32, groups of 32 tiles
  const i64 *group_e;
  const int32_t *group_pos;
};
struct AttrSpill {
  int32_t pos, cnt;
  i64 first, last, ns;
};

// A stack of open operators, one entry per lane of a warp (bottom = lane 0).
struct WStack {
  int cnt, reset;
  i64 e;
  int32_t pos;
};

// acc <- earlier (+) acc, all 32 lanes
__device__ __forceinline__ void wstack_combine(const WStack &ear, WStack &acc, bool *overflow) {
  if (acc.reset) return;
  const int lane = threadIdx.x & 31;
  int keep = ear.cnt;
  if (acc.cnt > 0) {
    const i64 e0 = __shfl_sync(0xffffffffu, acc.e, 0);
    // an earlier OP that ends exactly when the outermost later one does still encloses it
    keep = __popc(__ballot_sync(0xffffffffu, lane < ear.cnt && ear.e >= e0));
  }
  if (keep + acc.cnt > AT_CAP) {
    *overflow = true;
    keep = AT_CAP - acc.cnt;
  }
  const int src = lane - keep < 0 ? 0 : lane - keep;
  const i64 se = __shfl_sync(0xffffffffu, acc.e, src);
  const int32_t sp = __shfl_sync(0xffffffffu, acc.pos, src);
  acc.e = lane < keep ? ear.e : se;
  acc.pos = lane < keep ? ear.pos : sp;
  acc.cnt += keep;
  acc.reset = ear.reset;
}



// ---- kernel 1: the stack each tile leaves behind --------------------------------
// The operators of the tile's last lane that end no earlier than every later one.  A warp takes a
// tile, from its last row of 32 records to its first; nearly every row but the last is behind what
// later rows have raised the bar to, and costs its loads and one vote.  (A CTA per tile, with block
// barriers around its suffix maximum, took 170 us of 66.8 M records.)
template <int TILE>
__global__ void __launch_bounds__(AT_THREADS) k_attr_agg(AttrArgs a) {
  TA_PDL();
  if (ta_failed(a.status)) return;
  const int lane = threadIdx.x & 31;
  const int64_t tile = (int64_t)blockIdx.x * (AT_THREADS / 32) + (threadIdx.x >> 5);
  if (tile >= a.n_tiles) return;
  const int64_t tile_start = tile * TILE, vend = min(tile_start + TILE, a.n_valid);
  const int l = vend > tile_start ? tile_lane_search(a.lane_off, a.n_lanes, vend - 1) : -1;
  if (l < 0 || a.lane_domain[l] != 0) {
    if (lane == 0) a.agg_meta[tile] = 1 << 8;  // nothing carried past a device lane
    return;
  }
  const int64_t seg = a.lane_off[l], from = max(seg, tile_start);
  i64 bar = INT64_MIN;  // latest end so far
  int cnt = 0;
  i64 my_e = 0;         // entry `lane` of the stack, innermost first
  int32_t my_pos = 0;
  constexpr int AHEAD = 4;  // rows whose columns are in flight
  for (int64_t hi = vend; hi > from; hi -= 32 * AHEAD) {
    i64 e[AHEAD];
    bool op[AHEAD];
#pragma unroll
    for (int r = 0; r < AHEAD; r++) {
      const int64_t p = hi - 32 * (r + 1) + lane;
      op[r] = p >= from && a.kind[p] == TA_KIND_OP;
      e[r] = op[r] ? (i64)a.te[p] : 0;
    }
#pragma unroll
    for (int r = 0; r < AHEAD; r++) {
      // equal ends nest: the earlier operator encloses the later one
      u32 m = __ballot_sync(0xffffffffu, op[r] && e[r] >= bar);
      while (m) {
        const int src = 31 - __clz((int)m);
        m &= ~(1u << src);
        const i64 es = __shfl_sync(0xffffffffu, e[r], src);
        if (es < bar) continue;
        bar = es;
        if (lane == cnt) { my_e = es; my_pos = (int32_t)(hi - 32 * (r + 1) + src); }
        cnt++;
      }
    }
  }
  if (cnt > AT_CAP) {  // the outermost ones are lost: nesting this deep is reported anyway
    if (lane == 0) ta_set_err(a.status, TA_ERR_DEPTH);
    cnt = AT_CAP;
  }
  if (lane < cnt) {
    a.agg_e[(size_t)tile * AT_CAP + (cnt - 1 - lane)] = my_e;
    a.agg_pos[(size_t)tile * AT_CAP + (cnt - 1 - lane)] = my_pos;
  }
  if (lane == 0) a.agg_meta[tile] = cnt | ((seg >= tile_start ? 1 : 0) << 8);
}

// ---- kernel 2: the stack open at the start of every tile --------------------------
// An exclusive scan of the tile stacks under the stack monoid (wstack_combine; a stack whose
// reset flag is set cuts off everything before it, which is how lanes stay apart).  One fold
// over all tiles would be a serial chain as long as the longest host lane, so it is done as a
// tree with fan-out 32: fold groups of 32 stacks upwards until at most 32 remain, scan those
// with one warp, then unfold downwards.  Every step is one warp working through 32 staged
// stacks; no kernel waits for another.
struct StackArr {
  int32_t *meta;  // count | reset << 8
  i64 *e;
  int32_t *pos;
};
#define AT_FAN 32
struct StackStage {
  i64 e[4][AT_FAN][AT_CAP];
  int32_t pos[4][AT_FAN][AT_CAP];
  int meta[4][AT_FAN];
};
// lane i of the warp copies stack first + i into the stage (count 0 beyond n)
__device__ __forceinline__ void stack_stage(const StackArr &src, int64_t first, int64_t n, StackStage &st,
                                            int warp, int lane) {
  const int64_t t = first + lane;
  int m = 0;
  if (t < n) {
    m = src.meta[t];
    const int c = m & 0xFF;
#pragma unroll
    for (int k = 0; k < AT_CAP; k++)
      if (k < c) {
        st.e[warp][lane][k] = src.e[(size_t)t * AT_CAP + k];
        st.pos[warp][lane][k] = src.pos[(size_t)t * AT_CAP + k];
      }
  }
  st.meta[warp][lane] = m;
  __syncwarp();
}
__device__ __forceinline__ WStack stack_staged(const StackStage &st, int warp, int i, int lane) {
  WStack x;
  const int m = st.meta[warp][i];
  x.cnt = m & 0xFF;
  x.reset = (m >> 8) & 1;
  x.e = lane < x.cnt ? st.e[warp][i][lane] : 0;
  x.pos = lane < x.cnt ? st.pos[warp][i][lane] : 0;
  return x;
}
__device__ __forceinline__ WStack stack_load(const StackArr &src, int64_t t, int lane) {
  WStack x;
  const int m = src.meta[t];
  x.cnt = m & 0xFF;
  x.reset = (m >> 8) & 1;
  x.e = lane < x.cnt ? src.e[(size_t)t * AT_CAP + lane] : 0;
  x.pos = lane < x.cnt ? src.pos[(size_t)t * AT_CAP + lane] : 0;
  return x;
}
__device__ __forceinline__ void stack_store(const StackArr &dst, int64_t t, const WStack &x, int lane,
                                            bool count_only) {
  if (lane < x.cnt) {
    dst.e[(size_t)t * AT_CAP + lane] = x.e;
    dst.pos[(size_t)t * AT_CAP + lane] = x.pos;
  }
  if (lane == 0) dst.meta[t] = count_only ? x.cnt : (x.cnt | (x.reset << 8));
}

// parent[j] = child[32j] (+) ... (+) child[32j + 31]
__global__ void __launch_bounds__(128) k_attr_fold_up(StackArr child, int64_t n_child, StackArr parent,
                                                      int64_t n_parent, int32_t *status) {
  TA_PDL();
  __shared__ StackStage st;
  if (ta_failed(status)) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t j = (int64_t)blockIdx.x * 4 + warp;
  if (j >= n_parent) return;
  stack_stage(child, j * AT_FAN, n_child, st, warp, lane);
  bool overflow = false;
  WStack acc;
  acc.cnt = 0; acc.reset = 0; acc.e = 0; acc.pos = 0;
  const int cnt = (int)min((int64_t)AT_FAN, n_child - j * AT_FAN);
  for (int i = 0; i < cnt; i++) {
    WStack nxt = stack_staged(st, warp, i, lane);
    wstack_combine(acc, nxt, &overflow);
    acc = nxt;
  }
  stack_store(parent, j, acc, lane, false);
  if (overflow && lane == 0) ta_set_err(status, TA_ERR_DEPTH);
}

// one warp: start[i] = node[0] (+) ... (+) node[i - 1] for the few (at most AT_FAN) nodes of the top
// level, staged first (a chain of loads from memory took 18 us for 31 of them)
__global__ void __launch_bounds__(32) k_attr_fold_top(StackArr node, int64_t n, StackArr start,
                                                      int leaf, int32_t *status) {
  TA_PDL();
  __shared__ StackStage st;
  if (ta_failed(status)) return;
  const int lane = threadIdx.x & 31;
  stack_stage(node, 0, n, st, 0, lane);
  bool overflow = false;
  WStack acc;
  acc.cnt = 0; acc.reset = 0; acc.e = 0; acc.pos = 0;
  for (int i = 0; i < (int)n; i++) {
    stack_store(start, i, acc, lane, leaf != 0);
    WStack nxt = stack_staged(st, 0, i, lane);
    wstack_combine(acc, nxt, &overflow);
    acc = nxt;
  }
  if (overflow && lane == 0) ta_set_err(status, TA_ERR_DEPTH);
}

// child_start[32j + i] = parent_start[j] (+) child[32j] (+) ... (+) child[32j + i - 1]
__global__ void __launch_bounds__(128) k_attr_fold_down(StackArr child, int64_t n_child,
                                                        StackArr parent_start, int64_t n_parent,
                                                        StackArr child_start, int leaf, int32_t *status) {
  TA_PDL();
  __shared__ StackStage st;
  if (ta_failed(status)) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t j = (int64_t)blockIdx.x * 4 + warp;
  if (j >= n_parent) return;
  stack_stage(child, j * AT_FAN, n_child, st, warp, lane);
  bool overflow = false;
  WStack acc = stack_load(parent_start, j, lane);
  const int cnt = (int)min((int64_t)AT_FAN, n_child - j * AT_FAN);
  for (int i = 0; i < cnt; i++) {
    stack_store(child_start, j * AT_FAN + i, acc, lane, leaf != 0);
    WStack nxt = stack_staged(st, warp, i, lane);
    wstack_combine(acc, nxt, &overflow);
    acc = nxt;
  }
  if (overflow && lane == 0) ta_set_err(status, TA_ERR_DEPTH);
}

// ---- kernel 3: parent and depth of every host record, kernels of every operator ---------
// A warp takes a tile row by row, 32 records of ONE lane per row and one record per thread, and keeps
// the stack of operators open in front of the row in shared memory.  The innermost operator around a
// record is the nearest one in front of it that ends at or after the record's threshold: every thread
// starts from the operator just in front of its record and, while that has ended, jumps to that
// operator's own candidate (what lies between an operator and its candidate has ended for the
// operator, so also for whoever jumps over it); all 32 move at the same time, so a row takes the
// logarithm of its nesting in rounds of three shuffles.  What a row does not answer, the stack does.
// The kernels of the launches are added up on the way: an operator owns those of the launches
// directly inside it, so every one arrives while its operator is in the row or on the stack.
// (Four consecutive records per thread, each searched by a walk over a max-tree in shared memory and
// added to shared-memory rows by 64-bit atomics, took 660 warp instructions per 32 records, 1.33 ms
// of 66.8 M records; three atomics per kernel in memory, before that, 1.2 ms more.)
#define AS_LEVELS 64   // open operators a warp keeps; more than TA_MAX_DEPTH is an error anyway
#define AS_WARPS 8
#define AS_MORE 0x80000000u
struct AttrStack {
  i64 e[AS_LEVELS];      // end times, none above is greater than one below
  i64 first[AS_LEVELS], last[AS_LEVELS];
  u64 ns[AS_LEVELS];
  int32_t pos[AS_LEVELS];
  u32 cnt[AS_LEVELS];    // kernels; bit 31: k_attr_ops may add more, the row keeps its identities
  // what the launches of one row add: to the operators of the row (0..31), to the levels (32 + k);
  // times relative to the row's first kernel
  int32_t r_first[32 + AS_LEVELS], r_last[32 + AS_LEVELS];
  u32 r_ns[32 + AS_LEVELS], r_cnt[32 + AS_LEVELS];
};
__device__ __forceinline__ i64 shfl_i64(i64 v, int src) { return __shfl_sync(0xffffffffu, v, src); }

// rows of positions without a host record
__device__ __forceinline__ void attr_fill(const AttrArgs &a, int64_t from, int64_t to) {
  const int lane = threadIdx.x & 31;
#pragma unroll 2
  for (int64_t p = from + lane; p < to; p += 32) {
    a.parent[p] = -1;
    a.depth[p] = 0;
    a.op_n[p] = 0;
    a.op_first[p] = 0;
    a.op_last[p] = 0;
    a.op_ns[p] = 0;
  }
}
// levels [from, to) leave the stack: what they own is written, or noted for the rows of earlier tiles
// (the lowest `carried` levels).  open: later tiles may add to them.
__device__ __forceinline__ void attr_pop(const AttrArgs &a, const AttrStack &st, int from, int to, int carried, bool open) {
  const int lane = threadIdx.x & 31;
  for (int k = from + lane; k < to; k += 32) {
    const u32 c = st.cnt[k];
    const int32_t r = st.pos[k];
    if (k < carried) {
      if (c & ~AS_MORE)
        a.spill[atomicAdd(a.n_spill, 1u)] = AttrSpill{r, (int32_t)(c & ~AS_MORE), st.first[k], st.last[k], (i64)st.ns[k]};
    } else if (c || open) {
      a.op_n[r] = (int32_t)(c & ~AS_MORE);
      a.op_first[r] = st.first[k];
      a.op_last[r] = st.last[k];
      a.op_ns[r] = (i64)st.ns[k];
    }
  }
  __syncwarp();
}

// With fold_here the stacks in front of a tile are folded by the CTA that resolves it: the groups of 32
// tiles in front of its own and the tiles of the group in front of its first, at most 31 and 24, are
// dealt out over its warps, which leave eight partial folds on chip; every warp adds its CTA's tiles in
// front of its own.  Up to 1024 tiles this takes less than the two launches (k_attr_fold_top,
// k_attr_fold_down) it stands for.
struct StackPart {
  i64 e[AT_CAP];
  int32_t pos[AT_CAP];
  int cnt, reset;
};
// acc = acc (+) stacks [b, e) of an array, the next one's entries on their way while one is combined
__device__ __forceinline__ void attr_take(WStack &acc, const int32_t *meta, const i64 *es, const int32_t *ps,
                                          int64_t b, int64_t e, bool *overflow) {
  const int lane = threadIdx.x & 31;
  int m1 = 0;
  i64 e1 = 0;
  int32_t p1 = 0;
  auto ask = [&](int64_t t) {
    m1 = meta[t];
    if (lane < AT_CAP) { e1 = es[(size_t)t * AT_CAP + lane]; p1 = ps[(size_t)t * AT_CAP + lane]; }
  };
  if (b < e) ask(b);
  for (int64_t t = b; t < e; t++) {
    WStack x;
    x.cnt = m1 & 0xFF;
    x.reset = (m1 >> 8) & 1;
    x.e = lane < x.cnt ? e1 : 0;
    x.pos = lane < x.cnt ? p1 : 0;
    if (t + 1 < e) ask(t + 1);
    wstack_combine(acc, x, overflow);
    acc = x;
  }
}
__device__ __forceinline__ void attr_parts(const AttrArgs &a, int64_t tile0, StackPart *part) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int groups = (int)(tile0 >> 5), m = groups + (int)(tile0 & 31);
  const int b = warp * m / AS_WARPS, e = (warp + 1) * m / AS_WARPS;
  WStack acc;
  acc.cnt = 0; acc.reset = 0; acc.e = 0; acc.pos = 0;
  bool overflow = false;
  attr_take(acc, a.group_meta, a.group_e, a.group_pos, min(b, groups), min(e, groups), &overflow);
  const int64_t first = (int64_t)groups * 32 - groups;  // tile of element i behind the groups: first + i
  attr_take(acc, a.agg_meta, a.agg_e, a.agg_pos, first + max(b, groups), first + max(e, groups), &overflow);
  if (lane < AT_CAP) { part[warp].e[lane] = acc.e; part[warp].pos[lane] = acc.pos; }
  if (lane == 0) {
    part[warp].cnt = acc.cnt;
    part[warp].reset = acc.reset;
    if (overflow) ta_set_err(a.status, TA_ERR_DEPTH);
  }
}
__device__ __forceinline__ WStack attr_open(const AttrArgs &a, const StackPart *part, int64_t tile0, int64_t tile) {
  const int lane = threadIdx.x & 31;
  WStack acc;
  acc.cnt = 0; acc.reset = 0; acc.e = 0; acc.pos = 0;
  bool overflow = false;
  for (int w = 0; w < AS_WARPS; w++) {
    WStack x;
    x.cnt = part[w].cnt;
    x.reset = part[w].reset;
    x.e = lane < x.cnt ? part[w].e[lane] : 0;
    x.pos = lane < x.cnt ? part[w].pos[lane] : 0;
    wstack_combine(acc, x, &overflow);
    acc = x;
  }
  attr_take(acc, a.agg_meta, a.agg_e, a.agg_pos, tile0, tile, &overflow);
  if (overflow && lane == 0) ta_set_err(a.status, TA_ERR_DEPTH);
  return acc;
}

// kernels of an operator on the stack (one thread)
__device__ __forceinline__ void attr_level_add(AttrStack &st, int k, u32 cnt, i64 first, i64 last, u64 ns) {
  st.cnt[k] += cnt;
  st.first[k] = min(st.first[k], first);
  st.last[k] = max(st.last[k], last);
  st.ns[k] += ns;
}

template <int TILE>
__global__ void __launch_bounds__(AS_WARPS * 32, AS_MINB) k_attr_resolve(AttrArgs a) {
  TA_PDL();
  __shared__ AttrStack s_stack[AS_WARPS];
  __shared__ StackPart s_part[AS_WARPS];
  if (ta_failed(a.status)) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const u32 lt = (1u << lane) - 1u;
  const int64_t tile0 = (int64_t)blockIdx.x * AS_WARPS, tile = tile0 + warp;
  if (a.fold_here) {
    attr_parts(a, tile0, s_part);
    __syncthreads();
  }
  if (tile >= a.n_tiles) return;
  AttrStack &st = s_stack[warp];
  const int64_t tile_start = tile * TILE, tile_end = min(tile_start + TILE, a.n), vend = min(tile_end, a.n_valid);
  if (tile_start >= vend) {
    attr_fill(a, tile_start, tile_end);
    return;
  }
  for (int i = lane; i < 32 + AS_LEVELS; i += 32) {
    st.r_first[i] = INT_MAX; st.r_last[i] = INT_MIN; st.r_ns[i] = 0; st.r_cnt[i] = 0;
  }
  __syncwarp();
  int l = tile_lane_search(a.lane_off, a.n_lanes, tile_start);
  int64_t pos = tile_start;
  int depth = 0, carried = 0;  // levels on the stack; of these, the lowest ones come from earlier tiles
  if (a.lane_domain[l] == 0 && (int64_t)a.lane_off[l] < tile_start) {
    i64 open_e = 0;
    int32_t open_pos = 0;
    if (a.fold_here) {
      const WStack open = attr_open(a, s_part, tile0, tile);
      depth = carried = open.cnt;
      open_e = open.e;
      open_pos = open.pos;
    } else {
      depth = carried = a.carry_cnt[tile];
      if (lane < depth) {
        open_e = a.carry_e[(size_t)tile * AT_CAP + lane];
        open_pos = a.carry_pos[(size_t)tile * AT_CAP + lane];
      }
    }
    if (lane < depth) {
      st.e[lane] = open_e;
      st.pos[lane] = open_pos;
      st.first[lane] = INT64_MAX; st.last[lane] = INT64_MIN; st.ns[lane] = 0; st.cnt[lane] = 0;
    }
    __syncwarp();
  }
  while (pos < vend) {
    if (a.lane_domain[l] != 0) {
      const int64_t stop = min((int64_t)a.lane_dom_end[l], vend);
      attr_fill(a, pos, stop);
      pos = stop;
      l = a.lane_dom_next[l];
      continue;
    }
    const int64_t lane_end = a.lane_off[l + 1], seg_end = min(lane_end, vend);
    int dmax = 0;
    bool bad = false;
    // A row's columns are requested while the row in front of it is worked on, and so are the times of
    // its launches' kernels, whose positions come from one row further ahead.  (The join counts
    // kernels at launches only.)
    int kd1 = 9, nk1 = 0, nk2 = 0, kp2 = 0;
    i64 ts1 = 0, en1 = 0, ks1 = 0, ke1 = 0;
    auto ahead2 = [&](int64_t p) {
      nk2 = kp2 = 0;
      if (p < seg_end) { nk2 = a.kol[p]; kp2 = a.kernel_of[p]; }
    };
    auto ahead1 = [&](int64_t p) {
      kd1 = 9;
      if (p < seg_end) { kd1 = a.kind[p]; ts1 = a.ts[p]; en1 = a.te[p]; }
      nk1 = nk2;
      if (nk1 == 1) { ks1 = a.ts[kp2]; ke1 = a.te[kp2]; }
    };
    ahead2(pos + lane);
    ahead1(pos + lane);
    ahead2(pos + 32 + lane);
    for (; pos < seg_end; pos += 32) {
      const int64_t p = pos + lane;
      const bool in = p < seg_end, op = kd1 == TA_KIND_OP;
      const bool empty = !(en1 > ts1);
      const i64 e = en1, t = empty ? e : ts1 + 1, ks = ks1, ke = ke1;
      const int n_k = nk1;
      ahead1(p + 32);
      ahead2(p + 64);
      const u32 ops = __ballot_sync(0xffffffffu, op), empty_ops = __ballot_sync(0xffffffffu, op && empty);
      // nearest operator of the row
      int q = (ops & lt) ? 31 - __clz((int)(ops & lt)) : -1;
      i64 pe = 0;  // its end
      for (;;) {
        const int src = q < 0 ? 0 : q;
        pe = shfl_i64(e, src);
        const int up = __shfl_sync(0xffffffffu, q, src);
        const bool ended = in && q >= 0 && pe < t;
        if (!__any_sync(0xffffffffu, ended)) break;
        if (ended) q = up;
      }
      // else the stack: the highest of the levels that end at or after the threshold
      int par = q;  // 0..31: record of the row, 32 + k: level k, -1: none
      if (__any_sync(0xffffffffu, in && q < 0) && depth > 0) {
        int lo = 0, hi = depth;  // levels known to qualify / not known not to
        while (lo < hi) {
          const int mid = (lo + hi) >> 1;
          if (st.e[mid] >= t) lo = mid + 1;
          else hi = mid;
        }
        if (q < 0 && lo > 0) { par = 31 + lo; pe = st.e[lo - 1]; }
      }
      bad |= in && par >= 0 && pe < e;
      // level in the forest: distances to an ancestor, doubled until it is one whose level is known
      int d = par >= 32 ? par - 31 : par >= 0 ? 1 : 0, anc = q;
      if (!in) anc = -1;
      while (__any_sync(0xffffffffu, anc >= 0)) {
        const int src = anc < 0 ? 0 : anc;
        const int d2 = __shfl_sync(0xffffffffu, d, src), a2 = __shfl_sync(0xffffffffu, anc, src);
        if (anc >= 0) { d += d2; anc = a2; }
      }
      if (d > 255) d = 255;
      if (in) dmax = max(dmax, d);
      // kernels of the operators: 32-bit atomics on chip, a few operators' worth of neighbours at a
      // time (a vote and three warp reductions per operator took half of the kernel's instructions)
      u32 cnt = 0;
      i64 first = INT64_MAX, last = INT64_MIN;
      u64 ns = 0;
      u32 left = __ballot_sync(0xffffffffu, n_k == 1 && par >= 0);
      if (left) {
        const i64 base = shfl_i64(ks, __ffs((int)left) - 1);
        const i64 rs = ks - base, re = ke - base, dur = ke - ks;
        const bool mine = left >> lane & 1u;
        // times within a second of the row's first kernel and kernels below 67 ms
        const bool near = rs > -(1ll << 30) && re < (1ll << 30) && dur < (1ll << 26);
        if (__all_sync(0xffffffffu, !mine || near)) {
          if (mine) {
            atomicMin(&st.r_first[par], (int)rs);
            atomicMax(&st.r_last[par], (int)re);
            atomicAdd(&st.r_ns[par], (u32)dur);
            atomicAdd(&st.r_cnt[par], 1u);
          }
          __syncwarp();
          cnt = st.r_cnt[lane];
          if (cnt) {
            first = base + st.r_first[lane];
            last = base + st.r_last[lane];
            ns = st.r_ns[lane];
            st.r_first[lane] = INT_MAX; st.r_last[lane] = INT_MIN; st.r_ns[lane] = 0; st.r_cnt[lane] = 0;
          }
          for (int k = lane; k < depth; k += 32) {
            const u32 c = st.r_cnt[32 + k];
            if (!c) continue;
            attr_level_add(st, k, c, base + st.r_first[32 + k], base + st.r_last[32 + k], st.r_ns[32 + k]);
            st.r_first[32 + k] = INT_MAX; st.r_last[32 + k] = INT_MIN; st.r_ns[32 + k] = 0; st.r_cnt[32 + k] = 0;
          }
        } else {
          for (; left; left &= left - 1) {
            const int src = __ffs((int)left) - 1;
            const int key = __shfl_sync(0xffffffffu, par, src);
            const i64 f = shfl_i64(ks, src), g = shfl_i64(ke, src);
            if (key < 32) {
              if (lane == key) { cnt++; first = min(first, f); last = max(last, g); ns += (u64)(g - f); }
            } else if (lane == 0) {
              attr_level_add(st, key - 32, 1u, f, g, (u64)(g - f));
            }
          }
        }
        __syncwarp();
      }
      // launches with several kernels (graph replays): k_attr_ops meets their kernels one by one
      for (u32 many = __ballot_sync(0xffffffffu, n_k > 1 && par >= 0); many; many &= many - 1) {
        const int key = __shfl_sync(0xffffffffu, par, __ffs((int)many) - 1);
        if (key < 32) { if (lane == key) cnt |= AS_MORE; }
        else if (lane == 0) st.cnt[key - 32] |= AS_MORE;
      }
      __syncwarp();
      if (in) {
        a.parent[p] = par >= 32 ? st.pos[par - 32] : par >= 0 ? (int32_t)(pos + par) : -1;
        a.depth[p] = (uint8_t)d;
        a.op_n[p] = (int32_t)(cnt & ~AS_MORE);
        a.op_first[p] = cnt ? first : 0;
        a.op_last[p] = cnt ? last : 0;
        a.op_ns[p] = (i64)ns;
      }
      if (ops) {
        // the stack behind the row: the last operator and those around it, on what is left of the levels
        int c = 31 - __clz((int)ops);
        const i64 tc = shfl_i64(t, c);
        u32 open;
        int keep = 0;
        if (empty_ops >> c & 1u) {
          // it is empty: what ends at that instant may lie beside it, not around it; up the chain instead
          open = 0;
          while (c >= 0 && c < 32) {
            open |= 1u << c;
            c = __shfl_sync(0xffffffffu, par, c);
          }
          keep = c >= 32 ? c - 31 : 0;
        } else {
          // what still runs when it has begun is around it
          open = __ballot_sync(0xffffffffu, op && (lane == c || e >= tc));
          for (int k = lane; k < depth; k += 32) keep += st.e[k] >= tc;
          keep = depth <= 32 ? __popc(__ballot_sync(0xffffffffu, keep)) : (int)__reduce_add_sync(0xffffffffu, (u32)keep);
        }
        __syncwarp();  // (the row's zeros and parents are out before levels are written to or replaced)
        if (keep < depth) attr_pop(a, st, keep, depth, carried, false);
        if (carried > keep) carried = keep;
        const int at = keep + __popc(open & lt);
        if ((open >> lane & 1u) && at < AS_LEVELS) {
          st.e[at] = e;
          st.pos[at] = (int32_t)p;
          st.first[at] = first;
          st.last[at] = last;
          st.ns[at] = ns;
          st.cnt[at] = cnt;
        }
        depth = keep + __popc(open);
        if (depth > AS_LEVELS) {
          depth = AS_LEVELS;
          if (lane == 0) ta_set_err(a.status, TA_ERR_DEPTH);
        }
        __syncwarp();
      }
    }
    pos = seg_end;
    // the window's deepest record and partial overlap
    dmax = __reduce_max_sync(0xffffffffu, dmax);
    bad = __any_sync(0xffffffffu, bad);
    if (lane == 0) {
      ta_attr_summary *row = &a.sum[a.lane_window[l]];
      if (dmax > *(volatile int32_t *)&row->max_depth) atomicMax(&row->max_depth, dmax);
      if (bad) atomicOr(&row->bad_nesting, 1);
    }
    if (lane_end <= vend) {  // the lane is over: nothing stays open
      attr_pop(a, st, 0, depth, carried, false);
      depth = carried = 0;
      l++;
    }
  }
  attr_pop(a, st, 0, depth, carried, true);
  if (vend < tile_end) attr_fill(a, vend, tile_end);
}

// ---- device records inherit the operator of their launch ------------------------
// adds kernels to an operator's row in memory (whose first / last are identities while it has none)
__device__ __forceinline__ void attr_row_add(const AttrArgs &a, int32_t r, int cnt, i64 first, i64 last, i64 ns) {
  atomicAdd(&a.op_n[r], cnt);
  atomicAdd((u64 *)&a.op_ns[r], (u64)ns);
  atomicMin(&a.op_first[r], first);
  atomicMax(&a.op_last[r], last);
}
__device__ __forceinline__ void attr_spill(const AttrArgs &a) {
  const u32 m = *a.n_spill;
  for (u32 i = blockIdx.x * AT_THREADS + threadIdx.x; i < m; i += a.spill_blocks * AT_THREADS) {
    const AttrSpill x = a.spill[i];
    attr_row_add(a, x.pos, x.cnt, x.first, x.last, x.ns);
  }
}

// adds a group of device records to the row of their window
__device__ __forceinline__ void attr_emit(ta_attr_summary *sm, const u64 *t) {
  if (t[0]) atomicAdd((u64 *)&sm->n_attributed, t[0]);
  if (t[1]) atomicAdd((u64 *)&sm->n_no_launch, t[1]);
  if (t[2]) atomicAdd((u64 *)&sm->n_no_op, t[2]);
}
// A warp takes `rows` x 32 positions, 32 records of ONE lane per row, AO_ROWS rows at a time with the launches
// of the next ones on their way; no warp waits for another before the end.  (Four records per thread
// of a CTA's tile, the lanes walked by every thread behind two block barriers: 243 us of 66.8 M records and 67 of 16.8 M, where this
// takes 117 and 37; four CTAs per SM 124 and 37, eight 128 and 43; 8 rows 159 and 44, 32 rows 113 and 75.)
// MULTI: some launch has more than one kernel; those kernels are added to their operator here.
#define AO_ROWS 4
#define AO_MAX 16
template <bool MULTI>
__device__ __forceinline__ void attr_ops(const AttrArgs &a, int rows) {
  __shared__ u32 red[3][AT_THREADS / 32];
  __shared__ int red_w[AT_THREADS / 32];
  if (ta_failed(a.status)) return;
  if (blockIdx.x < a.spill_blocks) {
    attr_spill(a);
    return;
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t span = (int64_t)rows * 32;
  const int64_t begin = min(((int64_t)(blockIdx.x - a.spill_blocks) * (AT_THREADS / 32) + warp) * span, a.n);
  const int64_t end = min(begin + span, a.n), vend = min(end, a.n_valid);
  u32 cnt[3] = {0, 0, 0};  // attributed, no launch, no operator
  int cur = -1;            // window they are of
  auto flush = [&]() {
    u64 t[3];
#pragma unroll
    for (int k = 0; k < 3; k++) {
      t[k] = __reduce_add_sync(0xffffffffu, cnt[k]);
      cnt[k] = 0;
    }
    if (lane == 0) attr_emit(&a.sum[cur], t);
  };
  int l = begin < vend ? tile_lane_search(a.lane_off, a.n_lanes, begin) : 0;
  for (int64_t pos = begin; pos < vend;) {
    if (a.lane_domain[l] != 1) {  // host lanes hold no device record
      const int64_t stop = min((int64_t)a.lane_dom_end[l], vend);
      for (int64_t p = pos + lane; p < stop; p += 32) a.op_of[p] = -1;
      pos = stop;
      l = a.lane_dom_next[l];
      continue;
    }
    const int64_t lane_end = a.lane_off[l + 1], e = min(lane_end, vend);
    const int win = a.lane_window[l];
    if (win != cur) {
      if (cur >= 0) flush();
      cur = win;
    }
    // (launch_of is -1 wherever the record is no matched kernel or copy: the gather needs no kind)
    int lo[AO_ROWS], kd[AO_ROWS];
    auto ask = [&](int64_t p) {
#pragma unroll
      for (int r = 0; r < AO_ROWS; r++) {
        const int64_t q = p + 32 * r + lane;
        lo[r] = -1;
        kd[r] = 0;
        if (q < e) { lo[r] = a.launch_of[q]; kd[r] = a.kind[q]; }
      }
    };
    ask(pos);
    for (; pos < e; pos += 32 * AO_ROWS) {
      int op[AO_ROWS], from[AO_ROWS];
#pragma unroll
      for (int r = 0; r < AO_ROWS; r++) {
        from[r] = lo[r];
        op[r] = lo[r] >= 0 ? a.parent[lo[r]] : -1;
        cnt[1] += lo[r] < 0 && (kd[r] == TA_KIND_KERNEL || kd[r] == TA_KIND_MEMCPY);
      }
      ask(pos + 32 * AO_ROWS);
#pragma unroll
      for (int r = 0; r < AO_ROWS; r++) {
        const int64_t q = pos + 32 * r + lane;
        if (q >= e) continue;
        a.op_of[q] = op[r];
        cnt[0] += op[r] >= 0;
        cnt[2] += from[r] >= 0 && op[r] < 0;
        if (MULTI && op[r] >= 0 && a.kol[from[r]] > 1) {
          const i64 s = a.ts[q], t = a.te[q];
          attr_row_add(a, op[r], 1, s, t, t - s);
        }
      }
    }
    pos = e;
    if (lane_end == e) l++;
  }
  for (int64_t p = max(begin, vend) + lane; p < end; p += 32) a.op_of[p] = -1;  // dropped records
  // the CTA's figures: one addition where its warps are in one window
#pragma unroll
  for (int k = 0; k < 3; k++) {
    const u32 t = __reduce_add_sync(0xffffffffu, cnt[k]);
    if (lane == 0) red[k][warp] = t;
  }
  if (lane == 0) red_w[warp] = cur;
  __syncthreads();
  if (threadIdx.x != 0) return;
  u64 t[3] = {0, 0, 0};
  int w = -1;
  for (int x = 0; x < AT_THREADS / 32; x++) {
    if (red_w[x] < 0) continue;
    if (red_w[x] != w) {
      if (w >= 0) attr_emit(&a.sum[w], t);
      w = red_w[x];
      t[0] = t[1] = t[2] = 0;
    }
#pragma unroll
    for (int k = 0; k < 3; k++) t[k] += red[k][x];
  }
  if (w >= 0) attr_emit(&a.sum[w], t);
}

// operators that were open at the end of their tile and got no kernels from anywhere: no identities
// are left behind
__device__ __forceinline__ void attr_finalize(const AttrArgs &a, int64_t i) {
  const int64_t tile = i / AT_CAP;
  const int k = (int)(i - tile * AT_CAP);
  if (tile >= a.n_tiles || k >= (a.agg_meta[tile] & 0xFF)) return;
  const int32_t r = a.agg_pos[i];
  if (__ldcg(&a.op_n[r]) == 0) { a.op_first[r] = 0; a.op_last[r] = 0; }
}
__global__ void __launch_bounds__(256) k_attr_finalize(AttrArgs a, Tail tail) {
  TA_PDL();
  if (!ta_failed(a.status)) attr_finalize(a, (int64_t)blockIdx.x * 256 + threadIdx.x);
  run_tail(tail);
}
// With a tail the last CTA does the work of k_attr_finalize (of a few tiles).
template <bool MULTI, bool TAIL>
__global__ void __launch_bounds__(AT_THREADS, AT_OPS_MINB) k_attr_ops(AttrArgs a, int rows, Tail tail) {
  TA_PDL();
  attr_ops<MULTI>(a, rows);
  if (TAIL) run_tail(tail, [&] {
    if (ta_failed(a.status)) return;
    for (int64_t i = threadIdx.x; i < a.n_tiles * AT_CAP; i += AT_THREADS) attr_finalize(a, i);
  });
}

ta_status ta_run_attribute(ta_window *h, ta_attr_summary *out_summary) {
  const int64_t n = h->n, nn = n > 0 ? n : 1;
  const int W = h->W;
  cudaStream_t st = h->stream;
  // A warp takes a tile.  Small tiles keep a warp's chain of rows short: 128 records while the CTA folds the
  // stacks in front of its tiles itself (60 k records 400 us with 256, 387 with 128), 256 up to some
  // three million (1.2 M: 833 with 512, 822), 1024 from ten rounds of the 148 * 32 warps
  // k_attr_resolve keeps on the chip (66.8 M: 782 us of the kernel with 512, 750, and half the stacks); 512
  // between, where the last round's slowest warps show (16.8 M: 342 us of the kernel with 1024, 263; from
  // some 24 M on the call is 2 % faster with 1024: 28 M experts 579 and 571 us, prefill 698 and 669, 60 M
  // 1108 and 1074).
  const int per_tile = n <= 128ll * AT_FAN * AT_FAN ? 128 : n <= (3 << 20) ? 256 : n <= 10ll * 148 * 32 * 1024 ? 512 : 1024;
  const int64_t tiles = (n + per_tile - 1) / per_tile;
  size_t keep = 3 * Carver::pad(nn * 4) + Carver::pad(nn) + 3 * Carver::pad(nn * 8) + 256;
  void *kb = ta_dalloc(h, keep);
  if (!kb) return TA_ERR_OOM;
  Carver ck(kb);
  int32_t *parent = ck.take<int32_t>(nn), *op_of = ck.take<int32_t>(nn);
  uint8_t *depth = ck.take<uint8_t>(nn);
  int32_t *op_n = ck.take<int32_t>(nn);
  i64 *op_first = ck.take<i64>(nn), *op_last = ck.take<i64>(nn), *op_ns = ck.take<i64>(nn);
  ta_status zs;
  void *zb = ta_zalloc(h, Carver::pad((size_t)W * sizeof(ta_attr_summary)) + 256, &zs);
  if (!zb) return zs;
  Carver cz(zb);
  ta_attr_summary *d_sum = cz.take<ta_attr_summary>(W);
  u32 *n_spill = cz.take<u32>(1);

  const int64_t tt = tiles > 0 ? tiles : 1;
  size_t tb = Carver::pad(tt * AT_CAP * sizeof(AttrSpill)) + 2 * Carver::pad(tt * 4) + 2 * Carver::pad(tt * AT_CAP * 8) + 2 * Carver::pad(tt * AT_CAP * 4) + 256;
  // upper levels of the stack scan: node and start stacks per level
  std::vector<int64_t> level_n(1, tt);
  while (level_n.back() > AT_FAN) level_n.push_back((level_n.back() + AT_FAN - 1) / AT_FAN);
  for (size_t k = 1; k < level_n.size(); k++)
    tb += 2 * (Carver::pad(level_n[k] * 4) + Carver::pad(level_n[k] * AT_CAP * 8) +
               Carver::pad(level_n[k] * AT_CAP * 4));
  void *tmpb = ta_dalloc(h, tb);
  if (!tmpb) return TA_ERR_OOM;
  Carver ct(tmpb);
  AttrArgs a;
  memset(&a, 0, sizeof(a));
  a.agg_meta = ct.take<int32_t>(tt);
  a.carry_cnt = ct.take<int32_t>(tt);
  a.agg_e = ct.take<i64>(tt * AT_CAP);
  a.carry_e = ct.take<i64>(tt * AT_CAP);
  a.agg_pos = ct.take<int32_t>(tt * AT_CAP);
  a.carry_pos = ct.take<int32_t>(tt * AT_CAP);
  a.spill = ct.take<AttrSpill>(tt * AT_CAP);
  a.n_spill = n_spill;

  a.n = n; a.n_valid = h->n_valid; a.n_lanes = h->sorted.n_lanes; a.n_tiles = tiles;
  a.kind = h->sorted.kind; a.ts = h->sorted.ts_start; a.te = h->sorted.ts_end;
  a.lane_off = h->sorted.lane_off; a.lane_window = h->sorted.lane_window;
  a.lane_domain = h->sorted.lane_domain; a.lane_dom_end = h->d_lane_dom_end; a.lane_dom_next = h->d_lane_dom_next;
  a.parent = parent; a.depth = depth; a.sum = d_sum; a.status = h->d_status;
  a.launch_of = h->join.launch_of; a.kol = h->join.kernels_of_launch; a.kernel_of = h->d_kernel_of; a.op_of = op_of; a.op_n = op_n; a.op_first = op_first;
  a.op_last = op_last; a.op_ns = op_ns;
  int32_t words[ST_WORDS];
  std::vector<ta_attr_summary> hs(W);
  TA_TRY(ta_queue_d2h(h, words, h->d_status, sizeof(words)));
  TA_TRY(ta_queue_d2h(h, hs.data(), d_sum, W * sizeof(ta_attr_summary)));
  if (n > 0) {
    const unsigned wblocks = (unsigned)((tiles + AS_WARPS - 1) / AS_WARPS);
    ta_launch(per_tile == 128 ? k_attr_agg<128> : per_tile == 256 ? k_attr_agg<256> : per_tile == 512 ? k_attr_agg<512> : k_attr_agg<1024>, wblocks, AT_THREADS, 0, st, a);
    {
      // level 0 = tiles; fold upwards until at most AT_FAN stacks remain, scan those, unfold
      std::vector<StackArr> node(level_n.size()), start(level_n.size());
      node[0] = StackArr{a.agg_meta, a.agg_e, a.agg_pos};
      start[0] = StackArr{a.carry_cnt, a.carry_e, a.carry_pos};
      for (size_t k = 1; k < level_n.size(); k++) {
        const int64_t c = level_n[k];
        node[k] = StackArr{ct.take<int32_t>(c), ct.take<i64>(c * AT_CAP), ct.take<int32_t>(c * AT_CAP)};
        start[k] = StackArr{ct.take<int32_t>(c), ct.take<i64>(c * AT_CAP), ct.take<int32_t>(c * AT_CAP)};
      }
      const size_t top = level_n.size() - 1;
      a.fold_here = top <= 1;
      if (top == 1) { a.group_meta = node[1].meta; a.group_e = node[1].e; a.group_pos = node[1].pos; }
      for (size_t k = 1; k <= top; k++)
        ta_launch(k_attr_fold_up, (unsigned)((level_n[k] + 3) / 4), 128, 0, st, node[k - 1], level_n[k - 1], node[k], level_n[k], h->d_status);
      if (!a.fold_here)
        ta_launch(k_attr_fold_top, 1, 32, 0, st, node[top], level_n[top], start[top], 0, h->d_status);
      for (size_t k = top; k >= 1 && !a.fold_here; k--)
        ta_launch(k_attr_fold_down, (unsigned)((level_n[k] + 3) / 4), 128, 0, st, node[k - 1], level_n[k - 1], start[k], level_n[k], start[k - 1], k == 1 ? 1 : 0, h->d_status);
    }
    ta_launch(per_tile == 128 ? k_attr_resolve<128> : per_tile == 256 ? k_attr_resolve<256> : per_tile == 512 ? k_attr_resolve<512> : k_attr_resolve<1024>, wblocks, AS_WARPS * 32, 0, st, a);
    // (a tile owes something to few operators of earlier ones, as a rule)
    const int64_t sb = (tiles * 2 + AT_THREADS - 1) / AT_THREADS;
    a.spill_blocks = (unsigned)(sb < 148 * 2 ? sb : 148 * 2);
    // rows per warp: 16, fewer while that would be less than two rounds of the 148 * 48 warps on the chip
    int64_t rows = n / 32 / (148 * 96) / AO_ROWS * AO_ROWS;
    rows = rows < AO_ROWS ? AO_ROWS : rows > AO_MAX ? AO_MAX : rows;
    const unsigned ob = a.spill_blocks + (unsigned)((n + rows * AT_THREADS - 1) / (rows * AT_THREADS));
    // the last step in the last CTA of this one, for a few tiles (16 entries each)
    const int64_t entries = tiles * AT_CAP;
    Tail tail;
    if (entries <= 4 * AT_THREADS) tail = ta_tail(h, ob);
    auto ops = h->multi_launch ? (tail.m ? k_attr_ops<true, true> : k_attr_ops<true, false>)
                               : (tail.m ? k_attr_ops<false, true> : k_attr_ops<false, false>);
    ta_launch(ops, ob, AT_THREADS, 0, st, a, (int)rows, tail);
    if (tail.m == 0) {
      const int64_t fb = (entries + 255) / 256;
      ta_launch(k_attr_finalize, (unsigned)fb, 256, 0, st, a, ta_tail(h, fb));
    }
    TA_CHECK_CUDA(h, cudaGetLastError());
  }
  TA_TRY(ta_sync_fetch(h));
  ta_dfree(h, tmpb);
  bool any_bad = false, any_deep = words[ST_ERR] == TA_ERR_DEPTH;
  if (words[ST_ERR] && words[ST_ERR] != TA_ERR_DEPTH) return (ta_status)words[ST_ERR];
  if (any_deep)  // a data error of this call only: later calls start with a clean status word
    TA_CHECK_CUDA(h, cudaMemsetAsync(h->d_status, 0, sizeof(int32_t), st));
  for (int w = 0; w < W; w++) {
    if (hs[w].bad_nesting) any_bad = true;
    if (hs[w].max_depth > TA_MAX_DEPTH) any_deep = true;
    if (out_summary) out_summary[w] = hs[w];
  }
  h->attr.parent = parent;
  h->attr.depth = depth;
  h->attr.op_of = op_of;
  h->attr.op_first_start = (const int64_t *)op_first;
  h->attr.op_last_end = (const int64_t *)op_last;
  h->attr.op_kernel_ns = (const int64_t *)op_ns;
  h->attr.op_n_kernels = op_n;
  if (any_bad) return TA_ERR_BAD_NESTING;
  if (any_deep) return TA_ERR_DEPTH;
  return TA_OK;
}
