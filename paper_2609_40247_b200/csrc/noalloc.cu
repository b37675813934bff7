// ta_lane_gaps_noalloc: the stream-gap scan of ONE device lane for callers that
// must not allocate device memory (see include/ta.h).  Same arithmetic as the
// per-lane part of ta_stream_gaps; the sums, the tile descriptors of the chained
// max-scan, the tile counter and the status word live in a fixed file-scope device
// array instead of memory obtained from an allocator.  A call is one kernel and a host
// that watches the page-locked row the kernel's last tile writes (a second kernel where a
// lane's records do not end in ascending order).  There are two sets of sums: the last tile
// clears the set of the next call, which clears both itself when it does not follow a call that
// was alone on the device and succeeded.
// Bound by latency: 64 k records take 29 us through the Python binding, of which
// the kernel is 5 (two clearings, a scan, two copies back and a synchronisation: 62).
#include "ta_internal.cuh"

#include <cstring>
#include <mutex>

#define NA_THREADS 256
#define NA_ITEMS 8
#define NA_TILE (NA_THREADS * NA_ITEMS)
#define NA_MAX_RECORDS TA_NOALLOC_MAX_RECORDS
#define NA_MAX_TILES (NA_MAX_RECORDS / NA_TILE)
// tile of the scan-free run: small, so that a lane of 64 k records already keeps half the SMs busy
#define NF_ITEMS 4
#define NF_TILE (NA_THREADS * NF_ITEMS)

// what the kernels of a call add up
struct NaSums {
  u64 busy, idle, n_gaps, max_gap;
  i64 first_start, last_end;
  u32 tiles_done;      // tiles that have added their share: the last one writes the result
  u32 not_ascending;   // scan-free run: a record ends before the one in front of it
  int32_t status[ST_WORDS];
  u32 counter;         // tile tickets of the scan
  u32 pad[5];
};
static_assert(sizeof(NaSums) % 16 == 0, "cleared in words of 16 bytes");
// the result in page-locked host memory, next to the device row the caller asked for
struct NaHost {
  ta_lane_gaps row;
  int32_t err;
  u32 not_ascending;
  volatile u32 seq;  // the call's number, written last
};
struct NaScratch {
  NaSums sum[2];                // calls take them in turn
  u64 state[NA_MAX_TILES + 1];  // tile descriptors of the max-scan
  NaHost host;                  // stands in where no memory could be page-locked, and is copied
};

__device__ __forceinline__ NaSums *na_sums(NaScratch *sc, u32 seq) { return &sc->sum[seq & 1u]; }

// Every device that loads the library holds this array until the process exits.
// In host code `g_na_scratch` is only a stand-in for the symbol, not a device
// address: the address is looked up once per device with cudaGetSymbolAddress.
static __device__ __align__(256) unsigned char g_na_scratch[sizeof(NaScratch)];

// A tile's share to the sums; the last tile to do so writes the row and the host's copy of it.
__device__ __forceinline__ void na_finish(u64 sb, u64 si, u64 ng, u64 mg, int64_t n, u64 (*red)[8], NaScratch *sc,
                                          ta_lane_gaps *out, NaHost *host, u32 seq) {
  const int tid = threadIdx.x;
  sb = warp_reduce(sb, OpAdd());
  si = warp_reduce(si, OpAdd());
  ng = warp_reduce(ng, OpAdd());
  mg = warp_reduce(mg, OpMax());
  if ((tid & 31) == 0) { red[0][tid >> 5] = sb; red[1][tid >> 5] = si; red[2][tid >> 5] = ng; red[3][tid >> 5] = mg; }
  __syncthreads();
  if (tid != 0) return;
  u64 a = 0, b = 0, c = 0, d = 0;
  for (int w = 0; w < NA_THREADS / 32; w++) { a += red[0][w]; b += red[1][w]; c += red[2][w]; d = d > red[3][w] ? d : red[3][w]; }
  NaSums *s = na_sums(sc, seq);
  if (a) atomicAdd(&s->busy, a);
  if (b) atomicAdd(&s->idle, b);
  if (c) atomicAdd(&s->n_gaps, c);
  if (d) atomicMax(&s->max_gap, d);
  __threadfence();
  if (atomicAdd(&s->tiles_done, 1u) != gridDim.x - 1) return;
  __threadfence();
  ta_lane_gaps r;
  r.busy = (i64)__ldcg(&s->busy); r.idle = (i64)__ldcg(&s->idle); r.n_events = n;
  r.n_gaps = (i64)__ldcg(&s->n_gaps); r.max_gap = (i64)__ldcg(&s->max_gap);
  r.first_start = __ldcg(&s->first_start); r.last_end = __ldcg(&s->last_end);
  *out = r;
  uint4 *next = reinterpret_cast<uint4 *>(na_sums(sc, seq + 1));
#pragma unroll
  for (int k = 0; k < (int)(sizeof(NaSums) / 16); k++) next[k] = make_uint4(0, 0, 0, 0);
  host->row = r;
  host->err = __ldcg(&s->status[ST_ERR]);
  host->not_ascending = __ldcg(&s->not_ascending);
  __threadfence_system();
  host->seq = seq;
}

// One tile's records against the running maximum in front of each (pre: 0 = nothing before, else
// clipped end - W0 + 1).
template <int IT>
struct NaTile {
  i64 s[IT], ce[IT];
  u64 v[IT];
  u64 run;
  __device__ __forceinline__ void load(const int64_t *ts, const int64_t *te, int64_t p0, int64_t n, i64 W0, i64 W1) {
    run = 0;
#pragma unroll
    for (int j = 0; j < IT; j++) {
      s[j] = ce[j] = 0;
      v[j] = 0;
      if (p0 + j < n) {
        s[j] = ts[p0 + j];
        ce[j] = te[p0 + j];
      }
    }
#pragma unroll
    for (int j = 0; j < IT; j++)
      if (p0 + j < n) {
        ce[j] = ce[j] < W1 ? ce[j] : W1;
        const i64 rel = ce[j] - W0;
        v[j] = (u64)(rel > 0 ? rel : 0) + 1;
        run = run > v[j] ? run : v[j];
      }
  }
  __device__ __forceinline__ void walk(u64 pre, int64_t p0, int64_t n, i64 W0, i64 W1, int64_t *gap_before, NaSums *sum,
                                       u64 *sb, u64 *si, u64 *ng, u64 *mg, bool *descends) {
#pragma unroll
    for (int j = 0; j < IT; j++) {
      const int64_t p = p0 + j;
      if (p >= n) break;
      const i64 P = pre ? W0 + (i64)(pre - 1) : W0;
      const i64 gap = s[j] > P ? s[j] - P : 0;
      const i64 from = s[j] > P ? s[j] : P;
      const i64 busy = ce[j] > from ? ce[j] - from : 0;
      gap_before[p] = gap;
      *sb += (u64)busy;
      *si += (u64)gap;
      if (gap > 0) { ++*ng; *mg = *mg > (u64)gap ? *mg : (u64)gap; }
      if (p == 0) sum->first_start = s[j];
      if (p == n - 1) {
        const i64 Pm = P > ce[j] ? P : ce[j];
        const i64 tail = W1 - Pm;
        *si += (u64)tail;
        if (tail > 0) { ++*ng; *mg = *mg > (u64)tail ? *mg : (u64)tail; }
        sum->last_end = Pm;
      }
      *descends = *descends || v[j] < pre;
      pre = pre > v[j] ? pre : v[j];
    }
  }
};

// In-order streams end their records in ascending order: the running maximum in front of a record
// is the clipped end of its neighbour, and no tile waits for another.  Checked on the way.
__global__ void __launch_bounds__(NA_THREADS) k_lane_gaps_ascending(const int64_t *ts, const int64_t *te, int64_t n,
                                                                    i64 W0, i64 W1, int64_t *gap_before,
                                                                    ta_lane_gaps *out, NaScratch *sc, NaHost *host,
                                                                    u32 seq) {
  TA_PDL();
  __shared__ u64 red[4][8];
  const int64_t p0 = (int64_t)blockIdx.x * NF_TILE + (int64_t)threadIdx.x * NF_ITEMS;
  NaTile<NF_ITEMS> t;
  t.load(ts, te, p0, n, W0, W1);
  u64 pre = 0;
  if (p0 > 0 && p0 < n) {
    const i64 e = te[p0 - 1], c = (e < W1 ? e : W1) - W0;
    pre = (u64)(c > 0 ? c : 0) + 1;
  }
  u64 sb = 0, si = 0, ng = 0, mg = 0;
  bool descends = false;
  NaSums *sum = na_sums(sc, seq);
  t.walk(pre, p0, n, W0, W1, gap_before, sum, &sb, &si, &ng, &mg, &descends);
  if (descends) sum->not_ascending = 1u;
  na_finish(sb, si, ng, mg, n, red, sc, out, host, seq);
}

// Any lane: chained max-scan over tiles of 2048 records.
__global__ void __launch_bounds__(NA_THREADS) k_lane_gaps_noalloc(const int64_t *ts, const int64_t *te,
                                                                   int64_t n, i64 W0, i64 W1,
                                                                   int64_t *gap_before, ta_lane_gaps *out,
                                                                   NaScratch *sc, NaHost *host, u32 seq) {
  TA_PDL();
  __shared__ u64 tmp[33];
  __shared__ u64 red[4][8];
  __shared__ u64 s_excl;
  __shared__ int s_tile, s_fail;
  const int tid = threadIdx.x;
  NaSums *sum = na_sums(sc, seq);
  if (tid == 0) s_tile = (int)atomicAdd(&sum->counter, 1u);
  __syncthreads();
  const int tile = s_tile;
  const int64_t p0 = (int64_t)tile * NA_TILE + (int64_t)tid * NA_ITEMS;
  NaTile<NA_ITEMS> t;
  t.load(ts, te, p0, n, W0, W1);
  u64 tile_max;
  u64 thread_excl = block_scan_exclusive<OpMax>(t.run, OpMax(), tmp, &tile_max);
  if (tid < 32) {
    bool failed;
    u64 e = tile_lookback<OpMax>(sc->state, tile, tile_max, OpMax(), sum->status, &failed);
    if (tid == 0) { s_excl = e; s_fail = failed ? 1 : 0; }
  }
  __syncthreads();
  u64 sb = 0, si = 0, ng = 0, mg = 0;
  if (!s_fail) {  // a bounded wait that gave up: the status word says so, the tile writes nothing
    bool descends = false;
    t.walk(s_excl > thread_excl ? s_excl : thread_excl, p0, n, W0, W1, gap_before, sum, &sb, &si, &ng, &mg,
           &descends);
  }
  na_finish(sb, si, ng, mg, n, red, sc, out, host, seq);
}

// per device, set up by its first call: the address of the scratch array and the page-locked result
struct NaDevice {
  NaScratch *scratch;
  NaHost *host, *host_dev;
  u32 seq;
  u32 cleared_for;  // number of the call whose set of sums is clear, 0 = none is known to be
  int inside;       // calls in progress
  bool met;         // ... and two of them have been at the same time since there was none
};
static std::mutex g_na_guard;
static NaDevice g_na_device[64];

// clear: the call has to clear the sums itself.  na_leave ends what this begins.
static NaDevice *na_enter(u32 *seq, bool *clear) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
  std::lock_guard<std::mutex> lock(g_na_guard);
  NaDevice &d = g_na_device[dev];
  if (!d.scratch) {
    void *p = nullptr, *hp = nullptr, *hd = nullptr;
    if (cudaGetSymbolAddress(&p, g_na_scratch) != cudaSuccess || !p) {
      cudaGetLastError();
      return nullptr;
    }
    if (cudaHostAlloc(&hp, sizeof(NaHost), cudaHostAllocPortable | cudaHostAllocMapped) == cudaSuccess &&
        cudaHostGetDevicePointer(&hd, hp, 0) == cudaSuccess) {
      memset(hp, 0, sizeof(NaHost));
      d.host = (NaHost *)hp;
      d.host_dev = (NaHost *)hd;
    } else {
      cudaGetLastError();
      if (hp) cudaFreeHost(hp);
      d.host_dev = &((NaScratch *)p)->host;
    }
    d.scratch = (NaScratch *)p;
  }
  if (++d.seq == 0) ++d.seq;
  *seq = d.seq;
  *clear = d.inside > 0 || d.cleared_for != d.seq;
  d.cleared_for = 0;
  if (d.inside++ > 0) d.met = true;
  return &d;
}
// Calls that met on the device race for its sums (the caller's mistake): none of them leaves a set to
// the next.
static void na_leave(NaDevice *d, u32 seq, bool ok) {
  std::lock_guard<std::mutex> lock(g_na_guard);
  if (ok && !d->met && d->seq == seq) d->cleared_for = seq + 1 ? seq + 1 : 0;
  if (--d->inside == 0) d->met = false;
}
struct NaCall {
  NaDevice *d;
  u32 seq;
  bool clear, ok;
  NaCall() : d(nullptr), seq(0), clear(true), ok(false) { d = na_enter(&seq, &clear); }
  ~NaCall() { if (d) na_leave(d, seq, ok); }
};

extern "C" ta_status ta_lane_gaps_noalloc_host(const int64_t *ts_start, const int64_t *ts_end, int64_t n,
                                               int64_t win_t0, int64_t win_t1, int64_t *gap_before,
                                               ta_lane_gaps *lane_out, ta_lane_gaps *host_row, void *cuda_stream) {
  if (n < 0 || win_t0 >= win_t1 || !lane_out || (n > 0 && (!ts_start || !ts_end || !gap_before)))
    return TA_ERR_INVALID_ARG;
  if (((uintptr_t)lane_out | (n > 0 ? (uintptr_t)ts_start | (uintptr_t)ts_end | (uintptr_t)gap_before : 0)) & 7u)
    return TA_ERR_INVALID_ARG;  // 64-bit accesses
  if (n > NA_MAX_RECORDS) return TA_ERR_TOO_LARGE;  // the fixed scratch array covers no more
  if ((uint64_t)win_t1 - (uint64_t)win_t0 >= (1ull << 40)) return TA_ERR_TOO_LARGE;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  if (n == 0) {
    ta_lane_gaps empty = {0, win_t1 - win_t0, 0, 1, win_t1 - win_t0, 0, win_t0};
    if (cudaMemcpyAsync(lane_out, &empty, sizeof(empty), cudaMemcpyHostToDevice, st) != cudaSuccess)
      return TA_ERR_CUDA;
    if (host_row) *host_row = empty;
    return cudaStreamSynchronize(st) == cudaSuccess ? TA_OK : TA_ERR_CUDA;
  }
  NaCall call;
  NaDevice *d = call.d;
  if (!d) return TA_ERR_CUDA;
  const u32 seq = call.seq;
  NaScratch *sc = d->scratch;
  for (int scan = 0; scan < 2; scan++) {
    // the array keeps the previous call's contents: clear what must start at zero (a fill and the wait for
    // it in front of the kernel cost 1.4 us of 30)
    if ((scan || call.clear) && cudaMemsetAsync(sc, 0, scan ? sizeof(NaScratch) : sizeof(sc->sum), st) != cudaSuccess)
      return TA_ERR_CUDA;
    const int64_t tile = scan ? NA_TILE : NF_TILE;
    const unsigned tiles = (unsigned)((n + tile - 1) / tile);
    if (scan)
      ta_launch(k_lane_gaps_noalloc, tiles, NA_THREADS, 0, st, ts_start, ts_end, n, win_t0, win_t1, gap_before, lane_out, sc, d->host_dev, seq);
    else
      ta_launch(k_lane_gaps_ascending, tiles, NA_THREADS, 0, st, ts_start, ts_end, n, win_t0, win_t1, gap_before, lane_out, sc, d->host_dev, seq);
    if (cudaGetLastError() != cudaSuccess) return TA_ERR_CUDA;
    NaHost copy;
    const NaHost *h = d->host ? d->host : &copy;
    if (d->host) {
      TA_WAIT_SEQ(h->seq, seq, st);
    } else if (cudaMemcpyAsync(&copy, d->host_dev, sizeof(copy), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
               cudaStreamSynchronize(st) != cudaSuccess) {
      cudaGetLastError();
      return TA_ERR_CUDA;
    }
    if (h->seq != seq) return TA_ERR_CUDA;  // two calls overlapped
    std::atomic_thread_fence(std::memory_order_acquire);
    if (h->err) return (ta_status)h->err;
    if (host_row) *host_row = h->row;
    if (scan || !h->not_ascending) {
      call.ok = true;
      break;
    }
    if (d->host) d->host->seq = seq - 1;  // the scan announces itself again
  }
  return TA_OK;
}

extern "C" ta_status ta_lane_gaps_noalloc(const int64_t *ts_start, const int64_t *ts_end, int64_t n,
                                          int64_t win_t0, int64_t win_t1, int64_t *gap_before,
                                          ta_lane_gaps *lane_out, void *cuda_stream) {
  return ta_lane_gaps_noalloc_host(ts_start, ts_end, n, win_t0, win_t1, gap_before, lane_out, nullptr, cuda_stream);
}
