// C-ABI entry points (include/ta.h): argument checks, the handle, memory
// through the caller's allocator, call-order bookkeeping.  All arithmetic lives
// in the kernels of the other translation units.
#include <atomic>
#include <cstddef>
#include <cstring>
#include <mutex>
#include <new>

#include "ta_internal.cuh"

// Without caller callbacks memory comes from a private stream-ordered pool per device that
// keeps what it has been given (release threshold = everything): the default pool hands its
// memory back at every synchronisation, which makes each call pay for fresh gigabytes.
static cudaMemPool_t own_pool(int device) {
  static cudaMemPool_t pools[64] = {};
  static std::mutex guard;  // handles on different threads may arrive here together
  if (device < 0 || device >= 64) return nullptr;
  std::lock_guard<std::mutex> lock(guard);
  if (!pools[device]) {
    cudaMemPoolProps props;
    memset(&props, 0, sizeof(props));
    props.allocType = cudaMemAllocationTypePinned;
    props.handleTypes = cudaMemHandleTypeNone;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = device;
    cudaMemPool_t pool = nullptr;
    if (cudaMemPoolCreate(&pool, &props) != cudaSuccess) {
      cudaGetLastError();
      return nullptr;
    }
    unsigned long long keep = ~0ull;
    cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
    pools[device] = pool;
  }
  return pools[device];
}

// Blocks the library's own pool handed out are kept by exact size when they are released and
// given out again to a request of the same device, stream and size: successive windows ask for
// the same sizes in the same order, and the CUDA pool took 0.1 ms and more to carve a block of
// a new size out of what it holds (2.8 ms per 66.8 M record window).  A block is reused on the
// stream it was released on only, so stream order protects work still queued on it.  Blocks
// that no request has taken during the lifetime of the last two handles go back to the pool.
struct CachedBlock {
  void *p;
  size_t bytes;
  int device;
  cudaStream_t stream;
  unsigned long long gen;
};
static std::mutex g_cache_guard;
static std::vector<CachedBlock> g_cache;
static unsigned long long g_cache_gen = 0;

static void *cache_take(int device, cudaStream_t stream, size_t bytes) {
  std::lock_guard<std::mutex> lock(g_cache_guard);
  for (size_t i = 0; i < g_cache.size(); i++)
    if (g_cache[i].bytes == bytes && g_cache[i].device == device && g_cache[i].stream == stream) {
      void *p = g_cache[i].p;
      g_cache[i] = g_cache.back();
      g_cache.pop_back();
      return p;
    }
  return nullptr;
}
static void cache_put(int device, cudaStream_t stream, void *p, size_t bytes) {
  try {
    std::lock_guard<std::mutex> lock(g_cache_guard);
    g_cache.push_back(CachedBlock{p, bytes, device, stream, g_cache_gen});
  } catch (...) {  // no host memory to remember it by
    cudaFreeAsync(p, stream);
  }
}
// Called when a handle goes away.  Invariant: a block enters the cache only once the work that used it
// is done (ta_dfree is reached behind the wait that ends a call, and what it is given for later behind
// the next one; ta_free synchronises the stream), so handing it back to the pool below cannot race with
// a kernel of the stream it was used on - cudaFree itself does not wait for a stream-ordered allocation.
static void cache_age() {
  bool first = true;
  for (void *p = nullptr;; cudaFree(p)) {  // the stream the block was used on may no longer exist
    std::lock_guard<std::mutex> lock(g_cache_guard);
    if (first) g_cache_gen++;
    first = false;
    size_t i = 0;
    while (i < g_cache.size() && g_cache[i].gen + 2 >= g_cache_gen) i++;
    if (i == g_cache.size()) return;
    p = g_cache[i].p;
    g_cache[i] = g_cache.back();
    g_cache.pop_back();
  }
}

void *ta_dalloc(ta_window *h, size_t bytes) {
  if (bytes == 0) bytes = 256;
  if (h->allocs.size() == h->allocs.capacity()) {  // host memory first: a block must not be lost for want of it
    std::lock_guard<std::mutex> lock(h->alloc_guard);
    h->alloc_bytes.reserve(2 * h->allocs.size() + 32);
    h->allocs.reserve(2 * h->allocs.size() + 32);
  }
  void *p = nullptr;
  if (h->env.alloc) {
    p = h->env.alloc(bytes, h->env.ctx);
  } else if (!(p = cache_take(h->device, h->stream, bytes))) {
    cudaMemPool_t pool = own_pool(h->device);
    cudaError_t e = pool ? cudaMallocFromPoolAsync(&p, bytes, pool, h->stream)
                         : cudaMallocAsync(&p, bytes, h->stream);
    if (e != cudaSuccess) {
      cudaGetLastError();
      p = nullptr;
    }
  }
  if (p) {
    std::lock_guard<std::mutex> lock(h->alloc_guard);
    h->allocs.push_back(p);
    h->alloc_bytes.push_back(bytes);
  }
  return p;
}

void *ta_zpool(ta_window *h, size_t bytes) {
  const size_t need = Carver::pad(bytes ? bytes : 1);
  if (h->zero_used + need > h->zero_bytes) return nullptr;
  void *p = h->zero_pool + h->zero_used;
  h->zero_used += need;
  return p;
}
void *ta_zalloc(ta_window *h, size_t bytes, ta_status *st) {
  *st = TA_OK;
  void *p = ta_zpool(h, bytes);
  if (p) return p;
  p = ta_dalloc(h, bytes);
  if (!p) {
    *st = TA_ERR_OOM;
  } else if (cudaMemsetAsync(p, 0, bytes, h->stream) != cudaSuccess) {
    h->last_cuda = cudaGetLastError();
    *st = TA_ERR_CUDA;
    ta_dfree(h, p);
    p = nullptr;
  }
  return p;
}

static void release_one(ta_window *h, void *p, size_t bytes) {
  if (h->env.alloc) {
    if (h->env.release) h->env.release(p, h->env.ctx);
  } else {
    cache_put(h->device, h->stream, p, bytes);
  }
}

void ta_dfree(ta_window *h, void *p) {
  if (!p) return;
  size_t bytes = 0;
  {
    std::lock_guard<std::mutex> lock(h->alloc_guard);
    size_t i = 0;
    while (i < h->allocs.size() && h->allocs[i] != p) i++;
    if (i == h->allocs.size()) return;
    bytes = h->alloc_bytes[i];
    h->allocs[i] = h->allocs.back();
    h->allocs.pop_back();
    h->alloc_bytes[i] = h->alloc_bytes.back();
    h->alloc_bytes.pop_back();
  }
  release_one(h, p, bytes);
}

// Page-locked staging blocks are expensive to create (a system call and a page-table update
// each), so up to TA_PIN_KEEP of them are kept for the life of the process and handed from handle to handle.
#define TA_PIN_KEEP 32
#define TA_PIN_BYTES (512u << 10)  // and 64 bytes behind them for the number of the last fetch
static std::mutex g_pin_guard;
static unsigned char *g_pin_free[TA_PIN_KEEP];
static int g_pins_idle = 0;
static unsigned char *pin_take() {
  {
    std::lock_guard<std::mutex> lock(g_pin_guard);
    if (g_pins_idle > 0) return g_pin_free[--g_pins_idle];
  }
  void *p = nullptr;
  if (cudaHostAlloc(&p, TA_PIN_BYTES + 64, cudaHostAllocPortable | cudaHostAllocMapped) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;  // the copies then go straight to their (pageable) destinations
  }
  return (unsigned char *)p;
}
static void pin_put(unsigned char *p) {
  if (!p) return;
  {
    std::lock_guard<std::mutex> lock(g_pin_guard);
    if (g_pins_idle < TA_PIN_KEEP) {
      g_pin_free[g_pins_idle++] = p;
      return;
    }
  }
  cudaFreeHost(p);
}

// Writes up to TA_FETCH_MAX device regions into the mapped staging block: one launch in place of
// one copy each (a copy costs some six microseconds of stream time, however small).  The last CTA
// to finish writes the number of the fetch behind the data, which the host waits for (seq 0: the
// fetch is not the last of its call and nobody waits).
#define TA_FETCH_MAX 16
#define TA_FETCH_BYTES (128u << 10)
#define TA_FETCH_STRIPE (8u << 10)  // bytes per CTA
struct FetchList {
  const void *src[TA_FETCH_MAX];
  unsigned off[TA_FETCH_MAX], bytes[TA_FETCH_MAX];
};
__global__ void __launch_bounds__(256) k_collect(FetchList f, int m, unsigned char *pin_dev, u32 *ticket, u32 seq,
                                                 volatile u32 *seq_word) {
  TA_PDL();
  const unsigned lo = blockIdx.x * TA_FETCH_STRIPE;
  for (int e = 0; e < m; e++) {
    const unsigned b = f.bytes[e];
    if (lo >= b) continue;
    const unsigned hi = min(b, lo + TA_FETCH_STRIPE);
    const unsigned char *s = (const unsigned char *)f.src[e];
    unsigned char *d = pin_dev + f.off[e];
    if ((((uintptr_t)s | (uintptr_t)b) & 7u) == 0) {
      for (unsigned i = lo / 8 + threadIdx.x; i < hi / 8; i += blockDim.x)
        reinterpret_cast<u64 *>(d)[i] = reinterpret_cast<const u64 *>(s)[i];
    } else {
      for (unsigned i = lo + threadIdx.x; i < hi; i += blockDim.x) d[i] = s[i];
    }
  }
  if (!seq) return;
  __syncthreads();
  if (threadIdx.x != 0) return;
  __threadfence_system();
  if (gridDim.x > 1 && atomicInc(ticket, gridDim.x - 1) != gridDim.x - 1) return;  // (wraps back to 0)
  __threadfence_system();
  *seq_word = seq;
}
static volatile u32 *seq_word(unsigned char *pin) { return (volatile u32 *)(pin + TA_PIN_BYTES); }
static u32 next_seq(ResultStage &o) { return ++o.seq ? o.seq : ++o.seq; }
static void stage_open(ResultStage &o) {
  o.pin = pin_take();
  o.pin_dev = nullptr;
  if (o.pin) {
    void *dp = nullptr;
    if (cudaHostGetDevicePointer(&dp, o.pin, 0) == cudaSuccess) o.pin_dev = (unsigned char *)dp;
    else cudaGetLastError();
  }
  o.used = 0;
  o.seq = o.tail_seq = 0;
}
static void stage_clear(ResultStage &o) {
  o.pending.clear();
  o.fetch.clear();
  o.copies.clear();
  o.tail_seq = 0;
  o.used = 0;
}
static void stage_queue(ResultStage &o, void *dst, const void *dev_src, size_t bytes) {
  if (bytes == 0) return;
  const size_t need = (bytes + 15) & ~(size_t)15;
  if (!o.pin || o.used + need > TA_PIN_BYTES) {
    o.copies.push_back(ResultStage::Copy{dst, dev_src, bytes});
    return;
  }
  if (o.pin_dev && bytes <= TA_FETCH_BYTES)
    o.fetch.push_back(ResultStage::Fetch{dev_src, (unsigned)o.used, (unsigned)bytes});
  else
    o.copies.push_back(ResultStage::Copy{o.pin + o.used, dev_src, bytes});
  o.pending.push_back(ResultStage::Pending{dst, o.used, bytes});
  o.used += need;
}
// (at most TA_FETCH_MAX regions a launch; the last launch writes the number)
static ta_status stage_collect(ta_window *h, ResultStage &o, u32 seq) {
  for (size_t first = 0; first < o.fetch.size(); first += TA_FETCH_MAX) {
    FetchList f;
    memset(&f, 0, sizeof(f));
    const bool last = o.fetch.size() - first <= TA_FETCH_MAX;
    const unsigned m = last ? (unsigned)(o.fetch.size() - first) : TA_FETCH_MAX;
    unsigned most = 1;
    for (unsigned i = 0; i < m; i++) {
      const ResultStage::Fetch &q = o.fetch[first + i];
      f.src[i] = q.src; f.off[i] = q.off; f.bytes[i] = q.bytes;
      most = q.bytes > most ? q.bytes : most;
    }
    ta_launch(k_collect, (most + TA_FETCH_STRIPE - 1) / TA_FETCH_STRIPE, 256, 0, h->stream, f, (int)m, o.pin_dev,
              (u32 *)&h->d_status[ST_TICKET], last ? seq : 0u, seq_word(o.pin_dev));
  }
  o.fetch.clear();
  TA_CHECK_CUDA(h, cudaGetLastError());
  return TA_OK;
}
static ta_status stage_wait(ta_window *h, ResultStage &o) {
  // real copies are done when the stream is, not when a kernel's word appears
  if (!o.copies.empty()) o.tail_seq = 0;
  for (const ResultStage::Copy &c : o.copies)
    TA_CHECK_CUDA(h, cudaMemcpyAsync(c.dst, c.src, c.bytes, cudaMemcpyDeviceToHost, h->stream));
  o.copies.clear();
  u32 seq = o.tail_seq;
  o.tail_seq = 0;
  if (!o.fetch.empty()) {
    seq = next_seq(o);
    *seq_word(o.pin) = 0;
    TA_TRY(stage_collect(h, o, seq));
  } else if (!seq) {
    TA_CHECK_CUDA(h, cudaStreamSynchronize(h->stream));
    return TA_OK;
  }
  volatile u32 *word = seq_word(o.pin);
  TA_WAIT_SEQ(*word, seq, h->stream);
  if (*word != seq) TA_CHECK_CUDA(h, cudaStreamSynchronize(h->stream));
  std::atomic_thread_fence(std::memory_order_acquire);
  return *word == seq ? TA_OK : TA_ERR_CUDA;
}
// one wait, then everything to its destination
static ta_status stage_deliver(ta_window *h, ResultStage &o) {
  const ta_status fs = stage_wait(h, o);
  if (fs == TA_OK)
    for (const ResultStage::Pending &q : o.pending) memcpy(q.dst, o.pin + q.off, q.bytes);
  stage_clear(o);
  return fs;
}

ta_status ta_queue_d2h(ta_window *h, void *dst, const void *dev_src, size_t bytes) {
  stage_queue(h->out, dst, dev_src, bytes);
  return TA_OK;
}
Tail ta_tail(ta_window *h, int64_t grid) {
  ResultStage &o = h->out;
  Tail t;
  if (!o.pin_dev || o.fetch.empty() || o.fetch.size() > TA_TAIL_MAX || !o.copies.empty() || grid > 1024) return t;
  for (const ResultStage::Fetch &f : o.fetch)
    if (f.bytes > 4096 || (f.bytes & 3u)) return t;
  for (size_t i = 0; i < o.fetch.size(); i++) {
    t.src[i] = o.fetch[i].src;
    t.off[i] = o.fetch[i].off;
    t.bytes[i] = o.fetch[i].bytes;
  }
  t.m = (int)o.fetch.size();
  o.fetch.clear();
  t.pin_dev = o.pin_dev;
  t.ticket = (u32 *)&h->d_status[ST_TICKET];
  t.seq = o.tail_seq = next_seq(o);
  t.seq_word = seq_word(o.pin_dev);
  *seq_word(o.pin) = 0;
  return t;
}
ta_status ta_sync_fetch(ta_window *h) {
  TA_TRY(stage_deliver(h, h->out));
  for (void *p : h->deferred) ta_dfree(h, p);
  h->deferred.clear();
  return TA_OK;
}

ta_status ta_read_status(ta_window *h, int32_t *w) {
  TA_TRY(ta_queue_d2h(h, w, h->d_status, ST_WORDS * sizeof(int32_t)));
  return ta_sync_fetch(h);
}

void ta_dfree_later(ta_window *h, void *p) {
  if (p) h->deferred.push_back(p);
}

// Start of every entry point: copies an earlier call queued and never collected (it returned
// early with an error) must not be delivered to destinations that no longer exist.
// Also makes the handle's device current (it stays current when the call returns).
static ta_status begin_call(ta_window *h) {
  stage_clear(h->out);
  if (cudaSetDevice(h->device) != cudaSuccess) {
    h->last_cuda = cudaGetLastError();
    return TA_ERR_CUDA;
  }
  return TA_OK;
}

// ---- test hooks: the poll limit of device-side waits, and a wait that nothing ends ----
static std::atomic<int> g_ta_spin_limit{0};  // 0 = TA_SPIN_LIMIT; copied into each new handle's status word

// One warp looks back from tile 1 at a tile-0 descriptor that nothing publishes.
__global__ void k_selftest_wait(u64 *state, int32_t *status) {
  TA_PDL();
  bool failed;
  tile_lookback<OpAdd>(state, 1, 1ull, OpAdd(), status, &failed);
  if (threadIdx.x == 0) status[ST_LONG_RUN] = failed ? 1 : 0;
}

// ---- instrumentation: launch counter and event pairs around the radix passes ----
std::atomic<long long> g_ta_launches{0};
int g_ta_profile = 0;
static std::vector<cudaEvent_t> g_prof_events;  // begin, end, begin, end, ...
static size_t g_prof_used = 0;
static double g_prof_bytes = 0;  // algorithmic bytes of the timed passes

void ta_profile_mark(cudaStream_t st, int begin, double bytes) {
  if (begin) g_prof_bytes += bytes;
  if (g_prof_used == g_prof_events.size()) {
    cudaEvent_t e;
    if (cudaEventCreate(&e) != cudaSuccess) return;
    g_prof_events.push_back(e);
  }
  cudaEventRecord(g_prof_events[g_prof_used++], st);
}

// What the library throws are failed allocations of host memory (its tables grow with the windows); none
// leaves an entry point.
template <class F>
static ta_status no_throw(F f) {
  try {
    return f();
  } catch (...) {
    return TA_ERR_OOM;
  }
}
template <class F>
static ta_status run_call(ta_window *h, F f) {
  return no_throw([&]() -> ta_status {
    TA_TRY(begin_call(h));
    return f();
  });
}

extern "C" {

// Instrumentation helpers (they carry no work).  ta_profile_enable(1) makes the
// library record a CUDA event pair around every radix-sort pass and forgets the
// pairs recorded so far; ta_profile_radix reads them back (synchronises the
// events): number of passes timed and their summed duration in milliseconds.
void ta_profile_enable(int32_t on) {
  g_ta_profile = on;
  g_prof_used = 0;
  g_prof_bytes = 0;
}
int32_t ta_profile_radix(int64_t *n_passes, double *total_ms, double *total_bytes) {
  int64_t n = 0;
  double ms = 0;
  for (size_t i = 0; i + 1 < g_prof_used; i += 2) {
    if (cudaEventSynchronize(g_prof_events[i + 1]) != cudaSuccess) return -1;
    float t = 0;
    if (cudaEventElapsedTime(&t, g_prof_events[i], g_prof_events[i + 1]) != cudaSuccess) return -1;
    ms += t;
    n++;
  }
  if (n_passes) *n_passes = n;
  if (total_ms) *total_ms = ms;
  if (total_bytes) *total_bytes = g_prof_bytes;
  return 0;
}
int64_t ta_launch_count(void) { return g_ta_launches.load(); }

void ta_set_spin_limit(int32_t polls) { g_ta_spin_limit.store(polls > 0 ? polls : 0); }

ta_status ta_inject_device_error(ta_window *h, ta_status code) {
  if (!h || !h->d_status || code <= TA_OK || code > TA_ERR_BAD_NESTING) return TA_ERR_INVALID_ARG;
  if (cudaSetDevice(h->device) != cudaSuccess) return TA_ERR_CUDA;
  const int32_t c = (int32_t)code;
  TA_CHECK_CUDA(h, cudaMemcpyAsync(h->d_status + ST_ERR, &c, sizeof(c), cudaMemcpyHostToDevice, h->stream));
  TA_CHECK_CUDA(h, cudaStreamSynchronize(h->stream));
  return TA_OK;
}

ta_status ta_selftest_wait_timeout(void *cuda_stream, int32_t polls) {
  if (polls < 1 || polls > (1 << 20)) return TA_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  unsigned char *buf = nullptr;
  if (cudaMallocAsync((void **)&buf, 512, st) != cudaSuccess) {
    cudaGetLastError();
    return TA_ERR_OOM;
  }
  u64 *state = (u64 *)buf;                    // two descriptors, both EMPTY
  int32_t *status = (int32_t *)(buf + 256);   // ST_WORDS words
  int32_t words[ST_WORDS];
  memset(words, 0, sizeof(words));
  words[ST_SPIN] = polls;
  cudaError_t e = cudaMemsetAsync(buf, 0, 512, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(status, words, sizeof(words), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) {
    ta_launch(k_selftest_wait, 1, 32, 0, st, state, status);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(words, status, sizeof(words), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  cudaFreeAsync(buf, st);
  if (e != cudaSuccess) return TA_ERR_CUDA;
  // the kernel must have come back by itself, with the error recorded and nothing published
  if (words[ST_LONG_RUN] != 1) return TA_ERR_CUDA;
  return (ta_status)words[ST_ERR];
}

const char *ta_strerror(ta_status s) {
  switch (s) {
    case TA_OK: return "ok";
    case TA_ERR_INVALID_ARG: return "invalid argument";
    case TA_ERR_OOM: return "device allocation failed";
    case TA_ERR_CUDA: return "CUDA runtime error";
    case TA_ERR_ORDER: return "entry point called before its prerequisites";
    case TA_ERR_TOO_LARGE: return "size limit exceeded";
    case TA_ERR_OVERFLOW: return "internal table overflow";
    case TA_ERR_TIMEOUT: return "bounded device-side wait gave up";
    case TA_ERR_DEPTH: return "operator nesting deeper than TA_MAX_DEPTH";
    case TA_ERR_BAD_NESTING: return "partially overlapping ranges on one host thread";
  }
  return "unknown status";
}

int32_t ta_version(void) { return 1; }

static ta_status load_impl(ta_window *h, const ta_event *events, int32_t on_device,
                           ta_load_summary *out_summary) {
  const int64_t n = h->n;
  const int W = h->W;
  cudaStream_t st = h->stream;
  // one device block: [off | t0 | t1 | misc], filled by the planning kernel (by a copy when there
  // are many windows), and everything that starts at zero, cleared by that kernel too: [status | load
  // summaries | digit histograms | triple table | communicator table | pool for the later calls]
  const size_t up_words = (size_t)(W + 1) + 2 * (size_t)W + 16;
  // the pool: kernel counts (4 bytes per record), the join's table (some 2), the sort's descriptors (1.3),
  // bitmaps, lane tables and a few aggregate tables; what does not fit is cleared by itself
  // records per window and triple slot, as long as a window's counters (32 KB) are small beside its words
  h->cnt_windows = W == 1 || (W <= 1024 && n / W >= 8192) ? W : 0;
  const size_t cnt_bytes = (size_t)(h->cnt_windows ? h->cnt_windows : 1) * TA_TRIPLE_SLOTS * 4;
  h->zero_used = 0;
  h->zero_bytes = n <= TA_ZERO_POOL_RECORDS ? Carver::pad((size_t)n * 16 + (3u << 20)) : 0;
  size_t bytes = Carver::pad(up_words * 8) + Carver::pad(ST_WORDS * 4) +
                 Carver::pad(sizeof(TripleTable)) + Carver::pad(sizeof(CommTable)) +
                 Carver::pad(W * sizeof(ta_load_summary)) + 2 * Carver::pad(10 * 256 * 4) +
                 Carver::pad(cnt_bytes) + h->zero_bytes + 256;
  void *b = ta_dalloc(h, bytes);
  if (!b) return TA_ERR_OOM;
  Carver c(b);
  int64_t *up = c.take<int64_t>(up_words);
  h->d_off = up;
  h->d_t0 = up + (W + 1);
  h->d_t1 = h->d_t0 + W;
  h->d_misc = h->d_t1 + W;
  h->d_bin_offset = c.take<u32>(10 * 256);
  h->d_triples = c.take<TripleTable>(1);  // (only its first part, the slots, has to be cleared)
  char *zero_begin = (char *)h->d_triples->slots;
  static_assert(offsetof(TripleTable, slots) + sizeof(h->d_triples->slots) == sizeof(TripleTable), "slots come last");
  h->d_status = c.take<int32_t>(ST_WORDS);
  h->d_load_sum = c.take<ta_load_summary>(W);
  h->d_hist = c.take<u32>(10 * 256);
  h->d_slot_cnt = c.take<u32>(cnt_bytes / 4);
  h->zero_pool = c.take<char>(h->zero_bytes);
  h->d_comms = c.take<CommTable>(1);
  char *zero_end = (char *)h->d_comms + sizeof(h->d_comms->slots);
  static_assert(offsetof(CommTable, slots) == 0, "slots come first");
  static_assert(offsetof(TripleTable, slots) % 16 == 0 && sizeof(h->d_comms->slots) % 16 == 0, "cleared in 16-byte words");
  h->d_keys = (u64 *)ta_dalloc(h, (size_t)(n > 0 ? n : 1) * 8);
  if (!h->d_keys) return TA_ERR_OOM;

  if (!on_device) {
    h->events_copy = ta_dalloc(h, (size_t)(n > 0 ? n : 1) * sizeof(ta_event));
    if (!h->events_copy) return TA_ERR_OOM;
    if (n > 0)
      TA_TRY(ta_upload(h, h->events_copy, events, (size_t)n * sizeof(ta_event)));
    h->events = (const ta_event *)h->events_copy;
  } else {
    h->events = events;
  }
  if (W > TA_PLAN_WINDOWS) {
    std::vector<int64_t> host(h->h_off);
    host.insert(host.end(), h->h_t0.begin(), h->h_t0.end());
    host.insert(host.end(), h->h_t1.begin(), h->h_t1.end());
    // a pageable source is staged by the runtime before the call returns
    TA_CHECK_CUDA(h, cudaMemcpyAsync(up, host.data(), host.size() * 8, cudaMemcpyHostToDevice, st));
  }

  int32_t words[ST_WORDS];
  int64_t misc[16];
  std::vector<ta_load_summary> sums(W);
  h->h_comm_sorted.assign(TA_COMMS_AT_ONCE, 0);
  TA_TRY(ta_queue_d2h(h, misc, h->d_misc, sizeof(misc)));
  TA_TRY(ta_queue_d2h(h, h->h_comm_sorted.data(), h->d_comms->sorted_id, TA_COMMS_AT_ONCE * sizeof(u64)));
  TA_TRY(ta_queue_d2h(h, words, h->d_status, sizeof(words)));
  TA_TRY(ta_queue_d2h(h, sums.data(), h->d_load_sum, W * sizeof(ta_load_summary)));
  TA_TRY(ta_launch_discover(h, zero_begin, (size_t)(zero_end - zero_begin), g_ta_spin_limit.load()));
  TA_TRY(ta_sync_fetch(h));
  if (words[ST_ERR]) return (ta_status)words[ST_ERR];
  h->n_triples = words[ST_N_TRIPLES];
  h->n_pids = words[ST_N_PIDS];
  h->min_name = misc[0];
  h->max_name = misc[1];
  h->max_dur = misc[2];
  h->min_seq = misc[3];
  h->max_seq = misc[4];
  h->n_coll = misc[5];
  h->n_launch = misc[8];
  if (h->tkeep < 0) h->tkeep = (int)misc[6];
  h->n_comms = words[ST_N_COMMS];
  h->h_comm_sorted.resize((size_t)h->n_comms);
  if (h->n_comms > TA_COMMS_AT_ONCE) {  // rarely: the rest of the communicator ids
    TA_TRY(ta_queue_d2h(h, h->h_comm_sorted.data(), h->d_comms->sorted_id, (size_t)h->n_comms * sizeof(u64)));
    TA_TRY(ta_sync_fetch(h));
  }
  h->n_valid = 0;
  for (int w = 0; w < W; w++) {
    ta_load_summary &s = sums[w];
    s.n_events = h->h_off[w + 1] - h->h_off[w];
    s.n_valid = s.n_events - s.n_bad_kind - s.n_bad_interval - s.n_out_of_window;
    h->n_valid += s.n_valid;
    if (out_summary) out_summary[w] = s;
  }
  h->has_dropped = h->n_valid < n ? 1 : 0;
  TA_TRY(ta_launch_load(h, true));
  h->stage |= 1;
  return TA_OK;
}

ta_status ta_load_window(const ta_env *env, const ta_event *events, int64_t n,
                         int32_t events_on_device, const int64_t *win_off, const int64_t *win_t0,
                         const int64_t *win_t1, int32_t W, ta_load_summary *out_summary,
                         ta_window **handle) {
  if (!handle) return TA_ERR_INVALID_ARG;
  *handle = nullptr;
  if (!env || n < 0 || W < 1 || !win_off || !win_t0 || !win_t1 || (n > 0 && !events))
    return TA_ERR_INVALID_ARG;
  if (n >= (1ll << 31)) return TA_ERR_TOO_LARGE;
  if ((env->alloc == nullptr) != (env->release == nullptr)) return TA_ERR_INVALID_ARG;
  if (win_off[0] != 0 || win_off[W] != n) return TA_ERR_INVALID_ARG;
  for (int w = 0; w < W; w++) {
    if (win_off[w + 1] < win_off[w]) return TA_ERR_INVALID_ARG;
    if (win_t0[w] >= win_t1[w]) return TA_ERR_INVALID_ARG;
    if ((uint64_t)win_t1[w] - (uint64_t)win_t0[w] >= (1ull << 40)) return TA_ERR_TOO_LARGE;
  }
  ta_window *h = new (std::nothrow) ta_window();
  if (!h) return TA_ERR_OOM;
  h->env = *env;
  h->stream = (cudaStream_t)env->cuda_stream;
  h->device = env->device;
  h->last_cuda = cudaSuccess;
  h->n = n;
  h->W = W;
  h->stage = 0;
  h->events = nullptr;
  h->events_copy = nullptr;
  h->d_keys = nullptr;
  h->prekeys = 0;
  h->attr_status = 0;
  h->n_names = 0;
  h->d_names = nullptr;
  h->d_name_rank = nullptr;
  h->d_name_of = nullptr;
  h->d_op_gap_ns = nullptr;
  h->d_on_path = nullptr;
  h->d_status = nullptr;
  h->zero_bytes = h->zero_used = 0;
  *handle = h;
  return no_throw([&]() -> ta_status {
    stage_open(h->out);
    h->h_off.assign(win_off, win_off + W + 1);
    h->h_t0.assign(win_t0, win_t0 + W);
    h->h_t1.assign(win_t1, win_t1 + W);
    TA_TRY(begin_call(h));
    return load_impl(h, events, events_on_device, out_summary);
  });
}

ta_status ta_sort_timeline(ta_window *h, ta_sort_result *out) {
  if (!h || !out) return TA_ERR_INVALID_ARG;
  if (!(h->stage & 1) || (h->stage & 2)) return TA_ERR_ORDER;
  return run_call(h, [&]() -> ta_status {
    TA_TRY(ta_run_sort_timeline(h));
    h->stage |= 2;
    *out = h->sorted;
    return TA_OK;
  });
}

ta_status ta_correlate_launches(ta_window *h, ta_join_result *out, ta_join_summary *out_summary) {
  if (!h || !out) return TA_ERR_INVALID_ARG;
  if (!(h->stage & 2) || (h->stage & 4)) return TA_ERR_ORDER;
  return run_call(h, [&]() -> ta_status {
    TA_TRY(ta_run_correlate(h, out_summary));
    h->stage |= 4;
    *out = h->join;
    return TA_OK;
  });
}

ta_status ta_attribute_operators(ta_window *h, ta_attr_result *out, ta_attr_summary *out_summary) {
  if (!h || !out) return TA_ERR_INVALID_ARG;
  if (!(h->stage & 4) || (h->stage & 8)) return TA_ERR_ORDER;
  return run_call(h, [&]() -> ta_status {
    ta_status s = ta_run_attribute(h, out_summary);
    if (s != TA_OK && s != TA_ERR_DEPTH && s != TA_ERR_BAD_NESTING) return s;
    h->stage |= 8;
    h->attr_status = (int)s;
    *out = h->attr;
    return s;
  });
}

ta_status ta_stream_gaps(ta_window *h, int64_t min_gap_ns, ta_gap_result *out) {
  if (!h || !out) return TA_ERR_INVALID_ARG;
  if (!(h->stage & 2)) return TA_ERR_ORDER;
  return run_call(h, [&] { return ta_run_gaps(h, min_gap_ns, out); });
}

ta_status ta_aggregate_ops(ta_window *h, uint32_t kind_mask, int32_t value_sel, ta_agg_result *out) {
  if (!h || !out) return TA_ERR_INVALID_ARG;
  if (value_sel < 0 || value_sel > 3) return TA_ERR_INVALID_ARG;
  if ((value_sel == 1 || value_sel == 2) && kind_mask != (1u << TA_KIND_OP)) return TA_ERR_INVALID_ARG;
  if (!(h->stage & 2)) return TA_ERR_ORDER;
  if (value_sel == 1 && (!(h->stage & 8) || h->attr_status != 0)) return TA_ERR_ORDER;
  if (value_sel == 2 && !h->d_op_gap_ns) return TA_ERR_ORDER;
  if (value_sel == 3 && !h->d_on_path) return TA_ERR_ORDER;
  return run_call(h, [&] { return ta_run_aggregate(h, kind_mask, value_sel, out); });
}

ta_status ta_match_collectives(ta_window *h, const ta_comm_size *sizes, int32_t n_comms,
                               ta_coll_result *out) {
  if (!h || !out || n_comms < 0 || (n_comms > 0 && !sizes)) return TA_ERR_INVALID_ARG;
  if (!(h->stage & 2)) return TA_ERR_ORDER;
  return run_call(h, [&] { return ta_run_collectives(h, sizes, n_comms, out); });
}

ta_status ta_rollup_operators(ta_window *h, ta_rollup_result *out, ta_rollup_summary *out_summary) {
  if (!h || !out || !out_summary) return TA_ERR_INVALID_ARG;
  if (!(h->stage & 8) || h->attr_status != 0) return TA_ERR_ORDER;
  return run_call(h, [&] { return ta_run_rollup(h, out, out_summary); });
}

ta_status ta_operator_sol(ta_window *h, const double *flops, const double *bytes,
                          int32_t counts_on_device, double peak_flops, double peak_bw,
                          ta_sol_result *out, ta_sol_summary *out_summary) {
  if (!h || !out || !out_summary || (h->n > 0 && (!flops || !bytes))) return TA_ERR_INVALID_ARG;
  if (!(peak_flops > 0.0) || !(peak_bw > 0.0)) return TA_ERR_INVALID_ARG;
  if (!(h->stage & 8) || h->attr_status != 0) return TA_ERR_ORDER;
  return run_call(h, [&] { return ta_run_sol(h, flops, bytes, counts_on_device, peak_flops, peak_bw, out, out_summary); });
}

ta_status ta_blame_gaps(ta_window *h, const ta_gap_result *gaps, ta_blame_result *out,
                        ta_blame_summary *out_summary) {
  if (!h || !gaps || !out || !out_summary) return TA_ERR_INVALID_ARG;
  if (gaps->n_long_gaps < 0 || (gaps->n_long_gaps > 0 && !gaps->long_gaps)) return TA_ERR_INVALID_ARG;
  if (!(h->stage & 4)) return TA_ERR_ORDER;
  return run_call(h, [&] { return ta_run_blame(h, gaps, out, out_summary); });
}

ta_status ta_critical_path(ta_window *h, ta_critpath_result *out, ta_critpath_summary *out_summary) {
  if (!h || !out || !out_summary) return TA_ERR_INVALID_ARG;
  if (!(h->stage & 4)) return TA_ERR_ORDER;
  return run_call(h, [&] { return ta_run_critpath(h, out, out_summary); });
}

ta_status ta_device_overlap(ta_window *h, ta_overlap_result *out) {
  if (!h || !out) return TA_ERR_INVALID_ARG;
  if (!(h->stage & 2)) return TA_ERR_ORDER;
  return run_call(h, [&] { return ta_run_overlap(h, out); });
}

ta_status ta_fetch(ta_window *h, int32_t count, void *const *dst, const void *const *src, const uint64_t *bytes) {
  if (!h || count < 0 || (count > 0 && (!dst || !src || !bytes))) return TA_ERR_INVALID_ARG;
  if (cudaSetDevice(h->device) != cudaSuccess) {
    cudaGetLastError();
    return TA_ERR_CUDA;
  }
  // a block of its own: results are read while another thread is in a call on the handle, or reads as well
  ResultStage o;
  stage_open(o);
  const ta_status s = no_throw([&]() -> ta_status {
    for (int32_t i = 0; i < count; i++) stage_queue(o, dst[i], src[i], (size_t)bytes[i]);
    return stage_deliver(h, o);
  });
  if (s != TA_OK) cudaStreamSynchronize(h->stream);  // nothing queued may write to the block any more
  pin_put(o.pin);
  return s;
}

ta_status ta_block_of(ta_window *h, const void *p, void **base, uint64_t *bytes) {
  if (!h || !base || !bytes) return TA_ERR_INVALID_ARG;
  std::lock_guard<std::mutex> lock(h->alloc_guard);
  for (size_t i = 0; i < h->allocs.size(); i++) {
    const char *b = (const char *)h->allocs[i];
    if ((const char *)p >= b && (const char *)p < b + h->alloc_bytes[i]) {
      *base = h->allocs[i];
      *bytes = h->alloc_bytes[i];
      return TA_OK;
    }
  }
  return TA_ERR_INVALID_ARG;
}

// ---- a chunk of the caller's memory handed out piece by piece ----
struct ta_chunk {
  char *base;
  size_t bytes;
  void *(*alloc)(size_t, void *);
  void (*release)(void *, void *);
  void *ctx;
  struct Piece { size_t off, bytes; bool used; };
  std::vector<Piece> pieces;  // in address order, covering the chunk; free neighbours are merged
};
ta_chunk *ta_chunk_open(void *base, uint64_t bytes, void *(*alloc)(size_t, void *), void (*release)(void *, void *),
                        void *ctx) {
  if (!base || !alloc || !release) return nullptr;
  ta_chunk *c = new (std::nothrow) ta_chunk();
  if (!c) return nullptr;
  // pieces are as aligned as ta_env asks for, whatever the block is
  const size_t skip = (size_t)(-(uintptr_t)base & 255u);
  c->base = (char *)base + skip;
  c->bytes = bytes > skip ? (size_t)(bytes - skip) & ~(size_t)255 : 0;
  c->alloc = alloc;
  c->release = release;
  c->ctx = ctx;
  try {
    c->pieces.push_back(ta_chunk::Piece{0, c->bytes, false});
  } catch (...) {
    delete c;
    return nullptr;
  }
  return c;
}
void ta_chunk_close(ta_chunk *c) { delete c; }
void *ta_chunk_alloc(size_t bytes, void *chunk) {
  ta_chunk *c = (ta_chunk *)chunk;
  const size_t need = Carver::pad(bytes ? bytes : 1);
  size_t best = c->pieces.size();
  for (size_t i = 0; i < c->pieces.size(); i++)
    if (!c->pieces[i].used && c->pieces[i].bytes >= need &&
        (best == c->pieces.size() || c->pieces[i].bytes < c->pieces[best].bytes))
      best = i;
  if (best == c->pieces.size()) return c->alloc(bytes, c->ctx);
  const size_t off = c->pieces[best].off, rest = c->pieces[best].bytes - need;
  if (rest) {
    try {
      c->pieces.insert(c->pieces.begin() + best + 1, ta_chunk::Piece{off + need, rest, false});
    } catch (...) {  // no host memory to write the split down: the chunk stays as it is
      return c->alloc(bytes, c->ctx);
    }
  }
  c->pieces[best].bytes = need;
  c->pieces[best].used = true;
  return c->base + off;
}
void ta_chunk_release(void *ptr, void *chunk) {
  ta_chunk *c = (ta_chunk *)chunk;
  if ((char *)ptr < c->base || (char *)ptr >= c->base + c->bytes) {
    c->release(ptr, c->ctx);
    return;
  }
  const size_t off = (size_t)((char *)ptr - c->base);
  for (size_t i = 0; i < c->pieces.size(); i++) {
    if (c->pieces[i].off != off || !c->pieces[i].used) continue;
    c->pieces[i].used = false;
    if (i + 1 < c->pieces.size() && !c->pieces[i + 1].used) {
      c->pieces[i].bytes += c->pieces[i + 1].bytes;
      c->pieces.erase(c->pieces.begin() + i + 1);
    }
    if (i > 0 && !c->pieces[i - 1].used) {
      c->pieces[i - 1].bytes += c->pieces[i].bytes;
      c->pieces.erase(c->pieces.begin() + i);
    }
    return;
  }
}

void ta_free(ta_window *h) {
  if (!h) return;
  cudaSetDevice(h->device);
  cudaStreamSynchronize(h->stream);
  for (size_t i = 0; i < h->allocs.size(); i++) release_one(h, h->allocs[i], h->alloc_bytes[i]);
  h->allocs.clear();
  h->alloc_bytes.clear();
  pin_put(h->out.pin);
  const bool own = !h->env.alloc;
  delete h;
  if (own) cache_age();
  ta_upload_age();
}

}  // extern "C"
