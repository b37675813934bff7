// Host records to the device.  Page-locked memory is copied as it is.  Pageable memory (a file mapped
// or read by the caller, a numpy array) the driver copies through a staging buffer of its own with one
// thread, at 11 to 20 GB/s; here several threads copy pieces into a ring of page-locked buffers, each
// of which is on its way to the device as soon as it is full.  Bound by the host's memory
// bandwidth or the link (52 GB/s), whichever is less: 42 MB take 3.9 ms through the driver, 2.0 ms
// with memcpy into the buffers, 1.06 ms with streaming stores (0.77 from page-locked memory).
#include <emmintrin.h>

#include <algorithm>
#include <cstring>
#include <mutex>
#include <thread>

#include "ta_internal.cuh"

#define UP_PIECE (1u << 20)
#define UP_PIECES 24
#define UP_THREADS 6
#define UP_MIN (4u << 20)  // below this the threads cost more than they save
#define UP_RINGS 4         // rings (24 MB each) per device at most: the link is shared by more uploads than that anyway
#define UP_DEVICES 64

namespace {
struct Ring {
  unsigned char *buf;
  cudaEvent_t ev[UP_PIECES];
  bool used[UP_PIECES];  // an event of an earlier upload is recorded
  int device;
  unsigned long long last_used;  // number of the handle that used it last
};
std::mutex g_ring_guard;
Ring *g_idle[UP_DEVICES][UP_RINGS];  // an upload takes one out and puts it back
int g_made[UP_DEVICES];              // idle ones and those in use
unsigned long long g_handles = 0;

void ring_free(Ring *r) {
  for (int i = 0; i < UP_PIECES; i++)
    if (r->ev[i]) cudaEventDestroy(r->ev[i]);
  if (r->buf) cudaFreeHost(r->buf);
  delete r;
}
Ring *ring_make(int device) {
  Ring *r = new (std::nothrow) Ring();
  if (!r) return nullptr;
  r->device = device;
  void *p = nullptr;
  bool ok = cudaHostAlloc(&p, (size_t)UP_PIECE * UP_PIECES, cudaHostAllocPortable) == cudaSuccess;
  r->buf = (unsigned char *)p;
  for (int i = 0; i < UP_PIECES && ok; i++)
    if (cudaEventCreateWithFlags(&r->ev[i], cudaEventDisableTiming) != cudaSuccess) {
      r->ev[i] = nullptr;
      ok = false;
    }
  if (ok) return r;
  cudaGetLastError();
  ring_free(r);
  return nullptr;
}
// null: as many as there may be are in use, or there is no memory for one
Ring *ring_take(int device) {
  if (device < 0 || device >= UP_DEVICES) return nullptr;
  {
    std::lock_guard<std::mutex> lock(g_ring_guard);
    for (Ring *&idle : g_idle[device])
      if (idle) {
        Ring *r = idle;
        idle = nullptr;
        return r;
      }
    if (g_made[device] == UP_RINGS) return nullptr;
    g_made[device]++;
  }
  Ring *r = ring_make(device);
  if (!r) {
    std::lock_guard<std::mutex> lock(g_ring_guard);
    g_made[device]--;
  }
  return r;
}
void ring_put(Ring *r) {
  std::lock_guard<std::mutex> lock(g_ring_guard);
  r->last_used = g_handles;
  for (Ring *&idle : g_idle[r->device])
    if (!idle) {
      idle = r;
      return;
    }
}
}  // namespace

// Copies a piece past the caches: the device then reads it from memory.  Lines that are still dirty in
// some core's cache have to be snooped out of it one by one, which held the link at half its rate.
static void copy_piece(unsigned char *dst /* 64-byte aligned */, const unsigned char *src, size_t len) {
  size_t i = 0;
  for (; i + 64 <= len; i += 64) {
    const __m128i a = _mm_loadu_si128((const __m128i *)(src + i)), b = _mm_loadu_si128((const __m128i *)(src + i + 16));
    const __m128i c = _mm_loadu_si128((const __m128i *)(src + i + 32)), d = _mm_loadu_si128((const __m128i *)(src + i + 48));
    _mm_stream_si128((__m128i *)(dst + i), a);
    _mm_stream_si128((__m128i *)(dst + i + 16), b);
    _mm_stream_si128((__m128i *)(dst + i + 32), c);
    _mm_stream_si128((__m128i *)(dst + i + 48), d);
  }
  if (i < len) memcpy(dst + i, src + i, len - i);
  _mm_sfence();
}

// Rings no upload has asked for during the lifetime of the last 64 handles are given back.
void ta_upload_age() {
  Ring *out[UP_RINGS];
  int n = 0;
  {
    std::lock_guard<std::mutex> lock(g_ring_guard);
    g_handles++;
    for (int d = 0; d < UP_DEVICES && n == 0; d++)  // (of one device at a time)
      for (Ring *&idle : g_idle[d])
        if (idle && idle->last_used + 64 < g_handles) {
          out[n++] = idle;
          idle = nullptr;
          g_made[d]--;
        }
  }
  for (int i = 0; i < n; i++) ring_free(out[i]);
}

ta_status ta_upload(ta_window *h, void *dst, const void *src, size_t bytes) {
  cudaPointerAttributes at;
  memset(&at, 0, sizeof(at));
  const bool known = cudaPointerGetAttributes(&at, src) == cudaSuccess;
  if (!known) cudaGetLastError();
  Ring *r = nullptr;
  if (bytes >= UP_MIN && known && at.type == cudaMemoryTypeUnregistered) r = ring_take(h->device);
  if (!r) {
    TA_CHECK_CUDA(h, cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, h->stream));
    return TA_OK;
  }
  const size_t pieces = (bytes + UP_PIECE - 1) / UP_PIECE;
  std::atomic<size_t> next{0};
  std::atomic<int> failed{0};
  std::atomic<size_t> issued[UP_PIECES];  // 1 + last piece sent from the buffer
  for (int i = 0; i < UP_PIECES; i++) issued[i].store(0);
  auto work = [&]() {
    if (cudaSetDevice(h->device) != cudaSuccess) { failed.store(1); return; }
    for (;;) {
      const size_t c = next.fetch_add(1);
      if (c >= pieces || failed.load()) return;
      const int b = (int)(c % UP_PIECES);
      // the buffer's piece before has been sent off (pieces are drawn in order, so some thread is at
      // it or done with it), and has arrived
      while (c >= UP_PIECES && issued[b].load(std::memory_order_acquire) != c - UP_PIECES + 1)
        if (failed.load()) return;
      if ((c >= UP_PIECES || r->used[b]) && cudaEventSynchronize(r->ev[b]) != cudaSuccess) { failed.store(1); return; }
      const size_t off = c * (size_t)UP_PIECE, len = std::min((size_t)UP_PIECE, bytes - off);
      unsigned char *buf = r->buf + (size_t)b * UP_PIECE;
      copy_piece(buf, (const unsigned char *)src + off, len);
      if (cudaMemcpyAsync((unsigned char *)dst + off, buf, len, cudaMemcpyHostToDevice, h->stream) != cudaSuccess ||
          cudaEventRecord(r->ev[b], h->stream) != cudaSuccess) {
        failed.store(1);
        return;
      }
      issued[b].store(c + 1, std::memory_order_release);
    }
  };
  {
    // half of the host's cores at most, a thread per four pieces at most
    size_t threads = std::max<size_t>(1, std::min<size_t>(UP_THREADS, std::thread::hardware_concurrency() / 2));
    threads = std::min(threads, (pieces + 3) / 4);
    std::thread others[UP_THREADS];
    for (size_t t = 1; t < threads; t++) {
      try {
        others[t] = std::thread(work);
      } catch (...) {  // no more threads: those there are do the work
        break;
      }
    }
    work();
    for (std::thread &t : others)
      if (t.joinable()) t.join();
  }
  for (int i = 0; i < UP_PIECES; i++) r->used[i] = r->used[i] || issued[i].load() != 0;
  if (failed.load()) {
    h->last_cuda = cudaGetLastError();
    cudaStreamSynchronize(h->stream);  // what has been sent off still reads the buffers
  }
  ring_put(r);
  return failed.load() ? TA_ERR_CUDA : TA_OK;
}
