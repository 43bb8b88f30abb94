// Device buffers of packed handles, kept from a released handle for the next
// one on the same stream.
//
// A mask-training step packs, uses and releases a handle per layer.  With
// cudaMalloc (31 us each on this GPU) and cudaFree (28-59 us, and it waits for
// the whole device) for a handle's nine buffers, an 11008 x 4096 step spent
// half of its 0.93 ms there.
//
// Reuse is ordered by the stream: a buffer released by a handle that was used
// on one stream only (its gs_pack stream) may be handed to a later gs_pack on
// that stream without waiting, because everything the next owner queues runs
// after what the last one queued.  Streams are told apart by cudaStreamGetId,
// which is never reused, unlike the address of a destroyed stream.  A handle
// that was also used on another stream, or inside a graph capture (whose
// replays may run anywhere), gives its buffers to cudaFree, which waits for
// the device.
//
// What is kept is bounded (1 / 128 of the device's memory, oldest released
// first).  It goes back to the device when kPoolMaxAge other buffers have been
// taken or released since, when any allocation of the library finds the device
// full, and when the caller asks (gs_trim).  A program that neither packs nor
// releases handles any more keeps it until then.
#include "gs_common.cuh"

#include <mutex>

namespace gs {
namespace {

struct Idle {
  PoolBuf buf;
  PoolTag tag;
  uint64_t since;   // g_tick at its release
};

constexpr int kMaxIdle = 256;
constexpr uint64_t kPoolMaxAge = 8192;   // a handle takes and releases about nine

std::mutex g_pool_mu;
Idle g_idle[kMaxIdle];   // oldest first
int g_n_idle = 0;
size_t g_idle_bytes = 0;
uint64_t g_tick = 0;     // buffers taken and released so far

size_t idle_limit() {
  static const size_t limit = []() {
    size_t free_b = 0, total = 0;
    return cudaMemGetInfo(&free_b, &total) == cudaSuccess ? total / 128 : size_t(1) << 28;
  }();
  return limit;
}

// Allocation sizes: powers of two up to 1 MiB, then steps of at most 1 / 32 of
// the size, so that layers re-packed with another mask of the same density
// find each other's buffers.
size_t round_size(size_t b) {
  size_t s = 512;
  if (b <= (size_t(1) << 20)) {
    while (s < b) s <<= 1;
    return s;
  }
  size_t top = size_t(1) << 20;
  while (top * 2 <= b) top *= 2;
  const size_t step = top / 32;
  return (b + step - 1) / step * step;
}

bool same(const PoolTag& a, const PoolTag& b) {
  return a.valid && b.valid && a.device == b.device && a.stream_id == b.stream_id;
}

void drop(int i) {   // g_pool_mu held
  g_idle_bytes -= g_idle[i].buf.bytes;
  for (int k = i + 1; k < g_n_idle; ++k) g_idle[k - 1] = g_idle[k];
  --g_n_idle;
}

void free_on(int device, void* ptr) {
  int cur = -1;
  cudaGetDevice(&cur);
  if (cur != device) cudaSetDevice(device);
  cudaFree(ptr);
  if (cur >= 0 && cur != device) cudaSetDevice(cur);
}

// cudaFree of the oldest idle buffer that `which` asks for; false when there is none
template <class F>
bool release_oldest(F which) {
  Idle out;
  {
    std::lock_guard<std::mutex> lk(g_pool_mu);
    if (g_n_idle == 0 || !which()) return false;
    out = g_idle[0];
    drop(0);
  }
  free_on(out.tag.device, out.buf.ptr);
  return true;
}

void release_aged() {
  while (release_oldest([]() { return g_tick - g_idle[0].since > kPoolMaxAge; })) {
  }
}

}  // namespace

void pool_trim() {
  while (release_oldest([]() { return true; })) {
  }
}

cudaError_t device_malloc(void** ptr, size_t bytes) {
  *ptr = nullptr;
  cudaError_t e = cudaMalloc(ptr, bytes);
  if (e == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    pool_trim();
    e = cudaMalloc(ptr, bytes);
  }
  if (e != cudaSuccess) *ptr = nullptr;
  return e;
}

PoolTag pool_tag(int device, cudaStream_t s) {
  PoolTag t{device, false, 0};
  unsigned long long id = 0;
  if (cudaStreamGetId(s, &id) == cudaSuccess) {
    t.stream_id = id;
    t.valid = true;
  } else {
    cudaGetLastError();
  }
  return t;
}

cudaError_t pool_take(PoolBuf* buf, size_t bytes, const PoolTag& tag) {
  *buf = PoolBuf{nullptr, 0};
  const size_t want = round_size(bytes);
  {
    std::lock_guard<std::mutex> lk(g_pool_mu);
    ++g_tick;
    int best = -1;
    for (int i = 0; i < g_n_idle; ++i)
      if (same(g_idle[i].tag, tag) && g_idle[i].buf.bytes >= want && g_idle[i].buf.bytes - want <= want / 8 &&
          (best < 0 || g_idle[i].buf.bytes < g_idle[best].buf.bytes))
        best = i;
    if (best >= 0) {
      *buf = g_idle[best].buf;
      drop(best);
      return cudaSuccess;
    }
  }
  release_aged();
  void* ptr = nullptr;
  const cudaError_t e = device_malloc(&ptr, want);
  if (e == cudaSuccess) *buf = PoolBuf{ptr, want};
  return e;
}

void pool_give(const PoolBuf& buf, const PoolTag& tag) {
  if (!buf.ptr) return;
  bool kept = false;
  if (tag.valid && buf.bytes <= idle_limit()) {
    while (release_oldest([&]() { return g_n_idle == kMaxIdle || g_idle_bytes + buf.bytes > idle_limit(); })) {
    }
    std::lock_guard<std::mutex> lk(g_pool_mu);
    ++g_tick;
    if (g_n_idle < kMaxIdle) {
      g_idle[g_n_idle++] = Idle{buf, tag, g_tick};
      g_idle_bytes += buf.bytes;
      kept = true;
    }
  }
  if (!kept) free_on(tag.device, buf.ptr);
  release_aged();
}

}  // namespace gs
