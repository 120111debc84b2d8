// Device memory the library takes for itself: what a handle keeps (plans, split pointers) and the
// scratch of single calls.  It comes from one stream-ordered pool per device, because cudaMalloc and
// cudaFree cost 0.1 to 3 ms each (they map and unmap memory and wait for the device), more than the
// whole ingest of a small graph.
//
// The pool keeps at most kKeepInUse unused bytes while a handle is alive and kKeepIdle after the
// last one is gone.  What a destroyed handle held may still be read by kernels queued on any stream:
// it waits in a short list until the library next has the device idle (dg_graph_create waits for it
// anyway), or until the list reaches kMaxPending bytes.  Everything here is safe to call from several
// threads.
#include <mutex>

#include "dg_internal.cuh"

namespace dg {
namespace {

constexpr int kMaxDevices = 64;
constexpr size_t kKeepInUse = (size_t)4 << 30;
constexpr size_t kKeepIdle = (size_t)32 << 20;
constexpr int kMaxPendingBlocks = 64;
constexpr size_t kMaxPending = kKeepIdle;
constexpr int kPinnedWords = 128;  // one page

struct DevicePool {
  cudaMemPool_t pool = nullptr;
  int handles = 0;
  void* pending[kMaxPendingBlocks];
  int pending_count = 0;
  size_t pending_bytes = 0;
};

std::mutex g_mutex;
DevicePool g_pools[kMaxDevices];
// one page of host memory the device writes counters into, for the life of the process
HostCounters* g_pinned = nullptr;
enum : uint8_t { kWordFree = 0, kWordUsed = 1, kWordPending = 2 };  // pending: a copy may be on its way
uint8_t g_word_state[kPinnedWords];
uint8_t g_word_device[kPinnedWords];

// the device must be idle with respect to everything that is pending on it
void release_pending(DevicePool& d) {
  for (int i = 0; i < d.pending_count; ++i) cudaFreeAsync(d.pending[i], 0);
  d.pending_count = 0;
  d.pending_bytes = 0;
  const int device = (int)(&d - g_pools);
  for (int i = 0; i < kPinnedWords; ++i)
    if (g_word_state[i] == kWordPending && g_word_device[i] == device) g_word_state[i] = kWordFree;
}

cudaError_t keep(DevicePool& d, size_t bytes) {
  uint64_t v = bytes;
  return cudaMemPoolSetAttribute(d.pool, cudaMemPoolAttrReleaseThreshold, &v);
}

}  // namespace

cudaError_t pool_open(int device) {
  if (device < 0 || device >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_mutex);
  DevicePool& d = g_pools[device];
  if (!d.pool) {
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = device;
    if (cudaError_t e = cudaMemPoolCreate(&d.pool, &props)) {
      d.pool = nullptr;
      return e;
    }
  }
  if (d.handles == 0)
    if (cudaError_t e = keep(d, kKeepInUse)) return e;
  ++d.handles;
  return cudaSuccess;
}

void pool_close(int device) {
  std::lock_guard<std::mutex> lock(g_mutex);
  DevicePool& d = g_pools[device];
  if (--d.handles == 0) {
    keep(d, kKeepIdle);
    uint64_t reserved = 0;
    cudaMemPoolGetAttribute(d.pool, cudaMemPoolAttrReservedMemCurrent, &reserved);
    if (reserved > kKeepIdle) {
      cudaDeviceSynchronize();
      release_pending(d);
      cudaStreamSynchronize(0);
      cudaMemPoolTrimTo(d.pool, kKeepIdle);
    }
  }
}

void pool_device_is_idle(int device) {
  std::lock_guard<std::mutex> lock(g_mutex);
  release_pending(g_pools[device]);
}

cudaError_t pool_alloc(int device, size_t bytes, cudaStream_t s, void** out) {
  *out = nullptr;
  const cudaError_t e = cudaMallocFromPoolAsync(out, bytes ? bytes : 256, g_pools[device].pool, s);
  if (e != cudaSuccess) (void)cudaGetLastError();
  return e;
}

void pool_free(void* p, cudaStream_t s) {
  if (p) cudaFreeAsync(p, s);
}

void pool_retire(int device, void* p, size_t bytes) {
  if (!p) return;
  std::lock_guard<std::mutex> lock(g_mutex);
  DevicePool& d = g_pools[device];
  if (d.pending_count == kMaxPendingBlocks || d.pending_bytes + bytes > kMaxPending) {
    cudaDeviceSynchronize();
    release_pending(d);
    cudaFreeAsync(p, 0);
    return;
  }
  d.pending[d.pending_count++] = p;
  d.pending_bytes += bytes;
}

cudaError_t pinned_counters(int device, HostCounters** out) {
  std::lock_guard<std::mutex> lock(g_mutex);
  if (!g_pinned)
    if (cudaError_t e = cudaHostAlloc(&g_pinned, kPinnedWords * sizeof(HostCounters), cudaHostAllocPortable)) {
      g_pinned = nullptr;
      return e;
    }
  for (int i = 0; i < kPinnedWords; ++i) {
    if (g_word_state[i] != kWordFree) continue;
    g_word_state[i] = kWordUsed;
    g_word_device[i] = (uint8_t)device;
    *out = g_pinned + i;
    return cudaSuccess;
  }
  return cudaHostAlloc(out, sizeof(HostCounters), cudaHostAllocPortable);  // more handles than words
}

void pinned_counters_retire(HostCounters* p) {
  if (!p) return;
  std::lock_guard<std::mutex> lock(g_mutex);
  if (p >= g_pinned && p < g_pinned + kPinnedWords) {
    g_word_state[p - g_pinned] = kWordPending;
  } else {
    cudaDeviceSynchronize();
    cudaFreeHost(p);
  }
}

}  // namespace dg
