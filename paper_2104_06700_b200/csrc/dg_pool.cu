// Device memory the library takes for itself: what a handle keeps (plans, split pointers) and the
// scratch of single calls.  It comes from one stream-ordered pool per device, because cudaMalloc and
// cudaFree cost 0.1 to 3 ms each (they map and unmap memory and wait for the device), more than the
// whole ingest of a small graph.
//
// The pool keeps at most kKeepInUse unused bytes while a handle is alive and kKeepIdle after the
// last one is gone.  What a destroyed handle held may still be read by kernels queued on any stream:
// it waits on a list until the library next waits for the device (dg_graph_create does anyway), or
// until the list reaches kMaxPending bytes.  A wait frees what was on the list before it began and
// nothing that another thread adds meanwhile.  Everything here is safe to call from several threads.
#include <stdlib.h>

#include <mutex>

#include "dg_internal.cuh"

namespace dg {
namespace {

constexpr int kMaxDevices = 64;
constexpr size_t kKeepInUse = (size_t)4 << 30;
constexpr size_t kKeepIdle = (size_t)32 << 20;
constexpr size_t kMaxPending = kKeepIdle;
constexpr int kPinnedWords = 72;  // one page

// A device block, or a handle's pinned counters, that queued work may still use.
struct Retired {
  Retired* next;
  void* block;
  size_t bytes;
  HostCounters* counters;
};

struct DevicePool {
  cudaMemPool_t pool = nullptr;
  int handles = 0;
  Retired* pending = nullptr;
  size_t pending_bytes = 0;
};

std::mutex g_mutex;
DevicePool g_pools[kMaxDevices];
// one page of host memory the device writes counters into, for the life of the process
HostCounters* g_pinned = nullptr;
bool g_word_used[kPinnedWords];

bool in_page(const HostCounters* p) { return g_pinned && p >= g_pinned && p < g_pinned + kPinnedWords; }

cudaError_t keep(DevicePool& d, size_t bytes) {
  uint64_t v = bytes;
  return cudaMemPoolSetAttribute(d.pool, cudaMemPoolAttrReleaseThreshold, &v);
}

// No work uses it any more; its device is current.
void release(const Retired& r) {
  if (r.block) cudaFreeAsync(r.block, 0);
  if (!r.counters) return;
  if (in_page(r.counters)) {
    std::lock_guard<std::mutex> lock(g_mutex);
    g_word_used[r.counters - g_pinned] = false;
  } else {
    cudaFreeHost(r.counters);
  }
}

void retire(int device, const Retired& what) {
  Retired* r = static_cast<Retired*>(malloc(sizeof(Retired)));
  if (!r) {  // no list to put it on
    const DeviceScope scope(device);
    if (cudaDeviceSynchronize() == cudaSuccess) release(what);
    return;
  }
  *r = what;
  bool full;
  {
    std::lock_guard<std::mutex> lock(g_mutex);
    DevicePool& d = g_pools[device];
    r->next = d.pending;
    d.pending = r;
    d.pending_bytes += r->bytes;
    full = d.pending_bytes > kMaxPending;
  }
  if (full) (void)pool_wait(device);
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
  const DeviceScope scope(device);
  DevicePool& d = g_pools[device];
  uint64_t reserved = 0;
  {
    std::lock_guard<std::mutex> lock(g_mutex);
    if (--d.handles > 0) return;
    keep(d, kKeepIdle);
    cudaMemPoolGetAttribute(d.pool, cudaMemPoolAttrReservedMemCurrent, &reserved);
  }
  if (reserved > kKeepIdle && pool_wait(device) == cudaSuccess) {
    cudaStreamSynchronize(0);
    cudaMemPoolTrimTo(d.pool, kKeepIdle);
  }
}

// Waits for the device and frees what had been retired before.  The list is set aside first: work that another
// thread queues, and memory that it retires, while this one waits are not covered by the wait.
cudaError_t pool_wait(int device) {
  const DeviceScope scope(device);
  DevicePool& d = g_pools[device];
  Retired* r;
  {
    std::lock_guard<std::mutex> lock(g_mutex);
    r = d.pending;
    d.pending = nullptr;
    d.pending_bytes = 0;
  }
  const cudaError_t e = cudaDeviceSynchronize();
  while (r) {
    Retired* next = r->next;
    if (e == cudaSuccess) {
      release(*r);
      free(r);
    } else {  // not waited for (the calling thread captures a stream, say): back onto the list
      std::lock_guard<std::mutex> lock(g_mutex);
      r->next = d.pending;
      d.pending = r;
      d.pending_bytes += r->bytes;
    }
    r = next;
  }
  return e;
}

cudaError_t pool_alloc(int device, size_t bytes, cudaStream_t s, void** out) {
  *out = nullptr;
  const cudaError_t e = cudaMallocFromPoolAsync(out, bytes ? bytes : 256, g_pools[device].pool, s);
  if (e != cudaSuccess) (void)cudaGetLastError();
  return e;
}

cudaError_t scratch_alloc(const Graph* g, size_t bytes, cudaStream_t s, void** out) {
  *out = nullptr;
  if (bytes > (size_t)g->scratch_mb << 20) return cudaErrorMemoryAllocation;
  return pool_alloc(g->device, bytes, s, out);
}

void pool_free(void* p, cudaStream_t s) {
  if (p) cudaFreeAsync(p, s);
}

void pool_retire(int device, void* p, size_t bytes) {
  if (p) retire(device, Retired{nullptr, p, bytes, nullptr});
}

cudaError_t pinned_counters(HostCounters** out) {
  std::lock_guard<std::mutex> lock(g_mutex);
  if (!g_pinned)
    if (cudaError_t e = cudaHostAlloc(&g_pinned, kPinnedWords * sizeof(HostCounters), cudaHostAllocPortable)) {
      g_pinned = nullptr;
      return e;
    }
  for (int i = 0; i < kPinnedWords; ++i) {
    if (g_word_used[i]) continue;
    g_word_used[i] = true;
    *out = g_pinned + i;
    return cudaSuccess;
  }
  return cudaHostAlloc(out, sizeof(HostCounters), cudaHostAllocPortable);  // more handles than words
}

void pinned_counters_retire(int device, HostCounters* p) {
  if (p) retire(device, Retired{nullptr, nullptr, 0, p});
}

}  // namespace dg
