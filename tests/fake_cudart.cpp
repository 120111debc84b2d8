// A CUDA runtime without a GPU: the calls libdgagg makes, on host memory, with every call written down.  Kernels
// do not run.  Linked with the library's own object files it lets a test look at the host side alone: the order
// of waits and frees, the device that is current, and what happens when an allocation or a launch fails.
#include <cuda_runtime_api.h>

#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

namespace {
struct Event {
  std::string what;
  int device;
  void* pointer;
  size_t bytes;
};
std::vector<Event> g_events;
std::map<const void*, std::string> g_kernels;
int g_device = 0;
cudaError_t g_last = cudaSuccess;
void (*g_on_sync)() = nullptr;
size_t g_alloc_limit = ~(size_t)0;
size_t g_reserved = 0;
std::string g_failing;
int32_t g_totals[2] = {0, 0};
struct Call {
  dim3 grid, block;
  size_t shared;
  cudaStream_t stream;
};
std::vector<Call> g_calls;

cudaError_t fail(cudaError_t e) { return g_last = e; }
void note(const std::string& what, void* p = nullptr, size_t bytes = 0) {
  g_events.push_back(Event{what, g_device, p, bytes});
}
cudaError_t launch(const void* f, void** args) {
  const std::string& name = g_kernels[f];
  note(name);
  if (!g_failing.empty() && name.find(g_failing) != std::string::npos) return fail(cudaErrorLaunchOutOfResources);
  // the plan says how many rows it cut in its last argument
  if (name.find("plan_kernel") != std::string::npos) memcpy(*(int32_t**)args[10], g_totals, sizeof(g_totals));
  return cudaSuccess;
}
}  // namespace

extern "C" {
// ---- what a test sets and reads
void fake_on_sync(void (*f)()) { g_on_sync = f; }
void fake_alloc_limit(size_t bytes) { g_alloc_limit = bytes; }
void fake_failing_kernel(const char* name) { g_failing = name; }
void fake_plan_totals(int slots, int cut_rows) { g_totals[0] = slots, g_totals[1] = cut_rows; }
void fake_reserved(size_t bytes) { g_reserved = bytes; }
void fake_clear() { g_events.clear(); }
int fake_events() { return (int)g_events.size(); }
const char* fake_event(int i, int* device, void** pointer, size_t* bytes) {
  *device = g_events[i].device, *pointer = g_events[i].pointer, *bytes = g_events[i].bytes;
  return g_events[i].what.c_str();
}

// ---- the runtime
void** __cudaRegisterFatBinary(void*) { return (void**)&g_device; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*,
                            int*) {
  g_kernels[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t shared, cudaStream_t stream) {
  g_calls.push_back(Call{grid, block, shared, stream});
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* shared, void* stream) {
  const Call c = g_calls.back();
  g_calls.pop_back();
  *grid = c.grid, *block = c.block, *shared = c.shared, *(cudaStream_t*)stream = c.stream;
  return cudaSuccess;
}
cudaError_t cudaLaunchKernel(const void* f, dim3, dim3, void** args, size_t, cudaStream_t) { return launch(f, args); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void* f, void** args) { return launch(f, args); }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaGetLastError() {
  const cudaError_t e = g_last;
  g_last = cudaSuccess;
  return e;
}
const char* cudaGetErrorString(cudaError_t) { return "an error of the fake runtime"; }
cudaError_t cudaGetDevice(int* device) { return *device = g_device, cudaSuccess; }
cudaError_t cudaSetDevice(int device) { return g_device = device, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* value, cudaDeviceAttr attr, int) {
  *value = attr == cudaDevAttrMultiProcessorCount ? 148 : 126 << 20;
  return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() {
  note("sync");
  if (g_on_sync) g_on_sync();
  return cudaSuccess;
}
cudaError_t cudaMemPoolCreate(cudaMemPool_t* pool, const cudaMemPoolProps*) {
  return *pool = (cudaMemPool_t)&g_events, cudaSuccess;
}
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaMemPoolGetAttribute(cudaMemPool_t, cudaMemPoolAttr, void* value) {
  return *(uint64_t*)value = g_reserved, cudaSuccess;
}
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t) { return note("trim"), cudaSuccess; }
cudaError_t cudaMallocFromPoolAsync(void** p, size_t bytes, cudaMemPool_t, cudaStream_t) {
  if (bytes > g_alloc_limit) return fail(cudaErrorMemoryAllocation);
  *p = calloc(1, bytes);
  note("alloc", *p, bytes);
  return cudaSuccess;
}
// the memory stays, so that a test may look at what still points to it
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { return note("free", p), cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t bytes, unsigned) { return *p = calloc(1, bytes), cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { return note("free host", p), cudaSuccess; }
cudaError_t cudaMemsetAsync(void* p, int v, size_t bytes, cudaStream_t) { return memset(p, v, bytes), cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* to, const void* from, size_t bytes, cudaMemcpyKind, cudaStream_t) {
  note("copy", to, bytes);
  memcpy(to, from, bytes);
  return cudaSuccess;
}
cudaError_t cudaMemcpy2DAsync(void*, size_t, const void*, size_t, size_t, size_t, cudaMemcpyKind, cudaStream_t) {
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) { return *p = calloc(1, 16 << 20), cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return *s = nullptr, cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return *e = nullptr, cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
}
