// A stand-in for the CUDA runtime, for tests of the library's host code on a
// machine without a GPU: device memory is host memory filled with a pattern,
// copies and fills happen at once, kernels are recorded and not run.  Every
// call that allocates, frees, fills, copies, launches or waits goes to a log
// with its pointer, size and stream; allocations and device synchronisations
// can be made to fail, and fills and copies on a captured stream are only
// recorded.  fake_* are the test's own entry points.
#include <cuda_runtime_api.h>
#include <sys/mman.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <vector>

#define FAKE extern "C" __attribute__((visibility("default")))

namespace {
struct Entry {
  const char* what;
  const void* ptr;
  size_t bytes;
  void* stream;
};
std::recursive_mutex mu;
std::vector<Entry> entries;
std::map<void*, size_t> live;
size_t live_bytes = 0, total_bytes = (size_t)64 << 30;  // in use; the device's memory
size_t reported_total = (size_t)64 << 30;                       // what cudaMemGetInfo says of it
long long mallocs_left = -1;  // allocations that still succeed (negative: all)
cudaError_t sync_error = cudaSuccess;
int device = 0;
unsigned long long context = 1;  // 0: none is current yet; the next allocation or release makes one
cudaStream_t captured = nullptr;  // the stream being captured
thread_local struct { dim3 grid, block; size_t smem; void* stream; } config;

void note(const char* what, const void* p = nullptr, size_t bytes = 0, void* stream = nullptr) {
  std::lock_guard<std::recursive_mutex> lk(mu);
  entries.push_back({what, p, bytes, stream});
}
}  // namespace

FAKE int fake_log_size() { return (int)entries.size(); }
FAKE const char* fake_log_entry(int i, const void** p, size_t* bytes, void** stream) {
  *p = entries[i].ptr;
  *bytes = entries[i].bytes;
  *stream = entries[i].stream;
  return entries[i].what;
}
FAKE void fake_log_clear() { entries.clear(); }
FAKE void fake_set_mallocs_left(long long n) { mallocs_left = n; }
FAKE void fake_sync_error(int e) { sync_error = (cudaError_t)e; }
FAKE void fake_set_device(int d) { device = d; }
FAKE void fake_set_context(unsigned long long id) { context = id; }
FAKE void fake_set_captured(void* s) { captured = (cudaStream_t)s; }
FAKE void fake_set_total(size_t b) { total_bytes = b; }
FAKE void fake_set_reported_total(size_t b) { reported_total = b; }
FAKE size_t fake_live_bytes() {
  std::lock_guard<std::recursive_mutex> lk(mu);
  return live_bytes;
}

#define CUDA extern "C" __attribute__((visibility("default"))) cudaError_t

CUDA cudaMalloc(void** p, size_t bytes) {
  std::lock_guard<std::recursive_mutex> lk(mu);
  *p = nullptr;
  if (context == 0) context = 1;
  if (mallocs_left == 0 || live_bytes + bytes > total_bytes) {
    note("malloc failed", nullptr, bytes);
    return cudaErrorMemoryAllocation;
  }
  if (mallocs_left > 0) --mallocs_left;
  void* m = mmap(nullptr, bytes, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
  if (m == MAP_FAILED) return cudaErrorMemoryAllocation;
  memset(m, 0xa5, bytes < 4096 ? bytes : 4096);
  live[m] = bytes;
  live_bytes += bytes;
  *p = m;
  note("malloc", m, bytes);
  return cudaSuccess;
}
CUDA cudaFree(void* p) {
  std::lock_guard<std::recursive_mutex> lk(mu);
  if (context == 0) context = 1;
  if (!p) return cudaSuccess;
  auto it = live.find(p);
  if (it == live.end()) return note("free failed", p), cudaErrorInvalidValue;
  munmap(p, it->second);
  live_bytes -= it->second;
  live.erase(it);
  note("free", p);
  return cudaSuccess;
}
CUDA cudaMallocHost(void** p, size_t bytes) { return (*p = malloc(bytes)) ? cudaSuccess : cudaErrorMemoryAllocation; }
CUDA cudaFreeHost(void* p) { return free(p), cudaSuccess; }
CUDA cudaMemGetInfo(size_t* f, size_t* t) { return *f = total_bytes - live_bytes, *t = reported_total, cudaSuccess; }
namespace {
cudaError_t fill(void* p, int v, size_t n, void* s) {
  if (s && s == captured) return note("recorded", p, n, s), cudaSuccess;
  if (n && !p) return note("memset failed", p, n, s), cudaErrorInvalidValue;
  return memset(p, v, n), note("memset", p, n, s), cudaSuccess;
}
cudaError_t copy(void* d, const void* from, size_t n, void* s) {
  if (s && s == captured) return note("recorded", d, n, s), cudaSuccess;
  if (n && (!d || !from)) return note("memcpy failed", d, n, s), cudaErrorInvalidValue;
  return memcpy(d, from, n), note("memcpy", d, n, s), cudaSuccess;
}
}  // namespace
CUDA cudaMemset(void* p, int v, size_t n) { return fill(p, v, n, nullptr); }
CUDA cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t s) { return fill(p, v, n, s); }
CUDA cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { return copy(d, s, n, nullptr); }
CUDA cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t st) { return copy(d, s, n, st); }
CUDA cudaDeviceSynchronize() { return note("device sync"), sync_error; }
CUDA cudaStreamSynchronize(cudaStream_t s) {
  if (s && s == captured) return cudaErrorStreamCaptureUnsupported;
  return note("stream sync", nullptr, 0, s), cudaSuccess;
}
CUDA cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus* st) {
  return *st = s && s == captured ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone, cudaSuccess;
}
CUDA cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return *s = (cudaStream_t)malloc(1), cudaSuccess; }
CUDA cudaStreamDestroy(cudaStream_t s) { return free(s), cudaSuccess; }
CUDA cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
CUDA cudaEventCreate(cudaEvent_t* e) { return *e = (cudaEvent_t)malloc(1), cudaSuccess; }
CUDA cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return *e = (cudaEvent_t)malloc(1), cudaSuccess; }
CUDA cudaEventDestroy(cudaEvent_t e) { return free(e), cudaSuccess; }
CUDA cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
CUDA cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
CUDA cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { return *ms = 1.0f, cudaSuccess; }
CUDA cudaGetDevice(int* d) { return *d = device, cudaSuccess; }
CUDA cudaSetDevice(int d) { return device = d, note("set device"), cudaSuccess; }
CUDA cudaGetLastError() { return cudaSuccess; }
extern "C" __attribute__((visibility("default"))) const char* cudaGetErrorString(cudaError_t) { return "fake error"; }
extern "C" __attribute__((visibility("default"))) const char* cudaGetErrorName(cudaError_t) { return "fakeError"; }
CUDA cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrComputeCapabilityMajor   ? 10
       : a == cudaDevAttrComputeCapabilityMinor ? 3
       : a == cudaDevAttrMultiProcessorCount    ? 152
       : a == cudaDevAttrL2CacheSize            ? 129 << 20
                                                : 1;
  return cudaSuccess;
}
CUDA cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
CUDA cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t) { return *n = 2, cudaSuccess; }
CUDA cudaGetSymbolAddress(void** p, const void*) {
  static void* scratch = calloc(1, 32 << 20);
  return *p = scratch, cudaSuccess;
}
CUDA cudaLaunchCooperativeKernel(const void* f, dim3, dim3, void**, size_t, cudaStream_t s) {
  return note("launch", f, 0, s), cudaSuccess;
}
CUDA cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) { return note("launch", f, 0, c->stream), cudaSuccess; }
namespace {
int ctx_get_id(void*, unsigned long long* id) { return *id = context, 0; }
}  // namespace
CUDA cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long, cudaDriverEntryPointQueryResult* r) {
  *f = (void*)ctx_get_id;
  if (r) *r = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}

// what nvcc's host code calls for <<<>>> and at load time
CUDA __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void**, size_t, cudaStream_t s) { return note("launch", k, 0, s), cudaSuccess; }
CUDA __cudaGetKernel(cudaKernel_t* k, const void* f) { return *k = (cudaKernel_t)f, cudaSuccess; }
extern "C" __attribute__((visibility("default"))) unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t m, void* s) {
  return config = {g, b, m, s}, 0u;
}
CUDA __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* m, void* s) {
  return *g = config.grid, *b = config.block, *m = config.smem, *(void**)s = config.stream, cudaSuccess;
}
extern "C" __attribute__((visibility("default"))) void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
FAKE void __cudaRegisterFatBinaryEnd(void**) {}
FAKE void __cudaUnregisterFatBinary(void**) {}
FAKE void __cudaRegisterFunction(void**, const char*, char*, const char*, int, void*, void*, void*, void*, int*) {}
FAKE void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
