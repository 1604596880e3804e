#include "fake_cudart.h"

#include <cuda_runtime_api.h>

#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <set>
#include <string>

namespace fake {
int violations = 0, fail_alloc_at = 0;
bool capture = false;
std::size_t fail_over = 0;
const char* fail_kernel = nullptr;

namespace {
enum Kind { kPlain, kAsync, kHost };
struct Buffer {
  std::size_t bytes;
  Kind kind;
  cudaStream_t stream;
};
// leaked on purpose: the objects' registration code runs before any of this file's
std::map<void*, Buffer>& buffers() {
  static auto* m = new std::map<void*, Buffer>();
  return *m;
}
std::map<const void*, std::string>& names() {
  static auto* m = new std::map<const void*, std::string>();
  return *m;
}
std::map<std::string, int>& runs() {
  static auto* m = new std::map<std::string, int>();
  return *m;
}
std::set<cudaStream_t> busy;  // streams with work since they were waited for
bool capturing = false;
std::set<cudaStream_t> captured;                                // streams with work in the capture
std::map<std::uintptr_t, std::set<cudaStream_t>> graphs;        // ... in a graph (or its executable)
std::map<cudaStream_t, std::set<cudaStream_t>> flights;         // ... in the graphs running on a stream
std::map<cudaEvent_t, cudaStream_t> recorded;
int stream_waits = 0;
cudaError_t last = cudaSuccess;
std::uintptr_t next_handle = 0x1000;
struct {
  dim3 grid, block;
  std::size_t smem;
  cudaStream_t stream;
} config;

template <typename T>
T handle() {
  return reinterpret_cast<T>(next_handle += 16);
}
// Work on a stream: a copy or a kernel.
void work_on(cudaStream_t st) {
  if (capturing) {
    captured.insert(st);
    return;
  }
  busy.insert(st);
  for (const auto& f : flights)
    if (f.first != st && f.second.count(st)) {
      std::printf("violation: work on a stream beside the graph that runs its work elsewhere\n");
      ++violations;
    }
}
void waited_for(cudaStream_t st) {
  busy.erase(st);
  flights.erase(st);
}
void all_waited_for() {
  busy.clear();
  flights.clear();
}
cudaError_t allocate(void** p, std::size_t n, Kind kind, cudaStream_t st) {
  *p = nullptr;
  if (fail_alloc_at > 0 && --fail_alloc_at == 0) return last = cudaErrorMemoryAllocation;
  if (kind != kHost && fail_over && n > fail_over) return last = cudaErrorMemoryAllocation;
  *p = std::calloc(n ? n : 1, 1);
  if (!*p) return last = cudaErrorMemoryAllocation;
  buffers()[*p] = Buffer{n, kind, st};
  if (kind == kAsync) busy.insert(st);
  return cudaSuccess;
}
cudaError_t release(void* p, Kind kind, cudaStream_t st) {
  if (!p) return cudaSuccess;
  auto it = buffers().find(p);
  if (it == buffers().end() || it->second.kind != kind) {
    std::printf("violation: a buffer returned by the wrong call\n");
    ++violations;
    return last = cudaErrorInvalidValue;
  }
  if (kind == kAsync && st != it->second.stream && busy.count(it->second.stream)) {
    std::printf("violation: %zu bytes returned in another stream's order\n", it->second.bytes);
    ++violations;
  }
  std::free(p);
  buffers().erase(it);
  return cudaSuccess;
}
cudaError_t run(const void* fun, cudaStream_t st) {
  const std::string& n = names()[fun];
  if (fail_kernel && n.find(fail_kernel) != std::string::npos) {
    fail_kernel = nullptr;
    return last = cudaErrorLaunchOutOfResources;
  }
  ++runs()[n];
  work_on(st);
  return cudaSuccess;
}
}  // namespace

int waits() { return stream_waits; }
std::size_t live() { return buffers().size(); }
std::size_t held() {
  std::size_t n = 0;
  for (const auto& b : buffers()) n += b.second.bytes;
  return n;
}
int launched(const char* name) {
  int n = 0;
  for (const auto& r : runs())
    if (r.first.find(name) != std::string::npos) n += r.second;
  return n;
}
}  // namespace fake

using namespace fake;

extern "C" {

// registration and launches
void** __cudaRegisterFatBinary(void*) { return handle<void**>(); }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  names()[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* host) {
  *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(host));
  return cudaSuccess;
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, cudaStream_t st) {
  config = {grid, block, smem, st};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* st) {
  *grid = config.grid;
  *block = config.block;
  *smem = config.smem;
  *static_cast<cudaStream_t*>(st) = config.stream;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void**, size_t, cudaStream_t st) { return run(k, st); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* fun, void**) { return run(fun, c->stream); }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t) {
  *n = 2;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  *n = 2;
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void* sym) {
  *p = const_cast<void*>(sym);
  return cudaSuccess;
}

// device, errors
cudaError_t cudaGetDevice(int* d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : (a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 227 * 1024 : 1);
  return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() {
  all_waited_for();
  return cudaSuccess;
}
cudaError_t cudaGetLastError() {
  const cudaError_t e = last;
  last = cudaSuccess;
  return e;
}
const char* cudaGetErrorString(cudaError_t) { return "made to fail"; }

// memory
cudaError_t cudaMalloc(void** p, size_t n) { return allocate(p, n, kPlain, nullptr); }
cudaError_t cudaFree(void* p) {
  all_waited_for();  // waits for the device
  return release(p, kPlain, nullptr);
}
cudaError_t cudaMallocHost(void** p, size_t n) { return allocate(p, n, kHost, nullptr); }
cudaError_t cudaFreeHost(void* p) { return release(p, kHost, nullptr); }
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t st) { return allocate(p, n, kAsync, st); }
cudaError_t cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t, cudaStream_t st) { return allocate(p, n, kAsync, st); }
cudaError_t cudaFreeAsync(void* p, cudaStream_t st) { return release(p, kAsync, st); }
cudaError_t cudaMemPoolCreate(cudaMemPool_t* p, const cudaMemPoolProps*) {
  *p = handle<cudaMemPool_t>();
  return cudaSuccess;
}
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaMemPoolDestroy(cudaMemPool_t) { return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
  std::memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t st) {
  std::memcpy(d, s, n);
  work_on(st);
  return cudaSuccess;
}
cudaError_t cudaMemset(void*, int, size_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t st) {  // nothing reads the values
  work_on(st);
  return cudaSuccess;
}

// streams, events, graphs (without capture the library launches directly)
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  *s = handle<cudaStream_t>();
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  waited_for(s);
  return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t st, cudaEvent_t e, unsigned) {
  if (recorded.count(e) && recorded[e] != st) ++stream_waits;
  return cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* c) {
  *c = capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) {
  if (!capture || capturing) return last = cudaErrorNotSupported;
  capturing = true;
  captured.clear();
  return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
  *g = handle<cudaGraph_t>();
  capturing = false;
  graphs[reinterpret_cast<std::uintptr_t>(*g)] = captured;
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t g, unsigned long long) {
  *e = handle<cudaGraphExec_t>();
  graphs[reinterpret_cast<std::uintptr_t>(*e)] = graphs[reinterpret_cast<std::uintptr_t>(g)];
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t st) {
  for (cudaStream_t x : graphs[reinterpret_cast<std::uintptr_t>(e)]) {
    if (x != st && busy.count(x)) {
      std::printf("violation: a graph launched beside work on a stream whose work it runs\n");
      ++violations;
    }
    flights[st].insert(x);
  }
  work_on(st);
  return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) {
  *e = handle<cudaEvent_t>();
  return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t st) {
  if (!capturing) recorded[e] = st;
  return cudaSuccess;
}
cudaError_t cudaEventRecordWithFlags(cudaEvent_t e, cudaStream_t st, unsigned) { return cudaEventRecord(e, st); }
cudaError_t cudaEventSynchronize(cudaEvent_t e) {
  if (recorded.count(e)) waited_for(recorded[e]);
  return cudaSuccess;
}
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  *ms = 0.f;
  return cudaSuccess;
}

}  // extern "C"
