// A CUDA runtime for tests of libtp's host code without a GPU: linked into the
// library in the place of libcudart. Device memory is host memory, kernels do
// not run, and work stays "in flight" until fake_finish() (or a call that waits
// for it). What kernels would do to the host is played for the one kernel that
// reports: bounded_wait_kernel writes its error word when its work finishes.
#include <cuda_runtime_api.h>

#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <vector>

namespace {
struct Work {              // one launch, in flight or recorded into a graph
  int* word = nullptr;     // bounded_wait_kernel: the word to write, and with what
  int value = 0;
};
struct Event {
  uint64_t after = 0;      // complete once this many pieces of work have finished
};
struct Graph {
  std::vector<Work> work;
};

std::recursive_mutex mu;
std::map<const void*, int> limits;        // dynamic shared-memory limit of a kernel
std::vector<Work> flying;
uint64_t issued = 0, finished = 0;
cudaStream_t capturing = nullptr;
Graph* recording = nullptr;
int lowered = 0;
std::vector<uint64_t> seen[3];             // in order: partial sums given to kernels, counters reset, copies' targets
std::string last;                         // kernel launched last
int hosts = 0;                            // pinned allocations alive

// (built on first use: kernels are registered by other files' initialisers)
std::map<const void*, std::string>& names() {
  static std::map<const void*, std::string> m;
  return m;
}

void finish() {
  std::lock_guard<std::recursive_mutex> lk(mu);
  for (auto& w : flying)
    if (w.word && w.value) *w.word = w.value;
  finished += flying.size();
  flying.clear();
}

cudaError_t launch(const void* f, void** args, size_t smem, cudaStream_t st) {
  std::lock_guard<std::recursive_mutex> lk(mu);
  const std::string& n = names()[f];
  last = n;
  if (smem > 48 * 1024 && (!limits.count(f) || smem > (size_t)limits[f])) return cudaErrorInvalidValue;
  Work w;
  if (n.find("bounded_wait_kernel") != std::string::npos) {
    w.word = *static_cast<int**>(args[0]);
    w.value = *static_cast<bool*>(args[2]) ? 0 : 1;
  }
  if (n.find("residual_finish_kernel") != std::string::npos) seen[0].push_back(*static_cast<uint64_t*>(args[1]));
  if (recording && st == capturing) recording->work.push_back(w);
  else {
    flying.push_back(w);
    ++issued;
  }
  return cudaSuccess;
}

struct Config { dim3 g, b; size_t smem; cudaStream_t st; };
thread_local Config config;
int encode_tiled(...) { return 0; }
}  // namespace

extern "C" {
// ---- controls
void fake_finish() { finish(); }
int fake_lowered() { return lowered; }
int fake_hosts() { return hosts; }
const char* fake_last_kernel() { return last.c_str(); }
int64_t fake_seen(int which, uint64_t* out, int64_t room) {
  std::lock_guard<std::recursive_mutex> lk(mu);
  auto& v = seen[which];
  const int64_t n = (int64_t)v.size();
  for (int64_t i = 0; i < n && i < room; ++i) out[i] = v[i];
  v.clear();
  return n;
}

// ---- registration and launches
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  names()[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, struct CUstream_st* st) {
  config = {g, b, smem, st};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* st) {
  *g = config.g;
  *b = config.b;
  *smem = config.smem;
  *static_cast<cudaStream_t*>(st) = config.st;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(f));
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void** args, size_t smem, cudaStream_t st) {
  return launch(k, args, smem, st);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args) {
  return launch(f, args, c->dynamicSmemBytes, c->stream);
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
  std::lock_guard<std::recursive_mutex> lk(mu);
  if (a != cudaFuncAttributeMaxDynamicSharedMemorySize) return cudaSuccess;
  if (v > 232448) return cudaErrorInvalidValue;
  if (limits.count(f) && v < limits[f]) ++lowered;
  limits[f] = v;
  return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void*) {
  *a = {};
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t*) {
  *n = 1;
  return cudaSuccess;
}

// ---- device and memory
cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrComputeCapabilityMajor ? 10
       : a == cudaDevAttrComputeCapabilityMinor ? 3 : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 232448 : 0;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorName(cudaError_t) { return "fake"; }
const char* cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaMalloc(void** p, size_t n) { *p = std::calloc(n ? n : 1, 1); return cudaSuccess; }
cudaError_t cudaFree(void* p) { finish(); std::free(p); return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) {
  *p = std::calloc(n ? n : 1, 1);
  ++hosts;
  return cudaSuccess;
}
cudaError_t cudaMallocHost(void** p, size_t n) { return cudaHostAlloc(p, n, 0); }
cudaError_t cudaFreeHost(void* p) {
  finish();
  if (p) --hosts;
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { finish(); std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void*, size_t, cudaMemcpyKind, cudaStream_t) {
  std::lock_guard<std::recursive_mutex> lk(mu);
  seen[2].push_back(reinterpret_cast<uint64_t>(d));
  return cudaSuccess;
}
cudaError_t cudaMemset(void* d, int v, size_t n) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* d, int, size_t n, cudaStream_t) {
  std::lock_guard<std::recursive_mutex> lk(mu);
  if (n == sizeof(unsigned)) seen[1].push_back(reinterpret_cast<uint64_t>(d));
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) { *p = nullptr; return cudaErrorInvalidSymbol; }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* r) {
  *f = reinterpret_cast<void*>(encode_tiled);
  if (r) *r = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}

// ---- streams, events, graphs
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode*) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { finish(); return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = reinterpret_cast<cudaStream_t>(0x10); return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus* st) {
  *st = recording && s == capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode) {
  capturing = s;
  recording = new Graph();
  return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
  *g = reinterpret_cast<cudaGraph_t>(recording);
  recording = nullptr;
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t g, unsigned long long) {
  *e = reinterpret_cast<cudaGraphExec_t>(new Graph(*reinterpret_cast<Graph*>(g)));
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t) {
  std::lock_guard<std::recursive_mutex> lk(mu);
  for (auto& w : reinterpret_cast<Graph*>(e)->work) {
    flying.push_back(w);
    ++issued;
  }
  return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) { delete reinterpret_cast<Graph*>(g); return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) { delete reinterpret_cast<Graph*>(e); return cudaSuccess; }
cudaError_t cudaGraphGetNodes(cudaGraph_t, cudaGraphNode_t*, size_t* n) { *n = 0; return cudaSuccess; }
cudaError_t cudaGraphNodeGetType(cudaGraphNode_t, cudaGraphNodeType*) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = reinterpret_cast<cudaEvent_t>(new Event()); return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { delete reinterpret_cast<Event*>(e); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t) {
  std::lock_guard<std::recursive_mutex> lk(mu);
  reinterpret_cast<Event*>(e)->after = issued;
  return cudaSuccess;
}
cudaError_t cudaEventQuery(cudaEvent_t e) {
  std::lock_guard<std::recursive_mutex> lk(mu);
  return reinterpret_cast<Event*>(e)->after <= finished ? cudaSuccess : cudaErrorNotReady;
}
cudaError_t cudaEventSynchronize(cudaEvent_t) { finish(); return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }
}  // extern "C"
