// A stand-in for the CUDA runtime, linked with the library's host side (csrc/mixaq.cu) and fake_launch.cu: it counts what
// the host path asks for, checks the rules of stream capture, and fails a call on request.  Nothing runs on a device;
// pointers are never followed.
#include "fake.h"
#include <atomic>
#include <map>
#include <mutex>
#include <thread>

namespace {
struct Graph { int nodes; };
struct Capture { std::thread::id owner; cudaStream_t origin; };
std::mutex lock;                                   // of what follows
std::map<cudaStream_t, Capture> capturing;         // streams that are part of a capture
std::map<cudaEvent_t, cudaStream_t> event_origin;  // events recorded inside a capture: its origin stream
std::map<cudaStream_t, int> nodes;                 // kernels and copies captured so far, by origin
thread_local cudaError_t last_error = cudaSuccess;
long next_handle = 0x1000;

template <class T> T handle() { return reinterpret_cast<T>(next_handle += 16); }
cudaError_t fail(cudaError_t e) { last_error = e; return e; }
}  // namespace

extern "C" {
FakeCounts counts;
int fail_capture, fail_instantiate, fail_graph_launch;      // the call fails while this is set
unsigned fake_device_word;                                   // what copies to the host find in every 32-bit word of the device
FakeCopy last_copies[16];
cudaStream_t capture_origins[16];                            // of the newest captures
void fake_reset() { std::lock_guard<std::mutex> g(lock); const long live = counts.live_graphs; counts = FakeCounts(); counts.live_graphs = live; }
}

// work enqueued on a stream: part of a capture, or a direct launch
void enqueue(cudaStream_t st) {
  std::this_thread::yield();
  std::lock_guard<std::mutex> g(lock);
  auto it = capturing.find(st);
  if (it == capturing.end()) { ++counts.direct; return; }
  if (it->second.owner != std::this_thread::get_id()) ++counts.violations;
  ++nodes[it->second.origin];
  ++counts.captured;
  if (st != it->second.origin) ++counts.side_launches;
}

// ---- the runtime calls that csrc/mixaq.cu makes ----
extern "C" {
cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) { *p = reinterpret_cast<void*>(0x5000'0000'0000); return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t) { std::lock_guard<std::mutex> g(lock); *p = handle<void*>(); return cudaSuccess; }
cudaError_t cudaFree(void*) { return cudaSuccess; }
cudaError_t cudaMemset(void*, int, size_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t st) { enqueue(st); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* dst, const void* src, size_t n, cudaMemcpyKind kind, cudaStream_t st) {
  enqueue(st);
  if (kind == cudaMemcpyDeviceToHost) for (size_t i = 0; i < n / 4; ++i) static_cast<unsigned*>(dst)[i] = fake_device_word;
  std::lock_guard<std::mutex> g(lock);
  last_copies[counts.copies++ % 16] = {dst, src, n};
  return cudaSuccess;
}
cudaError_t cudaGetLastError() { cudaError_t e = last_error; last_error = cudaSuccess; return e; }
const char* cudaGetErrorString(cudaError_t) { return "fake error"; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { std::lock_guard<std::mutex> g(lock); *e = handle<cudaEvent_t>(); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 0.f; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t st) {
  std::lock_guard<std::mutex> g(lock);
  auto it = capturing.find(st);
  if (it == capturing.end()) event_origin.erase(e); else event_origin[e] = it->second.origin;
  return cudaSuccess;
}
cudaError_t cudaEventRecordWithFlags(cudaEvent_t, cudaStream_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t st, cudaEvent_t e, unsigned) {
  std::lock_guard<std::mutex> g(lock);
  auto it = event_origin.find(e);
  if (it != event_origin.end() && capturing.count(it->second)) {
    auto joined = capturing.find(st);
    if (joined != capturing.end() && joined->second.origin != it->second) ++counts.violations;
    if (joined == capturing.end()) capturing[st] = {std::this_thread::get_id(), it->second};
  }
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { std::lock_guard<std::mutex> g(lock); *s = handle<cudaStream_t>(); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t st, cudaStreamCaptureStatus* s) {
  std::lock_guard<std::mutex> g(lock);
  *s = capturing.count(st) ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t st, cudaStreamCaptureMode) {
  std::lock_guard<std::mutex> g(lock);
  if (fail_capture || !st || st == cudaStreamLegacy) return fail(cudaErrorStreamCaptureUnsupported);
  if (capturing.count(st)) { ++counts.violations; return fail(cudaErrorIllegalState); }
  capturing[st] = {std::this_thread::get_id(), st};
  nodes[st] = 0;
  capture_origins[counts.captures++ % 16] = st;
  return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t st, cudaGraph_t* graph) {
  std::lock_guard<std::mutex> g(lock);
  *graph = nullptr;
  auto it = capturing.find(st);
  if (it == capturing.end() || it->second.origin != st || it->second.owner != std::this_thread::get_id()) {
    ++counts.violations;
    return fail(cudaErrorIllegalState);
  }
  for (auto c = capturing.begin(); c != capturing.end();) c = c->second.origin == st ? capturing.erase(c) : std::next(c);
  *graph = reinterpret_cast<cudaGraph_t>(new Graph{nodes[st]});
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* exec, cudaGraph_t, unsigned long long) {
  std::lock_guard<std::mutex> g(lock);
  if (fail_instantiate) return fail(cudaErrorMemoryAllocation);
  *exec = handle<cudaGraphExec_t>();
  ++counts.instantiated; ++counts.live_graphs;
  return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t graph) { delete reinterpret_cast<Graph*>(graph); return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { std::lock_guard<std::mutex> g(lock); --counts.live_graphs; return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t st) {
  std::lock_guard<std::mutex> g(lock);
  if (fail_graph_launch) return fail(cudaErrorMemoryAllocation);
  if (capturing.count(st)) ++counts.violations;
  ++counts.graph_launches;
  return cudaSuccess;
}
// registration of the (unused) device code
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
char __cudaInitModule(void**) { return 1; }
}
