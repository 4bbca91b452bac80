// fake_cudart.cpp -- a CUDA runtime without a GPU, for tests of the library's
// host code: linked with its objects in place of the real runtime.  Device
// memory is host memory; kernels are counted, not run.  What it keeps of the
// real runtime is what a caller can get wrong:
//  * two devices; a launch, memory set or event on a stream needs the stream's
//    device to be current;
//  * copies from and to host memory are made when the stream is synchronised, not
//    before (the latest the real runtime may make them), and memory given back
//    with operator delete is overwritten;
//  * streams that are being captured take launches without running them, refuse
//    graphs and synchronisation, and a refused call ends the capture;
//  * the error of a failed call stays pending until cudaGetLastError.
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <map>
#include <set>
#include <vector>

#include <malloc.h>

#include <cuda_runtime_api.h>

void operator delete(void* p) noexcept {   // overwritten and never used again
  if (p) memset(p, 0xDD, malloc_usable_size(p));
}
void operator delete(void* p, size_t) noexcept { operator delete(p); }

namespace {
struct Stream {
  int device = 0;
  bool capturing = false, invalid = false;
  std::vector<std::function<void()>> pending;
};
thread_local int current = 0;
thread_local cudaError_t last = cudaSuccess;
std::set<Stream*> streams;
std::map<const void*, void*> symbols;
long long launches = 0, captured = 0, graph_launches = 0, last_blocks = 0;   // last_blocks: of the last plain launch
std::set<const void*> loaded;   // kernels the runtime has been asked about or has launched
long long cold_launches = 0;    // programmatic launches of kernels not loaded before
int fail_launch = 0;   // fails when it counts down to zero

cudaError_t ret(cudaError_t e) {
  if (e != cudaSuccess) last = e;
  return e;
}
Stream* of(cudaStream_t s) { return reinterpret_cast<Stream*>(s); }

// An operation enqueued on a stream: run by the next synchronisation.
cudaError_t enqueue(cudaStream_t st, bool needs_device, std::function<void()> f) {
  Stream* s = of(st);
  if (!s) {
    f();
    return cudaSuccess;
  }
  if (needs_device && s->device != current) return ret(cudaErrorInvalidResourceHandle);
  if (s->invalid) return ret(cudaErrorStreamCaptureInvalidated);
  if (s->capturing) ++captured;
  else s->pending.push_back(f);
  return cudaSuccess;
}
cudaError_t launch(cudaStream_t st) {
  if (fail_launch > 0 && --fail_launch == 0) return ret(cudaErrorLaunchOutOfResources);
  const cudaError_t e = enqueue(st, true, [] {});
  if (e == cudaSuccess) ++launches;
  return e;
}
struct Call {
  dim3 g, b;
  size_t smem;
  cudaStream_t st;
};
thread_local std::vector<Call> calls;
}  // namespace

extern "C" {
// --- control by the tests
void fake_set_device(int d) { current = d; }
int fake_device() { return current; }
void* fake_stream(int device) {
  Stream* s = new Stream();
  s->device = device;
  streams.insert(s);
  return s;
}
void fake_capture(void* s, int on) {
  static_cast<Stream*>(s)->capturing = on != 0;
  static_cast<Stream*>(s)->invalid = false;
}
int fake_capture_valid(void* s) { return !static_cast<Stream*>(s)->invalid; }
void fake_counts(long long* c) {
  c[0] = launches;
  c[1] = captured;
  c[2] = graph_launches;
  c[3] = last_blocks;
  c[4] = cold_launches;
}
void fake_fail_launch(int nth) { fail_launch = nth; }

// --- modules and launches
void** __cudaRegisterFatBinary(void*) {
  static void* h = nullptr;
  return &h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*, dim3*, int*) {}
void __cudaRegisterVar(void**, char* host, char*, const char*, int, size_t size, int, int) {
  symbols[host] = calloc(1, size);
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, cudaStream_t st) {
  calls.push_back({g, b, smem, st});
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* st) {
  const Call c = calls.back();
  calls.pop_back();
  *g = c.g;
  *b = c.b;
  *smem = c.smem;
  *static_cast<cudaStream_t*>(st) = c.st;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(f));
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3 g, dim3, void**, size_t, cudaStream_t st) {
  last_blocks = (int64_t)g.x * g.y * g.z;
  return launch(st);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
  if (loaded.insert(f).second) ++cold_launches;
  return launch(c->stream);
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes*, const void* f) {
  loaded.insert(f);
  return cudaSuccess;
}
cudaError_t cudaLaunchCooperativeKernel(const void*, dim3, dim3, void**, size_t, cudaStream_t st) { return launch(st); }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  *n = 4;
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void* s) {
  *p = symbols[s];
  return cudaSuccess;
}

// --- devices and errors
cudaError_t cudaGetDevice(int* d) {
  *d = current;
  return cudaSuccess;
}
cudaError_t cudaSetDevice(int d) {
  if (d < 0 || d > 1) return ret(cudaErrorInvalidDevice);
  current = d;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) {
  *v = 152;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() {
  const cudaError_t e = last;
  last = cudaSuccess;
  return e;
}
const char* cudaGetErrorString(cudaError_t) { return "fake error"; }

// --- memory
cudaError_t cudaMalloc(void** p, size_t n) {
  *p = calloc(1, n);
  return *p ? cudaSuccess : ret(cudaErrorMemoryAllocation);
}
cudaError_t cudaFree(void* p) {
  free(p);
  return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return cudaMalloc(p, n); }
cudaError_t cudaFreeHost(void* p) { return cudaFree(p); }
cudaError_t cudaHostGetDevicePointer(void** d, void* h, unsigned) {
  *d = h;
  return cudaSuccess;
}
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t st) {
  *p = calloc(1, n);
  return enqueue(st, false, [] {});
}
cudaError_t cudaFreeAsync(void* p, cudaStream_t st) { return enqueue(st, false, [p] { free(p); }); }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t st) {
  return enqueue(st, false, [=] { memcpy(d, s, n); });
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
  memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpy2DAsync(void* d, size_t dp, const void* s, size_t sp, size_t w, size_t h, cudaMemcpyKind,
                              cudaStream_t st) {
  return enqueue(st, false, [=] {
    for (size_t y = 0; y < h; ++y) memcpy(static_cast<char*>(d) + y * dp, static_cast<const char*>(s) + y * sp, w);
  });
}
cudaError_t cudaMemset(void* p, int v, size_t n) {
  memset(p, v, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t st) {
  return enqueue(st, true, [=] { memset(p, v, n); });
}

// --- streams, events, graphs
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* st, unsigned) {
  *st = static_cast<cudaStream_t>(fake_stream(current));
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t st) {
  Stream* s = of(st);
  if (!s) return cudaSuccess;
  if (s->capturing) {
    s->invalid = true;
    return ret(cudaErrorStreamCaptureUnsupported);
  }
  for (auto& f : s->pending) f();
  s->pending.clear();
  return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() {
  for (Stream* s : streams) cudaStreamSynchronize(reinterpret_cast<cudaStream_t>(s));
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t st) {
  cudaStreamSynchronize(st);
  streams.erase(of(st));
  return cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t st, cudaStreamCaptureStatus* c) {
  Stream* s = of(st);
  *c = !s || !s->capturing ? cudaStreamCaptureStatusNone
       : s->invalid        ? cudaStreamCaptureStatusInvalidated
                           : cudaStreamCaptureStatusActive;
  return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t st, cudaStreamCaptureMode) {
  if (of(st)->capturing) return ret(cudaErrorIllegalState);
  of(st)->capturing = true;
  return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t st, cudaGraph_t* g) {
  Stream* s = of(st);
  *g = s->invalid ? nullptr : reinterpret_cast<cudaGraph_t>(s);
  const bool bad = s->invalid;
  s->capturing = s->invalid = false;
  return bad ? ret(cudaErrorStreamCaptureInvalidated) : cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t g, unsigned long long) {
  *e = reinterpret_cast<cudaGraphExec_t>(g);
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t st) {
  if (of(st)->capturing) {
    of(st)->invalid = true;
    return ret(cudaErrorStreamCaptureUnsupported);
  }
  ++graph_launches;
  return enqueue(st, false, [] {});   // a graph knows its device
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) {
  *e = reinterpret_cast<cudaEvent_t>(malloc(1));
  return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t e) {
  free(e);
  return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t st) { return enqueue(st, true, [] {}); }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  *ms = 0.f;
  return cudaSuccess;
}
}
