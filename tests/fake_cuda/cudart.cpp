// A CUDA runtime without a device, preloaded in front of libcudart so that the library's host code runs
// on the CPU: "device" memory is host memory, every operation completes at once, and kernels do nothing
// except for the few of model.cu.  It keeps a record of what must not happen:
//
//  * a kernel launch or an asynchronous operation on a stream of its own while a memset, or a copy from
//    pageable memory, of the legacy stream may still be in flight (both may return before the device has
//    done them, and a non-blocking stream does not wait for the legacy one): only a synchronisation of the
//    legacy stream or a copy back ends that;
//  * a copy, a memset, a tensor map or a work list outside a live allocation.
#include <cuda.h>
#include <cuda_runtime_api.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <map>
#include <mutex>
#include <string>
#include <vector>

#include "model.h"

namespace {

std::recursive_mutex mu;
std::map<char*, size_t> live;
std::map<const void*, std::string> kernels;
std::vector<std::string> faults;
int pending = 0;         // legacy-stream operations that may be in flight
int legacy_waits = 0;    // how often the host waited for the legacy stream, and so for the caller's work on it
long mallocs = 0, fail_malloc = -1;
std::string trace;       // names of the kernels launched, one per line

struct Graph {
  std::vector<std::function<void()>> ops;
};
std::map<cudaStream_t, Graph*> capturing;

using Lock = std::lock_guard<std::recursive_mutex>;

}  // namespace
void fault(const std::string& what) { faults.push_back(what); }
namespace {

bool legacy(cudaStream_t s) { return s == nullptr || s == cudaStreamLegacy; }
bool inside(const void* p, size_t n) {
  auto it = live.upper_bound((char*)p);
  if (it == live.begin()) return false;
  --it;
  return (const char*)p + n <= it->first + it->second;
}
bool device(const void* p) { return inside(p, 0); }
void on_stream(cudaStream_t s, const std::string& what) {
  if (legacy(s) || !pending) return;
  fault(what + " with legacy-stream work possibly in flight");
  pending = 0;  // told once
}

cudaError_t launch(const void* f, void** args, cudaStream_t s) {
  Lock l(mu);
  const std::string k = kernels.count(f) ? kernels[f] : "?";
  auto run = body(k, args);
  auto op = [=] {
    trace += k + "\n";
    run();
  };
  if (capturing.count(s)) {
    capturing[s]->ops.push_back(op);
    return cudaSuccess;
  }
  on_stream(s, k);
  op();
  return cudaSuccess;
}

CUresult encode(CUtensorMap* m, CUtensorMapDataType t, cuuint32_t rank, void* base, const cuuint64_t* dims,
                const cuuint64_t* strides, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
  Lock l(mu);
  memset(m, 0, sizeof(*m));
  const size_t elem = t == CU_TENSOR_MAP_DATA_TYPE_UINT8 ? 1 : t == CU_TENSOR_MAP_DATA_TYPE_FLOAT32 ? 4 : 2;
  if (!inside(base, rank == 2 ? strides[0] * (dims[1] - 1) + dims[0] * elem : dims[0] * elem))
    fault("tensor map outside a live allocation");
  return CUDA_SUCCESS;
}

char symbol[1 << 21];

}  // namespace

bool in_device_memory(const void* p) { return device(p); }

extern "C" {

// ---- the tests' side
int fake_faults(char* buf, int n) {
  Lock l(mu);
  std::string s;
  for (auto& f : faults) s += f + "\n";
  snprintf(buf, n, "%s", s.c_str());
  return (int)faults.size();
}
// the n-th allocation from now fails (n < 0: none)
void fake_fail_malloc(long n) {
  Lock l(mu);
  fail_malloc = n < 0 ? -1 : mallocs + n;
}
long fake_mallocs() { return mallocs; }
int fake_legacy_waits() { return legacy_waits; }
size_t fake_live_bytes() {
  Lock l(mu);
  size_t b = 0;
  for (auto& a : live) b += a.second;
  return b;
}

// ---- registration and launches
void** __cudaRegisterFatBinary(void*) {
  static void* h[1];
  return h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  kernels[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
static thread_local struct {
  dim3 g, b;
  size_t smem;
  void* s;
} cfg;
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, struct CUstream_st* s) {
  cfg = {g, b, smem, s};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* s) {
  *g = cfg.g, *b = cfg.b, *smem = cfg.smem, *(void**)s = cfg.s;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void** args, size_t, cudaStream_t s) {
  return launch((const void*)k, args, s);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args) {
  return launch(f, args, c->stream);
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  *n = 1;
  return cudaSuccess;
}

// ---- device
cudaError_t cudaGetDevice(int* d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int) {
  memset(p, 0, sizeof(*p));
  p->major = 10;
  p->minor = 3;
  p->multiProcessorCount = 152;
  p->sharedMemPerBlockOptin = 232448;
  return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** fn, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* r) {
  *fn = (void*)encode;
  if (r) *r = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaMemGetInfo(size_t* f, size_t* t) {
  *f = *t = size_t(280) << 30;
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
  Lock l(mu);
  live[symbol] = sizeof(symbol);
  *p = symbol;
  return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
  Lock l(mu);
  memset(a, 0, sizeof(*a));
  a->type = device(p) ? cudaMemoryTypeDevice : cudaMemoryTypeUnregistered;
  return cudaSuccess;
}

// ---- memory
cudaError_t cudaMalloc(void** p, size_t n) {
  Lock l(mu);
  if (mallocs++ == fail_malloc) return cudaErrorMemoryAllocation;
  *p = aligned_alloc(512, (n + 511) / 512 * 512 + 512);
  memset(*p, 0xCD, n);  // as on the device, not zeros
  live[(char*)*p] = n;
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  Lock l(mu);
  if (!p) return cudaSuccess;
  if (!live.count((char*)p)) fault("free of what is not live");
  live.erase((char*)p);
  free(p);
  return cudaSuccess;
}
cudaError_t cudaMallocHost(void** p, size_t n) {
  *p = calloc(1, n);
  return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return cudaMallocHost(p, n); }
cudaError_t cudaFreeHost(void* p) {
  free(p);
  return cudaSuccess;
}
static void copy(void* d, const void* s, size_t n) {
  if (device(d) && !inside(d, n)) fault("copy beyond an allocation");
  if (device(s) && !inside(s, n)) fault("copy from beyond an allocation");
  memmove(d, s, n);
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
  Lock l(mu);
  if (device(d) && !device(s)) ++pending;
  if (!device(d)) pending = 0;
  copy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemset(void* d, int v, size_t n) {
  Lock l(mu);
  ++pending;
  if (!inside(d, n)) fault("memset beyond an allocation");
  memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t st) {
  Lock l(mu);
  on_stream(st, "copy");
  copy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t st) {
  Lock l(mu);
  on_stream(st, "memset");
  if (!inside(d, n)) fault("memset beyond an allocation");
  memset(d, v, n);
  return cudaSuccess;
}

// ---- streams, events, graphs
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  *s = (cudaStream_t)malloc(16);
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) {
  free(s);
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  Lock l(mu);
  if (legacy(s)) {
    pending = 0;
    ++legacy_waits;
  }
  return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode) {
  Lock l(mu);
  capturing[s] = new Graph;
  return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t* g) {
  Lock l(mu);
  *g = (cudaGraph_t)capturing[s];
  capturing.erase(s);
  return cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus* c) {
  Lock l(mu);
  *c = capturing.count(s) ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t g, unsigned long long) {
  *e = (cudaGraphExec_t) new Graph(*(Graph*)g);
  return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) {
  delete (Graph*)g;
  return cudaSuccess;
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) {
  delete (Graph*)e;
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t s) {
  Lock l(mu);
  on_stream(s, "graph");
  for (auto& op : ((Graph*)e)->ops) op();
  return cudaSuccess;
}
static int events = 0;
int fake_events() { return events; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) {
  Lock l(mu);
  ++events;
  *e = (cudaEvent_t)malloc(16);
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t e) {
  Lock l(mu);
  --events;
  free(e);
  return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t, cudaStream_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  *ms = 1.f;
  return cudaSuccess;
}

}  // extern "C"
