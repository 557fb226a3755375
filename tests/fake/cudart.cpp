// A CUDA runtime without a GPU for tests of the library's host code: device memory is host memory, kernels do
// nothing, and every call is written to a log (one line each) that the test reads.  Failures are made by counting
// allocations down to the one that returns cudaErrorMemoryAllocation.
#include <cuda_runtime.h>
#include <string.h>
#include <unistd.h>

#include <map>
#include <mutex>
#include <string>
#include <vector>

namespace {
std::mutex mu;
std::vector<std::string> lines;
// (the library registers its kernels while it is loaded, maybe before this file's own objects exist)
std::map<const void*, std::string>& names() {
  static auto* m = new std::map<const void*, std::string>;
  return *m;
}
std::string name_of(const void* f) {
  auto it = names().find(f);
  return it == names().end() ? "?" : it->second;
}
std::map<const void*, size_t> device;  // allocations, by address
int fail_in = -1, current_device = 0, slow = 0;
long next_id = 1;

std::string id(const void* p) { return std::to_string((unsigned long long)p); }
void note(const std::string& s) {
  std::lock_guard<std::mutex> lock(mu);
  lines.push_back(s);
}
template <typename T>
T fresh() {
  std::lock_guard<std::mutex> lock(mu);
  return (T)(uintptr_t)(next_id++ * 16);
}
bool is_device(const void* p) {
  std::lock_guard<std::mutex> lock(mu);
  auto it = device.upper_bound(p);
  if (it == device.begin()) return false;
  --it;
  return (const char*)p < (const char*)it->first + it->second;
}
cudaError_t allocate(void** p, size_t bytes, const char* what) {
  {
    std::lock_guard<std::mutex> lock(mu);
    if (fail_in >= 0 && fail_in-- == 0) {
      lines.push_back("nomem");
      return cudaErrorMemoryAllocation;
    }
    *p = calloc(bytes ? bytes : 1, 1);
    device[*p] = bytes ? bytes : 1;
  }
  note(std::string(what) + " " + id(*p) + " " + std::to_string(bytes));
  return cudaSuccess;
}
cudaError_t release(void* p) {
  if (!p) return cudaSuccess;
  {
    std::lock_guard<std::mutex> lock(mu);
    device.erase(p);
  }
  note("free " + id(p));
  free(p);
  return cudaSuccess;
}
struct Call {
  dim3 g, b;
  size_t smem;
  cudaStream_t st;
};
thread_local std::vector<Call> calls;
cudaError_t launched(const void* f, cudaStream_t st, size_t smem) {
  if (slow) usleep(slow);
  note("launch " + id(st) + " " + name_of(f) + " " + std::to_string(smem) + " " + std::to_string(current_device));
  return cudaSuccess;
}
}  // namespace

extern "C" {
// the test's side
void fake_clear() {
  std::lock_guard<std::mutex> lock(mu);
  lines.clear();
}
int fake_count() { return (int)lines.size(); }
const char* fake_line(int i) { return lines[(size_t)i].c_str(); }
void fake_fail_in(int n) { fail_in = n; }  // the (n + 1)-th allocation from now fails
void fake_slow(int us) { slow = us; }  // microseconds a launch takes
void fake_set_device(int d) { current_device = d; }
void* fake_malloc(size_t n) {
  void* p = nullptr;
  allocate(&p, n, "malloc");
  return p;
}

// the library's side
void** __cudaRegisterFatBinary(void*) {
  static void* h = nullptr;
  return &h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  names()[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, struct CUstream_st* st) {
  calls.push_back(Call{g, b, smem, st});
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* st) {
  const Call c = calls.back();
  calls.pop_back();
  *g = c.g;
  *b = c.b;
  *smem = c.smem;
  *(cudaStream_t*)st = c.st;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void**, size_t smem, cudaStream_t st) {
  return launched((const void*)k, st, smem);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
  return launched(f, c->stream, c->dynamicSmemBytes);
}
cudaError_t cudaLaunchCooperativeKernel(const void* f, dim3, dim3, void**, size_t smem, cudaStream_t st) {
  return launched(f, st, smem);
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "error of the runtime without a GPU"; }
const char* cudaGetErrorName(cudaError_t) { return "fake"; }
cudaError_t cudaGetDevice(int* d) {
  *d = current_device;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, enum cudaDeviceAttr, int) {
  *v = 152;
  return cudaSuccess;
}
cudaError_t cudaGetDeviceProperties(struct cudaDeviceProp* p, int) {
  memset(p, 0, sizeof(*p));
  strcpy(p->name, "fake");
  p->multiProcessorCount = 152;
  return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() {
  note("device_sync");
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void* f, enum cudaFuncAttribute, int v) {
  note("attribute " + std::to_string(current_device) + " " + name_of(f) + " " + std::to_string(v));
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t) {
  *n = 2;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  *n = 2;
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void* s) {
  *p = const_cast<void*>(s);
  return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** p, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult*) {
  *p = nullptr;
  return cudaErrorNotSupported;
}

cudaError_t cudaMalloc(void** p, size_t n) { return allocate(p, n, "malloc"); }
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { return allocate(p, n, "malloc"); }
cudaError_t cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t, cudaStream_t) { return allocate(p, n, "malloc"); }
cudaError_t cudaFree(void* p) { return release(p); }
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { return release(p); }
cudaError_t cudaMemPoolCreate(cudaMemPool_t* p, const struct cudaMemPoolProps*) {
  *p = fresh<cudaMemPool_t>();
  return cudaSuccess;
}
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, enum cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaMallocHost(void** p, size_t n) {
  *p = calloc(n ? n : 1, 1);
  return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return cudaMallocHost(p, n); }
cudaError_t cudaHostGetDevicePointer(void** d, void* h, unsigned) {
  *d = h;
  return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) {
  free(p);
  return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(struct cudaPointerAttributes* a, const void* p) {
  memset(a, 0, sizeof(*a));
  a->type = is_device(p) ? cudaMemoryTypeDevice : cudaMemoryTypeUnregistered;
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, enum cudaMemcpyKind, cudaStream_t st) {
  note("copy " + id(st) + " " + id(d));
  memmove(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, enum cudaMemcpyKind k) { return cudaMemcpyAsync(d, s, n, k, nullptr); }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
  memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaMemset(void* d, int v, size_t n) { return cudaMemsetAsync(d, v, n, nullptr); }

cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  *s = fresh<cudaStream_t>();
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  note("sync " + id(s));
  return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
  note("wait " + id(s) + " " + id(e));
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) {
  *e = fresh<cudaEvent_t>();
  return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
  note("record " + id(s) + " " + id(e));
  return cudaSuccess;
}
cudaError_t cudaEventRecordWithFlags(cudaEvent_t e, cudaStream_t s, unsigned) { return cudaEventRecord(e, s); }
cudaError_t cudaEventSynchronize(cudaEvent_t e) {
  note("sync_event " + id(e));
  return cudaSuccess;
}
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t a, cudaEvent_t b) {
  note("elapsed " + id(a) + " " + id(b));
  *ms = 1.f;
  return cudaSuccess;
}

cudaError_t cudaStreamBeginCapture(cudaStream_t s, enum cudaStreamCaptureMode) {
  note("capture " + id(s));
  return cudaSuccess;
}
cudaError_t cudaStreamBeginCaptureToGraph(cudaStream_t s, cudaGraph_t, const cudaGraphNode_t*, const cudaGraphEdgeData*,
                                          size_t, enum cudaStreamCaptureMode m) {
  return cudaStreamBeginCapture(s, m);
}
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t* g) {
  note("end_capture " + id(s));
  *g = fresh<cudaGraph_t>();
  return cudaSuccess;
}
cudaError_t cudaStreamGetCaptureInfo(cudaStream_t, enum cudaStreamCaptureStatus* st, unsigned long long*, cudaGraph_t*,
                                     const cudaGraphNode_t** deps, const cudaGraphEdgeData**, size_t* n) {
  *st = cudaStreamCaptureStatusActive;
  *deps = nullptr;
  *n = 0;
  return cudaSuccess;
}
cudaError_t cudaGraphCreate(cudaGraph_t* g, unsigned) {
  *g = fresh<cudaGraph_t>();
  return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphConditionalHandleCreate(cudaGraphConditionalHandle* h, cudaGraph_t, unsigned, unsigned) {
  *h = 1;
  return cudaSuccess;
}
cudaError_t cudaGraphAddNode(cudaGraphNode_t* n, cudaGraph_t, const cudaGraphNode_t*, const cudaGraphEdgeData*, size_t,
                             struct cudaGraphNodeParams* p) {
  static cudaGraph_t body;
  body = fresh<cudaGraph_t>();
  p->conditional.phGraph_out = &body;
  *n = fresh<cudaGraphNode_t>();
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t, unsigned long long) {
  *x = fresh<cudaGraphExec_t>();
  note("exec_new " + id(*x));
  return cudaSuccess;
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) {
  note("exec_del " + id(x));
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t x, cudaStream_t s) {
  note("exec_launch " + id(s) + " " + id(x));
  return cudaSuccess;
}
}
