// A stand-in for the CUDA runtime, linked with the library's own host objects (not with a GPU or a
// driver): device memory is host memory, copies and clears happen at once, kernels and graphs are only
// counted.  fake_fail(i) lets the i-th cudaGraphInstantiate from now on fail (0: none), fake_fail_new(i)
// the i-th operator new of the library, so that tests reach the paths behind such errors.
#include <cuda_runtime.h>

#include <atomic>
#include <cstdlib>
#include <cstring>
#include <new>

namespace {
std::atomic<long> g_launches{0}, g_graph_launches{0}, g_instantiates{0}, g_fail{0}, g_fail_new{0}, g_news{0}, g_copies{0};
std::atomic<int> g_error{0};
bool g_capturing = false;
long g_nodes = 0;
struct Graph {
  long nodes;
};
}  // namespace

void *operator new(std::size_t n) {
  ++g_news;
  if (g_fail_new > 0 && --g_fail_new == 0) throw std::bad_alloc();
  void *p = std::malloc(n ? n : 1);
  if (!p) throw std::bad_alloc();
  return p;
}
void *operator new[](std::size_t n) { return operator new(n); }
void *operator new(std::size_t n, const std::nothrow_t &) noexcept { return std::malloc(n ? n : 1); }
void operator delete(void *p) noexcept { std::free(p); }
void operator delete[](void *p) noexcept { std::free(p); }
void operator delete(void *p, std::size_t) noexcept { std::free(p); }
void operator delete[](void *p, std::size_t) noexcept { std::free(p); }

extern "C" {
void fake_fail(long i) { g_fail = i; }
void fake_fail_new(long i) {
  g_news = 0;
  g_fail_new = i;
}
long fake_news(void) { return g_news; }
long fake_count(int what) { return what == 0 ? g_launches : what == 1 ? g_graph_launches : what == 2 ? g_instantiates : g_copies; }

void **__cudaRegisterFatBinary(void *) {
  static void *h;
  return &h;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, void *, void *, void *, void *, int *) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void *) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *, dim3 *, size_t *, void *) { return cudaSuccess; }
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
static cudaError_t launched() {
  if (g_capturing) ++g_nodes;
  else ++g_launches;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void **, size_t, cudaStream_t) { return launched(); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *, const void *, void **) { return launched(); }

cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrComputeCapabilityMajor      ? 10
       : a == cudaDevAttrComputeCapabilityMinor    ? 3
       : a == cudaDevAttrMultiProcessorCount       ? 152
       : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 232448
                                                   : 0;
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int *d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) {
  *e = nullptr;
  return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) {
  *ms = 1.f;
  return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaFreeHost(void *p) {
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaMallocHost(void **p, size_t n) {
  *p = std::calloc(n, 1);
  return *p ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult *) {
  *f = nullptr;
  return cudaErrorNotSupported;
}
const char *cudaGetErrorString(cudaError_t) { return "fake error"; }
cudaError_t cudaGetLastError(void) { return (cudaError_t)g_error.exchange(0); }
cudaError_t cudaGetSymbolAddress(void **p, const void *) {
  *p = nullptr;
  return cudaErrorNotSupported;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) {
  g_capturing = true;
  g_nodes = 0;
  return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) {
  g_capturing = false;
  *g = (cudaGraph_t) new (std::nothrow) Graph{g_nodes};
  return cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s) {
  *s = cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
  *s = nullptr;
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t g, unsigned long long) {
  ++g_instantiates;
  if (g_fail > 0 && --g_fail == 0) {
    g_error = cudaErrorMemoryAllocation;
    return cudaErrorMemoryAllocation;
  }
  *x = (cudaGraphExec_t) new (std::nothrow) Graph(*(Graph *)g);
  return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) {
  std::free(g);
  return cudaSuccess;
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) {
  std::free(x);
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t x, cudaStream_t) {
  ++g_graph_launches;
  g_launches += ((Graph *)x)->nodes;
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) {
  if (n && !g_capturing) std::memcpy(d, s, n);
  ++g_copies;
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) {
  if (n && !g_capturing) std::memset(d, v, n);
  ++g_copies;
  return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *) {
  std::memset(a, 0, sizeof *a);
  return cudaSuccess;
}
}
