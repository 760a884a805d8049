// A CUDA runtime without a GPU, for tests of the library's host code: device
// memory is host memory, copies are copies, kernels do not run. Calls are
// counted by name, and one launch can be made to fail.
#include <cuda.h>
#include <cuda_runtime_api.h>

#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>

namespace {
std::mutex mu;
std::map<std::string, long> counts;
std::map<char *, size_t> device;  // allocations that count as device memory
long fail_in = -1;                // launches left until the one that fails
bool busy = false;                // events never complete
thread_local cudaError_t last = cudaSuccess;

void count(const char *name) {
  std::lock_guard<std::mutex> lock(mu);
  ++counts[name];
}
cudaError_t alloc(void **p, size_t n, bool dev) {
  *p = aligned_alloc(256, (n + 255) / 256 * 256 + 256);
  if (!*p) return cudaErrorMemoryAllocation;
  memset(*p, 0, n);
  std::lock_guard<std::mutex> lock(mu);
  if (dev) device[static_cast<char *>(*p)] = n;
  return cudaSuccess;
}
cudaError_t release(void *p) {
  std::lock_guard<std::mutex> lock(mu);
  device.erase(static_cast<char *>(p));
  free(p);
  return cudaSuccess;
}
cudaError_t launch() {
  std::lock_guard<std::mutex> lock(mu);
  ++counts["launch"];
  if (fail_in < 0 || fail_in-- > 0) return cudaSuccess;
  return last = cudaErrorLaunchOutOfResources;
}
CUresult encode(...) { return CUDA_SUCCESS; }
}  // namespace

extern "C" {
long fake_count(const char *name) {
  std::lock_guard<std::mutex> lock(mu);
  return counts[name];
}
void fake_reset(long fail_launch, int events_busy) {
  std::lock_guard<std::mutex> lock(mu);
  counts.clear();
  fail_in = fail_launch;
  busy = events_busy;
}

void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void *) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *, dim3 *, size_t *, void *) { return cudaSuccess; }
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void **, size_t, cudaStream_t) { return launch(); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *, const void *, void **) { return launch(); }
cudaError_t cudaLaunchCooperativeKernel(const void *, dim3, dim3, void **, size_t, cudaStream_t) { return launch(); }

cudaError_t cudaGetLastError(void) { cudaError_t e = last; last = cudaSuccess; return e; }
const char *cudaGetErrorString(cudaError_t e) { return e ? "a fake error" : "no error"; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode *) { return cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp *p, int) { memset(p, 0, sizeof *p); strcpy(p->name, "fake"); return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) { *n = 1; return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void **p, const void *) { static char a[256]; *p = a; return cudaSuccess; }
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **f, unsigned, unsigned long long, cudaDriverEntryPointQueryResult *r) {
  *f = reinterpret_cast<void *>(encode);
  if (r) *r = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
cudaError_t cudaMalloc(void **p, size_t n) { count("cudaMalloc"); return alloc(p, n, true); }
cudaError_t cudaMallocAsync(void **p, size_t n, cudaStream_t) { return alloc(p, n, true); }
cudaError_t cudaMallocHost(void **p, size_t n) { count("pinned"); return alloc(p, n, false); }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { count("pinned"); return alloc(p, n, false); }
cudaError_t cudaFree(void *p) { return release(p); }
cudaError_t cudaFreeAsync(void *p, cudaStream_t) { return release(p); }
cudaError_t cudaFreeHost(void *p) { return release(p); }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { count("copy"); memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) { count("copy"); memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpy2DAsync(void *d, size_t dp, const void *s, size_t sp, size_t w, size_t h, cudaMemcpyKind, cudaStream_t) {
  for (size_t i = 0; i < h; ++i) memcpy((char *)d + i * dp, (const char *)s + i * sp, w);
  return cudaSuccess;
}
cudaError_t cudaMemset(void *p, int v, size_t n) { memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t) { memset(p, v, n); return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *p) {
  memset(a, 0, sizeof *a);
  std::lock_guard<std::mutex> lock(mu);
  auto it = device.upper_bound(static_cast<char *>(const_cast<void *>(p)));
  const bool in = it != device.begin() && (--it, (const char *)p < it->first + it->second);
  a->type = in ? cudaMemoryTypeDevice : cudaMemoryTypeUnregistered;
  return cudaSuccess;
}
static int handle;
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = (cudaEvent_t)&handle; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { *e = (cudaEvent_t)&handle; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *t, cudaEvent_t, cudaEvent_t) { *t = 1; return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t) { return busy ? cudaErrorNotReady : cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { count("stream"); *s = (cudaStream_t)&handle; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
}
