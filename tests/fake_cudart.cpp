// A CUDA runtime without a GPU, for host-logic tests of the library: two devices
// (the current one per thread), memory that stays zero, streams and graphs that
// run nothing.  A launch is counted by kernel name and checked as the driver
// checks it: more than 48 KB of dynamic shared memory needs the limit raised on
// the device that is current, and a capturing stream takes launches only.
#include <cuda_runtime_api.h>
#include <sys/mman.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <set>
#include <string>
#include <utility>

namespace {
thread_local int g_device = 0;
thread_local cudaError_t g_last = cudaSuccess;
thread_local struct {
  dim3 grid, block;
  size_t smem;
  cudaStream_t stream;
} g_call;
int g_fail_attributes = 0;
std::map<std::pair<int, const void *>, int> g_limit;
std::map<const void *, std::string> g_name;
std::map<std::string, long long> g_launches, g_blocks;
long long g_total = 0;
std::map<cudaEvent_t, long long> g_events;
std::map<void *, size_t> g_sizes;
std::set<cudaStream_t> g_capturing;
long long g_handles = 0;

cudaError_t done(cudaError_t e) {
  if (e != cudaSuccess) g_last = e;
  return e;
}
void *handle() { return (void *)(0x1000 + 16 * ++g_handles); }
cudaError_t launch(const void *f, dim3 grid, size_t smem) {
  auto it = g_limit.find({g_device, f});
  if (smem > (size_t)(it == g_limit.end() ? 48 * 1024 : it->second))
    return done(cudaErrorInvalidValue);
  ++g_total;
  ++g_launches[g_name[f]];
  g_blocks[g_name[f]] = (long long)grid.x * grid.y * grid.z;
  return cudaSuccess;
}
cudaError_t copy(void *d, const void *s, size_t n, cudaMemcpyKind kind) {
  if (kind != cudaMemcpyDeviceToDevice) memcpy(d, s, n);
  return cudaSuccess;
}
}  // namespace

extern "C" {
// ---- what a test sets and reads
void fake_set_device(int d) { g_device = d; }
int fake_device(void) { return g_device; }
void fake_fail_attributes(int n) { g_fail_attributes = n; }
void fake_capture(void *s, int on) {
  if (on)
    g_capturing.insert((cudaStream_t)s);
  else
    g_capturing.erase((cudaStream_t)s);
}
long long fake_launches(const char *part) {
  long long n = 0;
  for (const auto &l : g_launches)
    if (l.first.find(part) != std::string::npos) n += l.second;
  return n;
}
long long fake_blocks(const char *part) {  // of the last such launch
  for (const auto &b : g_blocks)
    if (b.first.find(part) != std::string::npos) return b.second;
  return 0;
}

// ---- the runtime
cudaError_t cudaGetDevice(int *d) { *d = g_device; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { g_device = d; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : 0;
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute, int v) {
  if (g_fail_attributes > 0) {
    --g_fail_attributes;
    return done(cudaErrorInvalidValue);
  }
  g_limit[{g_device, f}] = v;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int,
                                                                   size_t, unsigned) {
  *n = 1;
  return cudaSuccess;
}
cudaError_t cudaMalloc(void **p, size_t n) {
  *p = mmap(nullptr, n, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
  if (*p == MAP_FAILED) return done(cudaErrorMemoryAllocation);
  g_sizes[*p] = n;
  return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
  if (p) munmap(p, g_sizes[p]);
  return cudaSuccess;
}
cudaError_t cudaMallocHost(void **p, size_t n) { *p = calloc(1, n); return cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaMemset(void *, int, size_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind k) { return copy(d, s, n, k); }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind k, cudaStream_t) {
  return copy(d, s, n, k);
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *) {
  memset(a, 0, sizeof(*a));
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void **p, const void *s) { *p = (void *)s; return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
  *s = (cudaStream_t)handle();
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  return g_capturing.count(s) ? done(cudaErrorStreamCaptureUnsupported) : cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) {
  *g = (cudaGraph_t)handle();
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *e, cudaGraph_t, unsigned long long) {
  *e = (cudaGraphExec_t)handle();
  return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t s) {
  return g_capturing.count(s) ? done(cudaErrorStreamCaptureUnsupported) : cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = (cudaEvent_t)handle(); return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t) { g_events[e] = g_total; return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t a, cudaEvent_t b) {
  *ms = (float)(g_events[b] - g_events[a]);  // a launch takes a millisecond
  return cudaSuccess;
}
const char *cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "fake error"; }
cudaError_t cudaGetLastError(void) {
  const cudaError_t e = g_last;
  g_last = cudaSuccess;
  return e;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **) {
  return launch(f, c->gridDim, c->dynamicSmemBytes);
}

// ---- what nvcc's host code calls
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, cudaStream_t s) {
  g_call = {g, b, smem, s};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *smem, void *s) {
  *g = g_call.grid;
  *b = g_call.block;
  *smem = g_call.smem;
  *(cudaStream_t *)s = g_call.stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3, void **, size_t smem, cudaStream_t) {
  return launch((const void *)k, grid, smem);
}
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
void __cudaRegisterFunction(void **, const char *f, char *, const char *name, int, uint3 *, uint3 *,
                            dim3 *, dim3 *, int *) {
  g_name[f] = name;
}
}
