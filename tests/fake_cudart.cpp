// A CUDA runtime without a device, for tests of the library's host code on the CPU: the objects of
// the library are linked with this file instead of the CUDA runtime.  Device memory is host memory
// (zeroed), streams run at once, and kernels do nothing but report their launch: the hook gets the
// kernel's name, its grid and the addresses of its arguments, and may write what the kernel would
// have written.  An allocation or a copy can be made to fail (fake_fail_alloc, fake_fail_copy), and the times between events
// are what the test says (fake_elapsed).
#include <cuda_runtime_api.h>
#include <string.h>

#include <map>
#include <set>
#include <string>
#include <vector>

#include <stdlib.h>

namespace {

typedef void (*Hook)(const char *kernel, const unsigned *grid, void **args);

struct Launch {
  std::string kernel;
  dim3 grid;
};
struct Graph {
  std::vector<Launch> launches;
};

std::map<const void *, std::string> g_names;   // host stub -> kernel
std::map<char *, size_t> g_device, g_pinned;   // allocations
std::vector<Launch> g_log;                     // launches that ran, graph replays included
std::vector<std::string> g_calls;              // copies and synchronisations
Hook g_hook = nullptr;
int64_t g_fail_at = 0, g_allocs = 0;
int64_t g_fail_copy = 0, g_copies = 0;
size_t g_free = size_t(64) << 30;
float g_elapsed = 1.f, g_elapsed_step = 0.f;
cudaError_t g_last = cudaSuccess;
Graph *g_capture = nullptr;
cudaStream_t g_capture_stream = nullptr;

cudaError_t set(cudaError_t e) {
  if (e != cudaSuccess) g_last = e;
  return e;
}

cudaError_t alloc(std::map<char *, size_t> &in, void **p, size_t n) {
  *p = nullptr;
  if (++g_allocs == g_fail_at) return set(cudaErrorMemoryAllocation);
  *p = calloc(1, n ? n : 1);
  if (!*p) return set(cudaErrorMemoryAllocation);
  in[static_cast<char *>(*p)] = n;
  return cudaSuccess;
}

cudaError_t give(std::map<char *, size_t> &in, void *p) {
  if (!p) return cudaSuccess;
  const auto it = in.find(static_cast<char *>(p));
  if (it == in.end()) return set(cudaErrorInvalidValue);
  in.erase(it);
  free(p);
  return cudaSuccess;
}

bool inside(const std::map<char *, size_t> &in, const void *q) {
  char *p = static_cast<char *>(const_cast<void *>(q));
  auto it = in.upper_bound(p);
  if (it == in.begin()) return false;
  --it;
  return p < it->first + it->second;
}

cudaError_t launch(const void *func, dim3 grid, void **args, cudaStream_t s) {
  const auto it = g_names.find(func);
  if (it == g_names.end()) return set(cudaErrorInvalidDeviceFunction);
  const Launch l{it->second, grid};
  if (g_capture && s == g_capture_stream) {
    g_capture->launches.push_back(l);
  } else {
    g_log.push_back(l);
  }
  const unsigned g[3] = {grid.x, grid.y, grid.z};
  if (g_hook) g_hook(l.kernel.c_str(), g, args);
  return cudaSuccess;
}

struct Config {
  dim3 grid, block;
  size_t smem;
  cudaStream_t s;
} g_config;

}  // namespace

extern "C" {

// ---- what the tests call

void fake_hook(Hook h) { g_hook = h; }
void fake_fail_alloc(int64_t n) {  // the n-th allocation from now on fails (0: none)
  g_allocs = 0;
  g_fail_at = n;
}
void fake_fail_copy(int64_t n) {  // the same for copies
  g_copies = 0;
  g_fail_copy = n;
}
int64_t fake_allocs() { return g_allocs; }
int64_t fake_device_blocks() { return (int64_t)g_device.size(); }
int64_t fake_device_bytes() {
  int64_t n = 0;
  for (const auto &b : g_device) n += (int64_t)b.second;
  return n;
}
int64_t fake_pinned_blocks() { return (int64_t)g_pinned.size(); }
int fake_on_device(const void *p) { return inside(g_device, p); }
void fake_set_free(int64_t n) { g_free = (size_t)n; }
void fake_elapsed(float first, float step) {  // of successive cudaEventElapsedTime calls
  g_elapsed = first;
  g_elapsed_step = step;
}
void fake_clear_log() {
  g_log.clear();
  g_calls.clear();
}
int64_t fake_log_size() { return (int64_t)g_log.size(); }
const char *fake_log_kernel(int64_t i) { return g_log[(size_t)i].kernel.c_str(); }
unsigned fake_log_grid(int64_t i) { return g_log[(size_t)i].grid.x; }
int64_t fake_calls(const char *name) {
  int64_t n = 0;
  for (const std::string &c : g_calls) n += c == name;
  return n;
}

// ---- registration and launches

void **__cudaRegisterFatBinary(void *) {
  static void *handle = nullptr;
  return &handle;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *, uint3 *,
                            dim3 *, dim3 *, int *) {
  g_names[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, cudaStream_t s) {
  g_config = Config{grid, block, smem, s};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void *s) {
  *grid = g_config.grid;
  *block = g_config.block;
  *smem = g_config.smem;
  *static_cast<cudaStream_t *>(s) = g_config.s;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *func) {
  *k = (cudaKernel_t)func;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3, void **args, size_t,
                               cudaStream_t s) {
  return launch((const void *)k, grid, args, s);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *func, void **args) {
  return launch(func, c->gridDim, args, c->stream);
}

// ---- device, memory

cudaError_t cudaGetDeviceCount(int *n) {
  *n = 1;
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int *d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrL2CacheSize ? 128 << 20 : 0;
  return cudaSuccess;  // (no memory pools: plain allocations)
}
cudaError_t cudaGetLastError() {
  const cudaError_t e = g_last;
  g_last = cudaSuccess;
  return e;
}
const char *cudaGetErrorString(cudaError_t) { return "an error of the stand-in runtime"; }
cudaError_t cudaMalloc(void **p, size_t n) { return alloc(g_device, p, n); }
cudaError_t cudaFree(void *p) { return give(g_device, p); }
cudaError_t cudaMallocFromPoolAsync(void **p, size_t n, cudaMemPool_t, cudaStream_t) {
  return alloc(g_device, p, n);
}
cudaError_t cudaFreeAsync(void *p, cudaStream_t) { return give(g_device, p); }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { return alloc(g_pinned, p, n); }
cudaError_t cudaFreeHost(void *p) { return give(g_pinned, p); }
cudaError_t cudaMemPoolCreate(cudaMemPool_t *, const cudaMemPoolProps *) {
  return set(cudaErrorNotSupported);
}
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void *) { return cudaSuccess; }
cudaError_t cudaMemGetInfo(size_t *f, size_t *t) {
  *f = g_free;
  *t = g_free;
  return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *p) {
  memset(a, 0, sizeof(*a));
  a->type = inside(g_device, p)   ? cudaMemoryTypeDevice
            : inside(g_pinned, p) ? cudaMemoryTypeHost
                                  : cudaMemoryTypeUnregistered;
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) {
  g_calls.push_back("copy");
  if (++g_copies == g_fail_copy || (n && (!d || !s))) return set(cudaErrorInvalidValue);
  memmove(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind k, cudaStream_t) {
  return cudaMemcpy(d, s, n, k);
}
cudaError_t cudaMemcpy2DAsync(void *d, size_t dp, const void *s, size_t sp, size_t w, size_t h,
                              cudaMemcpyKind, cudaStream_t) {
  g_calls.push_back("copy2d");
  for (size_t i = 0; i < h; ++i)
    memmove(static_cast<char *>(d) + i * dp, static_cast<const char *>(s) + i * sp, w);
  return cudaSuccess;
}
cudaError_t cudaMemset(void *d, int v, size_t n) {
  if (n && !d) return set(cudaErrorInvalidValue);
  memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { return cudaMemset(d, v, n); }
cudaError_t cudaMemset2DAsync(void *d, size_t pitch, int v, size_t w, size_t h, cudaStream_t) {
  for (size_t i = 0; i < h; ++i) memset(static_cast<char *>(d) + i * pitch, v, w);
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void **p, const void *) {
  static char scratch[1 << 20];
  *p = scratch;
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes *a, const void *) {
  memset(a, 0, sizeof(*a));
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *, int, size_t) {
  *n = 8;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *f, int t,
                                                                   size_t s, unsigned) {
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, f, t, s);
}
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult *) {
  return set(cudaErrorNotSupported);  // (no tensor maps: the staged direct form is not there)
}

// ---- streams, events, graphs

cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
  *s = (cudaStream_t)malloc(1);
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) {
  free((void *)s);
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) {
  g_calls.push_back("synchronise");
  return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) {
  *e = (cudaEvent_t)malloc(1);
  return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) {
  free((void *)e);
  return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t, cudaStream_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) {
  *ms = g_elapsed;
  g_elapsed += g_elapsed_step;
  return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode) {
  g_capture = new Graph();
  g_capture_stream = s;
  return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) {
  *g = (cudaGraph_t)g_capture;
  g_capture = nullptr;
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t g, unsigned long long) {
  *x = (cudaGraphExec_t) new Graph(*(Graph *)g);
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t x, cudaStream_t) {
  for (const Launch &l : ((Graph *)x)->launches) g_log.push_back(l);
  return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) {
  delete (Graph *)g;
  return cudaSuccess;
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) {
  delete (Graph *)x;
  return cudaSuccess;
}
cudaError_t cudaGraphGetNodes(cudaGraph_t, cudaGraphNode_t *, size_t *n) {
  *n = 0;  // (no event nodes: kernel statistics need eager launches here)
  return cudaSuccess;
}
cudaError_t cudaGraphNodeGetType(cudaGraphNode_t, cudaGraphNodeType *) {
  return set(cudaErrorInvalidValue);
}
cudaError_t cudaGraphEventRecordNodeGetEvent(cudaGraphNode_t, cudaEvent_t *) {
  return set(cudaErrorInvalidValue);
}
cudaError_t cudaGraphExecEventRecordNodeSetEvent(cudaGraphExec_t, cudaGraphNode_t, cudaEvent_t) {
  return set(cudaErrorInvalidValue);
}

}  // extern "C"
