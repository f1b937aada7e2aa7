// Host stand-in for the CUDA runtime calls that libcwell makes, for tests of
// its host logic without a GPU.  Loaded into the global symbol scope before the
// library (fake_runtime.py).  Device memory is host memory; kernels do not run.
// A launch moves the clock on by its kernel's cost and is written to a log with
// its stream and grid, as are event records and waits.  Refused as by the real runtime:
// more dynamic shared memory than the kernel was granted, and more device memory
// than there is.  A test can let a coming launch fail.
#include <cuda.h>
#include <cuda_runtime_api.h>
#include <dlfcn.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

namespace {
struct Event {
  double t = 0;
};
struct Graph {
  double cost = 0;
};
constexpr size_t SMEM_DEFAULT = 48 * 1024, SMEM_MAX = 227 * 1024;
std::map<const void *, std::string> kernels;
std::map<const void *, size_t> granted;
std::map<void *, size_t> blocks;
std::vector<std::pair<std::string, double>> costs;
size_t total = size_t(256) << 30, used = 0, peak = 0;
double now = 0, launch_us = 0;
Graph *capture = nullptr;
long fail_in = -1;  // launches until one fails
cudaError_t last = cudaSuccess;
std::string logbuf;
struct {
  dim3 grid, block;
  size_t smem;
  cudaStream_t stream;
} config;

void log(const char *what, const void *a, const void *b = nullptr, const char *s = "") {
  char line[64];
  snprintf(line, sizeof line, "%s %zx %zx ", what, (size_t)a, (size_t)b);
  logbuf += std::string(line) + s + "\n";
}
cudaError_t set(cudaError_t e) {
  if (e != cudaSuccess) last = e;
  return e;
}
}  // namespace

extern "C" {
// ---- what a test sets and reads
void fake_cost(const char *name, double us) { costs.insert(costs.begin(), {name, us}); }
void fake_launch_cost(double us) { launch_us = us; }  // of a launch that is not captured
void fake_total(size_t bytes) { total = bytes; }
void fake_fail_launch(long n) { fail_in = n; }
size_t fake_used() { return used; }
size_t fake_peak(int reset) {
  const size_t p = peak;
  if (reset) peak = used;
  return p;
}
const char *fake_log() { return logbuf.c_str(); }
void fake_log_clear() { logbuf.clear(); }

// ---- kernels
void **__cudaRegisterFatBinary(void *) {
  static void *h;
  return &h;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *,
                            int *) {
  kernels[host] = name;
}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, CUstream_st *stream) {
  config = {grid, block, smem, stream};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void *stream) {
  *grid = config.grid, *block = config.block, *smem = config.smem;
  *(cudaStream_t *)stream = config.stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *host) {
  *k = (cudaKernel_t)host;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3 block, void **, size_t smem, cudaStream_t s) {
  if (fail_in >= 0 && fail_in-- == 0) return set(cudaErrorLaunchOutOfResources);
  const size_t lim = granted.count(k) ? granted[k] : SMEM_DEFAULT;
  const unsigned threads = block.x * block.y * block.z;
  if (smem > lim || threads == 0 || threads > 1024 || grid.x == 0 || grid.x > 0x7fffffffu || grid.y == 0 ||
      grid.y > 65535 || grid.z == 0 || grid.z > 65535)
    return set(cudaErrorInvalidValue);
  const std::string &name = kernels[k];
  double us = 1;
  for (auto &c : costs)
    if (name.find(c.first) != std::string::npos) {
      us = c.second;
      break;
    }
  if (capture) capture->cost += us;
  else now += us + launch_us;
  log("launch", s, (void *)(size_t)grid.x, name.c_str());
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *f, enum cudaFuncAttribute a, int v) {
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) {
    if (v < 0 || (size_t)v > SMEM_MAX) return set(cudaErrorInvalidValue);
    granted[f] = v;
  }
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) {
  *n = 2;
  return cudaSuccess;
}

// ---- memory
cudaError_t cudaMalloc(void **p, size_t n) {
  *p = nullptr;
  if (used + n > total || !(*p = malloc(n))) return set(cudaErrorMemoryAllocation);
  blocks[*p] = n;
  used += n;
  peak = used > peak ? used : peak;
  return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
  if (!p) return cudaSuccess;
  auto it = blocks.find(p);
  if (it == blocks.end()) return set(cudaErrorInvalidValue);
  used -= it->second;
  blocks.erase(it);
  free(p);
  return cudaSuccess;
}
cudaError_t cudaMallocAsync(void **p, size_t n, cudaStream_t) { return cudaMalloc(p, n); }
cudaError_t cudaFreeAsync(void *p, cudaStream_t) { return cudaFree(p); }
cudaError_t cudaMemGetInfo(size_t *f, size_t *t) {
  *f = total - used, *t = total;
  return cudaSuccess;
}
cudaError_t cudaMemset(void *p, int v, size_t n) {
  memset(p, v, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t) { return cudaMemset(p, v, n); }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, enum cudaMemcpyKind) {
  memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, enum cudaMemcpyKind k, cudaStream_t) {
  return cudaMemcpy(d, s, n, k);
}
cudaError_t cudaMemcpy2D(void *d, size_t dp, const void *s, size_t sp, size_t w, size_t h, enum cudaMemcpyKind) {
  for (size_t r = 0; r < h; r++) memcpy((char *)d + r * dp, (const char *)s + r * sp, w);
  return cudaSuccess;
}
cudaError_t cudaMemcpy2DAsync(void *d, size_t dp, const void *s, size_t sp, size_t w, size_t h, enum cudaMemcpyKind k,
                              cudaStream_t) {
  return cudaMemcpy2D(d, dp, s, sp, w, h, k);
}
cudaError_t cudaMemcpyFromSymbolAsync(void *d, const void *, size_t n, size_t, enum cudaMemcpyKind, cudaStream_t) {
  return cudaMemset(d, 0, n);
}
cudaError_t cudaMemcpyToSymbolAsync(const void *, const void *, size_t, size_t, enum cudaMemcpyKind, cudaStream_t) {
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void **p, const void *) {
  static char scratch[1 << 20];
  *p = scratch;
  return cudaSuccess;
}

// ---- device, streams, events, graphs
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int *v, enum cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? (int)SMEM_MAX : 0;
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
  *s = (cudaStream_t) new int;
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) {
  delete (int *)s;
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  log("sync", s);
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) {
  *e = (cudaEvent_t) new Event;
  return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) {
  delete (Event *)e;
  return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
  ((Event *)e)->t = now;
  log("record", s, e);
  return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
  log("wait", s, e);
  return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t a, cudaEvent_t b) {
  *ms = (float)((((Event *)b)->t - ((Event *)a)->t) * 1e-3);
  return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, enum cudaStreamCaptureMode) {
  capture = new Graph;
  return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) {
  *g = (cudaGraph_t)capture;
  capture = nullptr;
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t g, unsigned long long) {
  *x = (cudaGraphExec_t) new Graph(*(Graph *)g);
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t x, cudaStream_t) {
  now += ((Graph *)x)->cost;
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

// ---- errors and the driver's tensor-map encoder
cudaError_t cudaGetLastError() {
  const cudaError_t e = last;
  last = cudaSuccess;
  return e;
}
const char *cudaGetErrorString(cudaError_t e) {
  return e == cudaErrorInvalidValue ? "invalid argument"
         : e == cudaErrorMemoryAllocation ? "out of memory"
         : e == cudaErrorLaunchOutOfResources ? "too many resources requested for launch" : "error";
}
static CUresult encode(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                       const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                       CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
  return CUDA_SUCCESS;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char *name, void **p, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult *q) {
  const bool known = !strcmp(name, "cuTensorMapEncodeTiled");
  *p = known ? (void *)encode : nullptr;
  *q = known ? cudaDriverEntryPointSuccess : cudaDriverEntryPointSymbolNotFound;
  return cudaSuccess;
}
}  // extern "C"
