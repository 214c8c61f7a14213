// fake_cudart.cpp -- the CUDA runtime calls libleiden makes, on host memory and
// without a device: copies copy, kernel launches do nothing but leave a line in
// a log, and a test can choose the current device, refuse launches of a kind,
// and say how many clusters fit.  Linked with the library's own objects in
// place of libcudart, it lets the host paths be tested where there is no GPU.
#include <cuda_runtime_api.h>
#include <stdlib.h>
#include <string.h>

#include <atomic>
#include <map>
#include <mutex>
#include <string>
#include <utility>

namespace {

int g_device = 0, g_sms = 152;
int g_max_cluster = 16;             // larger clusters never fit
bool g_refuse_coop = false, g_refuse_cluster = false;
cudaError_t g_last = cudaSuccess;
std::string g_log;
std::recursive_mutex g_mu;             // the server calls from its workers' threads
std::map<std::pair<int, const void *>, std::map<int, int>> g_attr;   // (device, kernel) -> attributes

std::map<const void *, std::string> &names() {
  static std::map<const void *, std::string> n;
  return n;
}

cudaError_t fail(cudaError_t e) {
  if (e != cudaSuccess) g_last = e;
  return e;
}

cudaError_t launch(const void *f, dim3 grid, dim3 block, size_t smem, int cluster, bool coop) {
  std::lock_guard<std::recursive_mutex> lock(g_mu);
  const auto &at = g_attr[{g_device, f}];
  auto have = [&](int a, int d) { auto i = at.find(a); return i == at.end() ? d : i->second; };
  cudaError_t e = cudaSuccess;
  // what the real runtime refuses for want of a function attribute
  if (smem > 48 * 1024 && (size_t)have(cudaFuncAttributeMaxDynamicSharedMemorySize, 0) < smem) e = cudaErrorInvalidValue;
  if (cluster > 8 && !have(cudaFuncAttributeNonPortableClusterSizeAllowed, 0)) e = cudaErrorInvalidClusterSize;
  if (cluster > g_max_cluster || (cluster > 1 && g_refuse_cluster)) e = cudaErrorInvalidClusterSize;
  if (coop && g_refuse_coop) e = cudaErrorCooperativeLaunchTooLarge;
  g_log += std::to_string(g_device) + " " + names()[f] + " grid " + std::to_string(grid.x) + " block " +
           std::to_string(block.x) + " smem " + std::to_string(smem) + " cluster " + std::to_string(cluster) +
           (coop ? " coop" : "") + (e == cudaSuccess ? " ok\n" : " refused\n");
  return fail(e);
}

struct Call { dim3 g, b; size_t m; cudaStream_t s; };
thread_local Call t_call;

void *token() {
  static char t[64];
  static std::atomic<unsigned> k{0};
  return &t[k++ % 64];
}

}  // namespace

extern "C" {

// ---- what a test sets and reads
void fake_reset() {
  g_device = 0; g_sms = 152; g_max_cluster = 16;
  g_refuse_coop = g_refuse_cluster = false;
  g_last = cudaSuccess;
  g_log.clear();
}
void fake_set_device(int d) { g_device = d; }
void fake_set_sms(int n) { g_sms = n; }
void fake_set_max_cluster(int n) { g_max_cluster = n; }
void fake_refuse(int coop, int cluster) { g_refuse_coop = coop != 0; g_refuse_cluster = cluster != 0; }
const char *fake_log() { return g_log.c_str(); }
int fake_pending_error() { return (int)g_last; }

// ---- registration and launches
void **__cudaRegisterFatBinary(void *) { return (void **)token(); }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, void *, void *, void *, void *, int *) {
  names()[host] = name;
}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t m, cudaStream_t s) {
  t_call = {g, b, m, s};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *m, void *s) {
  *g = t_call.g; *b = t_call.b; *m = t_call.m;
  *(cudaStream_t *)s = t_call.s;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void **, size_t m, cudaStream_t) {
  return launch((const void *)k, g, b, m, 1, false);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **) {
  int cluster = 1;
  bool coop = false;
  for (unsigned k = 0; k < c->numAttrs; k++) {
    if (c->attrs[k].id == cudaLaunchAttributeClusterDimension) cluster = (int)c->attrs[k].val.clusterDim.x;
    if (c->attrs[k].id == cudaLaunchAttributeCooperative) coop = c->attrs[k].val.cooperative != 0;
  }
  return launch(f, c->gridDim, c->blockDim, c->dynamicSmemBytes, cluster, coop);
}
cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute a, int v) {
  std::lock_guard<std::recursive_mutex> lock(g_mu);
  g_attr[{g_device, f}][(int)a] = v;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *f, const cudaLaunchConfig_t *c) {
  std::lock_guard<std::recursive_mutex> lock(g_mu);
  const auto &at = g_attr[{g_device, f}];
  auto have = [&](int a, int d) { auto i = at.find(a); return i == at.end() ? d : i->second; };
  const int cl = (int)c->attrs[0].val.clusterDim.x;
  *n = 0;
  if (cl > 8 && !have(cudaFuncAttributeNonPortableClusterSizeAllowed, 0)) return fail(cudaErrorInvalidClusterSize);
  if ((size_t)have(cudaFuncAttributeMaxDynamicSharedMemorySize, 48 * 1024) < c->dynamicSmemBytes)
    return fail(cudaErrorInvalidValue);
  *n = cl > g_max_cluster ? 0 : g_sms / cl;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *, int threads, size_t) {
  *n = (2048 / threads) >> g_device;   // devices differ
  return cudaSuccess;
}

// ---- memory: device and pinned memory are host memory, zeroed
cudaError_t cudaMalloc(void **p, size_t n) { *p = calloc(1, n ? n : 1); return *p ? cudaSuccess : fail(cudaErrorMemoryAllocation); }
cudaError_t cudaMallocHost(void **p, size_t n) { return cudaMalloc(p, n); }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { return cudaMalloc(p, n); }
cudaError_t cudaFree(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { memmove(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) { memmove(d, s, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { memset(d, v, n); return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void **p, const void *) { static char a[1 << 26]; *p = a; return cudaSuccess; }

// ---- device, streams, events, graphs
cudaError_t cudaGetDevice(int *d) { *d = g_device; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { g_device = d; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = g_sms; return cudaSuccess; }
cudaError_t cudaGetLastError() { const cudaError_t e = g_last; g_last = cudaSuccess; return e; }
const char *cudaGetErrorName(cudaError_t) { return "fake"; }
const char *cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = (cudaStream_t)token(); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = (cudaEvent_t)token(); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) { *g = (cudaGraph_t)token(); return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *e, cudaGraph_t, unsigned long long) { *e = (cudaGraphExec_t)token(); return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **, unsigned, unsigned long long, cudaDriverEntryPointQueryResult *) {
  return fail(cudaErrorNotSupported);
}

}  // extern "C"
