// A CUDA runtime without a device, for tests of the library's host side: allocations are counted against a capacity and never
// backed, copies from the device give zeros, launches are counted by kernel name, timings are what the test sets.
#include <cuda_runtime_api.h>

#include <cstdint>
#include <cstring>
#include <map>
#include <string>

namespace {
size_t g_capacity = SIZE_MAX, g_used = 0, g_peak = 0;
uintptr_t g_next = 0x100000000ull;
std::map<void *, size_t> g_live;
std::map<const void *, std::string> g_names;
std::map<std::string, int> g_launches;
int g_occupancy = 2;
float g_elapsed = 1.f;
dim3 g_grid, g_block;
void *g_set_args = nullptr;  // where the last training step's arguments went
}  // namespace

extern "C" {
void fake_capacity(size_t bytes) { g_capacity = bytes; }
size_t fake_used() { return g_used; }
size_t fake_peak(int reset) {
  const size_t p = g_peak;
  if (reset) g_peak = g_used;
  return p;
}
int fake_launches(const char *part, int reset) {
  int n = 0;
  for (auto &kv : g_launches)
    if (kv.first.find(part) != std::string::npos) n += kv.second;
  if (reset) g_launches.clear();
  return n;
}
void *fake_set_args() { return g_set_args; }
void fake_elapsed(float ms) { g_elapsed = ms; }

cudaError_t cudaMalloc(void **p, size_t n) {
  if (n > g_capacity || g_used > g_capacity - n) return cudaErrorMemoryAllocation;
  *p = reinterpret_cast<void *>(g_next);
  g_next += (n + 511) / 512 * 512;
  g_live[*p] = n;
  g_used += n;
  if (g_used > g_peak) g_peak = g_used;
  return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
  auto it = g_live.find(p);
  if (!p) return cudaSuccess;
  if (it == g_live.end()) return cudaErrorInvalidValue;
  g_used -= it->second;
  g_live.erase(it);
  return cudaSuccess;
}
cudaError_t cudaGetDeviceProperties(cudaDeviceProp *p, int) {
  std::memset(p, 0, sizeof *p);
  p->major = 10;
  p->minor = 3;
  p->multiProcessorCount = 152;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : 0;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) {
  *n = g_occupancy;
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int *d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void *dst, const void *, size_t n, cudaMemcpyKind k) {
  if (k == cudaMemcpyDeviceToHost) std::memset(dst, 0, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *dst, const void *src, size_t n, cudaMemcpyKind k, cudaStream_t) {
  return cudaMemcpy(dst, src, n, k);
}
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) {
  *ms = g_elapsed;
  return cudaSuccess;
}
const char *cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaMemset(void *, int, size_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) {
  *e = reinterpret_cast<cudaEvent_t>(1);
  return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
// captures and graphs end well and do nothing
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
  *s = reinterpret_cast<cudaStream_t>(1);
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) {
  *g = reinterpret_cast<cudaGraph_t>(1);
  return cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s) {
  *s = cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t, unsigned long long) {
  *x = reinterpret_cast<cudaGraphExec_t>(1);
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void **, const void *) { return cudaErrorNotSupported; }

// what nvcc's generated host code calls
void **__cudaRegisterFatBinary(void *) {
  static void *h;
  return &h;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) {
  g_names[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t, void *) {
  g_grid = g;
  g_block = b;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *smem, void *stream) {
  *g = g_grid;
  *b = g_block;
  *smem = 0;
  *static_cast<void **>(stream) = nullptr;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *host) {
  *k = reinterpret_cast<cudaKernel_t>(const_cast<void *>(host));
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void **args, size_t, cudaStream_t) {
  if (!g.x || !g.y || !g.z || !b.x || !b.y || !b.z || g.y > 65535 || g.z > 65535) return cudaErrorInvalidConfiguration;
  const std::string &name = g_names[reinterpret_cast<const void *>(k)];
  ++g_launches[name];
  if (name.find("k_set_args") != std::string::npos) std::memcpy(&g_set_args, args[1], sizeof g_set_args);
  return cudaSuccess;
}
cudaError_t cudaLaunchKernel(const void *f, dim3 g, dim3 b, void **a, size_t s, cudaStream_t st) {
  return __cudaLaunchKernel(reinterpret_cast<cudaKernel_t>(const_cast<void *>(f)), g, b, a, s, st);
}
}  // extern "C"
