// A CUDA runtime without a GPU, preloaded in front of the real one: device
// memory is host memory, copies are memcpy, kernels do not run.  It keeps what
// a runtime keeps per device (function attributes), refuses a launch that needs
// an attribute which its device lacks, and fails allocations on request, so
// that the library's host code can be tested on failures and on two devices.
#include <cuda_runtime_api.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <new>
#include <set>
#include <string>
#include <utility>

namespace {
std::recursive_mutex mu;
int device = 0;
const int kDevices = 2;
cudaError_t last = cudaSuccess;
long malloc_left = -1;  // allocations until one fails; -1: none
size_t fail_bytes = 0;  // and the smallest size that counts (0: all)
thread_local long new_left = -1;
std::map<const void*, std::string>& names() {
  static std::map<const void*, std::string> m;
  return m;
}
std::map<std::pair<int, const void*>, std::map<int, int>> attrs;
std::string log_;
long uploads = 0;

cudaError_t ret(cudaError_t e) {
  if (e != cudaSuccess) last = e;
  return e;
}
cudaError_t launch(const void* f, dim3 grid, dim3 block, size_t smem, int cluster) {
  std::lock_guard<std::recursive_mutex> lk(mu);
  auto& a = attrs[{device, f}];
  if (smem > 48 * 1024 && (size_t)a[cudaFuncAttributeMaxDynamicSharedMemorySize] < smem) return ret(cudaErrorInvalidValue);
  if (cluster > 8 && !a[cudaFuncAttributeNonPortableClusterSizeAllowed]) return ret(cudaErrorInvalidClusterSize);
  char line[160];
  std::snprintf(line, sizeof line, " %d %u %u %zu %d\n", device, grid.x, block.x, smem, cluster);
  log_ += names()[f] + line;
  return cudaSuccess;
}
struct Config {
  dim3 grid, block;
  size_t smem;
  cudaStream_t s;
};
thread_local Config config;
}  // namespace

// ---- the test's side --------------------------------------------------------------
extern "C" {
void fake_fail_malloc(long after, size_t bytes) {
  malloc_left = after;
  fail_bytes = bytes;
}
int fake_malloc_armed() { return malloc_left >= 0; }
void fake_fail_new(long after) { new_left = after; }
int fake_has_kernel(const char* part, const char* and_part) {  // a kernel whose name holds both
  for (const auto& n : names())
    if (n.second.find(part) != std::string::npos && n.second.find(and_part) != std::string::npos) return 1;
  return 0;
}
int fake_new_armed() { return new_left >= 0; }
void fake_clear_log() { log_.clear(); }
const char* fake_log() { return log_.c_str(); }  // kernel, device, grid, block, dynamic shared memory, cluster
long fake_uploads() { return uploads; }

// ---- the runtime's -----------------------------------------------------------------
void** __cudaRegisterFatBinary(void*) {
  static void* h = nullptr;
  return &h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* f, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  names()[f] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, cudaStream_t s) {
  config = Config{g, b, smem, s};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* s) {
  *g = config.grid;
  *b = config.block;
  *smem = config.smem;
  *(cudaStream_t*)s = config.s;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void**, size_t smem, cudaStream_t) {
  return launch((const void*)k, g, b, smem, 1);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
  int cluster = 1;
  for (unsigned i = 0; i < c->numAttrs; ++i)
    if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) cluster = (int)c->attrs[i].val.clusterDim.x;
  return launch(f, c->gridDim, c->blockDim, c->dynamicSmemBytes, cluster);
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
  std::lock_guard<std::recursive_mutex> lk(mu);
  attrs[{device, f}][a] = v;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void* f, const cudaLaunchConfig_t*) {
  std::lock_guard<std::recursive_mutex> lk(mu);
  *n = attrs[{device, f}][cudaFuncAttributeNonPortableClusterSizeAllowed] ? 4 : 0;
  return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t bytes) {
  std::lock_guard<std::recursive_mutex> lk(mu);
  if (malloc_left >= 0 && bytes >= fail_bytes && malloc_left-- == 0) return ret(cudaErrorMemoryAllocation);
  return (*p = std::aligned_alloc(256, (bytes + 255) / 256 * 256)) ? cudaSuccess : ret(cudaErrorMemoryAllocation);
}
cudaError_t cudaFree(void* p) {
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  ++uploads;
  std::memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
  std::memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) {
  *d = device;
  return cudaSuccess;
}
cudaError_t cudaSetDevice(int d) {
  if (d < 0 || d >= kDevices) return ret(cudaErrorInvalidDevice);
  device = d;
  return cudaSuccess;
}
cudaError_t cudaGetDeviceCount(int* n) {
  *n = kDevices;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) {
  *v = 152;
  return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaGetLastError() {
  const cudaError_t e = last;
  last = cudaSuccess;
  return e;
}
const char* cudaGetErrorString(cudaError_t e) { return e == cudaErrorMemoryAllocation ? "out of memory" : "error"; }
cudaError_t cudaGetSymbolAddress(void** p, const void* s) {
  *p = const_cast<void*>(s);
  return cudaSuccess;
}
static char handle;
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  *s = (cudaStream_t)&handle;
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* c) {
  *c = cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) {
  *e = (cudaEvent_t)&handle;
  return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  *ms = 1.0f;
  return cudaSuccess;
}
}

// the library's allocations on the host
void* operator new(std::size_t n) {
  if (new_left >= 0 && new_left-- == 0) throw std::bad_alloc();
  if (void* p = std::malloc(n ? n : 1)) return p;
  throw std::bad_alloc();
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }
