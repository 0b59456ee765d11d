// A stand-in for the CUDA runtime, for host checks of code that allocates and
// copies: device memory is host memory, and copies keep no more order than CUDA
// promises.  A pageable host-to-device cudaMemcpy returns when the source has
// been staged; its write happens when the legacy stream is waited for or takes
// its next device-to-host copy, and work on another stream (created
// non-blocking) does not wait for it.
#include "fake_cuda.h"

#include <cstdlib>
#include <cstring>
#include <functional>
#include <map>
#include <set>
#include <string>
#include <vector>

#include <cuda_runtime_api.h>

namespace fake {
size_t live = 0;
long allocs = 0;
bool full = false;
std::vector<Launch> launches;
}  // namespace fake
using namespace fake;

static std::map<const void*, std::string>& kernels() {  // names by their host entry (registered before main)
  static std::map<const void*, std::string> names;
  return names;
}
static std::map<char*, size_t> g_device;        // live device buffers
static std::set<void*> g_pinned;                // page-locked host buffers
static std::vector<std::function<void()>> g_legacy;  // writes of the legacy stream still to come

void fake::legacy_wait() {
  for (auto& f : g_legacy) f();
  g_legacy.clear();
}
static cudaError_t device_alloc(void** p, size_t n) {
  if (full) return cudaErrorMemoryAllocation;
  *p = std::malloc(n ? n : 1);
  std::memset(*p, 0xA5, n);
  g_device[static_cast<char*>(*p)] = n;
  live += n;
  ++allocs;
  return cudaSuccess;
}
static cudaError_t device_free(void* p) {
  auto it = g_device.find(static_cast<char*>(p));
  if (it == g_device.end()) return p ? cudaErrorInvalidValue : cudaSuccess;
  live -= it->second;
  g_device.erase(it);
  std::free(p);
  return cudaSuccess;
}
static void copy2d(void* d, size_t dp, const void* s, size_t sp, size_t w, size_t h) {
  for (size_t y = 0; y < h; ++y) std::memcpy((char*)d + y * dp, (const char*)s + y * sp, w);
}
// split_plane_kernel(pairs, f, g, n, join) on words of w bytes
static void split_plane(void** args, size_t w) {
  char *q = *(char**)args[0], *f = *(char**)args[1], *g = *(char**)args[2];
  const long long n = *(long long*)args[3];
  const bool join = *(int*)args[4] != 0;
  for (long long c = 0; c < n; ++c) {
    for (int k = 0; k < 2; ++k) {
      char *pair = q + (2 * c + k) * w, *one = (k ? g : f) + c * w;
      std::memcpy(join ? pair : one, join ? one : pair, w);
    }
  }
}

extern "C" {
cudaError_t cudaMalloc(void** p, size_t n) { return device_alloc(p, n); }
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { return device_alloc(p, n); }
cudaError_t cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t, cudaStream_t) { return device_alloc(p, n); }
cudaError_t cudaFree(void* p) { legacy_wait(); return device_free(p); }
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { return device_free(p); }
cudaError_t cudaMallocHost(void** p, size_t n) { *p = std::malloc(n); g_pinned.insert(*p); return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return cudaMallocHost(p, n); }
cudaError_t cudaFreeHost(void* p) { g_pinned.erase(p); std::free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind k) {
  if (k == cudaMemcpyHostToDevice && !g_pinned.count(const_cast<void*>(s))) {
    std::vector<char> staged((const char*)s, (const char*)s + n);
    g_legacy.push_back([d, staged = std::move(staged)]() { std::memcpy(d, staged.data(), staged.size()); });
    return cudaSuccess;
  }
  legacy_wait();
  std::memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t st) {
  if (!st) return cudaMemcpy(d, s, n, k);
  std::memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpy2D(void* d, size_t dp, const void* s, size_t sp, size_t w, size_t h, cudaMemcpyKind) {
  legacy_wait();
  copy2d(d, dp, s, sp, w, h);
  return cudaSuccess;
}
cudaError_t cudaMemcpy2DAsync(void* d, size_t dp, const void* s, size_t sp, size_t w, size_t h, cudaMemcpyKind,
                              cudaStream_t) {
  copy2d(d, dp, s, sp, w, h);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) { std::memset(p, v, n); return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)std::malloc(1); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { std::free(s); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { if (!s) legacy_wait(); return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)std::malloc(1); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { std::free(e); return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 0.0f; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "error"; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaErrorNotSupported; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t*) { return cudaErrorNotSupported; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t*, cudaGraph_t, unsigned long long) { return cudaErrorNotSupported; }
cudaError_t cudaGraphExecUpdate(cudaGraphExec_t, cudaGraph_t, cudaGraphExecUpdateResultInfo*) { return cudaErrorNotSupported; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
// kernel launches: recorded, and run if they split or join planes
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* cfg, const void* kernel, void**) {
  bool early = false;
  for (unsigned k = 0; k < cfg->numAttrs; ++k) early |= cfg->attrs[k].id == cudaLaunchAttributeProgrammaticStreamSerialization;
  launches.push_back({kernels()[kernel], early});
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t kernel, dim3, dim3, void** args, size_t, cudaStream_t st) {
  const std::string& name = kernels()[(const void*)kernel];
  launches.push_back({name, false});
  if (!st) legacy_wait();
  if (name.find("split_plane_kernelIyE") != name.npos) split_plane(args, 8);
  if (name.find("split_plane_kernelIjE") != name.npos) split_plane(args, 4);
  if (name.find("split_plane_kernelItE") != name.npos) split_plane(args, 2);
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) { *k = (cudaKernel_t)f; return cudaSuccess; }
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void*) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return cudaSuccess; }
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  kernels()[host] = name;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 1; return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  *n = 1;
  return cudaSuccess;
}
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
}
