// A CUDA runtime without a GPU, for tests of the library's host code (LD_PRELOAD): memory is host memory,
// kernels are recorded and not run. Allocations fail beyond a limit that the test sets. A copy from pageable
// memory is taken to reach the device only when its stream is waited for, as the runtime documents; a kernel
// launched on another stream before that is recorded as unordered.
#include <cuda_runtime_api.h>

#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>

namespace {
std::recursive_mutex mu;
using Lock = std::lock_guard<std::recursive_mutex>;
std::map<void*, size_t> live;            // device allocations
std::map<const void*, std::string> names;  // host function -> kernel name
std::map<uintptr_t, int> pending;        // stream -> copies not waited for
size_t used = 0, peak = 0, limit = SIZE_MAX;
long long fail_after = -1;               // device allocations that still succeed (-1: no count)
std::string log_, unordered;
uintptr_t next_stream = 16;
cudaError_t last = cudaSuccess;
struct Config {
  dim3 g, b;
  size_t smem;
  cudaStream_t s;
};
thread_local Config cfg[8];
thread_local int ncfg = 0;

cudaError_t alloc(void** p, size_t n) {
  Lock l(mu);
  *p = nullptr;
  if (used + n > limit || fail_after == 0) return last = cudaErrorMemoryAllocation;
  if (fail_after > 0) --fail_after;
  *p = std::malloc(n ? n : 1);
  live[*p] = n;
  used += n;
  peak = used > peak ? used : peak;
  return cudaSuccess;
}
cudaError_t release(void* p, const char* what) {
  Lock l(mu);
  if (!p) return cudaSuccess;
  auto it = live.find(p);
  if (it == live.end()) return last = cudaErrorInvalidValue;
  used -= it->second;
  live.erase(it);
  std::free(p);
  log_ += std::string(what) + "\n";
  return cudaSuccess;
}
cudaError_t copy(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t st, bool wait) {
  Lock l(mu);
  std::memcpy(d, s, n);
  if (k == cudaMemcpyHostToDevice) ++pending[(uintptr_t)st];
  else if (wait) pending.erase((uintptr_t)st);
  if (k == cudaMemcpyDeviceToHost) log_ += "read back\n";
  return cudaSuccess;
}
}  // namespace

extern "C" {
void fake_limit(size_t bytes) { limit = bytes; }
void fake_fail_after(long long n) { fail_after = n; }
size_t fake_used() { return used; }
size_t fake_peak() { return peak; }
void fake_reset() {
  Lock l(mu);
  log_.clear();
  unordered.clear();
  peak = used;
}
const char* fake_log() { return log_.c_str(); }
const char* fake_unordered() { return unordered.c_str(); }

void** __cudaRegisterFatBinary(void*) {
  static void* handle = nullptr;
  return &handle;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  names[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t m, cudaStream_t s) {
  cfg[ncfg++] = Config{g, b, m, s};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* m, void* s) {
  const Config c = cfg[--ncfg];
  *g = c.g;
  *b = c.b;
  *m = c.smem;
  *(cudaStream_t*)s = c.s;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void**, size_t, cudaStream_t s) {
  Lock l(mu);
  const std::string n = names[(const void*)k];
  log_ += "launch " + n + "\n";
  for (const auto& p : pending)
    if (p.second && p.first != (uintptr_t)s) {
      unordered += n + "\n";
      break;
    }
  return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t n) { return alloc(p, n); }
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { return alloc(p, n); }
cudaError_t cudaFree(void* p) { return release(p, "cudaFree"); }
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { return release(p, "cudaFreeAsync"); }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) {
  *p = std::calloc(1, n ? n : 1);
  return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) {
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaHostGetDevicePointer(void** d, void* h, unsigned) {
  *d = h;
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind k) { return copy(d, s, n, k, 0, true); }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t st) {
  return copy(d, s, n, k, st, false);
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t s) {
  Lock l(mu);
  std::memset(d, v, n);
  ++pending[(uintptr_t)s];
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  Lock l(mu);
  *s = (cudaStream_t)(next_stream += 16);
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  Lock l(mu);
  pending.erase((uintptr_t)s);
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) {
  *v = 152;
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaGetLastError() {
  const cudaError_t e = last;
  last = cudaSuccess;
  return e;
}
}
