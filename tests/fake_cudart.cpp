// A CUDA runtime without a device, preloaded into a CPU test's child process: memory is
// host memory, kernels do nothing, and every call is written to a trace.  It keeps the
// documented order of asynchronous work (a device memset, and a host-to-device copy from
// pageable memory, may still be under way when the call returns; only its own stream, or
// a synchronisation, orders later work after it) and notes every launch that is not
// ordered after a memset or copy.  Streams other than the legacy one are non-blocking.
#include <cuda_runtime.h>
#include <dlfcn.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <map>
#include <string>
#include <vector>

namespace {
struct Alloc {
  size_t id, bytes;
};
std::map<const char*, Alloc> g_allocs;
size_t g_next = 0, g_limit = ~size_t(0), g_streams = 0;
int g_capturing = 0;  // what cudaStreamIsCapturing answers for streams the library did not make
std::map<const void*, std::string> g_kernels;
std::map<const void*, size_t> g_smem;  // dynamic shared memory allowed, where it was set
std::vector<cudaStream_t> g_own;
struct Pending {
  cudaStream_t s;
  std::string what;
};
std::vector<Pending> g_pending;

void line(const std::string& t) {
  static FILE* f = fopen(getenv("FAKE_CUDART_TRACE"), "a");
  if (f) {
    fputs((t + "\n").c_str(), f);
    fflush(f);
  }
}
std::string place(const void* p) {
  auto it = g_allocs.upper_bound(static_cast<const char*>(p));
  if (it == g_allocs.begin()) return "host";
  --it;
  const size_t off = static_cast<const char*>(p) - it->first;
  if (off >= std::max<size_t>(it->second.bytes, 1)) return "host";
  return "#" + std::to_string(it->second.id) + "+" + std::to_string(off);
}
std::string name(cudaStream_t s) {
  char b[32];
  snprintf(b, sizeof b, "%p", (void*)s);
  return s == nullptr || s == cudaStreamLegacy ? "legacy" : b;
}
cudaStream_t plain(cudaStream_t s) { return s == cudaStreamLegacy ? nullptr : s; }
void pend(cudaStream_t s, const std::string& what) {
  line(what + " stream " + name(s));
  g_pending.push_back({plain(s), what});
}
void done(cudaStream_t s) {
  g_pending.erase(std::remove_if(g_pending.begin(), g_pending.end(), [&](const Pending& p) { return p.s == plain(s); }),
                  g_pending.end());
}
cudaError_t launch(const void* f, size_t smem, cudaStream_t s) {
  if (smem > (g_smem.count(f) ? g_smem[f] : 48 * 1024)) {
    line("TOO MUCH shared memory for " + g_kernels[f]);
    return cudaErrorInvalidValue;
  }
  const std::string k = g_kernels.count(f) ? g_kernels[f] : "?";
  line("launch " + k + " stream " + name(s));
  for (const Pending& p : g_pending)
    if (p.s != plain(s)) line("UNORDERED " + k + " stream " + name(s) + " after " + p.what + " stream " + name(p.s));
  return cudaSuccess;
}
int encode_tiled(...) { return 0; }
}  // namespace

extern "C" {
void fake_limit(size_t bytes) { g_limit = bytes; }  // cudaMalloc fails above this size
void fake_capturing(int on) { g_capturing = on; }
void fake_note(const char* t) { line(t); }

cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int) {
  memset(p, 0, sizeof *p);
  p->major = 10;
  p->minor = 3;
  p->multiProcessorCount = 152;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) {
    if (g_smem.count(f) && (size_t)v < g_smem[f]) line("LOWERED limit of " + g_kernels[f]);
    g_smem[f] = v;
  }
  return cudaSuccess;
}
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t bytes) {
  *p = nullptr;
  if (g_capturing) line("malloc in a capture");
  if (bytes > g_limit) {
    line("malloc refused " + std::to_string(bytes));
    return cudaErrorMemoryAllocation;
  }
  *p = malloc(std::max<size_t>(bytes, 1));
  memset(*p, 0xA5, bytes);
  g_allocs[static_cast<const char*>(*p)] = {g_next++, bytes};
  line("malloc " + place(*p) + " " + std::to_string(bytes));
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  if (!p) return cudaSuccess;
  line("free " + place(p));
  g_allocs.erase(static_cast<const char*>(p));
  free(p);
  return cudaSuccess;
}
cudaError_t cudaMemset(void* p, int v, size_t n) {
  memset(p, v, n);
  pend(nullptr, "memset " + place(p) + " " + std::to_string(n));
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t s) {
  memset(p, v, n);
  pend(s, "memset " + place(p) + " " + std::to_string(n));
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind k) {
  memcpy(d, s, n);
  if (k == cudaMemcpyHostToDevice) pend(nullptr, "copy to " + place(d) + " " + std::to_string(n));
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t st) {
  if (k != cudaMemcpyDeviceToDevice) memcpy(d, s, n);
  if (k == cudaMemcpyHostToDevice) pend(st, "copy to " + place(d) + " " + std::to_string(n));
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  *s = reinterpret_cast<cudaStream_t>(0x100000 + 16 * ++g_streams);
  g_own.push_back(*s);
  line("stream made " + name(*s));
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) {
  g_own.erase(std::remove(g_own.begin(), g_own.end(), s), g_own.end());
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) { done(s); return cudaSuccess; }
cudaError_t cudaDeviceSynchronize(void) { g_pending.clear(); return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus* st) {
  const bool own = std::find(g_own.begin(), g_own.end(), s) != g_own.end();
  *st = g_capturing && !own ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** p, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
  *p = reinterpret_cast<void*>(&encode_tiled);
  *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(f));
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void**, size_t smem, cudaStream_t s) { return launch(k, smem, s); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) { return launch(f, c->dynamicSmemBytes, c->stream); }
void __cudaRegisterFunction(void** h, const char* host, char* dev, const char* dname, int lim, uint3* a, uint3* b, dim3* c,
                            dim3* d, int* w) {
  g_kernels[host] = dname;
  using F = void (*)(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*, dim3*, int*);
  static F real = reinterpret_cast<F>(dlsym(RTLD_NEXT, "__cudaRegisterFunction"));
  if (real) real(h, host, dev, dname, lim, a, b, c, d, w);
}
}
