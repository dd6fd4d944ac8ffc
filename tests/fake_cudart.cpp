// A CUDA runtime without a GPU, for tests of the library's host code: "device" memory is host memory with a
// device ordinal, copies are memcpy, kernels do not run.  It keeps a log of copies and launches, refuses a
// launch whose dynamic shared memory is above the function's limit on the current device, and reports
// which launches were handed a watched pointer.  Linked with the library's object files in place of libcudart.
#include <cuda.h>
#include <cuda_runtime_api.h>

#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

#include "qg_internal.h"

namespace {

struct Mem {
  size_t n;
  int dev, type;
};
struct Entry {
  std::string what;  // "copy" or the kernel's mangled name
  const void *dst, *src;
  size_t n;
};
int g_dev = 0;
const void *g_watch = nullptr;
long long g_hits = 0;
std::map<uintptr_t, Mem> g_mem;
std::vector<Entry> g_log;
std::map<const void *, std::string> g_names;
std::map<std::pair<const void *, int>, size_t> g_limit;

void *take(size_t n, int dev, int type) {
  void *p = aligned_alloc(256, (n + 511) / 256 * 256);
  std::memset(p, 0, n);
  g_mem[(uintptr_t)p] = {n, dev, type};
  return p;
}

// Bytes of a kernel's first parameter that may be searched for a pointer (structures only).
size_t first_bytes(const std::string &name) {
  if (name.find("k_epi") != std::string::npos) return 64;  // the leading pointers of EpiArgs
  for (const char *k : {"k_s1", "k_s2", "k_s3", "k_s4", "k_s5", "k_gbus", "k_finish"})
    if (name.find(k) != std::string::npos)
      return name.find("df32") != std::string::npos ? sizeof(qg::Dev<float, qg::df32>) : sizeof(qg::Dev<double, double>);
  return 0;
}

cudaError_t launched(const void *func, void **args, size_t smem) {
  const std::string &name = g_names[func];
  const auto lim = g_limit.find({func, g_dev});
  if (smem > 48 * 1024 && (lim == g_limit.end() || smem > lim->second)) return cudaErrorInvalidValue;
  g_log.push_back({name, nullptr, nullptr, 0});
  if (g_watch)
    for (size_t o = 0, n = first_bytes(name); o + sizeof(void *) <= n; o += sizeof(void *)) {
      const void *p;
      std::memcpy(&p, static_cast<const char *>(args[0]) + o, sizeof(p));
      if (p == g_watch) {
        ++g_hits;
        break;
      }
    }
  return cudaSuccess;
}

CUresult encode(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
  return CUDA_SUCCESS;
}

}  // namespace

extern "C" {

// what the tests drive it with
void fake_set_device(int dev) { g_dev = dev; }
void *fake_alloc(size_t n, int dev, int type) { return take(n, dev, type); }
void fake_watch(const void *p) {
  g_watch = p;
  g_hits = 0;
  g_log.clear();
}
long long fake_hits() { return g_hits; }
// Copies into dst since the last fake_watch that came after the last launch.
long long fake_copies_to(const void *dst) {
  long long n = 0;
  for (const Entry &e : g_log) n = e.what != "copy" ? 0 : n + (e.dst == dst ? 1 : 0);
  return n;
}

cudaError_t cudaGetDevice(int *dev) { *dev = g_dev; return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int *n) { *n = 2; return cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp *p, int) {
  std::memset(p, 0, sizeof(*p));
  p->major = 10;
  p->minor = 3;
  p->multiProcessorCount = 152;
  return cudaSuccess;
}
cudaError_t cudaMalloc(void **p, size_t n) { *p = take(n, g_dev, cudaMemoryTypeDevice); return cudaSuccess; }
cudaError_t cudaFree(void *p) {
  if (g_mem.erase((uintptr_t)p)) std::free(p);
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) {
  std::memmove(d, s, n);
  g_log.push_back({"copy", d, s, n});
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind k, cudaStream_t) { return cudaMemcpy(d, s, n, k); }
cudaError_t cudaMemset(void *d, int v, size_t n) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *p) {
  std::memset(a, 0, sizeof(*a));
  auto it = g_mem.upper_bound((uintptr_t)p);
  if (it == g_mem.begin()) return cudaSuccess;  // cudaMemoryTypeUnregistered
  --it;
  if ((uintptr_t)p >= it->first + it->second.n) return cudaSuccess;
  a->type = (cudaMemoryType)it->second.type;
  a->device = it->second.dev;
  a->devicePointer = const_cast<void *>(p);
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute a, int v) {
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) g_limit[{f, g_dev}] = (size_t)v;
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void **p, const void *) { *p = take(size_t(32) << 20, g_dev, cudaMemoryTypeDevice); return cudaSuccess; }
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **p, unsigned, unsigned long long, cudaDriverEntryPointQueryResult *q) {
  *p = (void *)&encode;
  *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "refused by the fake runtime"; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s) { *s = cudaStreamCaptureStatusNone; return cudaSuccess; }

cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **args) { return launched(f, args, c->dynamicSmemBytes); }
static size_t g_call_smem;
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t smem, cudaStream_t) { g_call_smem = smem; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *smem, void *stream) {
  *g = *b = dim3{1, 1, 1};
  *smem = g_call_smem;
  *static_cast<cudaStream_t *>(stream) = nullptr;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) { *k = (cudaKernel_t)const_cast<void *>(f); return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void **args, size_t smem, cudaStream_t) {
  return launched((const void *)k, args, smem);
}
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, void *, void *, void *, void *, int *) {
  g_names[host] = name;
}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}

// not reached by the tests
cudaError_t cudaEventCreate(cudaEvent_t *) { return cudaErrorNotSupported; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaErrorNotSupported; }
cudaError_t cudaEventElapsedTime(float *, cudaEvent_t, cudaEvent_t) { return cudaErrorNotSupported; }
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaErrorNotSupported; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t, cudaStream_t, unsigned) { return cudaErrorNotSupported; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaErrorNotSupported; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaErrorNotSupported; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaErrorNotSupported; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *, cudaGraph_t, unsigned long long) { return cudaErrorNotSupported; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaErrorNotSupported; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *) { return cudaErrorNotSupported; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *, unsigned) { return cudaErrorNotSupported; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaErrorNotSupported; }

}  // extern "C"
