// A CUDA runtime on the host for the tests of the library's host code: device
// memory is zeroed host memory, kernels do nothing, and every stream is a
// queue that runs as late as the runtime's documentation allows.
//   - Copies, sets and launches run when their stream is waited for (or the
//     device is, as cudaFree does).  The source of a copy from pageable host
//     memory is staged at the call.
//   - cudaMemcpy to the device and cudaMemset go to the legacy stream, whose
//     queue non-blocking streams do not wait for; cudaMemcpy to the host
//     drains the legacy stream alone and copies.
// fake_fail_alloc makes one device allocation fail, fake_on_launch runs a
// function when a kernel whose name contains a text is launched.
#include <driver_types.h>
#include <vector_types.h>

#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <deque>
#include <functional>
#include <map>
#include <string>
#include <vector>

#include "fake_cudart.h"

namespace {

struct Stream {
  std::deque<std::function<void()>> queue;
};
Stream g_legacy;
std::vector<Stream *> g_streams;
std::map<uintptr_t, size_t> g_device, g_pinned;
std::map<const void *, std::string> g_names;
std::map<const void *, std::vector<unsigned char>> g_vars;
cudaError_t g_last = cudaSuccess;
long g_allocs = 0, g_fail_at = -1, g_unordered = 0;
size_t g_uploaded = 0;
bool g_fail_pinned = false;
std::string g_first_unordered, g_hook_name, g_fail_launch;
std::function<std::function<void()>(void **)> g_hook;
std::map<std::string, long> g_launches;
struct Config {
  dim3 grid, block;
  size_t smem;
  cudaStream_t stream;
} g_config;

Stream *of(cudaStream_t s) { return s ? reinterpret_cast<Stream *>(s) : &g_legacy; }
void drain(Stream *s) {
  while (!s->queue.empty()) {
    auto f = std::move(s->queue.front());
    s->queue.pop_front();
    f();
  }
}
void drain_all() {
  drain(&g_legacy);
  for (Stream *s : g_streams) drain(s);
}
cudaError_t done(cudaError_t e) {
  if (e != cudaSuccess) g_last = e;
  return e;
}
bool inside(const std::map<uintptr_t, size_t> &m, const void *p, size_t n = 0) {
  auto it = m.upper_bound((uintptr_t)p);
  if (it == m.begin()) return false;
  --it;
  return (uintptr_t)p + n <= it->first + it->second && (uintptr_t)p < it->first + it->second;
}
// a copy on stream s, its pageable host source staged now
cudaError_t enqueue_copy(Stream *s, void *dst, const void *src, size_t n, cudaMemcpyKind kind) {
  if ((kind == cudaMemcpyHostToDevice || kind == cudaMemcpyDeviceToDevice) && !inside(g_device, dst, n))
    return done(cudaErrorInvalidValue);
  if ((kind == cudaMemcpyDeviceToHost || kind == cudaMemcpyDeviceToDevice) && !inside(g_device, src, n))
    return done(cudaErrorInvalidValue);
  if (kind == cudaMemcpyHostToDevice) g_uploaded += n;
  if (kind == cudaMemcpyHostToDevice && !inside(g_pinned, src)) {
    std::vector<unsigned char> stage((const unsigned char *)src, (const unsigned char *)src + n);
    s->queue.push_back([dst, stage] { std::memcpy(dst, stage.data(), stage.size()); });
  } else {
    s->queue.push_back([dst, src, n] { std::memcpy(dst, src, n); });
  }
  return cudaSuccess;
}

}  // namespace

// ---- controls
void fake_fail_alloc(long k) {
  g_allocs = 0;
  g_fail_at = k;
}
long fake_allocs() { return g_allocs; }
long fake_unordered(std::string *first) {
  if (first) *first = g_first_unordered;
  return g_unordered;
}
void fake_on_launch(const char *name, std::function<void()> f) {
  fake_on_launch_args(name, [f](void **) { return f; });
}
void fake_on_launch_args(const char *name, std::function<std::function<void()>(void **)> f) {
  g_hook_name = name;
  g_hook = std::move(f);
}
void fake_fail_pinned(bool fail) { g_fail_pinned = fail; }
void fake_fail_launch(const char *name) { g_fail_launch = name; }
long fake_launches(const char *name) {
  long n = 0;
  for (auto &l : g_launches)
    if (l.first.find(name) != std::string::npos) n += l.second;
  return n;
}
size_t fake_device_bytes() {
  size_t n = 0;
  for (auto &p : g_device) n += p.second;
  return n;
}
size_t fake_uploaded() { return g_uploaded; }
void fake_settle() { drain_all(); }

// ---- the runtime
extern "C" {

cudaError_t cudaMalloc(void **p, size_t n) {
  if (g_allocs++ == g_fail_at) return done(cudaErrorMemoryAllocation);
  *p = std::calloc(n ? n : 1, 1);
  g_device[(uintptr_t)*p] = n;
  return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
  drain_all();
  if (!p) return cudaSuccess;
  if (!g_device.erase((uintptr_t)p)) return done(cudaErrorInvalidValue);
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) {
  if (g_fail_pinned) return done(cudaErrorMemoryAllocation);
  *p = std::calloc(n, 1);
  g_pinned[(uintptr_t)*p] = n;
  return cudaSuccess;
}
cudaError_t cudaMallocHost(void **p, size_t n) { return cudaHostAlloc(p, n, 0); }
cudaError_t cudaFreeHost(void *p) {
  drain_all();
  g_pinned.erase((uintptr_t)p);
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *dst, const void *src, size_t n, cudaMemcpyKind kind, cudaStream_t s) {
  const cudaError_t e = enqueue_copy(of(s), dst, src, n, kind);
  if (e == cudaSuccess && kind == cudaMemcpyDeviceToHost && !inside(g_pinned, dst)) drain(of(s));
  return e;
}
cudaError_t cudaMemcpy(void *dst, const void *src, size_t n, cudaMemcpyKind kind) {
  const cudaError_t e = enqueue_copy(&g_legacy, dst, src, n, kind);
  if (e == cudaSuccess && kind == cudaMemcpyDeviceToHost) drain(&g_legacy);
  return e;
}
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t s) {
  if (n && !inside(g_device, p, n)) return done(cudaErrorInvalidValue);
  of(s)->queue.push_back([p, v, n] { std::memset(p, v, n); });
  return cudaSuccess;
}
cudaError_t cudaMemset(void *p, int v, size_t n) { return cudaMemsetAsync(p, v, n, nullptr); }
cudaError_t cudaMemcpyToSymbolAsync(const void *sym, const void *src, size_t n, size_t off, cudaMemcpyKind,
                                    cudaStream_t s) {
  auto it = g_vars.find(sym);
  if (it == g_vars.end() || off + n > it->second.size()) return done(cudaErrorInvalidSymbol);
  unsigned char *dst = it->second.data() + off;
  std::vector<unsigned char> stage((const unsigned char *)src, (const unsigned char *)src + n);
  of(s)->queue.push_back([dst, stage] { std::memcpy(dst, stage.data(), stage.size()); });
  return cudaSuccess;
}
cudaError_t cudaMemcpyToSymbol(const void *sym, const void *src, size_t n, size_t off, cudaMemcpyKind kind) {
  return cudaMemcpyToSymbolAsync(sym, src, n, off, kind, nullptr);
}
cudaError_t cudaGetSymbolAddress(void **p, const void *sym) {
  auto it = g_vars.find(sym);
  if (it == g_vars.end()) return done(cudaErrorInvalidSymbol);
  *p = it->second.data();
  g_device[(uintptr_t)*p] = it->second.size();
  return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *p) {
  std::memset(a, 0, sizeof(*a));
  a->type = inside(g_device, p) ? cudaMemoryTypeDevice : inside(g_pinned, p) ? cudaMemoryTypeHost : cudaMemoryTypeUnregistered;
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
  g_streams.push_back(new Stream);
  *s = reinterpret_cast<cudaStream_t>(g_streams.back());
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) {
  drain(of(s));
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  drain(of(s));
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) {
  *e = reinterpret_cast<cudaEvent_t>(new Stream *(nullptr));
  return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
  *reinterpret_cast<Stream **>(e) = of(s);
  return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t e) {
  if (Stream *s = *reinterpret_cast<Stream **>(e)) drain(s);
  return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t e, unsigned) { return cudaEventSynchronize(e); }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) {
  *ms = 0.f;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() {
  const cudaError_t e = g_last;
  g_last = cudaSuccess;
  return e;
}
const char *cudaGetErrorName(cudaError_t) { return "fake error"; }
const char *cudaGetErrorString(cudaError_t) { return "fake error"; }
cudaError_t cudaGetDevice(int *d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int *n) {
  *n = 1;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) {
  *v = 4;
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) {
  *n = 1;
  return cudaSuccess;
}

// launches
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t m, cudaStream_t s) {
  g_config = Config{g, b, m, s};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *m, void *s) {
  *g = g_config.grid;
  *b = g_config.block;
  *m = g_config.smem;
  *reinterpret_cast<cudaStream_t *>(s) = g_config.stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) {
  *k = reinterpret_cast<cudaKernel_t>(const_cast<void *>(f));
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void **args, size_t, cudaStream_t s) {
  const std::string &name = g_names[reinterpret_cast<const void *>(k)];
  if (!g_fail_launch.empty() && name.find(g_fail_launch) != std::string::npos) return done(cudaErrorLaunchOutOfResources);
  ++g_launches[name];
  if (s && !g_legacy.queue.empty() && !g_unordered++) g_first_unordered = name;
  if (!g_hook_name.empty() && name.find(g_hook_name) != std::string::npos) of(s)->queue.push_back(g_hook(args));
  return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **args) {
  return __cudaLaunchKernel(reinterpret_cast<cudaKernel_t>(const_cast<void *>(f)), c->gridDim, c->blockDim, args,
                            c->dynamicSmemBytes, c->stream);
}
void **__cudaRegisterFatBinary(void *) {
  static void *handle;
  return &handle;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *,
                            int *) {
  g_names[host] = name;
}
void __cudaRegisterVar(void **, char *host, char *, const char *, int, size_t size, int, int) {
  g_vars[host].resize(size);
}

// graphs and captures: not part of these tests
#define NOT_HERE(name) \
  cudaError_t name() { return done(cudaErrorNotSupported); }
NOT_HERE(cudaGraphAddNode)
NOT_HERE(cudaGraphConditionalHandleCreate)
NOT_HERE(cudaGraphCreate)
NOT_HERE(cudaGraphDestroy)
NOT_HERE(cudaGraphExecDestroy)
NOT_HERE(cudaGraphInstantiate)
NOT_HERE(cudaGraphLaunch)
NOT_HERE(cudaStreamBeginCapture)
NOT_HERE(cudaStreamBeginCaptureToGraph)
NOT_HERE(cudaStreamEndCapture)
NOT_HERE(cudaStreamGetCaptureInfo)
NOT_HERE(cudaStreamUpdateCaptureDependencies)

}  // extern "C"
