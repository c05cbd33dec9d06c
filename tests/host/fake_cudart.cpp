// A stand-in for the CUDA runtime on a machine without a GPU, linked with the
// library's objects by tests/test_host_runtime.py.  Device memory is host
// memory, kernels are recorded and not run, and the calls behave as CUDA's
// documentation allows them to:
//   * asynchronous copies, from pageable memory too, are carried out when the
//     stream is next waited for;
//   * a function attribute belongs to the device that was current when it was
//     set, and a cluster of more than 8 CTAs needs it;
//   * a launch of zero blocks is an error.
// operator delete overwrites what it frees, so that a copy from freed memory shows.
#include <cuda_runtime_api.h>
#include <malloc.h>
#include <unistd.h>

#include <atomic>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <new>
#include <set>
#include <string>
#include <utility>
#include <vector>

namespace {
struct Op { int kind; void* dst; const void* src; size_t n; std::string then; };   // kind 0: copy, 1: copy from the host, 2: set
std::recursive_mutex mu;
std::vector<Op>& ops() { static auto* v = new std::vector<Op>; return *v; }
std::map<const char*, size_t>& device() { static auto* m = new std::map<const char*, size_t>; return *m; }
std::map<const void*, std::string>& names() { static auto* m = new std::map<const void*, std::string>; return *m; }
std::set<std::pair<int, const void*>>& wide() { static auto* s = new std::set<std::pair<int, const void*>>; return *s; }
std::string& log_() { static auto* s = new std::string; return *s; }
std::atomic<int> query_ms{0}, fail_new{-1}, cur_device{0};
thread_local cudaError_t last = cudaSuccess;
thread_local struct { dim3 g, b; size_t s; void* st; } conf;
long long changed = 0, copied = 0;

bool on_device(const void* p) {
  auto it = device().upper_bound((const char*)p);
  if (it == device().begin()) return false;
  --it;
  return (const char*)p < it->first + it->second;
}
void run_ops() {
  std::lock_guard<std::recursive_mutex> l(mu);
  for (Op& o : ops()) {
    if (o.kind == 2) { memset(o.dst, (int)(intptr_t)o.src, o.n); continue; }
    if (o.kind == 1) {
      copied += 1;
      if (memcmp(o.then.data(), o.src, o.n) != 0) changed += 1;
    }
    memmove(o.dst, o.src, o.n);
  }
  ops().clear();
}
cudaError_t err(cudaError_t e) { last = e; return e; }
cudaError_t launched(const void* f, dim3 g, dim3 b, unsigned cluster) {
  std::lock_guard<std::recursive_mutex> l(mu);
  if (g.x == 0 || g.y == 0 || g.z == 0 || b.x == 0 || b.x > 1024) return err(cudaErrorInvalidConfiguration);
  if (cluster > 8 && !wide().count({cur_device, f})) return err(cudaErrorInvalidClusterSize);
  log_() += names()[f] + " " + std::to_string(g.x) + " " + std::to_string(cluster) + "\n";
  return cudaSuccess;
}
unsigned cluster_of(const cudaLaunchConfig_t* c) {
  for (unsigned k = 0; k < c->numAttrs; ++k)
    if (c->attrs[k].id == cudaLaunchAttributeClusterDimension) return c->attrs[k].val.clusterDim.x;
  return 1;
}
}  // namespace

void* operator new(size_t n) {
  if (fail_new >= 0 && fail_new.fetch_sub(1) == 0) throw std::bad_alloc();
  void* p = malloc(n ? n : 1);
  if (!p) throw std::bad_alloc();
  return p;
}
void operator delete(void* p) noexcept {
  if (p) memset(p, 0xdd, malloc_usable_size(p));
  free(p);
}
void operator delete(void* p, size_t) noexcept { operator delete(p); }

extern "C" {
// the tests' side
void fake_set_device(int d) { cur_device = d; }
void fake_query_ms(int ms) { query_ms = ms; }
void fake_fail_new(int k) { fail_new = k; }                 // the k-th allocation from now throws; -1: none
long long fake_copied() { return copied; }                  // copies from the host carried out
long long fake_changed() { return changed; }                // those whose source was no longer what it was
const char* fake_launches() { return log_().c_str(); }      // a line per launch: name, blocks, CTAs a cluster
void fake_clear() { log_().clear(); }

// the runtime's side
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* f, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) { names()[f] = name; }
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t s, struct CUstream_st* st) { conf = {g, b, s, st}; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* s, void* st) {
  *g = conf.g; *b = conf.b; *s = conf.s; *(void**)st = conf.st;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void**, size_t, cudaStream_t) { return launched((const void*)k, g, b, 1); }
cudaError_t cudaLaunchKernel(const void* f, dim3 g, dim3 b, void**, size_t, cudaStream_t) { return launched(f, g, b, 1); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) { return launched(f, c->gridDim, c->blockDim, cluster_of(c)); }
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
  std::lock_guard<std::recursive_mutex> l(mu);
  if (a == cudaFuncAttributeNonPortableClusterSizeAllowed && v) wide().insert({cur_device, f});
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void* f, const cudaLaunchConfig_t* c) {
  std::lock_guard<std::recursive_mutex> l(mu);
  if (cluster_of(c) > 8 && !wide().count({cur_device, f})) return err(cudaErrorInvalidClusterSize);
  *n = 1;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  if (query_ms > 0) usleep(1000 * query_ms);
  *n = 4;
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) { *d = cur_device; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) { *v = a == cudaDevAttrMultiProcessorCount ? 152 : 0; return cudaSuccess; }
cudaError_t cudaGetLastError() { const cudaError_t e = last; last = cudaSuccess; return e; }
const char* cudaGetErrorString(cudaError_t) { return "an error of the stand-in runtime"; }
cudaError_t cudaGetSymbolAddress(void** p, const void* s) { *p = const_cast<void*>(s); return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) {
  std::lock_guard<std::recursive_mutex> l(mu);
  if (!(*p = calloc(n, 1))) return err(cudaErrorMemoryAllocation);
  device()[(const char*)*p] = n;
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  run_ops();
  std::lock_guard<std::recursive_mutex> l(mu);
  device().erase((const char*)p);
  free(p);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t) {
  std::lock_guard<std::recursive_mutex> l(mu);
  const bool host = k == cudaMemcpyHostToDevice && !on_device(s);
  ops().push_back({host ? 1 : 0, d, s, n, host ? std::string((const char*)s, n) : std::string()});
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
  run_ops();
  memmove(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemset(void* d, int v, size_t n) { run_ops(); memset(d, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
  std::lock_guard<std::recursive_mutex> l(mu);
  ops().push_back({2, d, (const void*)(intptr_t)v, n, {}});
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { run_ops(); return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) { *s = cudaStreamCaptureStatusNone; return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 0.f; return cudaSuccess; }
}
