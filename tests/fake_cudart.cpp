// A stand-in for the CUDA runtime, linked under the library's objects so that
// its host code runs without a GPU: device memory is host memory, kernels do
// nothing but fill the few counters the plan reads back (a tree of one leaf),
// and every stream's work is counted, so that a buffer given back while some
// stream may still use it, or used before it is there, is noticed.  Not a GPU
// model: maps stay zero.
#include <cuda_runtime_api.h>

#include <sys/mman.h>

#include <algorithm>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>

namespace {

std::mutex mu;
std::map<const void *, std::string> names;               // kernels by host function
struct Block {
  size_t n;
  int stream;  // pooled memory: whose order it was taken in, and after which operation
  long op;
};
std::map<const char *, Block> blocks;                    // live device memory
typedef std::map<int, long> Clock;                       // stream -> operations known done
std::map<int, Clock> streams;                            // what each stream is ordered after
std::map<cudaEvent_t, Clock> events;
Clock host;                                              // what the host has waited for
long ops = 0, unordered = 0, mallocs = 0, fail_malloc = -1, launches = 0, fail_launch = -1;
cudaError_t pending = cudaSuccess;
size_t pool_used = 0, pool_held = 0;
const size_t total_mem = 280ull << 30;
size_t others = 10ull << 30;  // taken by other processes and libraries
long next_stream = 1, next_event = 1;

int id(cudaStream_t s) { return (int)(intptr_t)s; }
void merge(Clock &a, const Clock &b) {
  for (const auto &kv : b) a[kv.first] = std::max(a[kv.first], kv.second);
}
void enqueue(cudaStream_t s) { streams[id(s)][id(s)] = ++ops; }
// Memory goes back in the order of stream s (or, s < 0, of the host alone):
// every operation of every stream has to be known done there.
void check_free(int s) {
  Clock known = host;
  if (s >= 0) merge(known, streams[s]);
  for (const auto &st : streams) {
    const auto own = st.second.find(st.first);
    if (own != st.second.end() && known[st.first] < own->second) {
      unordered++;
      return;
    }
  }
}
// Use of an address in the order of stream s: pooled memory is there only
// after the operation that took it from the pool.
void check_use(const void *p, int s) {
  auto it = blocks.upper_bound(static_cast<const char *>(p));
  if (it == blocks.begin()) return;
  --it;
  if (static_cast<const char *>(p) >= it->first + it->second.n || it->second.op == 0) return;
  Clock known = host;
  merge(known, streams[s]);
  if (known[it->second.stream] < it->second.op) unordered++;
}
cudaError_t get(void **p, size_t n, bool pooled, cudaStream_t s) {
  std::lock_guard<std::mutex> l(mu);
  if (mallocs++ == fail_malloc) return cudaErrorMemoryAllocation;
  // (never touched pages cost nothing: a queue of gigabytes is only an address range)
  *p = mmap(nullptr, n ? n : 1, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE,
            -1, 0);
  if (*p == MAP_FAILED) return cudaErrorMemoryAllocation;
  if (pooled) enqueue(s);
  blocks[static_cast<char *>(*p)] = Block{n ? n : 1, id(s), pooled ? ops : 0};
  if (pooled) {
    pool_used += n ? n : 1;
    pool_held = std::max(pool_held, pool_used);
  }
  return cudaSuccess;
}
void put(void *p, bool pooled) {
  const auto it = blocks.find(static_cast<char *>(p));
  if (it == blocks.end()) return;
  if (pooled) pool_used -= it->second.n;
  munmap(p, it->second.n);
  blocks.erase(it);
}
void copy(void *d, const void *s, size_t n) {
  if (n <= (size_t)64 << 20) memcpy(d, s, n);
}
// The counters a plan reads: one root leaf, active, without direct stars.
void kernel(const void *f, void **args) {
  const std::string &n = names[f];
  auto word = [&](int k) { return *static_cast<int32_t **>(args[k]); };
  if (n.find("k_tree_top") != std::string::npos) {
    int32_t *info = word(3);
    info[0] = info[1] = info[2] = 1;
  } else if (n.find("k_compact_leaves") != std::string::npos) {
    *word(6) = 1;
  }
}

}  // namespace

extern "C" {

long fake_unordered() { return unordered; }
long fake_pool_idle() { return (long)(pool_held - pool_used); }
long fake_total_memory() { return (long)total_mem; }
long fake_mallocs() { return mallocs; }
long fake_launches() { return launches; }
void fake_others(size_t bytes) { others = bytes; }
// the n-th allocation or launch from fake_reset on fails
void fake_fail_malloc(long n) { fail_malloc = n; }
void fake_fail_launch(long n) { fail_launch = n; }
void fake_reset() {
  std::lock_guard<std::mutex> l(mu);
  for (auto &s : streams) merge(host, s.second);
  unordered = mallocs = launches = 0;
  fail_malloc = fail_launch = -1;
  pool_held = pool_used;
  others = 10ull << 30;
}

// registration and launches
void **__cudaRegisterFatBinary(void *) {
  static void *h;
  return &h;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *f, char *, const char *name, int, uint3 *, uint3 *,
                            dim3 *, dim3 *, int *) {
  names[f] = name;
}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
static thread_local struct { dim3 g, b; size_t smem; cudaStream_t st; } cfg;
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, cudaStream_t st) {
  cfg = {g, b, smem, st};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *smem, void *st) {
  *g = cfg.g;
  *b = cfg.b;
  *smem = cfg.smem;
  *static_cast<cudaStream_t *>(st) = cfg.st;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void **args, size_t, cudaStream_t st) {
  std::lock_guard<std::mutex> l(mu);
  if (launches++ == fail_launch) return pending = cudaErrorLaunchOutOfResources;
  kernel((const void *)k, args);
  enqueue(st);
  return cudaSuccess;
}
cudaError_t cudaLaunchKernel(const void *f, dim3, dim3, void **args, size_t, cudaStream_t st) {
  return __cudaLaunchKernel((cudaKernel_t)f, dim3(), dim3(), args, 0, st);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **args) {
  return __cudaLaunchKernel((cudaKernel_t)f, dim3(), dim3(), args, 0, c->stream);
}
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes *a, const void *) {
  memset(a, 0, sizeof *a);
  a->ptxVersion = a->binaryVersion = 103;
  a->maxThreadsPerBlock = 1024;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int,
                                                                   size_t, unsigned) {
  *n = 2;
  return cudaSuccess;
}

// device, errors
cudaError_t cudaGetDevice(int *d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int *n) {
  *n = 1;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount    ? 152
       : a == cudaDevAttrL2CacheSize          ? 129 << 20
       : a == cudaDevAttrComputeCapabilityMajor ? 10
       : a == cudaDevAttrComputeCapabilityMinor ? 3
       : a == cudaDevAttrMaxGridDimX          ? INT32_MAX
                                              : 1 << 16;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() {
  const cudaError_t e = pending;
  pending = cudaSuccess;
  return e;
}
cudaError_t cudaPeekAtLastError() { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "fake runtime"; }
cudaError_t cudaMemGetInfo(size_t *f, size_t *t) {
  *f = total_mem - others - pool_held;
  *t = total_mem;
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void **, const void *) { return cudaErrorInvalidSymbol; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *, const void *) {
  return cudaErrorInvalidValue;
}

// memory
cudaError_t cudaMalloc(void **p, size_t n) { return get(p, n, false, nullptr); }
cudaError_t cudaMallocAsync(void **p, size_t n, cudaStream_t s) { return get(p, n, true, s); }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) {
  *p = calloc(n, 1);
  return cudaSuccess;
}
cudaError_t cudaFreeHost(void *p) {
  free(p);
  return cudaSuccess;
}
cudaError_t cudaFree(void *p) {  // (waits for the device)
  std::lock_guard<std::mutex> l(mu);
  for (auto &s : streams) merge(host, s.second);
  put(p, false);
  return cudaSuccess;
}
cudaError_t cudaFreeAsync(void *p, cudaStream_t s) {
  std::lock_guard<std::mutex> l(mu);
  check_free(id(s));
  put(p, true);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t st) {
  std::lock_guard<std::mutex> l(mu);
  check_use(d, id(st));
  check_use(s, id(st));
  copy(d, s, n);
  enqueue(st);
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) {
  std::lock_guard<std::mutex> l(mu);
  check_use(d, 0);
  check_use(s, 0);
  copy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemset(void *d, int v, size_t n) {
  std::lock_guard<std::mutex> l(mu);
  check_use(d, 0);
  if (n <= (size_t)1 << 20) memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t st) {
  std::lock_guard<std::mutex> l(mu);
  check_use(d, id(st));
  if (n <= (size_t)1 << 20) memset(d, v, n);
  enqueue(st);
  return cudaSuccess;
}
cudaError_t cudaDeviceGetDefaultMemPool(cudaMemPool_t *p, int) {
  *p = nullptr;
  return cudaSuccess;
}
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void *) { return cudaSuccess; }
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t keep) {
  std::lock_guard<std::mutex> l(mu);
  pool_held = std::max(pool_used, std::min(pool_held, keep));
  return cudaSuccess;
}
cudaError_t cudaMemPoolGetAttribute(cudaMemPool_t, cudaMemPoolAttr a, void *v) {
  std::lock_guard<std::mutex> l(mu);
  *static_cast<uint64_t *>(v) = a == cudaMemPoolAttrUsedMemCurrent ? pool_used : pool_held;
  return cudaSuccess;
}

// streams and events
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
  std::lock_guard<std::mutex> l(mu);
  *s = (cudaStream_t)(intptr_t)next_stream++;
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  std::lock_guard<std::mutex> l(mu);
  merge(host, streams[id(s)]);
  return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
  std::lock_guard<std::mutex> l(mu);
  merge(streams[id(s)], events[e]);
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) {
  std::lock_guard<std::mutex> l(mu);
  *e = (cudaEvent_t)(intptr_t)next_event++;
  return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
  std::lock_guard<std::mutex> l(mu);
  events[e] = streams[id(s)];
  return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t e) {
  std::lock_guard<std::mutex> l(mu);
  merge(host, events[e]);
  return cudaSuccess;
}
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) {
  *ms = 0.f;
  return cudaSuccess;
}

}  // extern "C"
