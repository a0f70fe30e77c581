// A CUDA runtime without a GPU, for tests of the library's host code on the CPU: device memory is host
// memory under a budget, kernels do nothing but are checked (a launch needs the shared memory that
// its function was opted in to on the current device) and counted, and errors are planted by the test.
// Linked with the library's objects in place of the runtime.
#include <cstdlib>
#include <cstring>
#include <cuda.h>
#include <cuda_runtime_api.h>

#include <map>
#include <mutex>
#include <set>
#include <string>
#include <utility>

namespace {
struct Block {
  size_t bytes;
  bool marked;
};
constexpr size_t DEFAULT_SMEM = 48 << 10, STATIC_SMEM = 256;
std::recursive_mutex g_mutex;
std::map<void *, Block> g_blocks;                               // cudaMalloc and pool blocks
std::set<void *> g_pool_blocks;
std::map<const void *, std::string> g_names;                    // host function -> kernel name
std::map<std::string, long> g_launches;
std::map<std::pair<const void *, int>, size_t> g_optin;         // (function, device) -> shared memory
size_t g_live = 0, g_peak = 0, g_budget = ~size_t(0);
size_t g_pool_used = 0, g_pool_held = 0, g_pool_keep = 0;       // of the one pool: blocks out, memory reserved
long g_mallocs = 0, g_fail_optin = 0;
bool g_capturing = false;
thread_local int t_device = 0;
thread_local cudaError_t t_last = cudaSuccess;
thread_local struct { dim3 grid, block; size_t smem; cudaStream_t stream; } t_call;

cudaError_t done(cudaError_t e) { return e == cudaSuccess ? e : t_last = e; }

cudaError_t launched(const void *func, size_t smem) {
  std::lock_guard<std::recursive_mutex> lock(g_mutex);
  auto it = g_optin.find({func, t_device});
  const size_t most = it == g_optin.end() ? DEFAULT_SMEM - STATIC_SMEM : it->second;
  if (smem > most) return done(cudaErrorInvalidValue);
  ++g_launches[g_names[func]];
  return cudaSuccess;
}

CUresult encode_tiled(CUtensorMap *map, CUtensorMapDataType, cuuint32_t, void *base, const cuuint64_t *, const cuuint64_t *,
                      const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                      CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
  std::memset(map, 0, sizeof *map);
  std::memcpy(map, &base, sizeof base);
  return CUDA_SUCCESS;
}
}  // namespace

extern "C" {
// ---- what the tests set and read
void fake_budget(size_t bytes) { g_budget = bytes; }
size_t fake_live() { return g_live; }
size_t fake_peak() {  // the most that was live since the last call
  const size_t peak = g_peak;
  g_peak = g_live;
  return peak;
}
long fake_mallocs() { return g_mallocs; }
void fake_mark() {
  for (auto &b : g_blocks) b.second.marked = true;
}
long fake_marked() {
  long n = 0;
  for (auto &b : g_blocks) n += b.second.marked;
  return n;
}
void fake_capturing(int on) { g_capturing = on != 0; }
void fake_fail_optin(long n) { g_fail_optin = n; }
size_t fake_pool_held() { return g_pool_held; }
long fake_launches(const char *part) {
  long n = 0;
  for (auto &l : g_launches)
    if (l.first.find(part) != std::string::npos) n += l.second;
  return n;
}

// ---- registration and launches
void **__cudaRegisterFatBinary(void *) {
  static void *handle;
  return &handle;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *,
                            int *) {
  g_names[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, struct CUstream_st *stream) {
  t_call = {grid, block, smem, stream};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void *stream) {
  *grid = t_call.grid, *block = t_call.block, *smem = t_call.smem;
  *static_cast<cudaStream_t *>(stream) = t_call.stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *kernel, const void *func) {
  *kernel = reinterpret_cast<cudaKernel_t>(const_cast<void *>(func));
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t kernel, dim3, dim3, void **, size_t smem, cudaStream_t) {
  return launched(kernel, smem);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *cfg, const void *func, void **) {
  return launched(func, cfg->dynamicSmemBytes);
}
cudaError_t cudaFuncSetAttribute(const void *func, cudaFuncAttribute attr, int value) {
  std::lock_guard<std::recursive_mutex> lock(g_mutex);
  if (attr != cudaFuncAttributeMaxDynamicSharedMemorySize) return cudaSuccess;
  if (g_fail_optin > 0) {
    --g_fail_optin;
    return done(cudaErrorUnknown);
  }
  g_optin[{func, t_device}] = value;
  return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes *a, const void *) {
  std::memset(a, 0, sizeof *a);
  a->sharedSizeBytes = STATIC_SMEM;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *, const cudaLaunchConfig_t *) {
  *n = 8;
  return cudaSuccess;
}

// ---- devices and errors
cudaError_t cudaGetDevice(int *dev) { return *dev = t_device, cudaSuccess; }
cudaError_t cudaSetDevice(int dev) { return t_device = dev, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 227 << 10 : 1;
  return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { return cudaStreamSynchronize(nullptr); }
cudaError_t cudaGetLastError() {
  const cudaError_t e = t_last;
  t_last = cudaSuccess;
  return e;
}
cudaError_t cudaPeekAtLastError() { return t_last; }
const char *cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "planted"; }
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **fn, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult *q) {
  *fn = reinterpret_cast<void *>(&encode_tiled);
  if (q) *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void **p, const void *) { return *p = nullptr, done(cudaErrorInvalidSymbol); }

// ---- memory
cudaError_t cudaMalloc(void **p, size_t bytes) {
  std::lock_guard<std::recursive_mutex> lock(g_mutex);
  ++g_mallocs;
  *p = nullptr;
  if (g_live + g_pool_held + bytes > g_budget) return done(cudaErrorMemoryAllocation);
  *p = std::aligned_alloc(1024, (bytes + 1023) / 1024 * 1024);
  std::memset(*p, 0, bytes < (1u << 22) ? bytes : (1u << 22));
  g_blocks[*p] = {bytes, false};
  g_live += bytes;
  if (g_live > g_peak) g_peak = g_live;
  return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
  std::lock_guard<std::recursive_mutex> lock(g_mutex);
  if (!p) return cudaSuccess;
  auto it = g_blocks.find(p);
  if (it == g_blocks.end()) return done(cudaErrorInvalidValue);
  g_live -= it->second.bytes;
  g_blocks.erase(it);
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaMemGetInfo(size_t *free_bytes, size_t *total) {
  *free_bytes = g_budget - g_live - g_pool_held;
  *total = g_budget;
  return cudaSuccess;
}
cudaError_t cudaMemPoolCreate(cudaMemPool_t *pool, const cudaMemPoolProps *) {
  static int one;
  *pool = reinterpret_cast<cudaMemPool_t>(&one);
  return cudaSuccess;
}
cudaError_t cudaMemPoolDestroy(cudaMemPool_t) { return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr a, void *v) {
  if (a == cudaMemPoolAttrReleaseThreshold) g_pool_keep = *static_cast<uint64_t *>(v);
  return cudaSuccess;
}
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t keep) {
  std::lock_guard<std::recursive_mutex> lock(g_mutex);
  g_pool_held = g_pool_used > keep ? g_pool_used : g_pool_held < keep ? g_pool_held : keep;
  return cudaSuccess;
}
cudaError_t cudaMallocFromPoolAsync(void **p, size_t bytes, cudaMemPool_t, cudaStream_t) {
  std::lock_guard<std::recursive_mutex> lock(g_mutex);
  const size_t more = g_pool_used + bytes > g_pool_held ? g_pool_used + bytes - g_pool_held : 0;
  if (g_live + g_pool_held + more > g_budget) return done(cudaErrorMemoryAllocation);
  g_pool_held += more;
  g_pool_used += bytes;
  *p = std::aligned_alloc(1024, (bytes + 1023) / 1024 * 1024);
  g_blocks[*p] = {bytes, false};
  return cudaSuccess;
}
cudaError_t cudaFreeAsync(void *p, cudaStream_t) {
  std::lock_guard<std::recursive_mutex> lock(g_mutex);
  g_pool_used -= g_blocks[p].bytes;
  g_blocks.erase(p);
  std::free(p);
  return cudaSuccess;
}
// a pool returns what it holds beyond its threshold when something is synchronised
cudaError_t cudaStreamSynchronize(cudaStream_t) {
  std::lock_guard<std::recursive_mutex> lock(g_mutex);
  const size_t keep = g_pool_used > g_pool_keep ? g_pool_used : g_pool_keep;
  if (g_pool_held > keep) g_pool_held = keep;
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { return std::memcpy(d, s, n), cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *, size_t n, cudaMemcpyKind, cudaStream_t) {
  if (n == 4) std::memset(d, 0, n);  // the device's error word
  return cudaSuccess;
}
cudaError_t cudaMemcpy2D(void *, size_t, const void *, size_t, size_t, size_t, cudaMemcpyKind) { return cudaSuccess; }
cudaError_t cudaMemcpy2DAsync(void *, size_t, const void *, size_t, size_t, size_t, cudaMemcpyKind, cudaStream_t) {
  return cudaSuccess;
}
cudaError_t cudaMemset(void *, int, size_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *, int, size_t, cudaStream_t) { return cudaSuccess; }

// ---- streams, events and graphs
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
  return *s = reinterpret_cast<cudaStream_t>(std::malloc(1)), cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) { return std::free(s), cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *st) {
  *st = g_capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) {
  return *g = reinterpret_cast<cudaGraph_t>(std::malloc(1)), cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t, unsigned long long) {
  return *x = reinterpret_cast<cudaGraphExec_t>(std::malloc(1)), cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) { return std::free(g), cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) { return std::free(x), cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) {
  ++g_launches["decode graph"];
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) {
  return *e = reinterpret_cast<cudaEvent_t>(std::malloc(1)), cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t e) { return std::free(e), cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { return *ms = 0.f, cudaSuccess; }
}
