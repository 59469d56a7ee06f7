// A CUDA runtime of two devices on the host, for tests of the library's host
// side without a GPU: memory is host memory, copies and clears happen at once,
// kernels do not run.  It keeps what the real runtime keeps per device (a
// kernel's shared-memory limit), refuses launches beyond it, and accounts for
// memory pools.  Linked with the library's own objects in place of cudart.
#include <cuda.h>
#include <cuda_runtime_api.h>
#include <sys/mman.h>

#include <algorithm>
#include <cstring>
#include <map>
#include <mutex>
#include <string>

namespace {

constexpr int kDevices = 2;
constexpr size_t kDefaultShared = 48 << 10;

std::mutex g_mu;
thread_local int t_dev = 0;
thread_local cudaError_t t_last = cudaSuccess;
std::map<const void*, std::string> g_names;
std::map<std::pair<int, const void*>, int> g_shared;  // (device, kernel) -> allowed dynamic shared memory
std::map<std::string, long> g_launched[kDevices];

struct Pool {
  size_t used = 0, reserved = 0;
};
struct Block {
  size_t bytes;
  Pool* pool;
  unsigned long long pinned;  // pinned memory: the id of its context, else 0
};
std::map<void*, Block> g_blocks;
size_t g_limit = SIZE_MAX;  // of a pool's reserved memory
unsigned long long g_ctx = 1;   // contexts have ids g_ctx + device; a reset moves on
long g_pinned_taken = 0, g_pinned_given = 0;

cudaError_t done(cudaError_t e) {
  if (e != cudaSuccess) t_last = e;
  return e;
}

cudaError_t take(void** p, size_t bytes, Pool* pool) {
  std::lock_guard<std::mutex> lock(g_mu);
  if (pool && pool->used + bytes > g_limit) return done(cudaErrorMemoryAllocation);
  void* m = mmap(nullptr, bytes ? bytes : 1, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
  if (m == MAP_FAILED) return done(cudaErrorMemoryAllocation);
  g_blocks[m] = Block{bytes ? bytes : 1, pool, 0};
  if (pool) {  // idle reserved memory serves any request, whatever blocks it lies in
    pool->used += bytes;
    pool->reserved = std::max(pool->reserved, pool->used);
  }
  *p = m;
  return cudaSuccess;
}

cudaError_t give(void* p) {
  if (!p) return cudaSuccess;
  std::lock_guard<std::mutex> lock(g_mu);
  auto it = g_blocks.find(p);
  if (it == g_blocks.end()) return done(cudaErrorInvalidValue);
  if (it->second.pool) it->second.pool->used -= it->second.bytes;
  munmap(p, it->second.bytes);
  g_blocks.erase(it);
  return cudaSuccess;
}

struct Launch {
  dim3 grid, block;
  size_t shared;
  void* stream;
};
thread_local Launch t_launch;

}  // namespace

extern "C" {

// ---- what the tests ask and set
void fake_limit(size_t bytes) { g_limit = bytes; }
long fake_launches(int dev, const char* part) {  // launches of kernels whose name contains part
  std::lock_guard<std::mutex> lock(g_mu);
  long n = 0;
  for (auto& e : g_launched[dev])
    if (e.first.find(part) != std::string::npos) n += e.second;
  return n;
}
long fake_pinned_taken(void) { return g_pinned_taken; }
long fake_pinned_given(void) { return g_pinned_given; }
void fake_reset(void) {  // a device reset: new contexts, pinned memory is gone
  std::lock_guard<std::mutex> lock(g_mu);
  g_ctx += kDevices;
  for (auto it = g_blocks.begin(); it != g_blocks.end();) {
    if (it->second.pinned) {
      munmap(it->first, it->second.bytes);
      it = g_blocks.erase(it);
    } else {
      ++it;
    }
  }
}
size_t fake_reserved(void) {
  std::lock_guard<std::mutex> lock(g_mu);
  size_t n = 0;
  std::map<Pool*, bool> seen;
  for (auto& b : g_blocks)
    if (b.second.pool && !seen[b.second.pool]) {
      seen[b.second.pool] = true;
      n += b.second.pool->reserved;
    }
  return n;
}

// ---- devices
cudaError_t cudaSetDevice(int dev) {
  if (dev < 0 || dev >= kDevices) return done(cudaErrorInvalidDevice);
  t_dev = dev;
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* dev) {
  *dev = t_dev;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, enum cudaDeviceAttr attr, int) {
  *v = attr == cudaDevAttrMultiProcessorCount ? 152 : 0;
  return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize(void) { return cudaSuccess; }
cudaError_t cudaGetLastError(void) {
  cudaError_t e = t_last;
  t_last = cudaSuccess;
  return e;
}
const char* cudaGetErrorString(cudaError_t e) { return e == cudaErrorInvalidValue ? "invalid argument" : "fake CUDA error"; }
static CUresult fake_ctx_current(CUcontext* c) {
  *c = (CUcontext)(g_ctx + t_dev);
  return CUDA_SUCCESS;
}
static CUresult fake_ctx_id(CUcontext c, unsigned long long* id) {
  *id = (unsigned long long)c;
  return CUDA_SUCCESS;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char* name, void** f, unsigned int, unsigned long long,
                                             enum cudaDriverEntryPointQueryResult* r) {
  *f = !std::strcmp(name, "cuCtxGetCurrent") ? (void*)fake_ctx_current
                                             : (!std::strcmp(name, "cuCtxGetId") ? (void*)fake_ctx_id : nullptr);
  if (r) *r = *f ? cudaDriverEntryPointSuccess : cudaDriverEntryPointSymbolNotFound;
  return cudaSuccess;
}

// ---- memory
cudaError_t cudaMalloc(void** p, size_t n) { return take(p, n, nullptr); }
cudaError_t cudaMallocHost(void** p, size_t n) { return take(p, n, nullptr); }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned int) {
  const cudaError_t e = take(p, n, nullptr);
  std::lock_guard<std::mutex> lock(g_mu);
  g_pinned_taken++;
  if (e == cudaSuccess) g_blocks[*p].pinned = g_ctx + t_dev;
  return e;
}
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { return take(p, n, nullptr); }
cudaError_t cudaFree(void* p) { return give(p); }
cudaError_t cudaFreeHost(void* p) {
  {
    std::lock_guard<std::mutex> lock(g_mu);
    g_pinned_given++;
  }
  return give(p);
}
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { return give(p); }
cudaError_t cudaMemPoolCreate(cudaMemPool_t* pool, const struct cudaMemPoolProps*) {
  *pool = (cudaMemPool_t)(new Pool);
  return cudaSuccess;
}
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, enum cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaMemPoolGetAttribute(cudaMemPool_t pool, enum cudaMemPoolAttr attr, void* v) {
  std::lock_guard<std::mutex> lock(g_mu);
  const Pool* P = (const Pool*)pool;
  *(unsigned long long*)v = attr == cudaMemPoolAttrUsedMemCurrent ? P->used : P->reserved;
  return cudaSuccess;
}
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t pool, size_t keep) {
  std::lock_guard<std::mutex> lock(g_mu);
  Pool* P = (Pool*)pool;
  P->reserved = std::min(P->reserved, std::max(P->used, keep));
  return cudaSuccess;
}
cudaError_t cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t pool, cudaStream_t) { return take(p, n, (Pool*)pool); }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, enum cudaMemcpyKind) {
  std::memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, enum cudaMemcpyKind k, cudaStream_t) { return cudaMemcpy(d, s, n, k); }
cudaError_t cudaMemset(void* d, int v, size_t n) {
  std::memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { return cudaMemset(d, v, n); }
cudaError_t cudaGetSymbolAddress(void** p, const void* s) {
  *p = (void*)s;
  return cudaSuccess;
}

// ---- streams, events, graphs: everything has happened when a call returns
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned int) {
  *s = (cudaStream_t)0x1000;
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned int) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, enum cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
  *g = (cudaGraph_t)0x2000;
  return cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t, enum cudaStreamCaptureStatus* s) {
  *s = cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaThreadExchangeStreamCaptureMode(enum cudaStreamCaptureMode*) { return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
  *e = (cudaGraphExec_t)0x3000;
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) {
  *e = (cudaEvent_t)0x4000;
  return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned int) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t, cudaStream_t, unsigned int) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  *ms = 1.0f;
  return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(struct cudaPointerAttributes* a, const void*) {
  std::memset(a, 0, sizeof(*a));
  a->type = cudaMemoryTypeHost;
  return cudaSuccess;
}

// ---- kernels
cudaError_t cudaFuncSetAttribute(const void* f, enum cudaFuncAttribute attr, int v) {
  std::lock_guard<std::mutex> lock(g_mu);
  if (attr == cudaFuncAttributeMaxDynamicSharedMemorySize) g_shared[{t_dev, f}] = v;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned int) {
  *n = 2;
  return cudaSuccess;
}
void** __cudaRegisterFatBinary(void*) {
  static void* handle;
  return &handle;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* f, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  std::lock_guard<std::mutex> lock(g_mu);
  g_names[f] = name;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t shared, struct CUstream_st* stream) {
  t_launch = Launch{grid, block, shared, stream};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* shared, void* stream) {
  *grid = t_launch.grid;
  *block = t_launch.block;
  *shared = t_launch.shared;
  *(void**)stream = t_launch.stream;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3 block, void**, size_t shared, cudaStream_t) {
  std::lock_guard<std::mutex> lock(g_mu);
  const void* f = (const void*)k;
  auto it = g_shared.find({t_dev, f});
  const size_t allowed = std::max(kDefaultShared, it == g_shared.end() ? (size_t)0 : (size_t)it->second);
  if (shared > allowed || !grid.x || !grid.y || !block.x || block.x > 1024) return done(cudaErrorInvalidValue);
  g_launched[t_dev][g_names[f]]++;
  return cudaSuccess;
}

}  // extern "C"
