// A CUDA runtime made of host memory for the tests of the library's host code:
// loaded before the library, its functions stand in for libcudart's.  Two
// devices with different SM counts; kernels do nothing but are checked and
// recorded; stream order is program order.  It refuses what the real runtime
// refuses: a launch with more than 48 KB of dynamic shared memory on a device
// where the kernel has no such attribute, a pool of a context that was reset,
// an allocation beyond the device's memory.
#include <cuda_runtime_api.h>
#include <cuda.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

namespace {
struct Block {
  size_t bytes;
  int dev;
  void* pool;
};
struct Pool {
  int dev, generation;
  size_t threshold, idle;
};
const int kDevices = 2;
const int kSms[kDevices] = {152, 20};
int g_dev = 0, g_generation[kDevices] = {1, 1};
size_t g_capacity = (size_t)64 << 30, g_used[kDevices];
std::map<void*, Block> g_blocks;
std::map<void*, Pool> g_pools;
std::map<std::pair<int, const void*>, int> g_smem;
std::map<const void*, std::string> g_names;
std::map<const void*, std::pair<size_t, void*>> g_symbols;   // size, device address
int g_launches, g_dead_pool_uses, g_blocking_copies;
unsigned g_max_persistent_grid;
const double* g_last_K;          // k_poses_float's second argument
double g_K[4];
bool g_have_K;
cudaError_t g_last = cudaSuccess;

cudaError_t set(cudaError_t e) {
  if (e != cudaSuccess) g_last = e;
  return e;
}

size_t idle_bytes(int dev) {
  size_t n = 0;
  for (auto& p : g_pools)
    if (p.second.dev == dev && p.second.generation == g_generation[dev]) n += p.second.idle;
  return n;
}

// `reuse`: the pool whose idle bytes serve the allocation
cudaError_t take(void** out, size_t n, Pool* reuse, void* pool) {
  *out = nullptr;
  const size_t from_idle = reuse ? (reuse->idle < n ? reuse->idle : n) : 0;
  if (g_used[g_dev] + idle_bytes(g_dev) + n - from_idle > g_capacity)
    return set(cudaErrorMemoryAllocation);
  if (reuse) reuse->idle -= from_idle;
  void* p = aligned_alloc(256, (n + 511) / 256 * 256);
  memset(p, 0, n);
  g_used[g_dev] += n;
  g_blocks[p] = Block{n, g_dev, pool};
  *out = p;
  return cudaSuccess;
}

cudaError_t drop(void* p) {
  auto it = g_blocks.find(p);
  if (it == g_blocks.end()) return set(cudaErrorInvalidValue);
  g_used[it->second.dev] -= it->second.bytes;
  auto pool = g_pools.find(it->second.pool);
  if (pool != g_pools.end()) {
    pool->second.idle += it->second.bytes;
    if (pool->second.idle > pool->second.threshold) pool->second.idle = pool->second.threshold;
  }
  free(p);
  g_blocks.erase(it);
  return cudaSuccess;
}

cudaError_t launch(const void* f, dim3 grid, dim3 block, void** args, size_t smem) {
  ++g_launches;
  if (smem > 48 * 1024) {
    auto it = g_smem.find({g_dev, f});
    if (it == g_smem.end() || (size_t)it->second < smem) return set(cudaErrorInvalidValue);
    if (grid.x * grid.y * grid.z > g_max_persistent_grid)
      g_max_persistent_grid = grid.x * grid.y * grid.z;
  }
  if (grid.x == 0 || block.x == 0) return set(cudaErrorInvalidConfiguration);
  if (g_names[f].find("k_poses_float") != std::string::npos) {
    // arguments: launch constants, intrinsics (or null), poses, m, out
    g_last_K = *(const double**)args[1];
    g_have_K = g_last_K != nullptr && ((size_t)g_last_K & 7) == 0;
    if (g_have_K) memcpy(g_K, g_last_K, sizeof g_K);
  }
  return cudaSuccess;
}

CUresult fake_encode(CUtensorMap* m, ...) {
  memset((void*)m, 0, sizeof *m);
  return CUDA_SUCCESS;
}
CUresult fake_ctx_id(CUcontext, unsigned long long* id) {
  *id = 1000ull * (g_dev + 1) + g_generation[g_dev];
  return CUDA_SUCCESS;
}
}  // namespace

extern "C" {
// the test's side
void fake_capacity(size_t bytes) { g_capacity = bytes; }
size_t fake_used(int dev) { return g_used[dev]; }
size_t fake_idle(int dev) { return idle_bytes(dev); }
int fake_dead_pool_uses() { return g_dead_pool_uses; }
int fake_pools() { return (int)g_pools.size(); }
int fake_blocking_copies() { return g_blocking_copies; }
unsigned fake_max_persistent_grid() { return g_max_persistent_grid; }
int fake_intrinsics(double* K) {   // what k_poses_float read; 1: by pointer, 0: none, -1: misaligned
  if (!g_last_K) return 0;
  if (!g_have_K) return -1;
  memcpy(K, g_K, sizeof g_K);
  return 1;
}

// registration
void** __cudaRegisterFatBinary(void*) {
  static void* h;
  return &h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*,
                            dim3*, dim3*, int*) {
  g_names[host] = name;
}
void __cudaRegisterVar(void**, char* host, char*, const char*, int, size_t n, int, int) {
  g_symbols[host] = {n, nullptr};
}
cudaError_t cudaGetSymbolAddress(void** p, const void* host) {
  auto& v = g_symbols[host];
  if (!v.second) v.second = aligned_alloc(256, (v.first + 255) / 256 * 256);
  *p = v.second;
  return cudaSuccess;
}

// launches
static dim3 s_grid, s_block;
static size_t s_smem;
static cudaStream_t s_stream;
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, cudaStream_t s) {
  s_grid = g, s_block = b, s_smem = smem, s_stream = s;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* s) {
  *g = s_grid, *b = s_block, *smem = s_smem, *(cudaStream_t*)s = s_stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void** a, size_t smem, cudaStream_t) {
  return launch((const void*)k, g, b, a, smem);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** a) {
  return launch(f, c->gridDim, c->blockDim, a, c->dynamicSmemBytes);
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute, int v) {
  g_smem[{g_dev, f}] = v;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t,
                                                                   unsigned) {
  *n = 1;
  return cudaSuccess;
}

// devices
cudaError_t cudaGetDevice(int* d) {
  *d = g_dev;
  return cudaSuccess;
}
cudaError_t cudaSetDevice(int d) {
  if (d < 0 || d >= kDevices) return set(cudaErrorInvalidDevice);
  g_dev = d;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int d) {
  *v = a == cudaDevAttrMultiProcessorCount ? kSms[d] : 1;
  return cudaSuccess;
}
cudaError_t cudaDeviceReset() {
  for (auto it = g_blocks.begin(); it != g_blocks.end();) {
    if (it->second.dev != g_dev) {
      ++it;
      continue;
    }
    free(it->first);
    it = g_blocks.erase(it);
  }
  g_used[g_dev] = 0;
  ++g_generation[g_dev];
  for (auto it = g_smem.begin(); it != g_smem.end();)
    it = it->first.first == g_dev ? g_smem.erase(it) : std::next(it);
  return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetLastError() {
  const cudaError_t e = g_last;
  g_last = cudaSuccess;
  return e;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char* name, void** f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
  *f = !strcmp(name, "cuTensorMapEncodeTiled") ? (void*)fake_encode
       : !strcmp(name, "cuCtxGetId")           ? (void*)fake_ctx_id
                                               : nullptr;
  *q = *f ? cudaDriverEntryPointSuccess : cudaDriverEntryPointSymbolNotFound;
  return cudaSuccess;
}

// memory
cudaError_t cudaMalloc(void** p, size_t n) { return take(p, n, nullptr, nullptr); }
cudaError_t cudaMallocHost(void** p, size_t n) {
  *p = calloc(1, n);
  return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) {
  free(p);
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) { return p ? drop(p) : cudaSuccess; }
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { return take(p, n, nullptr, nullptr); }
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { return drop(p); }
cudaError_t cudaMemPoolCreate(cudaMemPool_t* out, const cudaMemPoolProps* props) {
  *out = (cudaMemPool_t)malloc(1);
  g_pools[(void*)*out] = Pool{props->location.id, g_generation[props->location.id], 0, 0};
  return cudaSuccess;
}
cudaError_t cudaMemPoolDestroy(cudaMemPool_t p) {
  g_pools.erase((void*)p);
  return cudaSuccess;
}
static Pool* alive(cudaMemPool_t p) {
  auto it = g_pools.find((void*)p);
  if (it != g_pools.end() && it->second.generation == g_generation[it->second.dev])
    return &it->second;
  ++g_dead_pool_uses;
  return nullptr;
}
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t p, cudaMemPoolAttr, void* v) {
  Pool* q = alive(p);
  if (!q) return set(cudaErrorInvalidValue);
  q->threshold = (size_t)*(unsigned long long*)v;
  return cudaSuccess;
}
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t p, size_t n) {
  Pool* q = alive(p);
  if (!q) return set(cudaErrorInvalidValue);
  if (q->idle > n) q->idle = n;
  return cudaSuccess;
}
cudaError_t cudaMallocFromPoolAsync(void** out, size_t n, cudaMemPool_t p, cudaStream_t) {
  Pool* q = alive(p);
  if (!q) return set(cudaErrorInvalidValue);
  return take(out, n, q, (void*)p);
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
  memset(a, 0, sizeof *a);
  auto it = g_blocks.upper_bound((void*)p);
  if (it != g_blocks.begin()) {
    --it;
    if ((const char*)p < (const char*)it->first + it->second.bytes) {
      a->type = cudaMemoryTypeDevice;
      a->device = it->second.dev;
    }
  }
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
  ++g_blocking_copies;
  memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemset(void* d, int v, size_t n) {
  memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
  memset(d, v, n);
  return cudaSuccess;
}
}  // extern "C"
