// A stand-in for the CUDA runtime, linked with the library's objects so that
// its host code runs without a GPU: two devices, memory from calloc, kernels
// that do nothing.  It keeps what the tests ask about: which work is in flight
// on which stream of which device, and what the memory pools hold.
#include "fake_cudart.h"

#include <cuda_runtime_api.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <map>
#include <set>
#include <string>

namespace {

struct Stream {
  int device;
  uintptr_t handle;
  bool operator<(const Stream& o) const { return device != o.device ? device < o.device : handle < o.handle; }
};

struct Block {
  size_t bytes;
  int device;
  cudaMemPool_t pool;  // null: cudaMalloc
};

struct Pool {
  int device = 0;
  uint64_t threshold = 0;
  std::map<Stream, size_t> freed;  // freed, the host has not seen it complete
  size_t held = 0;                 // freed and complete
  size_t live = 0;
};

int g_device = 0;
std::set<Stream> g_busy;  // streams with work the host has not waited for
std::map<void*, Block> g_blocks;
std::map<cudaMemPool_t, Pool> g_pools;
std::map<const void*, std::string> g_kernels;
dim3 g_grid, g_block;
size_t g_shared;
cudaStream_t g_stream;
float g_elapsed = 1.f;

Stream here(cudaStream_t s) { return Stream{g_device, (uintptr_t)s}; }

// The host has seen everything up to now on the streams that `which` picks.
template <typename F>
void seen(F&& which) {
  for (auto it = g_busy.begin(); it != g_busy.end();) it = which(*it) ? g_busy.erase(it) : std::next(it);
  for (auto& p : g_pools) {
    Pool& pool = p.second;
    for (auto it = pool.freed.begin(); it != pool.freed.end();) {
      if (!which(it->first)) {
        ++it;
        continue;
      }
      pool.held += it->second;
      it = pool.freed.erase(it);
    }
    if (pool.held > pool.threshold) pool.held = pool.threshold;  // a synchronisation gives the rest back
  }
}

void forget(void* p, const Stream& order) {
  const Block b = g_blocks.at(p);
  for (const Stream& s : g_busy)
    if (s.device == b.device && (s.device != order.device || s.handle != order.handle)) ++fake::races;
  if (b.device != order.device) ++fake::wrong_device;
  g_blocks.erase(p);
  free(p);
  if (!b.pool) return;
  Pool& pool = g_pools.at(b.pool);
  pool.live -= b.bytes;
  pool.freed[order] += b.bytes;
}

}  // namespace

namespace fake {
size_t capacity = ~size_t(0);
int races = 0, wrong_device = 0, fail_set_attribute = 0;
std::map<std::string, unsigned> last_grid;

size_t reserved() {
  size_t n = 0;
  for (auto& p : g_pools) {
    n += p.second.live + p.second.held;
    for (auto& f : p.second.freed) n += f.second;
  }
  return n;
}
size_t used() {
  size_t n = reserved();
  for (auto& b : g_blocks) n += b.second.pool ? 0 : b.second.bytes;
  return n;
}
uint64_t lowest_threshold() {
  uint64_t t = ~0ull;
  for (auto& p : g_pools) t = p.second.threshold < t ? p.second.threshold : t;
  return t;
}
int blocks() { return (int)g_blocks.size(); }
bool from_pool(const void* p) {
  for (auto& b : g_blocks) {
    const char* at = (const char*)b.first;
    if (at <= (const char*)p && (const char*)p < at + b.second.bytes) return b.second.pool != nullptr;
  }
  return true;  // not a block at all
}
}  // namespace fake

extern "C" {

void** __cudaRegisterFatBinary(void*) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  const char* k = strstr(name, "k_");
  std::string s = k ? k : name;
  g_kernels[host] = s.substr(0, s.find_first_of("IE"));
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t shared, struct CUstream_st* s) {
  g_grid = grid;
  g_block = block;
  g_shared = shared;
  g_stream = s;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* shared, void* s) {
  *grid = g_grid;
  *block = g_block;
  *shared = g_shared;
  *(cudaStream_t*)s = g_stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3, void** args, size_t, cudaStream_t s) {
  const std::string& name = g_kernels.at((const void*)k);
  fake::last_grid[name] = grid.x;
  g_busy.insert(here(s));
  // What the autotuner measures: the query pass is the faster the more records
  // a tile has, everything else takes the same time.
  g_elapsed = name == "k_m_query" ? 1000.f / (float)*(const int*)args[3] : 1.f;
  return cudaSuccess;
}

cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaGetDeviceCount(int* n) {
  *n = 2;
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) {
  *d = g_device;
  return cudaSuccess;
}
cudaError_t cudaSetDevice(int d) {
  g_device = d;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) {
  *v = 8;  // multiprocessors
  return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() {
  const int d = g_device;
  seen([&](const Stream& s) { return s.device == d; });
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  const Stream me = here(s);
  seen([&](const Stream& o) { return o.device == me.device && o.handle == me.handle; });
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) {
  *e = (cudaEvent_t)malloc(1);
  return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t e) {
  free((void*)e);
  return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  *ms = g_elapsed;
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
  *p = nullptr;
  return cudaErrorInvalidSymbol;
}

cudaError_t cudaMemPoolCreate(cudaMemPool_t* pool, const cudaMemPoolProps* props) {
  *pool = (cudaMemPool_t)malloc(1);
  g_pools[*pool].device = props->location.id;
  return cudaSuccess;
}
cudaError_t cudaMemPoolDestroy(cudaMemPool_t pool) {
  g_pools.erase(pool);
  return cudaSuccess;
}
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t pool, cudaMemPoolAttr attr, void* v) {
  if (fake::fail_set_attribute > 0) {
    --fake::fail_set_attribute;
    return cudaErrorInvalidValue;
  }
  if (attr == cudaMemPoolAttrReleaseThreshold) g_pools.at(pool).threshold = *(uint64_t*)v;
  return cudaSuccess;
}
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t pool, size_t keep) {
  Pool& p = g_pools.at(pool);
  if (p.held > keep) p.held = keep;  // frees that the host has not seen complete stay
  return cudaSuccess;
}
static bool full(size_t n) { return fake::used() + n > fake::capacity; }
cudaError_t cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t pool, cudaStream_t) {
  Pool& from = g_pools.at(pool);
  const size_t reuse = from.held < n ? from.held : n;
  from.held -= reuse;
  if (full(n)) {
    from.held += reuse;
    return cudaErrorMemoryAllocation;
  }
  *p = calloc(n, 1);
  g_blocks[*p] = Block{n, g_pools.at(pool).device, pool};
  g_pools.at(pool).live += n;
  return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t n) {
  if (full(n)) return cudaErrorMemoryAllocation;
  *p = calloc(n, 1);
  g_blocks[*p] = Block{n, g_device, nullptr};
  return cudaSuccess;
}
cudaError_t cudaFreeAsync(void* p, cudaStream_t s) {
  forget(p, here(s));
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {  // waits for the pointer's device
  if (!p) return cudaSuccess;
  const int d = g_blocks.at(p).device;
  seen([&](const Stream& s) { return s.device == d; });
  forget(p, Stream{d, 0});
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t s) {
  g_busy.insert(here(s));
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* to, const void* from, size_t n, cudaMemcpyKind kind, cudaStream_t s) {
  g_busy.insert(here(s));
  if (kind == cudaMemcpyDeviceToHost || kind == cudaMemcpyHostToDevice) memcpy(to, from, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyToSymbolAsync(const void*, const void*, size_t, size_t, cudaMemcpyKind, cudaStream_t s) {
  g_busy.insert(here(s));
  return cudaSuccess;
}

}  // extern "C"
