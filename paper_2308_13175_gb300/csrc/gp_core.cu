// Context, errors and the device-wide scan used by the set-up paths.
#include <cstdio>
#include <map>
#include <mutex>
#include <string>
#include <utility>

#include "gp_internal.cuh"

gp_status gp_fail(gp_ctx* ctx, gp_status st, const std::string& msg) {
  if (ctx) ctx->err = msg;
  return st;
}

gp_status gp_cuda_fail(gp_ctx* ctx, cudaError_t e, const char* what) {
  std::string msg = std::string(what) + ": " + cudaGetErrorString(e);
  cudaGetLastError();  // clear a sticky launch error where possible
  return gp_fail(ctx, GP_ERR_CUDA, msg);
}

namespace {
struct DevicePool {
  cudaMemPool_t pool = nullptr;
  int64_t users = 0;
  gp_shown idle[GP_SHOWN_BLOCKS];  // blocks given back
  size_t idle_bytes = 0;
};
std::mutex g_pool_mutex;
std::map<int, DevicePool>& device_pools() {
  static std::map<int, DevicePool>* pools = new std::map<int, DevicePool>();  // outlives every context
  return *pools;
}
void drop_idle(DevicePool& d) {
  for (gp_shown& b : d.idle) {
    if (b.p) cudaFree(b.p);
    b = gp_shown{};
  }
  d.idle_bytes = 0;
}
void empty_pool(DevicePool& d) {
  drop_idle(d);
  if (d.pool) cudaMemPoolTrimTo(d.pool, 0);
}
}  // namespace

cudaError_t gp_pool_acquire(int device, cudaMemPool_t* pool) {
  std::lock_guard<std::mutex> lock(g_pool_mutex);
  DevicePool& d = device_pools()[device];
  if (!d.pool) {
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = device;
    cudaError_t e = cudaMemPoolCreate(&d.pool, &props);
    if (e != cudaSuccess) {
      d.pool = nullptr;
      return e;
    }
    uint64_t keep = GP_POOL_KEEP;
    e = cudaMemPoolSetAttribute(d.pool, cudaMemPoolAttrReleaseThreshold, &keep);
    if (e != cudaSuccess) {  // not left for the next context without its threshold
      cudaMemPoolDestroy(d.pool);
      d.pool = nullptr;
      return e;
    }
  }
  d.users += 1;
  *pool = d.pool;
  return cudaSuccess;
}

void gp_pool_release(int device) {
  std::lock_guard<std::mutex> lock(g_pool_mutex);
  DevicePool& d = device_pools()[device];
  if (d.users > 0) d.users -= 1;
  if (d.users == 0) empty_pool(d);
}

cudaError_t gp_shown_take(int device, size_t bytes, gp_shown* block) {
  *block = gp_shown{};
  std::lock_guard<std::mutex> lock(g_pool_mutex);
  DevicePool& d = device_pools()[device];
  gp_shown* best = nullptr;
  for (gp_shown& b : d.idle)
    if (b.p && b.bytes >= bytes && b.bytes <= 2 * bytes && (!best || b.bytes < best->bytes)) best = &b;
  if (best) {
    std::swap(*block, *best);
    d.idle_bytes -= block->bytes;
    return cudaSuccess;
  }
  DeviceScope scope(device);
  if (scope.err != cudaSuccess) return scope.err;
  void* p = nullptr;
  cudaError_t e = cudaMalloc(&p, bytes);
  if (e == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    empty_pool(d);
    e = cudaMalloc(&p, bytes);
  }
  if (e == cudaSuccess) *block = gp_shown{p, bytes};
  return e;
}

void gp_shown_give(int device, gp_shown* block) {
  const gp_shown b = *block;
  *block = gp_shown{};
  if (!b.p) return;
  std::lock_guard<std::mutex> lock(g_pool_mutex);
  DevicePool& d = device_pools()[device];
  if (d.users > 0 && d.idle_bytes + b.bytes <= GP_SHOWN_KEEP)
    for (gp_shown& slot : d.idle)
      if (!slot.p) {
        slot = b;
        d.idle_bytes += b.bytes;
        return;
      }
  cudaFree(b.p);
}

void gp_drop_kept(int device) {
  std::lock_guard<std::mutex> lock(g_pool_mutex);
  empty_pool(device_pools()[device]);
}

void gp_free_idle_done(int device) {
  cudaStreamSynchronize(nullptr);
  std::lock_guard<std::mutex> lock(g_pool_mutex);
  DevicePool& d = device_pools()[device];
  if (d.users == 0) empty_pool(d);
}

extern "C" gp_status gp_create(gp_ctx** out, int device, void* stream) {
  if (!out) return GP_ERR_ARG;
  *out = nullptr;
  int n = 0;
  if (cudaGetDeviceCount(&n) != cudaSuccess || device < 0 || device >= n) {
    cudaGetLastError();
    return GP_ERR_ARG;
  }
  gp_ctx* ctx = new (std::nothrow) gp_ctx();
  if (!ctx) return GP_ERR_OOM;
  ctx->device = device;
  ctx->stream = (cudaStream_t)stream;
  if (cudaSetDevice(device) != cudaSuccess ||
      cudaDeviceGetAttribute(&ctx->num_sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess ||
      gp_pool_acquire(device, &ctx->pool) != cudaSuccess) {
    cudaGetLastError();
    delete ctx;
    return GP_ERR_CUDA;
  }
  *out = ctx;
  return GP_OK;
}

extern "C" gp_status gp_set_stream(gp_ctx* ctx, void* stream) {
  if (!ctx) return GP_ERR_ARG;
  ctx->stream = (cudaStream_t)stream;
  return GP_OK;
}

extern "C" void gp_destroy(gp_ctx* ctx) {
  if (!ctx) return;
  if (ctx->live_bands > 0) {
    ctx->destroy_pending = true;
    return;
  }
  gp_ctx_release(ctx);
}

void gp_ctx_release(gp_ctx* ctx) {
  for (auto& r : ctx->prof) {
    if (r.start) cudaEventDestroy(r.start);
    if (r.stop) cudaEventDestroy(r.stop);
  }
  for (auto e : ctx->event_pool) cudaEventDestroy(e);
  gp_pool_release(ctx->device);
  delete ctx;
}

// ---------------------------------------------------------------- tracing
static cudaEvent_t prof_event(gp_ctx* ctx) {
  if (!ctx->event_pool.empty()) {
    cudaEvent_t e = ctx->event_pool.back();
    ctx->event_pool.pop_back();
    return e;
  }
  cudaEvent_t e = nullptr;
  if (cudaEventCreate(&e) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  return e;
}

void gp_prof_pre(gp_ctx* ctx) {
  if (!ctx->profiling) return;
  gp_prof_rec r{nullptr, prof_event(ctx), prof_event(ctx)};
  if (r.start) cudaEventRecord(r.start, ctx->stream);
  ctx->prof.push_back(r);
}

void gp_prof_post(gp_ctx* ctx, const char* name) {
  ++ctx->launches;
  if (!ctx->profiling || ctx->prof.empty()) return;
  gp_prof_rec& r = ctx->prof.back();
  r.name = name;
  if (r.stop) cudaEventRecord(r.stop, ctx->stream);
}

extern "C" gp_status gp_profile(gp_ctx* ctx, int enable) {
  if (!ctx) return GP_ERR_ARG;
  ctx->profiling = enable != 0;
  return GP_OK;
}

extern "C" int64_t gp_launch_count(const gp_ctx* ctx) { return ctx ? ctx->launches : -1; }

extern "C" gp_status gp_profile_read(gp_ctx* ctx, char* names, double* total_ms, int64_t* launches, int32_t max_kernels,
                                     int32_t* n_kernels) {
  if (!ctx) return GP_ERR_ARG;
  if (!n_kernels || (max_kernels > 0 && (!names || !total_ms || !launches)))
    return gp_fail(ctx, GP_ERR_ARG, "gp_profile_read: null pointer");
  GP_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
  std::vector<std::string> seen;
  std::vector<double> ms;
  std::vector<int64_t> cnt;
  for (auto& r : ctx->prof) {
    float t = 0.f;
    if (r.start && r.stop && r.name && cudaEventElapsedTime(&t, r.start, r.stop) == cudaSuccess) {
      size_t k = 0;
      while (k < seen.size() && seen[k] != r.name) ++k;
      if (k == seen.size()) {
        seen.emplace_back(r.name);
        ms.push_back(0.0);
        cnt.push_back(0);
      }
      ms[k] += t;
      cnt[k] += 1;
    } else {
      cudaGetLastError();
    }
    if (r.start) ctx->event_pool.push_back(r.start);
    if (r.stop) ctx->event_pool.push_back(r.stop);
  }
  ctx->prof.clear();
  *n_kernels = (int32_t)seen.size();
  for (size_t k = 0; k < seen.size() && (int32_t)k < max_kernels; ++k) {
    std::snprintf(names + 32 * k, 32, "%s", seen[k].c_str());
    total_ms[k] = ms[k];
    launches[k] = cnt[k];
  }
  return GP_OK;
}

extern "C" const char* gp_last_error(const gp_ctx* ctx) { return ctx ? ctx->err.c_str() : ""; }

extern "C" const char* gp_version(void) { return "gridpull-gb300 0.1"; }

// ------------------------------------------------------------------- scan
// Three-phase exclusive scan: per-block scans of SCAN_TILE elements, a
// recursive scan of the block totals, then a uniform add.
namespace {
constexpr int SCAN_THREADS = 512;
constexpr int SCAN_PER_THREAD = 4;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_PER_THREAD;

__global__ void k_scan_tiles(int32_t* __restrict__ data, int64_t n, int32_t* __restrict__ tile_sums) {
  __shared__ int32_t warp_tot[SCAN_THREADS / 32];
  int64_t base = (int64_t)blockIdx.x * SCAN_TILE + (int64_t)threadIdx.x * SCAN_PER_THREAD;
  int32_t v[SCAN_PER_THREAD];
  int32_t run = 0;
#pragma unroll
  for (int i = 0; i < SCAN_PER_THREAD; ++i) {
    int64_t idx = base + i;
    int32_t x = idx < n ? data[idx] : 0;
    v[i] = run;
    run += x;
  }
  // inclusive scan of per-thread totals across the block
  int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int32_t incl = run;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int32_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) warp_tot[wid] = incl;
  __syncthreads();
  if (wid == 0) {
    int32_t w = lane < SCAN_THREADS / 32 ? warp_tot[lane] : 0;
    int32_t wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int32_t y = __shfl_up_sync(0xffffffffu, wi, o);
      if (lane >= o) wi += y;
    }
    if (lane < SCAN_THREADS / 32) warp_tot[lane] = wi - w;  // exclusive warp offsets
    if (lane == SCAN_THREADS / 32 - 1) tile_sums[blockIdx.x] = wi;
  }
  __syncthreads();
  int32_t off = warp_tot[wid] + (incl - run);
#pragma unroll
  for (int i = 0; i < SCAN_PER_THREAD; ++i) {
    int64_t idx = base + i;
    if (idx < n) data[idx] = v[i] + off;
  }
}

__global__ void k_scan_add(int32_t* __restrict__ data, int64_t n, const int32_t* __restrict__ tile_offs) {
  int64_t idx = (int64_t)blockIdx.x * SCAN_TILE + threadIdx.x;
  int32_t add = tile_offs[blockIdx.x];
#pragma unroll
  for (int i = 0; i < SCAN_PER_THREAD; ++i, idx += SCAN_THREADS)
    if (idx < n) data[idx] += add;
}

}  // namespace

// Level l + 1 scans the tile sums of level l; the last level is one tile,
// whose sum is the total.
gp_status gp_exclusive_scan_i32(gp_ctx* ctx, int32_t* data, int64_t n, int64_t* total_host) {
  if (total_host) *total_host = 0;
  if (n <= 0) return GP_OK;
  constexpr int LEVELS = 4;  // SCAN_TILE^4 > 2^31
  int32_t* level[LEVELS + 1] = {data};
  int64_t len[LEVELS + 1] = {n};
  int depth = 0;
  gp_status st = GP_OK;
  cudaError_t e = cudaSuccess;
  do {
    const int64_t tiles = (len[depth] + SCAN_TILE - 1) / SCAN_TILE;
    if ((st = gp_alloc(ctx, &level[depth + 1], (size_t)tiles, "scan tile sums"))) break;
    k_scan_tiles<<<(unsigned)tiles, SCAN_THREADS, 0, ctx->stream>>>(level[depth], len[depth], level[depth + 1]);
    e = cudaGetLastError();
    len[++depth] = tiles;
  } while (e == cudaSuccess && len[depth] > 1 && depth < LEVELS);
  for (int l = depth - 2; l >= 0 && !st && e == cudaSuccess; --l) {
    k_scan_add<<<(unsigned)len[l + 1], SCAN_THREADS, 0, ctx->stream>>>(level[l], len[l], level[l + 1]);
    e = cudaGetLastError();
  }
  int32_t total = 0;
  if (!st && e == cudaSuccess) e = cudaMemcpyAsync(&total, level[depth], 4, cudaMemcpyDeviceToHost, ctx->stream);
  if (!st && e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
  for (int l = 1; l <= depth; ++l) gp_free(ctx, level[l]);
  if (st) return st;
  if (e != cudaSuccess) return gp_cuda_fail(ctx, e, "scan kernels");
  if (total_host) *total_host = total;
  return GP_OK;
}
