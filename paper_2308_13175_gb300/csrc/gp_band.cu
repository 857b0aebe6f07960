// gp_build_band: the uniform grid's near-surface band (Sec. 3 "Discrete
// Grids", the M1 pull bandwidth and the M2 TV bandwidth) stored as 8^3-vertex
// bricks, plus the band queries (info, init, export, values).
#include <algorithm>
#include <vector>

#include "gp_internal.cuh"

gp_status gp_build_points(gp_band* band, const float* pts_dev);  // gp_nn.cu

namespace {

// The cell and vertex sets are bit rows along x: 32 cells (or vertices) a
// word, row (y, z) starting at word (z n + y) W.  A byte per element took 16
// times the bytes in the dilation, and a thread per element: the kernels that
// make an object band on a 256^3 grid took 864 us, and the whole build is
// 0.8 ms shorter this way (7.96 -> 7.16 ms).
struct CellRows {
  int R, W;  // cells per axis, words per row
};
struct VertRows {
  int n, W;  // vertices per axis, words per row
};

__device__ __forceinline__ uint32_t row_tail(int n, int w) {  // the bits of word w that exist in a row of n
  const int left = n - 32 * w;
  return left >= 32 ? 0xffffffffu : (1u << left) - 1u;
}

__global__ void k_mark_occupied(const float* __restrict__ pts, int64_t J, CellRows g, uint32_t* __restrict__ occ) {
  int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= J) return;
  const float half_r = 0.5f * (float)g.R;
  int c[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    gp_cell1 p = gp_cell_exact(pts[3 * j + a], half_r);
    c[a] = min(max(p.c, 0), g.R - 1);
  }
  uint32_t* word = occ + ((int64_t)c[2] * g.R + c[1]) * g.W + (c[0] >> 5);
  const uint32_t bit = 1u << (c[0] & 31);
  if (!(*word & bit)) atomicOr(word, bit);  // a stale read only costs the atomic
}

// Sum of v over the block, added to *total by one thread.
__device__ __forceinline__ void add_count(int v, unsigned long long* total) {
  v = gp_warp_sum_i(v);
  if ((threadIdx.x & 31) == 0 && v) atomicAdd(total, (unsigned long long)v);
}

// v with every set bit spread s places up (0 <= s <= 31).
__device__ __forceinline__ unsigned long long spread_up(unsigned long long v, int s) {
  for (int done = 0; done < s;) {
    const int step = min(done + 1, s - done);
    v |= v << step;
    done += step;
  }
  return v;
}
__device__ __forceinline__ unsigned long long spread_down(unsigned long long v, int s) {
  for (int done = 0; done < s;) {
    const int step = min(done + 1, s - done);
    v |= v >> step;
    done += step;
  }
  return v;
}

// Dilation along x by m <= 31 cells (wider ones are several passes; Chebyshev
// dilations add up).  count (optional): the set bits of the input.
__global__ void k_dilate_x(const uint32_t* __restrict__ in, uint32_t* __restrict__ out, CellRows g, int m,
                           unsigned long long* count) {
  const int64_t n = (int64_t)g.R * g.R * g.W;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int bits = 0;
  if (i < n) {
    const int w = (int)(i % g.W);
    const uint32_t cur = in[i];
    const uint32_t lo = w > 0 ? in[i - 1] : 0u, hi = w + 1 < g.W ? in[i + 1] : 0u;
    const uint32_t up = (uint32_t)(spread_up(((unsigned long long)cur << 32) | lo, m) >> 32);
    const uint32_t down = (uint32_t)spread_down(((unsigned long long)hi << 32) | cur, m);
    out[i] = (up | down) & row_tail(g.R, w);
    bits = __popc(cur);
  }
  if (count) add_count(bits, count);
}

// Dilation along y (axis 1) or z (axis 2) by m.  count: the set bits of the
// output.
__global__ void k_dilate_rows(const uint32_t* __restrict__ in, uint32_t* __restrict__ out, CellRows g, int axis, int m,
                              unsigned long long* count) {
  const int64_t n = (int64_t)g.R * g.R * g.W;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int bits = 0;
  if (i < n) {
    const int64_t row = i / g.W;
    const int pos = axis == 1 ? (int)(row % g.R) : (int)(row / g.R);
    const int64_t stride = axis == 1 ? g.W : (int64_t)g.R * g.W;
    uint32_t v = 0u;
    for (int p = max(pos - m, 0); p <= min(pos + m, g.R - 1); ++p) v |= in[i + (p - pos) * stride];
    out[i] = v;
    bits = __popc(v);
  }
  if (count) add_count(bits, count);
}

__global__ void k_fill_rows(uint32_t* __restrict__ out, CellRows g) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < (int64_t)g.R * g.R * g.W) out[i] = row_tail(g.R, (int)(i % g.W));
}

// The corners of a set of cells: vertex (i, j, k) is one if any of the cells
// (i - dx, j - dy, k - dz), dx, dy, dz in {0, 1}, is in the set.
__global__ void k_corner_rows(const uint32_t* __restrict__ cells, CellRows g, VertRows v, uint32_t* __restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)v.n * v.n * v.W) return;
  const int w = (int)(i % v.W);
  const int64_t row = i / v.W;
  const int j = (int)(row % v.n), k = (int)(row / v.n);
  uint32_t bits = 0u;
#pragma unroll
  for (int d = 0; d < 4; ++d) {
    const int cj = j - (d & 1), ck = k - (d >> 1);
    if (cj < 0 || ck < 0 || cj >= g.R || ck >= g.R) continue;
    const uint32_t* r = cells + ((int64_t)ck * g.R + cj) * g.W;
    const uint32_t c = w < g.W ? r[w] : 0u;
    bits |= c | (c << 1) | (w > 0 ? r[w - 1] >> 31 : 0u);
  }
  out[i] = bits;
}

// The 8 bits of a vertex (or cell) row from position 8 b on.
__device__ __forceinline__ uint32_t row_byte(const uint32_t* __restrict__ row, int b) {
  return (row[b >> 2] >> (8 * (b & 3))) & 255u;
}

// Bricks that hold a required vertex: one of T, a trainable one or an axis
// neighbour of one of T.  A thread takes one z layer of a brick, its rows'
// neighbours in x and y, and the layers below and above for the outer two.
__global__ void k_brick_need(const uint32_t* __restrict__ tv, const uint32_t* __restrict__ train, VertRows v, int nb,
                             uint8_t* __restrict__ need) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)nb * nb * nb * 8) return;
  const int64_t b = i >> 3;
  const int bx = (int)(b % nb), by = (int)((b / nb) % nb), bz = (int)(b / ((int64_t)nb * nb));
  const int k = 8 * bz + (int)(i & 7);
  if (k >= v.n) return;
  const int R = v.n - 1;
  uint32_t any = 0u;
  auto row = [&](const uint32_t* s, int j, int kk) { return s + ((int64_t)kk * v.n + j) * v.W; };
  const int j1 = min(8 * by + 7, R);
#pragma unroll 4
  for (int j = 8 * by; j <= j1; ++j) {
    const uint32_t* t = row(tv, j, k);
    any |= row_byte(t, bx) | row_byte(row(train, j, k), bx);
    if (bx > 0) any |= row_byte(t, bx - 1) >> 7;
    if (8 * bx + 8 <= R) any |= row_byte(t, bx + 1) & 1u;
    if ((i & 7) == 0 && k > 0) any |= row_byte(row(tv, j, k - 1), bx);
    if ((i & 7) == 7 && k < R) any |= row_byte(row(tv, j, k + 1), bx);
  }
  if (by > 0) any |= row_byte(row(tv, 8 * by - 1, k), bx);
  if (8 * by + 8 <= R) any |= row_byte(row(tv, 8 * by + 8, k), bx);
  if (any) need[b] = 1;
}

__device__ __forceinline__ uint32_t compact3(uint32_t x) {  // every third bit -> contiguous
  x &= 0x09249249u;
  x = (x ^ (x >> 2)) & 0x030C30C3u;
  x = (x ^ (x >> 4)) & 0x0300F00Fu;
  x = (x ^ (x >> 8)) & 0x030000FFu;
  x = (x ^ (x >> 16)) & 0x000003FFu;
  return x;
}

// Morton-ordered flags of the needed bricks.
__global__ void k_morton_flags(const uint8_t* __restrict__ need, int nb, int64_t nm, int32_t* __restrict__ flags) {
  int64_t mi = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (mi >= nm) return;
  uint32_t bx = compact3((uint32_t)mi), by = compact3((uint32_t)(mi >> 1)), bz = compact3((uint32_t)(mi >> 2));
  int32_t f = 0;
  if (bx < (uint32_t)nb && by < (uint32_t)nb && bz < (uint32_t)nb)
    f = need[((int64_t)bz * nb + by) * nb + bx];
  flags[mi] = f;
}

__global__ void k_assign_slots(const uint8_t* __restrict__ need, const int32_t* __restrict__ offs, int nb,
                               int64_t nm, int32_t* __restrict__ table, int32_t* __restrict__ coord) {
  int64_t mi = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (mi >= nm) return;
  uint32_t bx = compact3((uint32_t)mi), by = compact3((uint32_t)(mi >> 1)), bz = compact3((uint32_t)(mi >> 2));
  if (bx >= (uint32_t)nb || by >= (uint32_t)nb || bz >= (uint32_t)nb) return;
  int64_t b = ((int64_t)bz * nb + by) * nb + bx;
  if (!need[b]) return;
  int32_t slot = offs[mi];
  table[b] = slot;
  coord[3 * slot + 0] = bx;
  coord[3 * slot + 1] = by;
  coord[3 * slot + 2] = bz;
}

// Slots of the 27 bricks around each brick (itself included), x fastest.
__global__ void k_brick_nbr(const int32_t* __restrict__ table, const int32_t* __restrict__ coord, int nb,
                            int64_t n_bricks, int32_t* __restrict__ nbr) {
  int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (a >= n_bricks * 27) return;
  int64_t slot = a / 27;
  int t = (int)(a - slot * 27);
  int bx = coord[3 * slot] + t % 3 - 1, by = coord[3 * slot + 1] + (t / 3) % 3 - 1, bz = coord[3 * slot + 2] + t / 9 - 1;
  int32_t v = -1;
  if ((unsigned)bx < (unsigned)nb && (unsigned)by < (unsigned)nb && (unsigned)bz < (unsigned)nb)
    v = table[((int64_t)bz * nb + by) * nb + bx];
  nbr[a] = v;
}

// A brick's masks, one thread per word (four rows of 8), 16 words a set.
__global__ void __launch_bounds__(256) k_brick_masks(const uint32_t* __restrict__ tv,
                                                     const uint32_t* __restrict__ train,
                                                     const uint32_t* __restrict__ pull, CellRows g, VertRows v,
                                                     const int32_t* __restrict__ coord, int64_t n_bricks,
                                                     uint32_t* __restrict__ masks, int32_t* __restrict__ active_flag,
                                                     unsigned long long* counts) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t slot = i >> 4;
  const int w = (int)(i & 15);
  uint32_t t = 0u, r = 0u, p = 0u;
  if (slot < n_bricks) {
    const int bx = coord[3 * slot], k = 8 * coord[3 * slot + 2] + (w >> 1);
#pragma unroll
    for (int y = 0; y < 4; ++y) {
      const int j = 8 * coord[3 * slot + 1] + 4 * (w & 1) + y;
      if (j >= v.n || k >= v.n) continue;
      const int64_t at = ((int64_t)k * v.n + j) * v.W;
      t |= row_byte(tv + at, bx) << (8 * y);
      r |= row_byte(train + at, bx) << (8 * y);
      if (j < g.R && k < g.R && 8 * bx < g.R)
        p |= row_byte(pull + ((int64_t)k * g.R + j) * g.W, bx) << (8 * y);
    }
    uint32_t* mk = masks + slot * 48;
    mk[w] = t;
    mk[16 + w] = r;
    mk[32 + w] = p;
  }
  const unsigned any = __ballot_sync(0xffffffffu, r != 0u);
  if (slot < n_bricks && w == 0) active_flag[slot] = (any >> (threadIdx.x & 16)) & 0xffffu ? 1 : 0;
  add_count(__popc(t), counts + 2);
  add_count(__popc(r), counts + 3);
}

__global__ void k_compact_active(const int32_t* __restrict__ flags, const int32_t* __restrict__ offs, int64_t n,
                                 int32_t* __restrict__ out) {
  int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (s < n && flags[s]) out[offs[s]] = (int32_t)s;
}

__global__ void k_init_sphere(float* __restrict__ D, const int32_t* __restrict__ coord, int64_t nslots, int R,
                              float cx, float cy, float cz, float radius, float noise, uint32_t k0, uint32_t k1) {
  int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (a >= nslots) return;
  int slot = (int)(a >> 9), l = (int)(a & 511);
  int i = coord[3 * slot] * 8 + (l & 7);
  int j = coord[3 * slot + 1] * 8 + ((l >> 3) & 7);
  int k = coord[3 * slot + 2] * 8 + (l >> 6);
  if (i > R || j > R || k > R) {
    D[a] = 0.f;
    return;
  }
  float h = 2.0f / (float)R;
  float x = -1.0f + h * (float)i - cx, y = -1.0f + h * (float)j - cy, z = -1.0f + h * (float)k - cz;
  float d = sqrtf(x * x + y * y + z * z) - radius;
  if (noise != 0.f) {
    uint64_t key = (uint64_t)i + (uint64_t)(R + 1) * ((uint64_t)j + (uint64_t)(R + 1) * (uint64_t)k);
    float3 zz = gp_box_muller3(gp_philox((uint32_t)key, (uint32_t)(key >> 32), 0u, 2u, k0, k1));
    d += noise * zz.x;
  }
  D[a] = d;
}

__global__ void k_export(const int32_t* __restrict__ coord, const uint32_t* __restrict__ masks, const float* __restrict__ D,
                         int64_t nslots, int R, int32_t* __restrict__ ijk, float* __restrict__ dout,
                         uint8_t* __restrict__ flags) {
  int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (a >= nslots) return;
  int slot = (int)(a >> 9), l = (int)(a & 511);
  int i = coord[3 * slot] * 8 + (l & 7);
  int j = coord[3 * slot + 1] * 8 + ((l >> 3) & 7);
  int k = coord[3 * slot + 2] * 8 + (l >> 6);
  if (ijk) {
    ijk[3 * a] = i;
    ijk[3 * a + 1] = j;
    ijk[3 * a + 2] = k;
  }
  if (dout) dout[a] = D[a];
  if (flags) {
    uint8_t f = 0;
    if (gp_mask_bit(masks, slot, 0, l)) f |= 1;
    if (gp_mask_bit(masks, slot, 1, l)) f |= 2;
    if (i <= R && j <= R && k <= R) f |= 4;
    if (gp_mask_bit(masks, slot, 2, l)) f |= 8;
    flags[a] = f;
  }
}

void band_free(gp_band* b) {
  if (!b) return;
  cudaDeviceSynchronize();  // any stream may have worked on the band
  gp_free_idle(b->brick_table);
  gp_free_idle(b->brick_coord);
  gp_free_idle(b->brick_nbr);
  gp_free_idle(b->masks);
  gp_free_idle(b->active);
  gp_shown_give(b->ctx->device, &b->shown);
  gp_free_idle(b->acc);
  gp_free_idle(b->qgrad);
  gp_free_idle(b->pts);
  gp_free_idle(b->pts_sorted);
  gp_free_idle(b->cell_table);
  gp_free_idle(b->cell_sup);
  gp_free_idle(b->cell_blk);
  gp_free_idle(b->cell_occ);
  gp_free_idle(b->sigma);
  gp_free_idle(b->seeds);
  gp_free_idle(b->perm);
  gp_free_idle(b->inv_perm);
  gp_free_idle(b->order_tiles);
  gp_free_idle(b->emit_order);
  gp_free_idle(b->emit_slot);
  gp_free_idle(b->emit_pts);
  gp_free_idle(b->partials);
  gp_free_idle(b->dev_ints);
  gp_free_idle_done(b->ctx->device);
  delete b;
}

struct TempBufs {
  gp_ctx* ctx;
  std::vector<void*> ptrs;
  explicit TempBufs(gp_ctx* c) : ctx(c) {}
  ~TempBufs() {
    for (void* p : ptrs) gp_free(ctx, p);
  }
  template <typename T>
  gp_status alloc(gp_ctx* c, T** p, size_t n, const char* what) {
    gp_status st = gp_alloc(c, p, n, what);
    if (!st) ptrs.push_back(*p);
    return st;
  }
};

gp_status build_band_sets(gp_band* b, const float* pts_dev) {
  gp_ctx* ctx = b->ctx;
  cudaStream_t s = ctx->stream;
  const int R = b->R;
  const int nb = b->nb;
  const int64_t nbr = (int64_t)nb * nb * nb;
  TempBufs tmp(ctx);
  const CellRows cr{R, (R + 31) / 32};
  const VertRows vr{R + 1, (R + 32) / 32};
  const int64_t nc = (int64_t)R * R * cr.W, nv = (int64_t)vr.n * vr.n * vr.W;
  uint32_t *occ = nullptr, *ping = nullptr, *pong = nullptr, *s1 = nullptr, *s2 = nullptr, *sx = nullptr;
  uint32_t *tv = nullptr, *train = nullptr;
  uint8_t* need = nullptr;
  unsigned long long* counts = nullptr;
  gp_status st;
  // Negative widths mean "every cell".
  const bool all1 = b->M1 < 0, all2 = b->M2 < 0;
  const int m1 = std::min(b->M1, R), m2 = std::min(b->M2, R);
  if ((st = tmp.alloc(ctx, &occ, nc, "occupied cells"))) return st;
  if ((st = tmp.alloc(ctx, &ping, nc, "cell rows"))) return st;
  if ((st = tmp.alloc(ctx, &pong, nc, "cell rows"))) return st;
  if ((st = tmp.alloc(ctx, &s1, nc, "pull cells"))) return st;
  if ((st = tmp.alloc(ctx, &counts, 8, "band counts"))) return st;
  GP_CUDA(ctx, cudaMemsetAsync(occ, 0, nc * sizeof(uint32_t), s));
  GP_CUDA(ctx, cudaMemsetAsync(counts, 0, 8 * sizeof(unsigned long long), s));
  GP_KERNEL(ctx, "k_mark_occupied", k_mark_occupied<<<gp_blocks(b->J, 256), 256, 0, s>>>(pts_dev, b->J, cr, occ));

  // The Chebyshev dilation of the occupied cells by m, one axis after another.
  auto dilate = [&](int m, uint32_t* out, unsigned long long* n_in, unsigned long long* n_out) -> gp_status {
    const uint32_t* in = occ;
    for (int left = m, first = 1; first || left > 0; first = 0) {
      const int step = std::min(left, 31);
      GP_KERNEL(ctx, "k_dilate_x", k_dilate_x<<<gp_blocks(nc, 256), 256, 0, s>>>(in, ping, cr, step, first ? n_in : nullptr));
      left -= step;
      std::swap(ping, pong);
      in = pong;
    }
    GP_KERNEL(ctx, "k_dilate_rows", k_dilate_rows<<<gp_blocks(nc, 256), 256, 0, s>>>(pong, ping, cr, 1, m, nullptr));
    GP_KERNEL(ctx, "k_dilate_rows", k_dilate_rows<<<gp_blocks(nc, 256), 256, 0, s>>>(ping, out, cr, 2, m, n_out));
    return GP_OK;
  };
  if ((st = dilate(all1 ? 0 : m1, s1, counts + 0, counts + 1))) return st;
  if (all1) GP_KERNEL(ctx, "k_fill_rows", k_fill_rows<<<gp_blocks(nc, 256), 256, 0, s>>>(s1, cr));
  s2 = s1;
  if (all2 != all1 || (!all1 && m2 != m1)) {
    if ((st = tmp.alloc(ctx, &s2, nc, "TV cells"))) return st;
    if (all2)
      GP_KERNEL(ctx, "k_fill_rows", k_fill_rows<<<gp_blocks(nc, 256), 256, 0, s>>>(s2, cr));
    else if ((st = dilate(m2, s2, nullptr, nullptr)))
      return st;
  }
  // The trainable cells are the wider of the two sets.
  sx = all1 || (!all2 && m1 > m2) ? s1 : s2;
  if ((st = tmp.alloc(ctx, &tv, nv, "TV vertices"))) return st;
  GP_KERNEL(ctx, "k_corner_rows", k_corner_rows<<<gp_blocks(nv, 256), 256, 0, s>>>(s2, cr, vr, tv));
  train = tv;
  if (sx != s2) {
    if ((st = tmp.alloc(ctx, &train, nv, "trainable vertices"))) return st;
    GP_KERNEL(ctx, "k_corner_rows", k_corner_rows<<<gp_blocks(nv, 256), 256, 0, s>>>(sx, cr, vr, train));
  }
  if ((st = tmp.alloc(ctx, &need, nbr, "brick flags"))) return st;
  GP_CUDA(ctx, cudaMemsetAsync(need, 0, nbr, s));
  GP_KERNEL(ctx, "k_brick_need", k_brick_need<<<gp_blocks(8 * nbr, 256), 256, 0, s>>>(tv, train, vr, nb, need));

  // Slots in Morton order of the brick coordinates.
  int nbm = 1;
  while (nbm < nb) nbm <<= 1;
  const int64_t nm = (int64_t)nbm * nbm * nbm;
  int32_t* mflags = nullptr;
  if ((st = tmp.alloc(ctx, &mflags, nm, "morton flags"))) return st;
  GP_KERNEL(ctx, "k_morton_flags", k_morton_flags<<<gp_blocks(nm, 256), 256, 0, s>>>(need, nb, nm, mflags));
  int64_t n_bricks = 0;
  if ((st = gp_exclusive_scan_i32(ctx, mflags, nm, &n_bricks))) return st;
  b->n_bricks = n_bricks;
  if ((st = gp_alloc(ctx, &b->brick_table, nbr, "brick table"))) return st;
  GP_CUDA(ctx, cudaMemsetAsync(b->brick_table, 0xFF, nbr * sizeof(int32_t), s));
  if ((st = gp_alloc(ctx, &b->brick_coord, 3 * n_bricks, "brick coords"))) return st;
  GP_KERNEL(ctx, "k_assign_slots", k_assign_slots<<<gp_blocks(nm, 256), 256, 0, s>>>(need, mflags, nb, nm, b->brick_table, b->brick_coord));
  if ((st = gp_alloc(ctx, &b->brick_nbr, 27 * n_bricks, "brick neighbours"))) return st;
  if (n_bricks > 0)
    GP_KERNEL(ctx, "k_brick_nbr", k_brick_nbr<<<gp_blocks(27 * n_bricks, 256), 256, 0, s>>>(b->brick_table, b->brick_coord, nb, n_bricks, b->brick_nbr));

  if ((st = gp_alloc(ctx, &b->masks, 48 * n_bricks, "brick masks"))) return st;
  int32_t *aflag = nullptr, *aoffs = nullptr;
  if ((st = tmp.alloc(ctx, &aflag, n_bricks, "active flags"))) return st;
  if ((st = tmp.alloc(ctx, &aoffs, n_bricks, "active offsets"))) return st;
  if (n_bricks > 0) {
    GP_KERNEL(ctx, "k_brick_masks", k_brick_masks<<<gp_blocks(16 * n_bricks, 256), 256, 0, s>>>(tv, train, s1, cr, vr, b->brick_coord, n_bricks, b->masks, aflag, counts));
    GP_CUDA(ctx, cudaMemcpyAsync(aoffs, aflag, n_bricks * sizeof(int32_t), cudaMemcpyDeviceToDevice, s));
  }
  int64_t n_active = 0;
  if ((st = gp_exclusive_scan_i32(ctx, aoffs, n_bricks, &n_active))) return st;
  b->n_active = n_active;
  if ((st = gp_alloc(ctx, &b->active, n_active, "active list"))) return st;
  if (n_bricks > 0) {
    GP_KERNEL(ctx, "k_compact_active", k_compact_active<<<gp_blocks(n_bricks, 256), 256, 0, s>>>(aflag, aoffs, n_bricks, b->active));
  }
  unsigned long long hc[8];
  GP_CUDA(ctx, cudaMemcpyAsync(hc, counts, sizeof(hc), cudaMemcpyDeviceToHost, s));
  GP_CUDA(ctx, cudaStreamSynchronize(s));
  b->n_occ = (int64_t)hc[0];
  b->n_pull = all1 ? (int64_t)R * R * R : (int64_t)hc[1];
  b->V_tv = (int64_t)hc[2];
  b->V_trainable = (int64_t)hc[3];
  return GP_OK;
}

}  // namespace

extern "C" gp_status gp_build_band(gp_ctx* ctx, const float* pts_dev, int64_t J, const gp_grid_desc* desc,
                                   gp_band** out) {
  if (!ctx) return GP_ERR_ARG;
  if (!out || !pts_dev || !desc) return gp_fail(ctx, GP_ERR_ARG, "gp_build_band: null argument");
  *out = nullptr;
  int R = desc->R;
  if (R < 8 || R > 2048 || (R & (R - 1)))
    return gp_fail(ctx, GP_ERR_ARG, "gp_build_band: R must be a power of two in [8, 2048]");
  if (J < 1 || J >= (int64_t(1) << 31)) return gp_fail(ctx, GP_ERR_ARG, "gp_build_band: J must be in [1, 2^31)");
  if (desc->knn_k < 0 || desc->knn_k > 64) return gp_fail(ctx, GP_ERR_ARG, "gp_build_band: knn_k must be in [0, 64]");
  if (desc->nn_grid < 0 || desc->nn_grid > 1024)
    return gp_fail(ctx, GP_ERR_ARG, "gp_build_band: nn_grid must be in [0, 1024]");
  GP_CUDA(ctx, cudaSetDevice(ctx->device));
  gp_band* b = new (std::nothrow) gp_band();
  if (!b) return gp_fail(ctx, GP_ERR_OOM, "gp_build_band: host allocation");
  b->ctx = ctx;
  b->R = R;
  b->M1 = desc->M1;
  b->M2 = desc->M2;
  b->nb = R / 8 + 1;
  b->knn_k = desc->knn_k;
  b->flags = desc->flags;
  b->J = J;
  b->G = desc->nn_grid;
  gp_status st = build_band_sets(b, pts_dev);
  int64_t V = b->V_stored();
  if (!st) st = gp_alloc_shown(ctx, &b->shown, &b->D, 4 * (size_t)V, "values and Adam moments");
  if (!st) {
    b->D_alt = b->D + V;
    b->m = b->D + 2 * V;
    b->v = b->D + 3 * V;
  }
  if (!st && (b->flags & GP_BAND_DETERMINISTIC)) st = gp_alloc(ctx, &b->acc, 2 * V, "fixed-point accumulator");
  if (!st) st = gp_alloc(ctx, &b->qgrad, V, "query gradient");
  if (!st) st = gp_alloc(ctx, &b->partials, (size_t)GP_MAX_PARTIAL_BLOCKS * 8, "partials");
  if (!st) st = gp_alloc(ctx, &b->dev_ints, GP_DI_COUNT, "device ints");
  if (!st) {
    cudaStream_t s = ctx->stream;
    cudaError_t e = cudaMemsetAsync(b->D, 0, 4 * V * sizeof(float), s);
    if (e == cudaSuccess && b->acc) e = cudaMemsetAsync(b->acc, 0, 2 * V * sizeof(unsigned long long), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(b->qgrad, 0, V * sizeof(float), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(b->dev_ints, 0, GP_DI_COUNT * sizeof(int32_t), s);
    if (e != cudaSuccess) st = gp_cuda_fail(ctx, e, "gp_build_band: memset");
  }
  if (!st) st = gp_build_points(b, pts_dev);
  if (!st) {
    cudaError_t e = cudaStreamSynchronize(ctx->stream);
    if (e != cudaSuccess) st = gp_cuda_fail(ctx, e, "gp_build_band: synchronise");
  }
  if (st) {
    band_free(b);
    return st;
  }
  ctx->live_bands += 1;
  *out = b;
  return GP_OK;
}

extern "C" void gp_band_destroy(gp_band* band) {
  if (!band) return;
  gp_ctx* ctx = band->ctx;
  cudaSetDevice(ctx->device);
  band_free(band);
  cudaGetLastError();
  ctx->live_bands -= 1;
  if (ctx->live_bands == 0 && ctx->destroy_pending) gp_ctx_release(ctx);
}

extern "C" gp_status gp_band_get_info(const gp_band* b, gp_band_info* out) {
  if (!b || !out) return GP_ERR_ARG;
  out->R = b->R;
  out->nb = b->nb;
  out->n_bricks = b->n_bricks;
  out->n_active_bricks = b->n_active;
  out->V_stored = b->V_stored();
  out->V_trainable = b->V_trainable;
  out->V_tv = b->V_tv;
  out->n_pull_cells = b->n_pull;
  out->n_occupied_cells = b->n_occ;
  out->J = b->J;
  out->nn_grid = b->G;
  out->knn_k = b->knn_k;
  return GP_OK;
}

extern "C" gp_status gp_band_init_sphere(gp_band* b, float cx, float cy, float cz, float radius, float noise_std,
                                         uint64_t seed) {
  if (!b) return GP_ERR_ARG;
  gp_ctx* ctx = b->ctx;
  int64_t V = b->V_stored();
  if (V == 0) return GP_OK;
  GP_KERNEL(ctx, "k_init_sphere", k_init_sphere<<<gp_blocks(V, 256), 256, 0, ctx->stream>>>(b->D, b->brick_coord, V, b->R, cx, cy, cz, radius,
                                                            noise_std, (uint32_t)seed, (uint32_t)(seed >> 32)));
  return GP_OK;
}

extern "C" gp_status gp_band_set_values(gp_band* b, const float* d_dev) {
  if (!b) return GP_ERR_ARG;
  if (!d_dev) return gp_fail(b->ctx, GP_ERR_ARG, "gp_band_set_values: null values");
  GP_CUDA(b->ctx, cudaMemcpyAsync(b->D, d_dev, b->V_stored() * sizeof(float), cudaMemcpyDeviceToDevice,
                                  b->ctx->stream));
  return GP_OK;
}

extern "C" gp_status gp_band_export(const gp_band* b, int32_t* ijk_dev, float* d_dev, uint8_t* flags_dev) {
  if (!b) return GP_ERR_ARG;
  gp_ctx* ctx = b->ctx;
  int64_t V = b->V_stored();
  if (V == 0 || (!ijk_dev && !d_dev && !flags_dev)) return GP_OK;
  GP_KERNEL(ctx, "k_export", k_export<<<gp_blocks(V, 256), 256, 0, ctx->stream>>>(b->brick_coord, b->masks, b->D, V, b->R, ijk_dev, d_dev,
                                                       flags_dev));
  return GP_OK;
}

extern "C" gp_status gp_band_values(gp_band* b, float** d_dev, float** m_dev, float** v_dev) {
  if (!b) return GP_ERR_ARG;
  if (d_dev) *d_dev = b->D;
  if (m_dev) *m_dev = b->m;
  if (v_dev) *v_dev = b->v;
  return GP_OK;
}

extern "C" gp_status gp_band_reset_adam(gp_band* b) {
  if (!b) return GP_ERR_ARG;
  int64_t V = b->V_stored();
  GP_CUDA(b->ctx, cudaMemsetAsync(b->m, 0, V * sizeof(float), b->ctx->stream));
  GP_CUDA(b->ctx, cudaMemsetAsync(b->v, 0, V * sizeof(float), b->ctx->stream));
  return GP_OK;
}

extern "C" gp_status gp_band_check(gp_band* b) {
  if (!b) return GP_ERR_ARG;
  gp_ctx* ctx = b->ctx;
  int32_t flag = 0;
  GP_CUDA(ctx, cudaMemcpyAsync(&flag, b->dev_ints + GP_DI_ERROR, 4, cudaMemcpyDeviceToHost, ctx->stream));
  GP_CUDA(ctx, cudaMemsetAsync(b->dev_ints + GP_DI_ERROR, 0, 4, ctx->stream));
  GP_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
  if (flag & GP_EF_TIMEOUT) return gp_fail(ctx, GP_ERR_TIMEOUT, "a bounded device wait gave up");
  if (flag & (GP_EF_NUMERIC | GP_EF_RANGE))
    return gp_fail(ctx, GP_ERR_NUMERIC, "a device numeric or range check fired");
  return GP_OK;
}
