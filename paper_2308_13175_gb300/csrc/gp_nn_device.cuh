// Device side of the exact nearest-point search (shared by gp_nn.cu and
// gp_multi.cu): the cell list with its block bounds, the float32 screen with
// its proven margins, the search of one query by one thread and the float64
// tie-break.  The exactness argument is in the header of gp_nn.cu.
#pragma once

#include <math.h>

#include "gp_internal.cuh"

constexpr float NN_EPS = 3.814697265625e-06f;  // 2^-18
constexpr float NN_TINY = 1e-30f;
// A hint more than this many cells away (twice as many where the query's own
// block is empty) is passed over: it says nothing about where the nearest point
// is, and the ball of what is found beside it holds much of the cloud (262,144
// queries among 100,000 points of a surface, random points as hints: 7,200 us,
// and 160 with them passed over).  A query's own source point lies within four
// sigma, six cells at the usual 50 neighbours and 6.5 points a cell.
constexpr float NN_FAR_HINT = 8.f;

// The cloud in a uniform grid of G^3 cells, grouped into blocks of 4^3 cells
// and super-blocks of 4^3 blocks.  Only what holds points is stored.
//
// The points of a cell lie in chunks of four, 64 bytes each: (x0..x3),
// (y0..y3), (z0..z3) and the four original indices; the last chunk of a cell
// is filled up with points at infinity (index -1), whose distance +inf never
// compares below another.  A chunk is three 16-byte loads, and its four
// distances twelve two-wide float32 instructions (four 16-byte loads and 24
// instructions with the points as records of four floats).  The parts are
// rotated by the chunk's number (nn_part), so that lanes reading the same part
// of chunks anywhere spread over the banks: 1,500,001 queries among 2 M points
// took 491 us with it, 520 us in a fixed order.
//
// A block with points has a record of two float4,
//   (n.x, n.y, n.z, lo), (hi, first occupied cell, occupancy mask: 2 words),
// the plane n . p in [lo, hi] holding for every point p of the block (n a unit
// vector, the normal of the block's best plane, or 0 with lo = hi = 0), bit
// 16 z + 4 y + x of the mask telling whether that cell of the block holds
// points.  The k-th occupied cell's chunks are occ[first + k] up to
// occ[first + k + 1].
struct NNGrid {
  const float4* __restrict__ pts;     // 4 per chunk
  const int32_t* __restrict__ occ;    // first chunk of each occupied cell, one more entry per block
  const float4* __restrict__ blk;     // the records of the blocks with points
  const int32_t* __restrict__ table;  // nbk^3: record of the block, -1 where it holds no point
  const unsigned long long* __restrict__ sup;  // nsup^3: which blocks of a super-block hold points
  int G, nbk, nsup;
  float half_g;  // G / 2
  float cs;      // 2 / G
};

__device__ __forceinline__ int nn_cell(float x, const NNGrid& g) {
  float t = __fmul_rn(__fadd_rn(x, 1.0f), g.half_g);
  int c = (t < 0.f) ? -1 : (int)floorf(fminf(t, 1.0e6f));
  return min(max(c, 0), g.G - 1);
}

// Lower bound on the distance from q to any point outside the box of cells
// [c - r, c + r]; returns +inf when the box covers the whole grid.
__device__ __forceinline__ float nn_gap(const float q[3], const int c[3], int r, const NNGrid& g) {
  float gap = INFINITY;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if (c[a] - r > 0) {
      float lo = -1.0f + (float)(c[a] - r) * g.cs;
      gap = fminf(gap, q[a] - lo);
    }
    if (c[a] + r < g.G - 1) {
      float hi = -1.0f + (float)(c[a] + r + 1) * g.cs;
      gap = fminf(gap, hi - q[a]);
    }
  }
  return gap;
}

// sqrt(max(x, 0)) in one instruction: within a relative 1e-6 of the root, which
// the factor 1.000001 and the additive margin (>= 2e-5) wherever it is used as
// a radius cover.
__device__ __forceinline__ float nn_root(float x) {
  float r;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(fmaxf(x, 0.f)));
  return r;
}

__device__ __forceinline__ float nn_margin(const float q[3]) {
  float m = fmaxf(fabsf(q[0]), fmaxf(fabsf(q[1]), fabsf(q[2])));
  return 1e-5f * (2.0f + m);
}

__device__ __forceinline__ double nn_d64(const float q[3], float x, float y, float z) {
  double dx = __dsub_rn((double)q[0], (double)x);
  double dy = __dsub_rn((double)q[1], (double)y);
  double dz = __dsub_rn((double)q[2], (double)z);
  return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}

// The float32 distance of the screen, in the order of the two-wide form.
__device__ __forceinline__ float nn_d32(const float q[3], float x, float y, float z) {
  const float dx = __fsub_rn(x, q[0]), dy = __fsub_rn(y, q[1]), dz = __fsub_rn(z, q[2]);
  return __fmaf_rn(dz, dz, __fmaf_rn(dy, dy, __fmul_rn(dx, dx)));
}

// -q, twice per axis, for the two-wide distances.
struct NNQuery {
  unsigned long long x, y, z;
};
__device__ __forceinline__ unsigned long long nn_twice(float v) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(v));
  return r;
}
__device__ __forceinline__ NNQuery nn_query(const float q[3]) {
  return NNQuery{nn_twice(-q[0]), nn_twice(-q[1]), nn_twice(-q[2])};
}
__device__ __forceinline__ void nn_d32x2(unsigned long long x, unsigned long long y, unsigned long long z,
                                         const NNQuery& q, float& d0, float& d1) {
  asm("{\n .reg .b64 a, b, c;\n"
      " add.rn.f32x2 a, %2, %5;\n add.rn.f32x2 b, %3, %6;\n add.rn.f32x2 c, %4, %7;\n"
      " mul.rn.f32x2 a, a, a;\n fma.rn.f32x2 a, b, b, a;\n fma.rn.f32x2 a, c, c, a;\n"
      " mov.b64 {%0, %1}, a;\n}\n"
      : "=f"(d0), "=f"(d1)
      : "l"(x), "l"(y), "l"(z), "l"(q.x), "l"(q.y), "l"(q.z));
}
// Where part k (0: x, 1: y, 2: z, 3: index) of chunk c lies, in float4.
__host__ __device__ __forceinline__ int64_t nn_part(int64_t c, int k) {
  return 4 * c + ((k + (int)(c >> 1)) & 3);
}

// Where part k of a point of a block lies, in floats: `at` is its place counted
// from the block's first chunk (4 chunk + place in the chunk).  A cell's last
// chunk is filled up, so places counted from the start of the cloud pass 2^31
// for clouds that gp_build_band takes; a block's own stay below 2^32.
__host__ __device__ __forceinline__ int64_t nn_place(int64_t first_chunk, uint32_t at, int k) {
  return 4 * nn_part(first_chunk + (at >> 2), k) + (at & 3u);
}

// Part k of the point at place i (4 chunk + place in the chunk).
__device__ __forceinline__ float nn_value(const float4* __restrict__ pts, int64_t i, int k) {
  return __ldg(reinterpret_cast<const float*>(pts + nn_part(i >> 2, k)) + (i & 3));
}

// The distances of chunk c's four points.
__device__ __forceinline__ void nn_chunk(const float4* __restrict__ pts, const NNQuery& q, int c, float d[4]) {
  const ulonglong2* p = reinterpret_cast<const ulonglong2*>(pts + 4 * (int64_t)c);
  const int r = c >> 1;
  const ulonglong2 X = __ldg(p + (r & 3)), Y = __ldg(p + ((r + 1) & 3)), Z = __ldg(p + ((r + 2) & 3));
  nn_d32x2(X.x, Y.x, Z.x, q, d[0], d[1]);
  nn_d32x2(X.y, Y.y, Z.y, q, d[2], d[3]);
}

// The pruning radius squared that a known float32 distance d gives.
__device__ __forceinline__ float nn_thr(float d) { return d * (1.0f + 8.0f * NN_EPS) + NN_TINY; }

// The cells [lo, hi] (grid coordinates) of block (bx, by, bz) as a mask.
__host__ __device__ __forceinline__ unsigned long long nn_box_mask(const int lo[3], const int hi[3], int bx, int by,
                                                                   int bz) {
  const int xl = lo[0] - 4 * bx > 0 ? lo[0] - 4 * bx : 0, xh = hi[0] - 4 * bx < 3 ? hi[0] - 4 * bx : 3;
  const int yl = lo[1] - 4 * by > 0 ? lo[1] - 4 * by : 0, yh = hi[1] - 4 * by < 3 ? hi[1] - 4 * by : 3;
  const int zl = lo[2] - 4 * bz > 0 ? lo[2] - 4 * bz : 0, zh = hi[2] - 4 * bz < 3 ? hi[2] - 4 * bz : 3;
  if (xl > xh || yl > yh || zl > zh) return 0ull;
  const uint32_t x = ((2u << xh) - (1u << xl)) * 0x11111111u;
  const uint32_t y = ((16u << (4 * yh)) - (1u << (4 * yl))) * 0x00010001u;
  const unsigned long long xy = (unsigned long long)(x & y);
  const unsigned long long z = (~0ull >> (48 - 16 * zh)) & (~0ull << (16 * zl));
  return (xy | (xy << 32)) & z;
}

// A stored block: its occupancy and first occupied cell.
struct NNBlock {
  unsigned long long mask;
  int first;
};

__device__ __forceinline__ NNBlock nn_block(float4 B) {
  return NNBlock{(unsigned long long)__float_as_uint(B.z) | ((unsigned long long)__float_as_uint(B.w) << 32),
                 __float_as_int(B.y)};
}

// Takes from m its lowest cell and the ones after it up to the next occupied
// cell of the block that is not in m: their chunks are one range [a, b).
__device__ __forceinline__ void nn_pop_cells(const NNGrid& g, const NNBlock& k, unsigned long long& m, int& a, int& b) {
  const unsigned long long low = m & (0ull - m);
  const unsigned long long stop = k.mask & ~m & (0ull - low);
  const unsigned long long run = m & ((stop & (0ull - stop)) - 1ull);  // all of m without a stop
  const int32_t* o = g.occ + k.first + __popcll(k.mask & (low - 1ull));
  m ^= run;
  a = __ldg(o);
  b = __ldg(o + __popcll(run));
}

// The cells of stored block bi at (bx, by, bz) that can hold a point within
// squared distance thr of q.  Every point p of the block has n . p in
// [lo, hi], so |p - q| is at least the gap h from n . q to that interval, and
// what of p - q is across n is at most l = sqrt(thr - h^2) long: along axis a,
// p_a - q_a lies in n_a [lo - n.q, hi - n.q] +- l sqrt(1 - n_a^2).  On a flat
// patch this leaves a disc around the foot of q where the ball around q would
// take every cell that reaches into it from below.  The margin covers the
// rounding of the dot products and of the cell faces, 1e-3 that of the root's
// argument near n_a = 1.
__device__ __forceinline__ unsigned long long nn_block_cells(const float q[3], float thr, float margin,
                                                             const NNGrid& g, int bi, int bx, int by, int bz,
                                                             NNBlock& k) {
  const float4 A = __ldg(g.blk + 2 * (int64_t)bi), B = __ldg(g.blk + 2 * (int64_t)bi + 1);
  k = nn_block(B);
  if (!(thr < INFINITY)) return k.mask;
  const float nq = A.x * q[0] + A.y * q[1] + A.z * q[2];
  const float dlo = A.w - nq - margin, dhi = B.x - nq + margin;
  const float h = fmaxf(fmaxf(dlo, -dhi), 0.f);
  const float rem = thr - h * h;
  if (!(rem >= 0.f)) return 0ull;
  const float l = nn_root(rem) * 1.000001f + margin, rad = nn_root(thr) * 1.000001f + margin;
  const float n[3] = {A.x, A.y, A.z};
  int lo[3], hi[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const float u = n[a] * dlo, v = n[a] * dhi;
    const float w = l * (nn_root(1.0f - n[a] * n[a]) + 1e-3f) + margin;
    lo[a] = nn_cell(q[a] + fmaxf(fminf(u, v) - w, -rad), g);
    hi[a] = nn_cell(q[a] + fminf(fmaxf(u, v) + w, rad), g);
  }
  return k.mask & nn_box_mask(lo, hi, bx, by, bz);
}

// Visit every cell of ring r (Chebyshev shell of cells) around cell c that
// holds points.  Blocks that lie whole within the rings before are stepped over
// along x, so that a ring takes the blocks of its shell, not of its box: the
// build of 300,001 points, one of them 150 cells from the rest, k = 50, takes 312 ms,
// 2,228 with the box (100,000 points side by side: 402 and 393 us of k_knn_sigma).
template <typename F>
__device__ __forceinline__ void nn_ring(const int c[3], int r, const NNGrid& g, F&& visit) {
  int lo[3], hi[3], li[3], hj[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    lo[a] = max(c[a] - r, 0);
    hi[a] = min(c[a] + r, g.G - 1);
    li[a] = c[a] - r + 1;
    hj[a] = c[a] + r - 1;
  }
  const int from = (li[0] + 3) >> 2, to = (hj[0] - 3) >> 2;
  for (int bz = lo[2] >> 2; bz <= hi[2] >> 2; ++bz)
    for (int by = lo[1] >> 2; by <= hi[1] >> 2; ++by) {
      const bool in = 4 * bz >= li[2] && 4 * bz + 3 <= hj[2] && 4 * by >= li[1] && 4 * by + 3 <= hj[1];
      for (int bx = lo[0] >> 2; bx <= hi[0] >> 2; ++bx) {
        if (in && bx >= from && bx <= to) {
          bx = to;
          continue;
        }
        const int bi = __ldg(g.table + ((int64_t)bz * g.nbk + by) * g.nbk + bx);
        if (bi < 0) continue;
        const NNBlock k = nn_block(__ldg(g.blk + 2 * (int64_t)bi + 1));
        unsigned long long m = k.mask & nn_box_mask(lo, hi, bx, by, bz);
        if (r > 0) m &= ~nn_box_mask(li, hj, bx, by, bz);
        while (m) {
          int a, b;
          nn_pop_cells(g, k, m, a, b);
          visit(a, b);
        }
      }
    }
}

// Lower bound on |p_a - q_a| for any point p in super-block s along one axis
// (those at the grid's ends extend to infinity outwards).
__device__ __forceinline__ float nn_super_gap(float qa, int s, const NNGrid& g, float margin) {
  const float lo = -1.0f + (float)(16 * s) * g.cs, hi = lo + 16.0f * g.cs;
  float d = 0.f;
  if (s > 0 && qa < lo) d = lo - qa;
  if (s < g.nsup - 1 && qa > hi) d = qa - hi;
  return fmaxf(d - margin, 0.f);
}

// Visit the cells of the blocks sm of super-block (sx, sy, sz) that can hold a
// point within squared distance thr of q (thr is read live).
template <typename F>
__device__ __forceinline__ void nn_super(const float q[3], const NNGrid& g, float margin, const float& thr, int sx, int sy,
                                         int sz, unsigned long long sm, F&& visit) {
  while (sm) {
    const int bit = __ffsll((long long)sm) - 1;
    sm &= sm - 1ull;
    const int bx = 4 * sx + (bit & 3), by = 4 * sy + ((bit >> 2) & 3), bz = 4 * sz + (bit >> 4);
    const int bi = __ldg(g.table + ((int64_t)bz * g.nbk + by) * g.nbk + bx);
    NNBlock k;
    unsigned long long m = nn_block_cells(q, thr, margin, g, bi, bx, by, bz, k);
    while (m) {
      int a, b;
      nn_pop_cells(g, k, m, a, b);
      visit(a, b);
    }
  }
}

// Visit the cells that can hold a point within squared distance thr of q, thr
// known: the blocks that the box of that ball meets, in super-blocks the ball
// meets (of a query far outside, the box is most of the grid: 20,000 queries at
// six radii 22.7 ms without that test, 13.2 with it).  It ranks near ties, in which
// a lane works by itself while its warp waits: with nn_walk, which tests every
// block of the super-block, 200,000 queries with 8-way ties took 1,419 us, now
// 676, and 262,144 queries among a noisy object's points 116, now 89 (as a
// function of its own, to save registers: 581 and 92).
template <typename F>
__device__ __forceinline__ void nn_ball(const float q[3], const NNGrid& g, float margin, float thr, F&& visit) {
  const float rad = nn_root(thr) * 1.000001f + margin;
  int lo[3], hi[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    lo[a] = nn_cell(q[a] - rad, g) >> 2;
    hi[a] = nn_cell(q[a] + rad, g) >> 2;
  }
  for (int sz = lo[2] >> 2; sz <= hi[2] >> 2; ++sz)
    for (int sy = lo[1] >> 2; sy <= hi[1] >> 2; ++sy)
      for (int sx = lo[0] >> 2; sx <= hi[0] >> 2; ++sx) {
        const float dx = nn_super_gap(q[0], sx, g, margin), dy = nn_super_gap(q[1], sy, g, margin),
                    dz = nn_super_gap(q[2], sz, g, margin);
        if (dx * dx + dy * dy + dz * dz > thr) continue;
        nn_super(q, g, margin, thr, sx, sy, sz,
                 __ldg(g.sup + ((int64_t)sz * g.nsup + sy) * g.nsup + sx) & nn_box_mask(lo, hi, sx, sy, sz), visit);
      }
}

// Visit, in rings of super-blocks around q, the cells that can hold a point
// within squared distance thr of q (thr is read live and may start at +inf).
template <typename F>
__device__ __forceinline__ void nn_walk(const float q[3], const NNGrid& g, float margin, const float& thr, F&& visit) {
  const int c[3] = {nn_cell(q[0], g) >> 4, nn_cell(q[1], g) >> 4, nn_cell(q[2], g) >> 4};
  for (int r = 0;; ++r) {
    if (r > 0) {
      float gap = INFINITY;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        if (c[a] - r >= 0) gap = fminf(gap, nn_super_gap(q[a], c[a] - r, g, margin));
        if (c[a] + r < g.nsup) gap = fminf(gap, nn_super_gap(q[a], c[a] + r, g, margin));
      }
      if (!(gap < INFINITY) || gap * gap > thr) break;
    }
    for (int sz = max(c[2] - r, 0); sz <= min(c[2] + r, g.nsup - 1); ++sz)
      for (int sy = max(c[1] - r, 0); sy <= min(c[1] + r, g.nsup - 1); ++sy) {
        const bool face = sz == c[2] - r || sz == c[2] + r || sy == c[1] - r || sy == c[1] + r;
        for (int sx = c[0] - r; sx <= c[0] + r; sx += (face || r == 0) ? 1 : 2 * r) {
          if (sx < 0 || sx >= g.nsup) continue;
          const unsigned long long sm = __ldg(g.sup + ((int64_t)sz * g.nsup + sy) * g.nsup + sx);
          if (!sm) continue;
          const float dx = nn_super_gap(q[0], sx, g, margin), dy = nn_super_gap(q[1], sy, g, margin),
                      dz = nn_super_gap(q[2], sz, g, margin);
          if (dx * dx + dy * dy + dz * dz > thr) continue;
          nn_super(q, g, margin, thr, sx, sy, sz, sm, visit);
        }
      }
  }
}

// The best float32 distance seen (b1, of a point of chunk c1) and the smallest
// of any other point (b2).  No chunk is met twice.
struct NNTop {
  float b1, b2;
  int c1;
};

__device__ __forceinline__ void nn_scan(NNTop& t, const NNQuery& q, const NNGrid& g, int c) {
  float d[4];
  nn_chunk(g.pts, q, c, d);
  const float l0 = fminf(d[0], d[1]), h0 = fmaxf(d[0], d[1]), l1 = fminf(d[2], d[3]), h1 = fmaxf(d[2], d[3]);
  const float m = fminf(l0, l1);                                   // the chunk's best
  const float m2 = fminf(fmaxf(l0, l1), fminf(h0, h1));            // and its runner-up
  t.b2 = fminf(fminf(t.b2, m2), fmaxf(t.b1, m));
  if (m < t.b1) {
    t.b1 = m;
    t.c1 = c;
  }
}

// A block with points near q, where the block q lies in has none: of the first
// ring of super-blocks around q with any, the one whose centre is nearest.
static __device__ __noinline__ int nn_near_block(float q0, float q1, float q2, const NNGrid& g) {
  const int c[3] = {nn_cell(q0, g) >> 4, nn_cell(q1, g) >> 4, nn_cell(q2, g) >> 4};
  float best = INFINITY;
  int at = -1;
  for (int r = 0; r < g.nsup && at < 0; ++r)
    for (int sz = max(c[2] - r, 0); sz <= min(c[2] + r, g.nsup - 1); ++sz)
      for (int sy = max(c[1] - r, 0); sy <= min(c[1] + r, g.nsup - 1); ++sy) {
        const bool face = sz == c[2] - r || sz == c[2] + r || sy == c[1] - r || sy == c[1] + r;
        for (int sx = c[0] - r; sx <= c[0] + r; sx += (face || r == 0) ? 1 : 2 * r) {
          if (sx < 0 || sx >= g.nsup) continue;
          unsigned long long sm = __ldg(g.sup + ((int64_t)sz * g.nsup + sy) * g.nsup + sx);
          while (sm) {
            const int bit = __ffsll((long long)sm) - 1;
            sm &= sm - 1ull;
            const int bx = 4 * sx + (bit & 3), by = 4 * sy + ((bit >> 2) & 3), bz = 4 * sz + (bit >> 4);
            const float dx = q0 - (-1.0f + (float)(4 * bx + 2) * g.cs), dy = q1 - (-1.0f + (float)(4 * by + 2) * g.cs),
                        dz = q2 - (-1.0f + (float)(4 * bz + 2) * g.cs);
            const float d = dx * dx + dy * dy + dz * dz;
            if (at < 0 || d < best) {
              best = d;
              at = bx | by << 8 | bz << 16;
            }
          }
        }
      }
  return at;
}

// Whether the block q lies in holds no point.
__device__ __forceinline__ bool nn_block_empty(const float q[3], const NNGrid& g) {
  const int bx = nn_cell(q[0], g) >> 2, by = nn_cell(q[1], g) >> 2, bz = nn_cell(q[2], g) >> 2;
  return __ldg(g.table + ((int64_t)bz * g.nbk + by) * g.nbk + bx) < 0;
}

// Step 1 of a search: a first point.  hint: index of a cloud point
// to start from (-1: none); a record of `seeds` is a point s and its normal n
// as three 10-bit signed fractions of 511 (0: unknown).  The nearest point is
// expected around the foot of q on the tangent plane of s, then, if that lies
// outside, on the near face of the slab of the block there (of the block of s,
// where that one holds no point; a block that is not flat leaves the place as it
// is: on its middle plane instead, 300,000 hinted queries in a volume of a million
// points took 139 us, 93 now, in a thick shell 185, now 143); the
// points of the 2^3 cells nearest to that place are scanned, or those of the
// whole block where these are empty.  A query without a hint tends to lie on
// the surface (a mesh scored against a cloud); within half a cell of the plane
// its ball is small and the one cell it is in is scanned.  Returns the block scanned
// and where: record << 8 | (0: 2^3 cells, 1: all, 2: one cell) << 6 | lowest
// scanned cell in the block, all bits set if there is no block.
template <bool COUNT>
__device__ __forceinline__ int nn_first(const float q[3], int hint, int64_t J, const float4* __restrict__ seeds,
                                        const NNGrid& g, NNTop& t, int& work) {
  t = NNTop{INFINITY, INFINITY, -1};
  float f[3] = {q[0], q[1], q[2]};
  float4 s = make_float4(q[0], q[1], q[2], 0.f);
  bool hinted = hint >= 0 && hint < J;
  if (hinted) {
    const float4 p = __ldg(seeds + hint);
    const float d = nn_d32(q, p.x, p.y, p.z), far = NN_FAR_HINT * g.cs;
    if (COUNT) ++work;
    hinted = d <= far * far || (d <= 4.f * far * far && nn_block_empty(q, g));
    if (hinted) {
      s = p;
      const int w = __float_as_int(s.w);
      const float n0 = (float)((w << 22) >> 22) * (1.0f / 511.0f), n1 = (float)((w << 12) >> 22) * (1.0f / 511.0f),
                  n2 = (float)((w << 2) >> 22) * (1.0f / 511.0f);
      const float h = (q[0] - s.x) * n0 + (q[1] - s.y) * n1 + (q[2] - s.z) * n2;
      f[0] -= h * n0;
      f[1] -= h * n1;
      f[2] -= h * n2;
    }
  }
  int bx = nn_cell(f[0], g) >> 2, by = nn_cell(f[1], g) >> 2, bz = nn_cell(f[2], g) >> 2;
  int bi = __ldg(g.table + ((int64_t)bz * g.nbk + by) * g.nbk + bx);
  if (bi < 0) {
    bx = nn_cell(s.x, g) >> 2;
    by = nn_cell(s.y, g) >> 2;
    bz = nn_cell(s.z, g) >> 2;
    bi = __ldg(g.table + ((int64_t)bz * g.nbk + by) * g.nbk + bx);
    if (bi < 0) {
      const int at = nn_near_block(q[0], q[1], q[2], g);
      if (at < 0) return -1;
      bx = at & 255;
      by = (at >> 8) & 255;
      bz = at >> 16;
      bi = __ldg(g.table + ((int64_t)bz * g.nbk + by) * g.nbk + bx);
    }
  }
  const float4 A = __ldg(g.blk + 2 * (int64_t)bi), B = __ldg(g.blk + 2 * (int64_t)bi + 1);
  const NNBlock k = nn_block(B);
  const float n[3] = {A.x, A.y, A.z};
  const float nf = A.x * f[0] + A.y * f[1] + A.z * f[2];
  const float off = fminf(fmaxf(nf, A.w), B.x) - nf;
  const int corner[3] = {4 * bx, 4 * by, 4 * bz};
  const float h = n[0] * q[0] + n[1] * q[1] + n[2] * q[2] - 0.5f * (A.w + B.x);
  int how = !hinted && fabsf(h) < 0.5f * g.cs ? 2 : 0;
  int lo[3], hi[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    // the 2 cells nearest to the place along this axis (or its cell), inside the block
    const int c = nn_cell(f[a] + off * n[a] - (how ? 0.f : 0.5f * g.cs), g);
    lo[a] = min(max(c, corner[a]), corner[a] + (how ? 3 : 2));
    hi[a] = lo[a] + (how ? 0 : 1);
  }
  unsigned long long m = k.mask & nn_box_mask(lo, hi, bx, by, bz);
  if (!m) {
    m = k.mask;
    how = 1;
  }
  const NNQuery q2 = nn_query(q);
  int cur = 0, end = 0;
  while (true) {
    if (cur >= end) {
      if (!m) break;
      nn_pop_cells(g, k, m, cur, end);
      if (COUNT) work += 4 * (end - cur);
    }
    nn_scan(t, q2, g, cur++);
  }
  return (bi << 8) | (how << 6) | ((lo[0] & 3) | ((lo[1] & 3) << 2) | ((lo[2] & 3) << 4));
}

// A warp's shared state in step 2: its 32 queries with their bounds, and the
// two queues.
struct NNWarp {
  float4 q[32];                 // x, y, z, pruning radius squared
  unsigned long long key1[32];  // best distance (float bits), then its chunk
  unsigned int key2[32];        // best distance of any other point (float bits)
  int first[32];                // where step 1 scanned
  int lo[32], hi[32];           // blocks the ball meets, 8 bits an axis
  int off[32];                  // first super-block of each query in the warp's list
  int2 range[64];               // chunks to scan: first, query | count << 5
  int block[64];                // blocks to test: coordinates, 8 bits an axis | query << 24
};

// Step 2 for a warp's queries: the blocks the ball of the best distance meets,
// cut to the cells that can hold a nearer point (nn_block_cells), without
// those step 1 scanned.  What one query needs here varies by a factor of ten
// and more within a warp (its work grows with the cube of its distance), so
// the work of all 32 is laid out in three lists that the lanes share evenly:
// the super-blocks of all the balls, the blocks with points these hold, and
// the ranges of at most two chunks their cells come to.  A list is worked
// through 32 entries at a time as soon as it has as many.  A point within its
// query's bound (few are) goes to the query's two keys by atomics in shared
// memory: the smaller key stays, the larger goes on to the second.
//
// Measured (GB300, seeded batches, whole search): with one thread walking its
// query's rows of cells, 8 of 32 lanes active, 1,116 us for 2,097,152 queries
// among 10 M points and 206 us for 262,144 among 100,000; with step 2 lane by
// lane 730 and 210; shared 503 and 111 (488 and 86 as the search stands).  It is
// then bound by the L1, for which a lane's chunk is a line of its own, and by issue
// (75% of the L1's throughput and 64% of the issue slots with 1,500,001 queries; 52%
// and 64% with 262,144, which leave latency).
// Sorting a block's queries by radius instead of sharing gave 700 and 190.
template <bool COUNT>
__device__ __forceinline__ void nn_rest(const float q[3], const NNGrid& g, bool go, int first, NNTop& t, NNWarp& sh,
                                        int& work) {
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const unsigned below = (1u << lane) - 1u;
  int total = 0;
  {
    const float thr = nn_thr(t.b1);
    const float rad = nn_root(thr) * 1.000001f + nn_margin(q);
    int lo = 0, hi = 0, n = go ? 1 : 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int l = nn_cell(q[a] - rad, g) >> 2, h = nn_cell(q[a] + rad, g) >> 2;
      lo |= l << (8 * a);
      hi |= h << (8 * a);
      n *= (h >> 2) - (l >> 2) + 1;
    }
    __syncwarp();
    sh.q[lane] = make_float4(q[0], q[1], q[2], thr);
    sh.key1[lane] = ((unsigned long long)__float_as_uint(t.b1) << 32) | (unsigned)t.c1;
    sh.key2[lane] = __float_as_uint(t.b2);
    sh.first[lane] = first;
    sh.lo[lane] = lo;
    sh.hi[lane] = hi;
    int incl = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(FULL, incl, o);
      if (lane >= o) incl += y;
    }
    sh.off[lane] = incl - n;
    total = __shfl_sync(FULL, incl, 31);
    __syncwarp();
  }
  int base = 0, nb = 0, nr = 0;  // super-blocks taken, entries of the two queues
  unsigned long long sm = 0;     // this lane's super-block's blocks still to queue
  int at = 0;                    // its lowest block | query << 24
  while (true) {
    while (nb < 32) {
      unsigned some = __ballot_sync(FULL, sm != 0ull);
      if (!some) {
        if (base >= total) break;
        const int idx = base + lane;
        base += 32;
        if (idx < total) {
          int o = 0;
#pragma unroll
          for (int step = 16; step > 0; step >>= 1)
            if (sh.off[o + step] <= idx) o += step;
          const int lw = sh.lo[o], hw = sh.hi[o];
          const int lo[3] = {lw & 255, (lw >> 8) & 255, lw >> 16}, hi[3] = {hw & 255, (hw >> 8) & 255, hw >> 16};
          const unsigned nx = (hi[0] >> 2) - (lo[0] >> 2) + 1, ny = (hi[1] >> 2) - (lo[1] >> 2) + 1;
          const unsigned l = idx - sh.off[o], yz = l / nx;
          const int sx = (lo[0] >> 2) + (int)(l - yz * nx), sy = (lo[1] >> 2) + (int)(yz % ny),
                    sz = (lo[2] >> 2) + (int)(yz / ny);
          sm = __ldg(g.sup + ((int64_t)sz * g.nsup + sy) * g.nsup + sx) & nn_box_mask(lo, hi, sx, sy, sz);
          at = (4 * sx) | (4 * sy << 8) | (4 * sz << 16) | (o << 24);
        }
        continue;
      }
      if (sm) {
        const int bit = __ffsll((long long)sm) - 1;
        sm &= sm - 1ull;
        sh.block[nb + __popc(some & below)] = at + ((bit & 3) | ((bit >> 2) & 3) << 8 | (bit >> 4) << 16);
      }
      nb += __popc(some);
    }
    if (nb == 0 && nr == 0) break;
    const bool last = nb <= 32 && base >= total && !__any_sync(FULL, sm != 0ull);
    const int take = min(nb, 32);
    nb -= take;
    if (go) sh.q[lane].w = nn_thr(__uint_as_float((unsigned)(sh.key1[lane] >> 32)));  // the bounds reached so far
    __syncwarp();
    unsigned long long m = 0ull;
    NNBlock k{0ull, 0};
    int o = 0, a = 0, n = 0;
    if (lane < take) {
      const int e = sh.block[nb + lane];
      const int bx = e & 255, by = (e >> 8) & 255, bz = (e >> 16) & 255;
      o = (int)((unsigned)e >> 24);
      const float4 Q = sh.q[o];
      const float qo[3] = {Q.x, Q.y, Q.z};
      const int bi = __ldg(g.table + ((int64_t)bz * g.nbk + by) * g.nbk + bx);
      m = nn_block_cells(qo, Q.w, nn_margin(qo), g, bi, bx, by, bz, k);
      const int f = sh.first[o];
      if (bi == (int)((unsigned)f >> 8)) {
        const int l0[3] = {f & 3, (f >> 2) & 3, (f >> 4) & 3};
        const int e = (f & 128) ? 0 : 1;
        const int h0[3] = {l0[0] + e, l0[1] + e, l0[2] + e};
        m &= (f & 64) ? 0ull : ~nn_box_mask(l0, h0, 0, 0, 0);
      }
    }
    __syncwarp();
    while (true) {
      if (n == 0 && m) {
        int b;
        nn_pop_cells(g, k, m, a, b);
        n = b - a;
        if (COUNT) work += 4 * n;
      }
      const unsigned some = __ballot_sync(FULL, n > 0);
      if (n > 0) {
        const int c = min(n, 2);
        sh.range[nr + __popc(some & below)] = make_int2(a, o | c << 5);
        a += c;
        n -= c;
      }
      nr += __popc(some);
      const bool flush = last && !some;
      if (nr >= 32 || (flush && nr > 0)) {
        const int r = min(nr, 32);
        nr -= r;
        __syncwarp();
        if (lane < r) {
          const int2 e = sh.range[nr + lane];
          const int w = e.y & 31;
          const float4 Q = sh.q[w];
          const float qo[3] = {Q.x, Q.y, Q.z};
          const NNQuery q2 = nn_query(qo);
          const int c2 = (e.y >> 5) > 1 ? e.x + 1 : e.x;
          float d[2][4];
          nn_chunk(g.pts, q2, e.x, d[0]);
          nn_chunk(g.pts, q2, c2, d[1]);
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            const float l0 = fminf(d[j][0], d[j][1]), h0 = fmaxf(d[j][0], d[j][1]);
            const float l1 = fminf(d[j][2], d[j][3]), h1 = fmaxf(d[j][2], d[j][3]);
            const float lm = fminf(l0, l1);
            if (lm <= Q.w && (j == 0 || c2 != e.x)) {
              const float m2 = fminf(fmaxf(l0, l1), fminf(h0, h1));
              const unsigned long long key =
                  ((unsigned long long)__float_as_uint(lm) << 32) | (unsigned)(j ? c2 : e.x);
              const unsigned long long was = atomicMin(&sh.key1[w], key);
              atomicMin(&sh.key2[w], min((unsigned)((was > key ? was : key) >> 32), __float_as_uint(m2)));
            }
          }
        }
        __syncwarp();
      }
      if (!some && !(flush && nr > 0)) break;
    }
    if (last) break;
  }
  __syncwarp();
  if (go) {
    const unsigned long long k1 = sh.key1[lane];
    t.b1 = __uint_as_float((unsigned)(k1 >> 32));
    t.c1 = (int)(unsigned)k1;
    t.b2 = __uint_as_float(sh.key2[lane]);
  }
}

// The answer of a searched query: its index and point.  At a near tie
// (another point within the float32 margin of the best) every point within
// the margin is ranked by its float64 distance and index.  -1 if no point
// compares below +inf.
template <bool COUNT>
__device__ __forceinline__ int nn_answer(const float q[3], const NNGrid& g, const NNTop& t, float s[3], int& work) {
  if (t.c1 < 0) return -1;
  const NNQuery q2 = nn_query(q);
  const float tie = t.b1 * (1.0f + 2.0f * NN_EPS) + NN_TINY;
  int64_t at = 0;  // 4 chunk + place
  if (t.b2 > tie) {
    float d[4];
    nn_chunk(g.pts, q2, t.c1, d);
    at = 4 * (int64_t)t.c1 + (d[0] == t.b1 ? 0 : d[1] == t.b1 ? 1 : d[2] == t.b1 ? 2 : 3);
  } else {
    double bd = INFINITY;
    int bj = 0x7fffffff;
    const float thr = nn_thr(t.b1);
    nn_ball(q, g, nn_margin(q), thr, [&](int a, int b) {
      if (COUNT) work += 4 * (b - a);
      for (int c = a; c < b; ++c) {
        float d[4];
        nn_chunk(g.pts, q2, c, d);
        for (int k = 0; k < 4; ++k) {
          if (!(d[k] <= tie)) continue;
          const int64_t i = 4 * (int64_t)c + k;
          const int j = __float_as_int(nn_value(g.pts, i, 3));
          const double dd = nn_d64(q, nn_value(g.pts, i, 0), nn_value(g.pts, i, 1), nn_value(g.pts, i, 2));
          if (dd < bd || (dd == bd && j < bj)) {
            bd = dd;
            bj = j;
            at = i;
          }
        }
      }
    });
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) s[a] = nn_value(g.pts, at, a);
  return __float_as_int(nn_value(g.pts, at, 3));
}

__device__ __forceinline__ bool nn_query_ok(const float q[3]) {
  return fabsf(q[0]) <= 1e18f && fabsf(q[1]) <= 1e18f && fabsf(q[2]) <= 1e18f;
}

// The search of a warp's 32 queries, one a lane, all lanes together (ok: this
// lane has one).  Step 1 lane by lane, step 2 shared; a query that step 1
// leaves without a bound (a block of points no distance to which compares
// below +inf) walks the rings instead.
template <bool COUNT>
__device__ __forceinline__ int nn_search(const float q[3], bool ok, int hint, int64_t J,
                                         const float4* __restrict__ seeds, const NNGrid& g, NNWarp& sh, float s[3],
                                         int& work) {
  NNTop t{INFINITY, INFINITY, -1};
  int first = -1;
  bool go = false;
  if (ok) {
    first = nn_first<COUNT>(q, hint, J, seeds, g, t, work);
    go = t.b1 < INFINITY;
    if (!go) {
      const NNQuery q2 = nn_query(q);
      float thr = INFINITY;
      t = NNTop{INFINITY, INFINITY, -1};
      nn_walk(q, g, nn_margin(q), thr, [&](int a, int b) {
        if (COUNT) work += 4 * (b - a);
        for (int c = a; c < b; ++c) nn_scan(t, q2, g, c);
        thr = nn_thr(t.b1);
      });
    }
  }
  __syncwarp();
  nn_rest<COUNT>(q, g, go, first, t, sh, work);
  return ok ? nn_answer<COUNT>(q, g, t, s, work) : -1;
}

__host__ __device__ __forceinline__ int nn_pack_normal(float x, float y, float z) {
  return ((int)lrintf(x * 511.0f) & 1023) | (((int)lrintf(y * 511.0f) & 1023) << 10) |
         (((int)lrintf(z * 511.0f) & 1023) << 20);
}

inline NNGrid make_grid(const gp_band* b) {
  NNGrid g;
  g.pts = b->pts_sorted;
  g.occ = b->cell_occ;
  g.blk = b->cell_blk;
  g.table = b->cell_table;
  g.sup = b->cell_sup;
  g.G = b->G;
  g.nbk = (b->G + 3) / 4;
  g.nsup = (b->G + 15) / 16;
  g.half_g = 0.5f * (float)b->G;
  g.cs = 2.0f / (float)b->G;
  return g;
}
