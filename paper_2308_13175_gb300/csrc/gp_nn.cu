// Nearest surface point NN(q) (Eq. 4) and the per-point sampling sigma
// (distance to the k-th nearest other point), both by an exact search over a
// uniform cell list of the cloud.  The paper organises the points in a KD-tree
// (Sec. 3 "Discrete Grids"); a GPU walks a uniform grid far better than a
// pointer-chasing tree, and the search below is exact all the same.
//
// Exactness of gp_nn.  The answer is defined in float64:
//   D_j = ((qx-sx)^2 + (qy-sy)^2) + (qz-sz)^2 from the float32 inputs,
//   NN = argmin_j D_j, ties to the lowest j.
// The scan works in float32.  With E_j the exact squared distance, the float32
// value is within a relative 5u (u = 2^-24) of E_j (plus an absolute 1e-30
// covering underflow) and the float64 value within 3*2^-53.  Keeping the
// smallest float32 distance b1 and the second smallest b2 over all scanned
// points: if b2 > b1 (1 + 2 eps) + 1e-30 with eps = 2^-18 >> 5u, every other
// point has E_k > E_j1 (1 + eps), hence a larger float64 value, so the point of
// b1 is the float64 answer.  Otherwise (a near tie, e.g. duplicate points) the
// cells within the margin are visited again and every point within it is
// ranked by its float64 value and index.  A cell is left out only if no point
// of it can be within sqrt(b1 (1 + 8 eps)) of q: its super-block or block does
// not meet that ball, or the plane of its block keeps its points out of it
// (nn_block_cells), each taken with a rounding margin of 1e-5 (2 + |q|_inf).
#include <algorithm>
#include <cmath>

#include "gp_internal.cuh"
#include "gp_nn_device.cuh"

namespace {

__device__ __forceinline__ int nn_local_cell(float4 p, const NNGrid& g) {
  return (nn_cell(p.x, g) & 3) | ((nn_cell(p.y, g) & 3) << 2) | ((nn_cell(p.z, g) & 3) << 4);
}

__global__ void k_point_blocks(const float* __restrict__ pts, int64_t J, NNGrid g, int32_t* __restrict__ bid,
                               int32_t* __restrict__ counts) {
  int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= J) return;
  const int bx = nn_cell(pts[3 * j], g) >> 2, by = nn_cell(pts[3 * j + 1], g) >> 2, bz = nn_cell(pts[3 * j + 2], g) >> 2;
  const int32_t c = (int32_t)(((int64_t)bz * g.nbk + by) * g.nbk + bx);
  bid[j] = c;
  atomicAdd(counts + c, 1);
}

__global__ void k_point_scatter(const float* __restrict__ pts, int64_t J, const int32_t* __restrict__ bid,
                                const int32_t* __restrict__ start, int32_t* __restrict__ cursor,
                                float4* __restrict__ by_block) {
  int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= J) return;
  int32_t c = bid[j];
  int32_t pos = start[c] + atomicAdd(cursor + c, 1);
  by_block[pos] = make_float4(pts[3 * j], pts[3 * j + 1], pts[3 * j + 2], __int_as_float((int)j));
}

// A vector of least spread of the points with covariance S (00, 01, 02, 11,
// 12, 22): cyclic Jacobi rotations (Golub and Van Loan, "Matrix Computations",
// the two-sided 2 x 2 rotation that zeroes one off-diagonal entry), then the
// column of the smallest diagonal entry.  Any vector serves: it only shapes
// bounds and seeds.
__device__ __forceinline__ void least_spread(const float S[6], float n[3]) {
  float A[3][3] = {{S[0], S[1], S[2]}, {S[1], S[3], S[4]}, {S[2], S[4], S[5]}};
  float V[3][3] = {{1.f, 0.f, 0.f}, {0.f, 1.f, 0.f}, {0.f, 0.f, 1.f}};
  const float scale = fabsf(S[0]) + fabsf(S[3]) + fabsf(S[5]);
#pragma unroll 1
  for (int sweep = 0; sweep < 6; ++sweep) {
#pragma unroll
    for (int e = 0; e < 3; ++e) {
      const int p = e == 2 ? 1 : 0, q = e == 0 ? 1 : 2, r = 3 - p - q;
      const float apq = A[p][q];
      if (!(fabsf(apq) > 1e-9f * scale)) continue;
      const float tau = (A[q][q] - A[p][p]) / (2.f * apq);
      const float t = (tau >= 0.f ? 1.f : -1.f) / (fabsf(tau) + sqrtf(1.f + tau * tau));
      const float c = rsqrtf(1.f + t * t), s = t * c;
      A[p][p] -= t * apq;
      A[q][q] += t * apq;
      A[p][q] = A[q][p] = 0.f;
      const float arp = A[r][p], arq = A[r][q];
      A[r][p] = A[p][r] = c * arp - s * arq;
      A[r][q] = A[q][r] = s * arp + c * arq;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const float vp = V[k][p], vq = V[k][q];
        V[k][p] = c * vp - s * vq;
        V[k][q] = s * vp + c * vq;
      }
    }
  }
  const int m = A[0][0] <= A[1][1] ? (A[0][0] <= A[2][2] ? 0 : 2) : (A[1][1] <= A[2][2] ? 1 : 2);
#pragma unroll
  for (int k = 0; k < 3; ++k) n[k] = m == 0 ? V[k][0] : m == 1 ? V[k][1] : V[k][2];
  const float len = sqrtf(n[0] * n[0] + n[1] * n[1] + n[2] * n[2]);
  const float inv = len > 0.5f && len < 2.f ? 1.f / len : 0.f;
#pragma unroll
  for (int k = 0; k < 3; ++k) n[k] = inv > 0.f ? n[k] * inv : 0.f;
}

// A block's 64 cell counts, in shared memory, from its points [first, last)
// (unsigned: the last of J < 2^31 points plus a warp's stride).
__device__ __forceinline__ void block_histogram(const NNGrid& g, const float4* __restrict__ by_block, uint32_t first,
                                                uint32_t last, unsigned* cell) {
  const int lane = threadIdx.x & 31;
  __syncwarp();
  cell[lane] = 0;
  cell[lane + 32] = 0;
  __syncwarp();
  for (uint32_t p = first + lane; p < last; p += 32) atomicAdd(cell + nn_local_cell(by_block[p], g), 1u);
  __syncwarp();
}

constexpr int NN_BUILD_WARPS = 4;
// Blocks a warp takes at a time: with 32, a cloud's blocks with points, which
// lie side by side, met in few warps.  k_block_build over 100,000 points in 46
// blocks a side: 69 us with 32, 39 with 8; k_block_count: 16 and 11.
constexpr int NN_BUILD_RUN = 8;
enum { NN_C_BLOCKS, NN_C_OCC, NN_C_CHUNKS, NN_C_ALL };

// Each warp takes 8 consecutive blocks of the grid and works through those
// with points.  Pass 1: gives them their records' numbers and counts their
// occupied cells (one more each) and chunks.
__global__ void __launch_bounds__(32 * NN_BUILD_WARPS) k_block_count(NNGrid g, const int32_t* __restrict__ start,
                                                                     const float4* __restrict__ by_block, int64_t nblk,
                                                                     int32_t* __restrict__ table,
                                                                     int32_t* __restrict__ totals) {
  __shared__ unsigned s_cell[NN_BUILD_WARPS][64];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int64_t b0 = ((int64_t)blockIdx.x * NN_BUILD_WARPS + w) * NN_BUILD_RUN; b0 < nblk;
       b0 += (int64_t)gridDim.x * NN_BUILD_WARPS * NN_BUILD_RUN) {
    const int64_t mine = lane < NN_BUILD_RUN ? b0 + lane : nblk;
    const int f = mine < nblk ? start[mine] : 0, l = mine < nblk ? start[mine + 1] : 0;
    const unsigned some = __ballot_sync(0xffffffffu, l > f);
    int base = 0, occ = 0, chunks = 0;
    if (lane == 0 && some) base = atomicAdd(totals + NN_C_BLOCKS, __popc(some));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (mine < nblk) table[mine] = l > f ? base + __popc(some & ((1u << lane) - 1u)) : -1;
    for (unsigned left = some; left; left &= left - 1u) {
      const int k = __ffs(left) - 1;
      block_histogram(g, by_block, __shfl_sync(0xffffffffu, f, k), __shfl_sync(0xffffffffu, l, k), s_cell[w]);
      const unsigned n0 = s_cell[w][lane], n1 = s_cell[w][lane + 32];
      occ += (n0 > 0) + (n1 > 0) + (lane == 0);
      chunks += (int)((n0 + 3u) >> 2) + (int)((n1 + 3u) >> 2);
    }
    occ = gp_warp_sum_i(occ);
    chunks = gp_warp_sum_i(chunks);
    if (lane == 0 && some) {
      atomicAdd(totals + NN_C_OCC, occ);
      atomicAdd(totals + NN_C_CHUNKS, chunks);
    }
  }
}

// Pass 2: the chunks of the cells, the first chunk of each occupied cell, the
// occupancy, and the plane the points lie along.  Blocks with a point outside
// the grid's cube (kept in the boundary cells) get no plane, so that every
// coordinate of a bounded block is at most 1.01.
__global__ void __launch_bounds__(32 * NN_BUILD_WARPS) k_block_build(
    NNGrid g, const int32_t* __restrict__ start, const float4* __restrict__ by_block, int64_t nblk,
    const int32_t* __restrict__ table, int32_t* __restrict__ totals, float* __restrict__ pts, int32_t* __restrict__ occ,
    float4* __restrict__ blk, unsigned long long* __restrict__ sup) {
  __shared__ unsigned s_cell[NN_BUILD_WARPS][64];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  unsigned* cell = s_cell[w];
  for (int64_t b0 = ((int64_t)blockIdx.x * NN_BUILD_WARPS + w) * NN_BUILD_RUN; b0 < nblk;
       b0 += (int64_t)gridDim.x * NN_BUILD_WARPS * NN_BUILD_RUN) {
    const int64_t mine = lane < NN_BUILD_RUN ? b0 + lane : nblk;
    const int fl = mine < nblk ? start[mine] : 0, ll = mine < nblk ? start[mine + 1] : 0;
    for (unsigned left = __ballot_sync(0xffffffffu, ll > fl); left; left &= left - 1u) {
      const int kb = __ffs(left) - 1;
      const uint32_t first = __shfl_sync(0xffffffffu, fl, kb), last = __shfl_sync(0xffffffffu, ll, kb);
      const int64_t b = b0 + kb;
      const int bi = table[b];
      const int bx = (int)(b % g.nbk), by = (int)((b / g.nbk) % g.nbk), bz = (int)(b / ((int64_t)g.nbk * g.nbk));
      const float c0 = -1.0f + (4 * bx + 2) * g.cs, c1 = -1.0f + (4 * by + 2) * g.cs, c2 = -1.0f + (4 * bz + 2) * g.cs;
      block_histogram(g, by_block, first, last, cell);
      // Exclusive scans of the cells' chunks and occupancy, two consecutive
      // cells per lane, and the block's share of the arrays.
      const unsigned n0 = cell[2 * lane], n1 = cell[2 * lane + 1];
      const int h0 = (int)((n0 + 3u) >> 2), h1 = (int)((n1 + 3u) >> 2);
      int incl = h0 + h1;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      const unsigned e = __ballot_sync(0xffffffffu, n0 > 0), d = __ballot_sync(0xffffffffu, n1 > 0);
      const int nocc = __popc(e) + __popc(d);
      int base = 0, o0 = 0;
      if (lane == 31) base = atomicAdd(totals + NN_C_CHUNKS, incl);
      if (lane == 31) o0 = atomicAdd(totals + NN_C_OCC, nocc + 1);
      base = __shfl_sync(0xffffffffu, base, 31);
      o0 = __shfl_sync(0xffffffffu, o0, 31);
      const int at0 = base + incl - h0 - h1, at1 = at0 + h0;
      const unsigned below = (1u << lane) - 1u;
      const int k0 = __popc(e & below) + __popc(d & below);
      if (n0) occ[o0 + k0] = at0;
      if (n1) occ[o0 + k0 + (n0 > 0)] = at1;
      if (lane == 31) occ[o0 + nocc] = base + incl;
      __syncwarp();
      cell[2 * lane] = 4u * (unsigned)(at0 - base);  // the cell's next place (nn_place)
      cell[2 * lane + 1] = 4u * (unsigned)(at1 - base);
      __syncwarp();
      float m[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
      bool inside = true;
      for (uint32_t p = first + lane; p < last; p += 32) {
        const float4 P = by_block[p];
        const unsigned at = atomicAdd(cell + nn_local_cell(P, g), 1u);
        const float v[4] = {P.x, P.y, P.z, P.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) pts[nn_place(base, at, k)] = v[k];
        inside = inside && fabsf(P.x) <= 1.01f && fabsf(P.y) <= 1.01f && fabsf(P.z) <= 1.01f;
        const float x = P.x - c0, y = P.y - c1, z = P.z - c2;
        m[0] += x;
        m[1] += y;
        m[2] += z;
        m[3] += x * x;
        m[4] += x * y;
        m[5] += x * z;
        m[6] += y * y;
        m[7] += y * z;
        m[8] += z * z;
      }
      __syncwarp();
      // The places left in each cell's last chunk.
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const unsigned end = 4u * (unsigned)((k ? at1 + h1 : at0 + h0) - base);
        for (unsigned at = cell[2 * lane + k]; at < end; ++at) {
#pragma unroll
          for (int j = 0; j < 4; ++j) pts[nn_place(base, at, j)] = j < 3 ? INFINITY : __int_as_float(-1);
        }
      }
      inside = __all_sync(0xffffffffu, inside);
      float n[3] = {0.f, 0.f, 0.f};
      if (inside) {
        const float inv = 1.0f / (float)(last - first);
#pragma unroll
        for (int k = 0; k < 9; ++k) m[k] = gp_warp_sum(m[k]) * inv;
        const float S[6] = {m[3] - m[0] * m[0], m[4] - m[0] * m[1], m[5] - m[0] * m[2],
                            m[6] - m[1] * m[1], m[7] - m[1] * m[2], m[8] - m[2] * m[2]};
        least_spread(S, n);
      }
      float lo = INFINITY, hi = -INFINITY;
      for (uint32_t p = first + lane; p < last; p += 32) {
        const float4 P = by_block[p];
        const float v = n[0] * P.x + n[1] * P.y + n[2] * P.z;
        lo = fminf(lo, v);
        hi = fmaxf(hi, v);
      }
#pragma unroll
      for (int k = 16; k > 0; k >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, k));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, k));
      }
      if (lane == 0) {
        if (!inside) lo = hi = 0.f;
        unsigned long long mask = 0ull;
        for (int k = 0; k < 32; ++k)
          mask |= ((unsigned long long)((e >> k) & 1u) | ((unsigned long long)((d >> k) & 1u) << 1)) << (2 * k);
        blk[2 * (int64_t)bi] = make_float4(n[0], n[1], n[2], lo);
        blk[2 * (int64_t)bi + 1] = make_float4(hi, __int_as_float(o0), __uint_as_float((uint32_t)mask),
                                               __uint_as_float((uint32_t)(mask >> 32)));
        atomicOr(sup + ((int64_t)(bz >> 2) * g.nsup + (by >> 2)) * g.nsup + (bx >> 2),
                 1ull << ((bx & 3) | ((by & 3) << 2) | ((bz & 3) << 4)));
      }
    }
  }
}

// Chunk c's points relative to q, four at a time: 16-byte loads, four of them
// (the fourth for the indices), instead of 4 bytes for each part of each point.
struct NNFour {
  float dx[4], dy[4], dz[4];
  int idx[4];
};
__device__ __forceinline__ NNFour nn_four(const float4* __restrict__ pts, int64_t c, const float q[3]) {
  const float4 x = __ldg(pts + nn_part(c, 0)), y = __ldg(pts + nn_part(c, 1)), z = __ldg(pts + nn_part(c, 2)),
               i = __ldg(pts + nn_part(c, 3));
  return {{x.x - q[0], x.y - q[0], x.z - q[0], x.w - q[0]},
          {y.x - q[1], y.y - q[1], y.z - q[1], y.w - q[1]},
          {z.x - q[2], z.y - q[2], z.z - q[2], z.w - q[2]},
          {__float_as_int(i.x), __float_as_int(i.y), __float_as_int(i.z), __float_as_int(i.w)}};
}

// sigma_j: distance to the k-th nearest other point, by a bounded max-heap.
// Bound by its dependent local-memory reads and their divergence; a chunk's
// candidates are told from the rest by one test each, so that only lanes with
// one enter the heap.  100,000 points, k = 50: 478 -> 394 us with this and the
// 16-byte loads (k_normals 221 -> 139).  A warp a point, distances gathered in
// shared memory and the k-th selected by bisection with ballots, both kernels in
// one: 1,168 us.
__global__ void __launch_bounds__(128) k_knn_sigma(NNGrid g, int64_t chunks, int k, float* __restrict__ sigma) {
  int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 4 * chunks) return;
  const int self = __float_as_int(nn_value(g.pts, t, 3));
  if (self < 0) return;
  float heap[64];
  int cnt = 0;
  if (k <= 0) {
    sigma[self] = 0.f;
    return;
  }
  float q[3] = {nn_value(g.pts, t, 0), nn_value(g.pts, t, 1), nn_value(g.pts, t, 2)};
  int c[3] = {nn_cell(q[0], g), nn_cell(q[1], g), nn_cell(q[2], g)};
  float margin = nn_margin(q);
  float top = 0.f;  // heap[0]
  for (int r = 0; r <= g.G; ++r) {
    nn_ring(c, r, g, [&](int a, int b) {
      for (int64_t ch = a; ch < b; ++ch) {
        const NNFour f = nn_four(g.pts, ch, q);
        float ds[4];
        unsigned in = 0;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          ds[u] = f.dx[u] * f.dx[u] + f.dy[u] * f.dy[u] + f.dz[u] * f.dz[u];
          if (f.idx[u] >= 0 && 4 * ch + u != t && (cnt < k || ds[u] < top)) in |= 1u << u;
        }
        for (; in; in &= in - 1u) {
          const int u = __ffs(in) - 1;
          const float d = u == 0 ? ds[0] : u == 1 ? ds[1] : u == 2 ? ds[2] : ds[3];
          int i = 0;
          if (cnt < k) {
            // sift up
            i = cnt++;
            while (i > 0) {
              int par = (i - 1) >> 1;
              if (heap[par] >= d) break;
              heap[i] = heap[par];
              i = par;
            }
          } else if (d < top) {
            // replace root, sift down
            while (true) {
              int l = 2 * i + 1;
              if (l >= k) break;
              int m = (l + 1 < k && heap[l + 1] > heap[l]) ? l + 1 : l;
              if (heap[m] <= d) break;
              heap[i] = heap[m];
              i = m;
            }
          } else {
            continue;
          }
          heap[i] = d;
          top = heap[0];
        }
      }
    });
    if (cnt == k) {
      float gap = nn_gap(q, c, r, g);
      if (gap == INFINITY) break;
      float gs = gap - margin;
      if (gs > 0.f && gs * gs > top * (1.0f + 8.0f * NN_EPS) + NN_TINY) break;
    } else if (nn_gap(q, c, r, g) == INFINITY) {
      break;
    }
  }
  sigma[self] = cnt > 0 ? sqrtf(top) : 0.f;
}

// Normal of each point: direction of least spread of the points within
// sigma_j (its k-nearest-neighbour ball), by PCA.  Used only to seed gp_nn:
// written with the point, packed, as its record of `seeds`.
__global__ void __launch_bounds__(128) k_normals(NNGrid g, int64_t chunks, const float* __restrict__ sigma,
                                                 float4* __restrict__ seeds) {
  int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 4 * chunks) return;
  const int self = __float_as_int(nn_value(g.pts, t, 3));
  if (self < 0) return;
  const float q[3] = {nn_value(g.pts, t, 0), nn_value(g.pts, t, 1), nn_value(g.pts, t, 2)};
  const int c[3] = {nn_cell(q[0], g), nn_cell(q[1], g), nn_cell(q[2], g)};
  const float rad = sigma[self];
  const float r2 = rad * rad * 1.000001f;
  const float margin = nn_margin(q);
  float m[3] = {0, 0, 0}, S[6] = {0, 0, 0, 0, 0, 0};
  int cnt = 0;
  for (int r = 0; r <= g.G; ++r) {
    nn_ring(c, r, g, [&](int a, int b) {
      for (int64_t ch = a; ch < b; ++ch) {
        const NNFour f = nn_four(g.pts, ch, q);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float dx = f.dx[u], dy = f.dy[u], dz = f.dz[u];
          if (dx * dx + dy * dy + dz * dz > r2) continue;
          m[0] += dx;
          m[1] += dy;
          m[2] += dz;
          S[0] += dx * dx;
          S[1] += dx * dy;
          S[2] += dx * dz;
          S[3] += dy * dy;
          S[4] += dy * dz;
          S[5] += dz * dz;
          ++cnt;
        }
      }
    });
    float gap = nn_gap(q, c, r, g);
    if (gap == INFINITY || gap - margin > rad) break;
  }
  float n[3] = {0.f, 0.f, 0.f};
  if (cnt >= 3) {
    const float inv = 1.0f / (float)cnt;
    for (int a = 0; a < 3; ++a) m[a] *= inv;
    const float C[6] = {S[0] * inv - m[0] * m[0], S[1] * inv - m[0] * m[1], S[2] * inv - m[0] * m[2],
                        S[3] * inv - m[1] * m[1], S[4] * inv - m[1] * m[2], S[5] * inv - m[2] * m[2]};
    least_spread(C, n);
  }
  seeds[self] = make_float4(q[0], q[1], q[2], __int_as_float(nn_pack_normal(n[0], n[1], n[2])));
}

// Records of a cloud without normals: the points themselves.
__global__ void k_seed_points(const float* __restrict__ pts, int64_t J, float4* __restrict__ seeds) {
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j < J) seeds[j] = make_float4(pts[3 * j], pts[3 * j + 1], pts[3 * j + 2], 0.f);
}

// Four warps a block, 8 blocks an SM at 64 registers; 64 or 256 threads, and
// 10 blocks an SM at fewer registers, were within 2% on every batch measured.
constexpr int NN_THREADS = 128;

// One lane per query (nn_search works on a warp's 32 together).  Queries with a
// NaN, infinite or huge coordinate (whose squared distances would overflow
// float32) get -1 and a NaN surface point.  COUNT: also add the number of point
// distances evaluated (seeds, cells and tie-break) to *work_total, for
// measurement; the search is the same.
template <bool COUNT>
__global__ void __launch_bounds__(NN_THREADS, 8) k_nn(NNGrid g, const float* __restrict__ qin, int64_t n,
                                                      const int32_t* __restrict__ hint, int64_t J,
                                                      const float4* __restrict__ seeds, int32_t* __restrict__ nn_out,
                                                      float* __restrict__ rec, Grid band, int32_t* __restrict__ nvalid,
                                                      unsigned long long* __restrict__ work_total) {
  __shared__ NNWarp s_warp[NN_THREADS / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t first = (int64_t)blockIdx.x * NN_THREADS + 32 * warp;
  const int64_t i = first + lane;
  const float nan = __int_as_float(0x7fc00000);
  float q[3] = {nan, nan, nan}, s[3] = {nan, nan, nan};
  int h = -1;
  if (i < n) {
    q[0] = qin[3 * i];
    q[1] = qin[3 * i + 1];
    q[2] = qin[3 * i + 2];
    if (hint) h = __ldg(hint + i);
  }
  int work = 0;
  const int best = nn_search<COUNT>(q, nn_query_ok(q), h, J, seeds, g, s_warp[warp], s, work);
  if (nn_out && i < n) nn_out[i] = best;
  if (nvalid) {
    Cells C;
    const unsigned v = __ballot_sync(0xffffffffu, best >= 0 && classify(band, q, s, C));
    if (lane == 0 && v) atomicAdd(nvalid, __popc(v));
  }
  if (rec) {
    // Through shared memory, so that the warp's records are written in lines.
    float* out = reinterpret_cast<float*>(&s_warp[warp]);
    static_assert(sizeof(NNWarp) >= 32 * 6 * sizeof(float), "record staging");
    __syncwarp();
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      out[6 * lane + a] = q[a];
      out[6 * lane + 3 + a] = s[a];
    }
    __syncwarp();
    const int64_t left = 6 * (n - first);
#pragma unroll
    for (int k = lane; k < 32 * 6; k += 32)
      if (k < left) rec[6 * first + k] = out[k];
  }
  if (COUNT) {
    unsigned long long w = (unsigned long long)work;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
    if (lane == 0 && w) atomicAdd(work_total, w);
  }
}

// Emission order of the spatial batches: point indices sorted by the Morton
// code of their cell-list cell (ties by index), so that consecutive points, and
// the queries drawn around them, stay close in all three directions.  A radix
// sort of (code, index), 8 bits a pass from the lowest, each pass stable: the
// digits of a tile are counted, the counts scanned over digits and tiles, and
// the tile's pairs written in order.  (On the host, with a comparison sort of
// 64-bit keys, the order took 4 of the 8 ms that a band of 100,000 points took
// to build.)
constexpr int RS_THREADS = 256, RS_WARPS = RS_THREADS / 32;
constexpr int RS_ROUNDS = 16;                     // 32 pairs a warp and round
constexpr int RS_TILE = RS_THREADS * RS_ROUNDS;

__device__ __forceinline__ uint32_t nn_spread3(uint32_t x) {  // bit k to bit 3 k (10 bits)
  x = (x | x << 16) & 0x030000FFu;
  x = (x | x << 8) & 0x0300F00Fu;
  x = (x | x << 4) & 0x030C30C3u;
  return (x | x << 2) & 0x09249249u;
}

__global__ void k_emit_keys(const float* __restrict__ pts, int64_t J, NNGrid g, uint32_t* __restrict__ key,
                            int32_t* __restrict__ order) {
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= J) return;
  key[j] = nn_spread3(nn_cell(pts[3 * j], g)) | nn_spread3(nn_cell(pts[3 * j + 1], g)) << 1 |
           nn_spread3(nn_cell(pts[3 * j + 2], g)) << 2;
  order[j] = (int32_t)j;
}

__global__ void __launch_bounds__(RS_THREADS) k_radix_count(const uint32_t* __restrict__ key, int64_t n, int shift,
                                                            int64_t ntiles, int32_t* __restrict__ counts) {
  __shared__ int hist[256];
  hist[threadIdx.x] = 0;
  __syncthreads();
  const int64_t base = (int64_t)blockIdx.x * RS_TILE;
  for (int k = 0; k < RS_ROUNDS; ++k) {
    const int64_t i = base + k * RS_THREADS + threadIdx.x;
    if (i < n) atomicAdd(hist + ((key[i] >> shift) & 255u), 1);
  }
  __syncthreads();
  counts[(int64_t)threadIdx.x * ntiles + blockIdx.x] = hist[threadIdx.x];
}

__global__ void __launch_bounds__(GP_ORDER_THREADS) k_radix_scan(int32_t* __restrict__ counts, int64_t n) {
  gp_block_scan_inplace(counts, n);
}

__global__ void __launch_bounds__(RS_THREADS) k_radix_scatter(const uint32_t* __restrict__ key,
                                                              const int32_t* __restrict__ val, int64_t n, int shift,
                                                              int64_t ntiles, const int32_t* __restrict__ offs,
                                                              uint32_t* __restrict__ key_out,
                                                              int32_t* __restrict__ val_out) {
  __shared__ int at[RS_WARPS][256];  // pairs of each digit per warp, then the next place of each
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int k = lane; k < 256; k += 32) at[w][k] = 0;
  __syncwarp();
  const int64_t base = (int64_t)blockIdx.x * RS_TILE + (int64_t)w * (32 * RS_ROUNDS) + lane;
  for (int r = 0; r < RS_ROUNDS; ++r) {
    const int64_t i = base + 32 * r;
    if (i < n) atomicAdd(&at[w][(key[i] >> shift) & 255u], 1);
  }
  __syncthreads();
  {
    int run = offs[(int64_t)threadIdx.x * ntiles + blockIdx.x];
    for (int k = 0; k < RS_WARPS; ++k) {
      const int c = at[k][threadIdx.x];
      at[k][threadIdx.x] = run;
      run += c;
    }
  }
  __syncthreads();
  for (int r = 0; r < RS_ROUNDS; ++r) {
    const int64_t i = base + 32 * r;
    const bool mine = i < n;
    const uint32_t k = mine ? key[i] : 0u;
    const int d = mine ? (int)((k >> shift) & 255u) : 256;  // lanes past the end share a digit of their own
    const unsigned peers = __match_any_sync(0xffffffffu, d);
    const int before = __popc(peers & ((1u << lane) - 1u));
    const int pos = mine ? at[w][d] + before : 0;
    __syncwarp();
    if (mine) {
      if (before == 0) at[w][d] = pos + __popc(peers);
      key_out[pos] = k;
      val_out[pos] = val[i];
    }
    __syncwarp();
  }
}

// Points and sigma in emission order, for the sampler's coalesced reads.
__global__ void k_emit_pts(const int32_t* __restrict__ order, const float* __restrict__ pts,
                           const float* __restrict__ sigma, int64_t J, float4* __restrict__ out) {
  const int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (u >= J) return;
  const int64_t j = order[u];
  out[u] = make_float4(pts[3 * j], pts[3 * j + 1], pts[3 * j + 2], sigma[j]);
}

}  // namespace

static gp_status build_emit_order(gp_band* b) {
  gp_ctx* ctx = b->ctx;
  cudaStream_t s = ctx->stream;
  const int64_t J = b->J, ntiles = (J + RS_TILE - 1) / RS_TILE;
  int bits = 0;  // per axis
  while ((1 << bits) < b->G) ++bits;
  uint32_t* key[2] = {nullptr, nullptr};
  int32_t *val[2] = {nullptr, nullptr}, *counts = nullptr;
  gp_status st = gp_alloc(ctx, &val[0], J, "emission order");
  if (!st) st = gp_alloc(ctx, &val[1], J, "emission order");
  if (!st) st = gp_alloc(ctx, &key[0], J, "emission keys");
  if (!st) st = gp_alloc(ctx, &key[1], J, "emission keys");
  if (!st) st = gp_alloc(ctx, &counts, 256 * ntiles, "emission digit counts");
  cudaError_t e = cudaSuccess;
  int cur = 0;
  if (!st) {
    k_emit_keys<<<gp_blocks(J, 256), 256, 0, s>>>(b->pts, J, make_grid(b), key[0], val[0]);
    for (int shift = 0; shift < 3 * bits; shift += 8, cur ^= 1) {
      k_radix_count<<<(unsigned)ntiles, RS_THREADS, 0, s>>>(key[cur], J, shift, ntiles, counts);
      k_radix_scan<<<1, GP_ORDER_THREADS, 0, s>>>(counts, 256 * ntiles);
      k_radix_scatter<<<(unsigned)ntiles, RS_THREADS, 0, s>>>(key[cur], val[cur], J, shift, ntiles, counts,
                                                             key[cur ^ 1], val[cur ^ 1]);
    }
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  }
  gp_free(ctx, key[0]);
  gp_free(ctx, key[1]);
  gp_free(ctx, counts);
  gp_free(ctx, val[cur ^ 1]);
  if (st || e != cudaSuccess) {
    gp_free(ctx, val[cur]);
    return st ? st : gp_cuda_fail(ctx, e, "emission order");
  }
  b->emit_order = val[cur];
  return GP_OK;
}

constexpr double NN_POINTS_PER_CELL = 6.5;

// Point copy, cell list and sigma (called by gp_build_band).
gp_status gp_build_points(gp_band* b, const float* pts_dev) {
  gp_ctx* ctx = b->ctx;
  cudaStream_t s = ctx->stream;
  const int64_t J = b->J;
  if (b->G <= 0) {
    // About 6.5 points per occupied cell of the search grid (5 to 10 are within
    // 5% of one another on the benchmark clouds, 3 and 14 up to 25% slower).
    // The cloud is a surface, so the cells it occupies at grid G are
    // about n_occ (G / R)^2, n_occ being its occupied cells at the band's R.
    // That estimate fails for a cloud too sparse to cover its surface at R
    // (n_occ near J); there sqrt(J / 3) cells per axis, the bound that served
    // such clouds before, is the smaller one and is taken.
    const double occ = (double)std::max<int64_t>(b->n_occ, 1);
    const double g_area = (double)b->R * std::sqrt((double)J / (NN_POINTS_PER_CELL * occ));
    const double g_count = std::sqrt((double)J / 3.0);
    const int G = (int)std::min(g_area, g_count);
    b->G = std::min(std::max(G, 4), 512);
  }
  const int G = b->G;
  const int nbk = (G + 3) / 4, nsup = (G + 15) / 16;
  const int64_t nblk = (int64_t)nbk * nbk * nbk, nsb = (int64_t)nsup * nsup * nsup;
  gp_status st;
  if ((st = gp_alloc(ctx, &b->pts, 3 * J, "points"))) return st;
  GP_CUDA(ctx, cudaMemcpyAsync(b->pts, pts_dev, 3 * J * sizeof(float), cudaMemcpyDeviceToDevice, s));
  if ((st = gp_alloc(ctx, &b->cell_table, nblk, "cell blocks"))) return st;
  if ((st = gp_alloc(ctx, &b->cell_sup, nsb, "cell super-blocks"))) return st;
  if ((st = gp_alloc(ctx, &b->seeds, J, "search seeds"))) return st;
  int32_t *bid = nullptr, *start = nullptr, *cursor = nullptr;  // the block totals follow the cursors
  float4* by_block = nullptr;
  st = gp_alloc(ctx, &bid, J, "point blocks");
  if (!st) st = gp_alloc(ctx, &start, nblk + 1, "block starts");
  if (!st) st = gp_alloc(ctx, &cursor, nblk + NN_C_ALL, "block cursors");
  if (!st) st = gp_alloc(ctx, &by_block, J, "points by block");
  cudaError_t e = cudaSuccess;
  NNGrid g = make_grid(b);
  if (!st) {
    e = cudaMemsetAsync(start, 0, (nblk + 1) * sizeof(int32_t), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(cursor, 0, (nblk + NN_C_ALL) * sizeof(int32_t), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(b->cell_sup, 0, nsb * sizeof(unsigned long long), s);
    if (e == cudaSuccess) {
      k_point_blocks<<<gp_blocks(J, 256), 256, 0, s>>>(b->pts, J, g, bid, start);
      e = cudaGetLastError();
    }
  }
  int64_t total = 0;
  int32_t totals[NN_C_ALL] = {0, 0, 0};
  if (!st && e == cudaSuccess) st = gp_exclusive_scan_i32(ctx, start, nblk + 1, &total);
  const unsigned grid = gp_blocks(nblk, NN_BUILD_RUN * NN_BUILD_WARPS, 16 * (int64_t)ctx->num_sms);
  int32_t* tot_dev = cursor ? cursor + nblk : nullptr;
  if (!st && e == cudaSuccess) {
    k_point_scatter<<<gp_blocks(J, 256), 256, 0, s>>>(b->pts, J, bid, start, cursor, by_block);
    k_block_count<<<grid, 32 * NN_BUILD_WARPS, 0, s>>>(g, start, by_block, nblk, b->cell_table, tot_dev);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(totals, tot_dev, sizeof(totals), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(tot_dev, 0, sizeof(totals), s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  }
  b->n_chunks = totals[NN_C_CHUNKS];
  if (!st && e == cudaSuccess) st = gp_alloc(ctx, &b->cell_blk, 2 * (size_t)totals[NN_C_BLOCKS], "cell block records");
  if (!st && e == cudaSuccess) st = gp_alloc(ctx, &b->cell_occ, totals[NN_C_OCC], "occupied cells");
  if (!st && e == cudaSuccess) st = gp_alloc(ctx, &b->pts_sorted, 4 * (size_t)b->n_chunks, "sorted points");
  if (!st && e == cudaSuccess) {
    k_block_build<<<grid, 32 * NN_BUILD_WARPS, 0, s>>>(g, start, by_block, nblk, b->cell_table, tot_dev,
                                                       reinterpret_cast<float*>(b->pts_sorted), b->cell_occ,
                                                       b->cell_blk, b->cell_sup);
    e = cudaGetLastError();
  }
  cudaStreamSynchronize(s);
  gp_free(ctx, bid);
  gp_free(ctx, start);
  gp_free(ctx, cursor);
  gp_free(ctx, by_block);
  if (st) return st;
  if (e != cudaSuccess) return gp_cuda_fail(ctx, e, "point cell list");
  g = make_grid(b);
  if (b->knn_k == 0)
    GP_KERNEL(ctx, "k_seed_points", k_seed_points<<<gp_blocks(J, 256), 256, 0, s>>>(b->pts, J, b->seeds));
  if (b->knn_k > 0) {
    if ((st = gp_alloc(ctx, &b->sigma, J, "sigma"))) return st;
    if ((st = gp_alloc(ctx, &b->perm, J, "permutation"))) return st;
    if ((st = gp_alloc(ctx, &b->inv_perm, J, "inverse permutation"))) return st;
    if ((st = gp_alloc(ctx, &b->order_tiles, (J + GP_ORDER_TILE - 1) / GP_ORDER_TILE + 1, "order tiles"))) return st;
    if ((st = build_emit_order(b))) return st;
    if ((st = gp_alloc(ctx, &b->emit_slot, J, "emission slots"))) return st;
    int k = (int)std::min<int64_t>(b->knn_k, J - 1);
    GP_KERNEL(ctx, "k_knn_sigma", k_knn_sigma<<<gp_blocks(4 * b->n_chunks, 128), 128, 0, s>>>(g, b->n_chunks, k, b->sigma));
    GP_KERNEL(ctx, "k_normals", k_normals<<<gp_blocks(4 * b->n_chunks, 128), 128, 0, s>>>(g, b->n_chunks, b->sigma, b->seeds));
    if ((st = gp_alloc(ctx, &b->emit_pts, J, "emission points"))) return st;
    GP_KERNEL(ctx, "k_emit_pts", k_emit_pts<<<gp_blocks(J, 256), 256, 0, s>>>(b->emit_order, b->pts, b->sigma, J,
                                                                            b->emit_pts));
  }
  return GP_OK;
}

extern "C" gp_status gp_band_sigma(const gp_band* b, float* sigma_dev) {
  if (!b) return GP_ERR_ARG;
  if (!sigma_dev) return gp_fail(b->ctx, GP_ERR_ARG, "gp_band_sigma: null output");
  if (!b->sigma) return gp_fail(b->ctx, GP_ERR_STATE, "gp_band_sigma: band built with knn_k = 0");
  GP_CUDA(b->ctx, cudaMemcpyAsync(sigma_dev, b->sigma, b->J * sizeof(float), cudaMemcpyDeviceToDevice,
                                  b->ctx->stream));
  return GP_OK;
}

// The launch of gp_nn; work_total (device, NULL = not counted) receives the
// number of point distances evaluated.
static gp_status nn_launch(gp_band* b, const float* q_dev, int64_t n, const int32_t* hint_dev, int32_t* nn_dev,
                           float* rec_dev, int32_t* nvalid_dev, unsigned long long* work_total) {
  gp_ctx* ctx = b->ctx;
  NNGrid g = make_grid(b);
  Grid band;
  band.table = b->brick_table;
  band.masks = b->masks;
  band.D = b->D;
  band.nb = b->nb;
  band.R = b->R;
  band.half_r = 0.5f * (float)b->R;
#define GP_NN(C_) \
  k_nn<C_><<<gp_blocks(n, NN_THREADS), NN_THREADS, 0, ctx->stream>>>(g, q_dev, n, hint_dev, b->J, b->seeds, nn_dev, \
                                                                     rec_dev, band, nvalid_dev, work_total)
  // Large seeded batches are traced under a name of their own.
  if (work_total)
    GP_KERNEL(ctx, "k_nn_count", GP_NN(true));
  else if (hint_dev && n >= (int64_t(1) << 20))
    GP_KERNEL(ctx, "k_nn_sorted", GP_NN(false));
  else
    GP_KERNEL(ctx, "k_nn", GP_NN(false));
#undef GP_NN
  return GP_OK;
}

extern "C" gp_status gp_nn(gp_band* b, const float* q_dev, int64_t n, const int32_t* hint_dev, int32_t* nn_dev,
                           float* rec_dev, int32_t* nvalid_dev) {
  if (!b) return GP_ERR_ARG;
  gp_ctx* ctx = b->ctx;
  if (n < 0 || n >= (int64_t(1) << 31)) return gp_fail(ctx, GP_ERR_ARG, "gp_nn: n must be in [0, 2^31)");
  if (nvalid_dev) GP_CUDA(ctx, cudaMemsetAsync(nvalid_dev, 0, sizeof(int32_t), ctx->stream));
  if (n == 0) return GP_OK;
  if (!q_dev || (!nn_dev && !rec_dev)) return gp_fail(ctx, GP_ERR_ARG, "gp_nn: null pointer");
  return nn_launch(b, q_dev, n, hint_dev, nn_dev, rec_dev, nvalid_dev, nullptr);
}

extern "C" gp_status gp_nn_work(gp_band* b, const float* q_dev, int64_t n, const int32_t* hint_dev,
                                int32_t* nn_dev, int64_t* work_host) {
  if (!b) return GP_ERR_ARG;
  gp_ctx* ctx = b->ctx;
  if (n < 0 || n >= (int64_t(1) << 31)) return gp_fail(ctx, GP_ERR_ARG, "gp_nn_work: n must be in [0, 2^31)");
  if (!work_host || !nn_dev || (n > 0 && !q_dev)) return gp_fail(ctx, GP_ERR_ARG, "gp_nn_work: null pointer");
  *work_host = 0;
  if (n == 0) return GP_OK;
  unsigned long long* dev = nullptr;
  gp_status st = gp_alloc(ctx, &dev, 1, "gp_nn_work counter");
  if (st) return st;
  cudaError_t e = cudaMemsetAsync(dev, 0, sizeof(unsigned long long), ctx->stream);
  if (e == cudaSuccess) {
    st = nn_launch(b, q_dev, n, hint_dev, nn_dev, nullptr, nullptr, dev);
    unsigned long long h = 0;
    if (!st) e = cudaMemcpyAsync(&h, dev, sizeof(h), cudaMemcpyDeviceToHost, ctx->stream);
    if (!st && e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
    *work_host = (int64_t)h;
  }
  gp_free(ctx, dev);
  if (st) return st;
  if (e != cudaSuccess) return gp_cuda_fail(ctx, e, "gp_nn_work");
  return GP_OK;
}
