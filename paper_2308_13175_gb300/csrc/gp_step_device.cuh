// Device functions of the step shared by the single-band kernels (gp_step.cu)
// and the many-band kernels (gp_multi.cu): Eq. 3 interpolation, the per-record
// forward + hand-written backward, one brick of the L_TV sweep, one Adam update.
// The formulas are stated in the header comment of gp_step.cu.
#pragma once

#include <string.h>

#include "gp_internal.cuh"

constexpr float NORM_FLOOR = 1e-12f;
// Deterministic sums: each contribution v is split into two integers, hi in
// units of 2^-20 and lo in units of 2^-60 (fix_split), accumulated with 64-bit
// integer atomics (exact, so the order of the additions does not matter).
// The sum is hi * 2^-20 + lo * 2^-60: a resolution of 2^-60; a contribution
// of magnitude 2^42 (FIX_LIMIT) or more, or a non-finite one, raises
// GP_EF_NUMERIC instead.
constexpr double FIX_HI = 1048576.0;                     // 2^20
constexpr double FIX_LO = 1152921504606846976.0;         // 2^60
constexpr double FIX_LIMIT = 4398046511104.0;            // 2^42

struct Eval {
  float f;
  float gt[3];  // df/dt (t = local coordinate in cell units)
};

// The slots of the bricks that hold the corners of cell c (corner
// k = dx + 2 dy + 4 dz), slot being the cell's own.  Only corners in a
// neighbouring brick are looked up; -1 where that brick is not stored.  One
// path serves all cells, here and in the loads and sums below: with a path each
// for cells inside a brick (by x mod 4) and across bricks, the lanes of a warp
// took them all in turn (k_query_ilp: 206 -> 164 us for 2,097,152 records of a
// 1024^3 band, 49 -> 40 us for 262,144 in no order on a 256^3 one, 521 -> 468 us
// for 4,194,304 with the fixed-point sums; k_m_query 334 -> 226 us).
__device__ __forceinline__ void cell_slots(const Grid& G, const int c[3], int slot, int s[8]) {
  const int ox = (c[0] & 7) == 7 ? 1 : 0, oy = (c[1] & 7) == 7 ? G.nb : 0, oz = (c[2] & 7) == 7 ? G.nb * G.nb : 0;
  const int32_t* T = G.table + ((int64_t)(c[2] >> 3) * G.nb + (c[1] >> 3)) * G.nb + (c[0] >> 3);
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int off = ((k & 1) ? ox : 0) + ((k & 2) ? oy : 0) + ((k & 4) ? oz : 0);
    s[k] = slot;
    if (off) s[k] = __ldg(T + off);
  }
}

// Place of corner k of cell c in its brick.
__device__ __forceinline__ int corner_local(const int c[3], int k) {
  return gp_local(c[0] + (k & 1), c[1] + ((k >> 1) & 1), c[2] + (k >> 2));
}

// The 8 corner values, along x in pairs: one 8-byte load at even x (both lie
// in one brick), two single ones at odd x (an aligned 16-byte load for all of
// them holds twice the registers: 178 -> 234 us on the first of those batches).
// A missing brick turns ok false.
__device__ __forceinline__ void load_corners_at(const Grid& G, const int c[3], const int s[8], float d[8], bool& ok) {
  const bool even = (c[0] & 1) == 0;
#pragma unroll
  for (int e = 0; e < 8; e += 2) {
    const bool have = s[e] >= 0 && s[e + 1] >= 0;
    if (!have) ok = false;
    const float* lo = G.D + ((int64_t)(have ? s[e] : s[0]) * 512 + corner_local(c, e));
    const float* hi = G.D + ((int64_t)(have ? s[e + 1] : s[0]) * 512 + corner_local(c, e + 1));
    if (even) {
      const float2 v = __ldg(reinterpret_cast<const float2*>(lo));
      d[e] = v.x;
      d[e + 1] = v.y;
    } else {
      d[e] = __ldg(lo);
      d[e + 1] = __ldg(hi);
    }
  }
}

__device__ __forceinline__ void load_corners(const Grid& G, const int c[3], int slot, float d[8], bool& ok) {
  int s[8];
  cell_slots(G, c, slot, s);
  load_corners_at(G, c, s, d, ok);
}

// Trilinear interpolation of Eq. 3.  f is a lerp along x, then y, then z.
// Each gradient component is the bilinear blend, over the other two axes, of
// the four cell-edge differences along its own axis: a difference of two close
// grid values is exact (Sterbenz), so no component suffers the cancellation
// that differencing two interpolated values would bring.
__device__ __forceinline__ float lerp1(float t, float a, float b) { return fmaf(t, b - a, a); }

__device__ __forceinline__ Eval trilerp(const float d[8], const float t[3]) {
  Eval r;
  float e00 = lerp1(t[0], d[0], d[1]), e10 = lerp1(t[0], d[2], d[3]);
  float e01 = lerp1(t[0], d[4], d[5]), e11 = lerp1(t[0], d[6], d[7]);
  r.f = lerp1(t[2], lerp1(t[1], e00, e10), lerp1(t[1], e01, e11));
  // x edges at (y,z) = 00, 10, 01, 11
  float a00 = d[1] - d[0], a10 = d[3] - d[2], a01 = d[5] - d[4], a11 = d[7] - d[6];
  r.gt[0] = lerp1(t[2], lerp1(t[1], a00, a10), lerp1(t[1], a01, a11));
  // y edges at (x,z) = 00, 10, 01, 11
  float b00 = d[2] - d[0], b10 = d[3] - d[1], b01 = d[6] - d[4], b11 = d[7] - d[5];
  r.gt[1] = lerp1(t[2], lerp1(t[0], b00, b10), lerp1(t[0], b01, b11));
  // z edges at (x,y) = 00, 10, 01, 11
  float c00 = d[4] - d[0], c10 = d[5] - d[1], c01 = d[6] - d[2], c11 = d[7] - d[3];
  r.gt[2] = lerp1(t[1], lerp1(t[0], c00, c10), lerp1(t[0], c01, c11));
  return r;
}

// Two adjacent floats added as one 8-byte vector reduction (address 8-byte aligned).
__device__ __forceinline__ void red_add_v2(float* addr, float a, float b) {
  asm volatile("red.global.add.v2.f32 [%0], {%1, %2};\n" ::"l"(addr), "f"(a), "f"(b) : "memory");
}
// Four adjacent floats as one 16-byte vector reduction (address 16-byte aligned).
__device__ __forceinline__ void red_add_v4(float* addr, float a, float b, float c, float d) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};\n" ::"l"(addr), "f"(a), "f"(b), "f"(c), "f"(d)
               : "memory");
}

// Deterministic sums: each contribution v is taken exactly (to 2^-60) into
// two integers, hi in units of 2^-20 and lo in units of 2^-60 with
// hi 2^40 + lo = v 2^60 rounded toward zero below 2^-60, by integer
// arithmetic on v's bits.  Integer sums do not depend on the order of the
// additions.  Returns false for a non-finite v or |v| >= 2^42 (FIX_LIMIT).
// Integer arithmetic only, so the host build (a CPU test of its boundaries)
// computes the same integers as the device.
__host__ __device__ __forceinline__ bool fix_split(float v, long long& hi, long long& lo) {
#ifdef __CUDA_ARCH__
  const uint32_t u = __float_as_uint(v);
#else
  uint32_t u;
  memcpy(&u, &v, sizeof(u));
#endif
  const int ex = (int)((u >> 23) & 0xffu);
  if (ex == 0xff) return false;
  long long m = (long long)(u & 0x7fffffu);
  int e;
  if (ex == 0) {
    e = -149;
  } else {
    m |= 0x800000ll;
    e = ex - 150;
  }
  hi = 0;
  lo = 0;
  if (m == 0) return true;
  const int sh = e + 60;  // v 2^60 = m 2^sh, m < 2^24
  // |v| >= 2^42 exactly when e >= 19 (m >= 2^23 for a normal v), i.e. sh >= 79;
  // below that hi = m 2^(sh - 40) < 2^62 fits its 64-bit word.
  if (sh >= 79) return false;
  if (sh >= 40) {
    hi = m << (sh - 40);
  } else if (sh >= 0) {
    const long long val = m << sh;  // < 2^63
    hi = val >> 40;
    lo = val & ((1ll << 40) - 1);
  } else if (sh > -64) {
    lo = m >> (-sh);
  }
  if (u >> 31) {
    hi = -hi;
    lo = -lo;
  }
  return true;
}

// dL/dd_c of the cell's corner c = dx + 2 dy + 4 dz from dL/df = A and
// dL/dt = Gt at local coordinate t: A w_c(t) + sum_a Gt_a dw_c/dt_a, per x edge
// the part that both corners share and the difference along x.
__device__ __forceinline__ void corner_values(const float t[3], float A, const float Gt[3], float v[8]) {
  const float wy[2] = {1.f - t[1], t[1]}, wz[2] = {1.f - t[2], t[2]};
  const float gy[2] = {Gt[1] * wz[0], Gt[1] * wz[1]}, gz[2] = {Gt[2] * wy[0], Gt[2] * wy[1]};
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const int dy = e & 1, dz = e >> 1;
    const float wyz = wy[dy] * wz[dz];
    const float p = fmaf(A, wyz, (dy ? gy[dz] : -gy[dz]) + (dz ? gz[dy] : -gz[dy])), q = Gt[0] * wyz;
    v[2 * e] = fmaf(p, 1.f - t[0], -q);
    v[2 * e + 1] = fmaf(p, t[0], q);
  }
}

// One contribution into the fixed-point sums.
__device__ __forceinline__ void scatter_fixed(unsigned long long* __restrict__ acc, int32_t* __restrict__ err,
                                              int64_t at, float v) {
  long long hi, lo;
  if (!fix_split(v, hi, lo)) {
    atomicOr(err, GP_EF_NUMERIC);
    return;
  }
  if (hi) atomicAdd(acc + 2 * at, (unsigned long long)hi);
  if (lo) atomicAdd(acc + 2 * at + 1, (unsigned long long)lo);
}

// Scatter of one cell's 8 corner contributions: computed once, then per edge
// one vector reduction (8 bytes at even x, 16 bytes from x - 1 at x = 1 mod 4,
// the outer two lanes adding zero) or, at x = 3 mod 4, two single ones.  Every
// corner is stored: load_corners found them.
template <bool DET>
__device__ __forceinline__ void scatter8(const Grid& G, float* __restrict__ grad, unsigned long long* __restrict__ acc,
                                         int32_t* __restrict__ err, const int c[3], const int s[8], const float t[3],
                                         float A, const float Gt[3]) {
  float v[8];
  corner_values(t, A, Gt, v);
  const int xm = c[0] & 3;
#pragma unroll
  for (int e = 0; e < 8; e += 2) {
    const int64_t lo = (int64_t)s[e] * 512 + corner_local(c, e), hi = (int64_t)s[e + 1] * 512 + corner_local(c, e + 1);
    if (DET) {
      scatter_fixed(acc, err, lo, v[e]);
      scatter_fixed(acc, err, hi, v[e + 1]);
      continue;
    }
    if (xm == 1) red_add_v4(grad + lo - 1, 0.f, v[e], v[e + 1], 0.f);
    if (!(xm & 1)) red_add_v2(grad + lo, v[e], v[e + 1]);
    if (xm == 3) {
      atomicAdd(grad + lo, v[e]);
      atomicAdd(grad + hi, v[e + 1]);
    }
  }
}

// Where a record's corner contributions go: straight to the gradient with
// global reductions (float atomics, or the two-word fixed point).
template <bool DET>
struct GlobalSink {
  const Grid& G;
  float* __restrict__ grad;
  unsigned long long* __restrict__ acc;
  int32_t* __restrict__ err;
  __device__ __forceinline__ void cell(const int c[3], int, const int s[8], const float t[3], float A,
                                       const float Gt[3]) {
    scatter8<DET>(G, grad, acc, err, c, s, t, A, Gt);
  }
};

// One step record: classify it, evaluate Eq. 3 at q and at s, add its loss
// terms to sp / sg / ss and (GRAD) scatter its gradient to the 8 + 8 corners,
// scaled by w = 1/B_v (the fixed-point sums too: a contribution below 2^-20
// then has no high word, and most corners take one 64-bit atomic, not two).
//
// The validity test is the one of classify(), with its memory reads arranged
// for latency: both brick slots are read together, then both pull-mask words
// and all 16 corner values together (the corners of a record that turns out
// invalid are read for nothing).
// l_grad = 1 - n . n_s (Eq. 7) without the cancellation of 1 - cos near
// cos = 1: 1 - n.m = |n - m|^2 / 2 + (1 - |n|^2) / 2 + (1 - |m|^2) / 2, whose
// last two terms vanish for a unit vector (a gradient above the floor).  The
// difference n - m of two close unit vectors is computed almost exactly.
__device__ __forceinline__ float grad_term(const float n[3], const float m[3], bool n_unit, bool m_unit) {
  const float d0 = n[0] - m[0], d1 = n[1] - m[1], d2 = n[2] - m[2];
  float l = 0.5f * (d0 * d0 + d1 * d1 + d2 * d2);
  if (!n_unit) l += 0.5f * (1.0f - (n[0] * n[0] + n[1] * n[1] + n[2] * n[2]));
  if (!m_unit) l += 0.5f * (1.0f - (m[0] * m[0] + m[1] * m[1] + m[2] * m[2]));
  return l;
}

// The backward pass of one record from its forward quantities.  With
// u = r / |r| (0 at r = 0), for the pull term dL/df = -w u.n and
// dL/dn = -w f u - w gamma n_s, for the gradient term dL/dn_s = -w gamma n;
// through n = g / |g|, dL/dg = (I - n n^T) dL/dn / |g| (dL/dn / 1e-12 below the
// floor), and dL/dt = dL/dg R/2.  For a unit n the projections are taken from
// small differences instead of differences of large terms:
//   u.n = ((q - s).n - f) / |r|,  (I - n n^T) u = ((q - s) - ((q - s).n) n) / |r|,
//   (I - n n^T) n_s = (n_s - n) - ((n_s - n).n) n,
// which are the same quantities, but keep float32 accuracy when |f| >> |q - s|
// or n ~ n_s (the residual r = (q - s) - f n loses the small perpendicular
// part of q - s to the rounding of f n).
__device__ __forceinline__ void backward_terms(const float q[3], const float s[3], float f, const float nv[3],
                                               const float ns[3], float lp, float inv, float invs, bool big,
                                               bool bigs, float w, float gamma, float half_r, float Gq[3],
                                               float Gs[3], float& dfq) {
  const float ilp = lp > 0.f ? 1.0f / lp : 0.f;
  const float d[3] = {q[0] - s[0], q[1] - s[1], q[2] - s[2]};
  if (big) {
    const float dn = d[0] * nv[0] + d[1] * nv[1] + d[2] * nv[2];
    const float e[3] = {ns[0] - nv[0], ns[1] - nv[1], ns[2] - nv[2]};
    const float en = e[0] * nv[0] + e[1] * nv[1] + e[2] * nv[2];
    dfq = -w * (dn - f) * ilp;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float u_perp = (d[a] - dn * nv[a]) * ilp;
      const float ns_perp = e[a] - en * nv[a];
      Gq[a] = (-w * f * u_perp - w * gamma * ns_perp) * inv * half_r;
    }
  } else {
    const float r[3] = {d[0] - f * nv[0], d[1] - f * nv[1], d[2] - f * nv[2]};
    const float un = (r[0] * nv[0] + r[1] * nv[1] + r[2] * nv[2]) * ilp;
    dfq = -w * un;
#pragma unroll
    for (int a = 0; a < 3; ++a) Gq[a] = (-w * f * r[a] * ilp - w * gamma * ns[a]) * inv * half_r;
  }
  if (bigs) {
    const float e[3] = {nv[0] - ns[0], nv[1] - ns[1], nv[2] - ns[2]};
    const float en = e[0] * ns[0] + e[1] * ns[1] + e[2] * ns[2];
#pragma unroll
    for (int a = 0; a < 3; ++a) Gs[a] = -w * gamma * (e[a] - en * ns[a]) * invs * half_r;
  } else {
#pragma unroll
    for (int a = 0; a < 3; ++a) Gs[a] = -w * gamma * nv[a] * invs * half_r;
  }
}

// A record between the phases of its evaluation.  The three phases issue
// the record's dependent loads level by level - the brick slots (phase a),
// then the pull-mask words and the 16 corner values (phase b) - so that a
// thread working on several records issues all of one level's loads before it
// waits for any of them.
struct RecState {
  float q[3], s[3];
  Cells C;
  int lq, ls;
  uint32_t wq, ws;
  float dq[8], ds[8];
  int sq[8], ss[8];  // the corners' brick slots (not set by the windowed forms)
  bool ok;       // still a candidate for a valid record
  bool corners;  // every corner was found in the band
};

__device__ __forceinline__ void rec_phase_a(const Grid& G, const float q[3], const float s[3], bool active,
                                            RecState& R) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    R.q[a] = q[a];
    R.s[a] = s[a];
  }
  R.ok = active && classify_cells(G, q, s, R.C);
  if (!R.ok) return;
  R.C.slot_q = gp_brick_slot(G.table, G.nb, R.C.cq[0], R.C.cq[1], R.C.cq[2]);
  R.C.slot_s = gp_brick_slot(G.table, G.nb, R.C.cs[0], R.C.cs[1], R.C.cs[2]);
  cell_slots(G, R.C.cq, R.C.slot_q, R.sq);
  cell_slots(G, R.C.cs, R.C.slot_s, R.ss);
}

__device__ __forceinline__ void rec_phase_b(const Grid& G, RecState& R) {
  if (!R.ok) return;
  if (R.C.slot_q < 0 || R.C.slot_s < 0) {
    R.ok = false;
    return;
  }
  R.lq = gp_local(R.C.cq[0], R.C.cq[1], R.C.cq[2]);
  R.ls = gp_local(R.C.cs[0], R.C.cs[1], R.C.cs[2]);
  R.wq = __ldg(G.masks + (int64_t)R.C.slot_q * 48 + 32 + (R.lq >> 5));
  R.ws = __ldg(G.masks + (int64_t)R.C.slot_s * 48 + 32 + (R.ls >> 5));
  R.corners = true;
  load_corners_at(G, R.C.cq, R.sq, R.dq, R.corners);
  load_corners_at(G, R.C.cs, R.ss, R.ds, R.corners);
}

// Validity (cell(q) and cell(s) in the pull band, Sec. 3), the forward terms
// and, with GRAD, the backward pass into the sink.  Returns whether the
// record is valid.
template <bool GRAD, class Sink>
__device__ __forceinline__ bool rec_phase_c(const Grid& G, RecState& R, float w, float beta, float gamma,
                                            Sink& sink, int32_t* __restrict__ err, float& sp, float& sg,
                                            float& ss) {
  if (!R.ok) return false;
  if (!((R.wq >> (R.lq & 31)) & 1u) || !((R.ws >> (R.ls & 31)) & 1u)) return false;
  if (!R.corners) {
    atomicOr(err, GP_EF_RANGE);
    return false;
  }
  const float* q = R.q;
  const float* s = R.s;
  const Cells& C = R.C;
  Eval eq = trilerp(R.dq, C.tq);
  Eval es = trilerp(R.ds, C.ts);
  float g[3] = {eq.gt[0] * G.half_r, eq.gt[1] * G.half_r, eq.gt[2] * G.half_r};
  float gs[3] = {es.gt[0] * G.half_r, es.gt[1] * G.half_r, es.gt[2] * G.half_r};
  float gl = sqrtf(g[0] * g[0] + g[1] * g[1] + g[2] * g[2]);
  float gls = sqrtf(gs[0] * gs[0] + gs[1] * gs[1] + gs[2] * gs[2]);
  float inv = 1.0f / fmaxf(gl, NORM_FLOOR), invs = 1.0f / fmaxf(gls, NORM_FLOOR);
  float nv[3] = {g[0] * inv, g[1] * inv, g[2] * inv};
  float ns[3] = {gs[0] * invs, gs[1] * invs, gs[2] * invs};
  float f = eq.f, fs = es.f;
  float r[3] = {(q[0] - s[0]) - f * nv[0], (q[1] - s[1]) - f * nv[1], (q[2] - s[2]) - f * nv[2]};
  float lp = sqrtf(r[0] * r[0] + r[1] * r[1] + r[2] * r[2]);
  bool big = gl > NORM_FLOOR, bigs = gls > NORM_FLOOR;
  sp += lp;
  sg += grad_term(nv, ns, big, bigs);
  ss += fabsf(fs);
  if (!GRAD) return true;
  float Gq[3], Gs[3], dfq;
  backward_terms(q, s, f, nv, ns, lp, inv, invs, big, bigs, w, gamma, G.half_r, Gq, Gs, dfq);
  float dfs = fs > 0.f ? w * beta : (fs < 0.f ? -w * beta : 0.f);
  sink.cell(C.cq, C.slot_q, R.sq, C.tq, dfq, Gq);
  sink.cell(C.cs, C.slot_s, R.ss, C.ts, dfs, Gs);
  return true;
}

template <bool GRAD, class Sink>
__device__ __forceinline__ bool query_record_to(const Grid& G, const float q[3], const float s[3], float w,
                                                float beta, float gamma, Sink& sink, int32_t* __restrict__ err,
                                                float& sp, float& sg, float& ss) {
  RecState R;
  rec_phase_a(G, q, s, true, R);
  rec_phase_b(G, R);
  return rec_phase_c<GRAD>(G, R, w, beta, gamma, sink, err, sp, sg, ss);
}

// The record with its contributions reduced straight into the gradient.
template <bool DET, bool GRAD>
__device__ __forceinline__ bool query_record(const Grid& G, const float q[3], const float s[3], float w, float beta,
                                             float gamma, float* __restrict__ grad,
                                             unsigned long long* __restrict__ acc, int32_t* __restrict__ err,
                                             float& sp, float& sg, float& ss) {
  GlobalSink<DET> sink{G, grad, acc, err};
  return query_record_to<GRAD>(G, q, s, w, beta, gamma, sink, err, sp, sg, ss);
}

// The L_TV sweep, one brick at a time per warp.  With 1/TV of T vertices (0
// elsewhere) the gradient of a vertex is
//   dTV/dd_i = sum over its in-grid axis neighbours n of
//              (d_i - d_n) (1/TV_i + 1/TV_n),
// so a brick needs 1/TV on its 8^3 vertices and on the six layers that touch
// it, and these need the values two vertices out along an axis and one along
// two.  The warp stages those values and the T masks of the brick and its six
// face neighbours in shared memory (cp.async), computes 1/TV there, then the
// gradient.  A lane works on four vertices along x at a time and keeps its
// column of values along z in registers, so a stencil costs about 3.5 shared
// words a vertex instead of 7 (a thread per vertex was bound by them).
//
// Every array moves once: values in, gradient out, 8 bytes a stored slot.
// Warps share nothing, so a block has no barriers; 20 of them an SM hide each
// other's copies.
//
// The band stores every in-grid axis neighbour of a T vertex, so a value the
// sums use is always present: absent bricks are staged as zeros.  In bricks at
// the grid's boundary the vertices just outside take the values of their
// in-grid neighbours (difference 0); padding slots get gradient 0 and, with
// VALUES, out() their own values.
constexpr int TV_SWEEP_THREADS = 128;
constexpr int TV_SWEEP_WARPS = TV_SWEEP_THREADS / 32;
constexpr int TV_BLOCKS_PER_SM = 5;  // resident blocks per SM: 43 KB of shared memory; at most 102 registers (92 to 96 used)
constexpr int TV_DENSE = 144 * 8;    // rows (y, z) in [-2, 9]^2, x in [0, 8)
constexpr int TV_SIDE = 100 * 2;     // rows (y, z) in [-1, 8]^2: x = -2, -1 or x = 8, 9
constexpr int TV_COPIES = 264 + 192; // 16-byte pieces of rows, 8-byte pieces of the sides
constexpr int TV_PLAN = (TV_COPIES + 31) / 32;  // per lane

// Brick b as the sweep sees it: values, masks, its row of the 27-neighbour
// table (3x3x3, x fastest, -1 absent), grid size and origin vertex.
struct TvBrick {
  const float* D;
  const uint32_t* masks;
  const int32_t* nbr;
  int R, ox, oy, oz;
};

struct TvWarp {
  __align__(16) float d[TV_DENSE + 2 * TV_SIDE];  // values: rows, then the low and the high side
  __align__(16) float inv[100 * 8];               // 1/TV: rows (y, z) in [-1, 8]^2
  float side[2][64];                              // 1/TV at x = -1 and x = 8: index 8 z + y
  __align__(16) uint32_t T[7 * 16];               // T masks: the brick, -x, +x, -y, +y, -z, +z
};
struct TvShared {
  TvWarp w[TV_SWEEP_WARPS];
  uint32_t plan[TV_PLAN * 32];  // region | local << 5 | destination << 14 | 16 bytes << 25 | valid << 26
};

__device__ __forceinline__ void cp_async_ca8(void* smem, const void* gmem, int src_bytes) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(sa), "l"(gmem), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async_cg16(void* smem, const void* gmem, int src_bytes) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(sa), "l"(gmem), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

__device__ __forceinline__ int tv_row(int y, int z) { return ((z + 2) * 12 + (y + 2)) * 8; }   // in TvWarp::d
__device__ __forceinline__ int tv_side(int s, int y, int z) {                                  // the side's pair
  return TV_DENSE + s * TV_SIDE + ((z + 1) * 10 + (y + 1)) * 2;
}
__device__ __forceinline__ int tv_irow(int y, int z) { return ((z + 1) * 10 + (y + 1)) * 8; }  // in TvWarp::inv

// The copies of a brick, the same for each: entry e of the plan.
__device__ __forceinline__ uint32_t tv_plan_entry(int e) {
  if (e >= TV_COPIES) return 0u;
  int y, z, dx, x, dst;
  const bool big = e < 264;
  if (big) {
    // Rows: 96 with z in [0, 8), y in [-2, 9]; 20 with z = -1, 8, y in
    // [-1, 8]; 16 with z = -2, 9, y in [0, 8).  Two pieces each.
    const int r = e >> 1;
    if (r < 96) {
      z = r / 12;
      y = r % 12 - 2;
    } else if (r < 116) {
      z = r < 106 ? -1 : 8;
      y = (r - 96) % 10 - 1;
    } else {
      z = r < 124 ? -2 : 9;
      y = (r - 116) % 8;
    }
    dx = 1;
    x = 4 * (e & 1);
    dst = ((z + 2) * 12 + (y + 2)) * 8 + x;
  } else {
    // Sides: 80 rows with z in [0, 8), y in [-1, 8]; 16 with z = -1, 8, y in [0, 8).
    const int k = e - 264, s = k / 96, r = k % 96;
    if (r < 80) {
      z = r / 10;
      y = r % 10 - 1;
    } else {
      z = r < 88 ? -1 : 8;
      y = (r - 80) % 8;
    }
    dx = 2 * s;
    x = s ? 0 : 6;
    dst = TV_DENSE + s * TV_SIDE + ((z + 1) * 10 + (y + 1)) * 2;
  }
  const uint32_t reg = ((z >> 3) + 1) * 9 + ((y >> 3) + 1) * 3 + dx;
  const uint32_t loc = ((z & 7) << 6) | ((y & 7) << 3) | x;
  return reg | (loc << 5) | ((uint32_t)dst << 14) | ((big ? 1u : 0u) << 25) | (1u << 26);
}

// Boundary bricks: the vertices one step outside the grid take the value of
// the in-grid vertex next to them.
__device__ __forceinline__ void tv_close_grid(float* d, const TvBrick& bk, int lane) {
  auto copy_y = [&](int to, int from) {  // rows y = from to y = to, all z
    for (int k = lane; k < 96; k += 32) {
      const int z = (k >> 3) - 2, x = k & 7;
      d[tv_row(to, z) + x] = d[tv_row(from, z) + x];
    }
    if (to >= -1 && to <= 8)
      for (int k = lane; k < 40; k += 32)
        d[tv_side(k / 20, to, (k % 20) / 2 - 1) + (k & 1)] = d[tv_side(k / 20, from, (k % 20) / 2 - 1) + (k & 1)];
    __syncwarp();
  };
  auto copy_z = [&](int to, int from) {
    for (int k = lane; k < 96; k += 32) {
      const int y = (k >> 3) - 2, x = k & 7;
      d[tv_row(y, to) + x] = d[tv_row(y, from) + x];
    }
    if (to >= -1 && to <= 8)
      for (int k = lane; k < 40; k += 32)
        d[tv_side(k / 20, (k % 20) / 2 - 1, to) + (k & 1)] = d[tv_side(k / 20, (k % 20) / 2 - 1, from) + (k & 1)];
    __syncwarp();
  };
  const int lx = bk.R - bk.ox, ly = bk.R - bk.oy, lz = bk.R - bk.oz;  // the last in-grid vertex
  if (bk.ox == 0 || lx <= 8) {
    for (int k = lane; k < 100; k += 32) {
      const int y = k % 10 - 1, z = k / 10 - 1;
      if (bk.ox == 0) d[tv_side(0, y, z) + 1] = d[tv_row(y, z)];
      if (lx == 0) d[tv_row(y, z) + 1] = d[tv_row(y, z)];
      if (lx == 8) d[tv_side(1, y, z) + 1] = d[tv_side(1, y, z)];
    }
    __syncwarp();
  }
  if (bk.oy == 0) copy_y(-1, 0);
  if (ly <= 8) copy_y(ly + 1, ly);
  if (bk.oz == 0) copy_z(-1, 0);
  if (lz <= 8) copy_z(lz + 1, lz);
}

__device__ __forceinline__ float4 tv_ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }

// 1/TV of a quad from its values and those of its 6 axis neighbours (the
// squared differences added in the order -x, +x, -y, +y, -z, +z), 0 where the
// bit of T is clear; tsum: the sum of TV.
__device__ __forceinline__ float4 tv_inv4(float4 c, float left, float right, float4 ym, float4 yp, float4 zm,
                                          float4 zp, uint32_t bits, float& tsum) {
  const float v[6] = {left, c.x, c.y, c.z, c.w, right};
  const float a[4][4] = {{ym.x, yp.x, zm.x, zp.x}, {ym.y, yp.y, zm.y, zp.y},
                         {ym.z, yp.z, zm.z, zp.z}, {ym.w, yp.w, zm.w, zp.w}};
  float out[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float d = v[k + 1];
    float e = d - v[k];
    float s = e * e;
    e = d - v[k + 2];
    s = fmaf(e, e, s);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      e = d - a[k][j];
      s = fmaf(e, e, s);
    }
    const bool in = (bits >> k) & 1u;
    out[k] = in && s > 0.f ? rsqrtf(s) : 0.f;
    tsum += in ? s * out[k] : 0.f;
  }
  return make_float4(out[0], out[1], out[2], out[3]);
}

// The gradient of a quad, unscaled, in the same order of neighbours.
__device__ __forceinline__ float4 tv_grad4(float4 c, float left, float right, float4 ym, float4 yp, float4 zm,
                                           float4 zp, float4 ic, float ileft, float iright, float4 iym, float4 iyp,
                                           float4 izm, float4 izp) {
  const float v[6] = {left, c.x, c.y, c.z, c.w, right}, w[6] = {ileft, ic.x, ic.y, ic.z, ic.w, iright};
  const float a[4][4] = {{ym.x, yp.x, zm.x, zp.x}, {ym.y, yp.y, zm.y, zp.y},
                         {ym.z, yp.z, zm.z, zp.z}, {ym.w, yp.w, zm.w, zp.w}};
  const float b[4][4] = {{iym.x, iyp.x, izm.x, izp.x}, {iym.y, iyp.y, izm.y, izp.y},
                         {iym.z, iyp.z, izm.z, izp.z}, {iym.w, iyp.w, izm.w, izp.w}};
  float out[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float d = v[k + 1], own = w[k + 1];
    float g = (d - v[k]) * (own + w[k]);
    g = fmaf(d - v[k + 2], own + w[k + 2], g);
#pragma unroll
    for (int j = 0; j < 4; ++j) g = fmaf(d - a[k][j], own + b[k][j], g);
    out[k] = g;
  }
  return make_float4(out[0], out[1], out[2], out[3]);
}

// The sweep over work items 0 .. n - 1, dealt to the warps of the grid in
// turn.  src.brick(i) gives item i's TvBrick.  For each of the brick's 128
// quads q (vertices 4 q .. 4 q + 3) one lane calls fetch(i, q), whose loads the
// stencil work then hides, and out(i, q, d, g, fetched) with the quad's values
// and unscaled gradient; done(i, tsum) is called by every lane after each item
// with its share of the sum of TV_i.  All lanes of the warp call these together.
// GRAD = false: the sums only (no layers, no fetch, no out).  VALUES: out() uses d.
template <bool GRAD, bool VALUES, class Src, class Fetch, class Out, class Done>
__device__ __forceinline__ void tv_sweep(const Src& src, int64_t n, TvShared& sh, Fetch&& fetch, Out&& out,
                                         Done&& done) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int e = threadIdx.x; e < TV_PLAN * 32; e += TV_SWEEP_THREADS) sh.plan[e] = tv_plan_entry(e);
  __syncthreads();
  TvWarp& s = sh.w[wid];
  const int xq = lane & 1, y = (lane >> 1) & 7, z0 = 4 * (lane >> 4);
  const int64_t stride = (int64_t)gridDim.x * TV_SWEEP_WARPS;
  int64_t i = (int64_t)blockIdx.x * TV_SWEEP_WARPS + wid;
  if (i >= n) return;
  TvBrick bk = src.brick(i);
  int nbr = lane < 27 ? __ldg(bk.nbr + lane) : -1;
  while (true) {
    // Copies of item i.
#pragma unroll 5
    for (int k = 0; k < TV_PLAN; ++k) {
      const uint32_t t = sh.plan[lane + 32 * k];
      const int sl = __shfl_sync(0xffffffffu, nbr, t & 31);
      if (!(t >> 26)) continue;
      const float* from = sl >= 0 ? bk.D + (int64_t)sl * 512 + ((t >> 5) & 511) : bk.D;
      float* to = &s.d[(t >> 14) & 2047];
      if ((t >> 25) & 1)
        cp_async_cg16(to, from, sl >= 0 ? 16 : 0);
      else
        cp_async_ca8(to, from, sl >= 0 ? 8 : 0);
    }
    {
      const int f = lane >> 2;  // the brick, -x, +x, -y, +y, -z, +z
      const int reg = f == 0 ? 13 : f == 1 ? 12 : f == 2 ? 14 : f == 3 ? 10 : f == 4 ? 16 : f == 5 ? 4 : 22;
      const int sl = __shfl_sync(0xffffffffu, nbr, reg);
      if (lane < 28)
        cp_async_cg16(&s.T[4 * lane], sl >= 0 ? bk.masks + (int64_t)sl * 48 + 4 * (lane & 3) : bk.masks,
                      sl >= 0 ? 16 : 0);
    }
    // The next item's neighbours are fetched meanwhile.
    const int64_t next = i + stride;
    TvBrick nk = bk;
    int nnbr = -1;
    if (next < n) {
      nk = src.brick(next);
      if (lane < 27) nnbr = __ldg(nk.nbr + lane);
    }
    cp_async_wait_all();
    __syncwarp();
    const bool edge = bk.ox == 0 || bk.oy == 0 || bk.oz == 0 || bk.ox + 8 >= bk.R || bk.oy + 8 >= bk.R ||
                      bk.oz + 8 >= bk.R;
    if (edge) tv_close_grid(s.d, bk, lane);

    // 1/TV of the brick's own quads, up a lane's column z0 .. z0 + 3.
    float tsum = 0.f, none = 0.f;
    {
      float4 zm = tv_ld4(s.d + tv_row(y, z0 - 1) + 4 * xq), c = tv_ld4(s.d + tv_row(y, z0) + 4 * xq);
#pragma unroll 2
      for (int z = z0; z < z0 + 4; ++z) {
        const int r = tv_row(y, z);
        const float4 zp = tv_ld4(s.d + r + 96 + 4 * xq);
        const float left = s.d[xq ? r + 3 : tv_side(0, y, z) + 1], right = s.d[xq ? tv_side(1, y, z) : r + 4];
        const float4 iv = tv_inv4(c, left, right, tv_ld4(s.d + r - 8 + 4 * xq), tv_ld4(s.d + r + 8 + 4 * xq), zm, zp,
                                  s.T[2 * z + (y >> 2)] >> (8 * (y & 3) + 4 * xq), tsum);
        if (GRAD) *reinterpret_cast<float4*>(s.inv + tv_irow(y, z) + 4 * xq) = iv;
        zm = c;
        c = zp;
      }
    }
    if (GRAD) {
    // The layers y = -1, 8 and z = -1, 8: 16 quads each.
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int f = (lane >> 4) + 2 * k, t = (lane >> 1) & 7;
      const int fy = f == 0 ? -1 : f == 1 ? 8 : t, fz = f == 2 ? -1 : f == 3 ? 8 : t;
      const int r = tv_row(fy, fz);
      const float left = s.d[xq ? r + 3 : tv_side(0, fy, fz) + 1], right = s.d[xq ? tv_side(1, fy, fz) : r + 4];
      const uint32_t bits = s.T[16 * (f + 3) + 2 * (fz & 7) + ((fy & 7) >> 2)] >> (8 * (fy & 3) + 4 * xq);
      *reinterpret_cast<float4*>(s.inv + tv_irow(fy, fz) + 4 * xq) =
          tv_inv4(tv_ld4(s.d + r + 4 * xq), left, right, tv_ld4(s.d + r - 8 + 4 * xq), tv_ld4(s.d + r + 8 + 4 * xq),
                  tv_ld4(s.d + r - 96 + 4 * xq), tv_ld4(s.d + r + 96 + 4 * xq), bits, none);
    }
    // The layers x = -1 and x = 8: 64 vertices each.
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int sd = k >> 1, v = lane + 32 * (k & 1), fy = v & 7, fz = v >> 3;
      const int at = tv_side(sd, fy, fz) + (sd ? 0 : 1);  // the layer's value; its outer neighbour beside it
      const float d = s.d[at];
      const float xm = sd ? s.d[tv_row(fy, fz) + 7] : s.d[at - 1], xp = sd ? s.d[at + 1] : s.d[tv_row(fy, fz)];
      float e = d - xm, q = e * e;
      e = d - xp;
      q = fmaf(e, e, q);
      e = d - s.d[at - 2];
      q = fmaf(e, e, q);
      e = d - s.d[at + 2];
      q = fmaf(e, e, q);
      e = d - s.d[at - 20];
      q = fmaf(e, e, q);
      e = d - s.d[at + 20];
      q = fmaf(e, e, q);
      const bool in = (s.T[16 * (1 + sd) + 2 * fz + (fy >> 2)] >> (8 * (fy & 3) + (sd ? 0 : 7))) & 1u;
      s.side[sd][v] = in && q > 0.f ? rsqrtf(q) : 0.f;
    }
    __syncwarp();
    // The gradient.
    float4 zm = tv_ld4(s.d + tv_row(y, z0 - 1) + 4 * xq), c = tv_ld4(s.d + tv_row(y, z0) + 4 * xq);
    float4 izm = tv_ld4(s.inv + tv_irow(y, z0 - 1) + 4 * xq), ic = tv_ld4(s.inv + tv_irow(y, z0) + 4 * xq);
#pragma unroll 2
    for (int z = z0; z < z0 + 4; ++z) {
      const int r = tv_row(y, z), ir = tv_irow(y, z), q = (z * 8 + y) * 2 + xq;
      auto got = fetch(i, q);
      const float4 zp = tv_ld4(s.d + r + 96 + 4 * xq), izp = tv_ld4(s.inv + ir + 80 + 4 * xq);
      const float left = s.d[xq ? r + 3 : tv_side(0, y, z) + 1], right = s.d[xq ? tv_side(1, y, z) : r + 4];
      const float ileft = xq ? s.inv[ir + 3] : s.side[0][8 * z + y], iright = xq ? s.side[1][8 * z + y] : s.inv[ir + 4];
      float4 g = tv_grad4(c, left, right, tv_ld4(s.d + r - 8 + 4 * xq), tv_ld4(s.d + r + 8 + 4 * xq), zm, zp, ic, ileft,
                          iright, tv_ld4(s.inv + ir - 8 + 4 * xq), tv_ld4(s.inv + ir + 8 + 4 * xq), izm, izp);
      float4 own = c;
      if (edge) {
        const bool row = bk.oy + y <= bk.R && bk.oz + z <= bk.R;
        const int x = bk.ox + 4 * xq;
        g.x = row && x <= bk.R ? g.x : 0.f;
        g.y = row && x + 1 <= bk.R ? g.y : 0.f;
        g.z = row && x + 2 <= bk.R ? g.z : 0.f;
        g.w = row && x + 3 <= bk.R ? g.w : 0.f;
        if (VALUES) {
          // Not those that tv_close_grid put beside the grid.
          const int slot = __shfl_sync(0xffffffffu, nbr, 13);
          if (!row || x + 3 > bk.R) {
            const float4 held = __ldg(reinterpret_cast<const float4*>(bk.D + (int64_t)slot * 512 + 4 * q));
            own.x = row && x <= bk.R ? c.x : held.x;
            own.y = row && x + 1 <= bk.R ? c.y : held.y;
            own.z = row && x + 2 <= bk.R ? c.z : held.z;
            own.w = held.w;
          }
        }
      }
      out(i, q, own, g, got);
      zm = c;
      c = zp;
      izm = ic;
      ic = izp;
    }
    }
    done(i, tsum);
    if (next >= n) break;
    __syncwarp();  // every lane is done with the staged brick
    i = next;
    bk = nk;
    nbr = nnbr;
  }
}

// One Adam step (Kingma and Ba; Sec. 4 "Details") of one vertex, the bias
// corrections given as their reciprocals ibc = 1 / (1 - beta^t):
//   m <- b1 m + (1 - b1) g,  v <- b2 v + (1 - b2) g^2,
//   d <- d - lr (m ibc1) / (sqrt(v ibc2) + eps).
// The root is x rsqrt(x) and the division __fdividef: a few ulp each, far
// inside the step's tolerance, and neither has a slow path.
__device__ __forceinline__ float adam_elem(float g, float& m, float& v, float d, float lr, float b1, float b2,
                                           float eps, float ibc1, float ibc2) {
  const float mm = fmaf(b1, m, (1.0f - b1) * g);
  const float vv = fmaf(b2, v, (1.0f - b2) * g * g);
  m = mm;
  v = vv;
  const float mh = mm * ibc1, vh = vv * ibc2;
  const float root = (vh > 0.f && vh < INFINITY) ? vh * rsqrtf(vh) : vh;
  return d - __fdividef(lr * mh, root + eps);
}

// Adam on the trainable vertices among 4q .. 4q + 3 of brick `slot` (q in
// [0, 128)): one 16-byte load and store per array.  Vertices of the quad that
// are not trainable are written back unchanged.
__device__ __forceinline__ void adam_quad(int slot, int q, const uint32_t* __restrict__ masks,
                                          const float* __restrict__ grad, float* __restrict__ D,
                                          float* __restrict__ m, float* __restrict__ v, float lr, float b1, float b2,
                                          float eps, float ibc1, float ibc2) {
  const uint32_t bits = (__ldg(masks + (int64_t)slot * 48 + 16 + (q >> 3)) >> ((4 * q) & 31)) & 15u;
  if (!bits) return;
  const int64_t a = (int64_t)slot * 512 + 4 * q;
  const float4 g4 = __ldg(reinterpret_cast<const float4*>(grad + a));
  float4 m4 = *reinterpret_cast<const float4*>(m + a);
  float4 v4 = *reinterpret_cast<const float4*>(v + a);
  float4 d4 = *reinterpret_cast<const float4*>(D + a);
  const float* gp = reinterpret_cast<const float*>(&g4);
  float* mp = reinterpret_cast<float*>(&m4);
  float* vp = reinterpret_cast<float*>(&v4);
  float* dp = reinterpret_cast<float*>(&d4);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    if (!((bits >> k) & 1u)) continue;
    dp[k] = adam_elem(gp[k], mp[k], vp[k], dp[k], lr, b1, b2, eps, ibc1, ibc2);
  }
  *reinterpret_cast<float4*>(m + a) = m4;
  *reinterpret_cast<float4*>(v + a) = v4;
  *reinterpret_cast<float4*>(D + a) = d4;
}
