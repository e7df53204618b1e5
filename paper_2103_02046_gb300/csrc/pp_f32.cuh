// Pieces shared by the FP32 short-range kernels: record loads, reductions, the error-free split of
// force terms and the fitted erfc(x) e^{x^2}.
#pragma once

#include <algorithm>
#include <cmath>

#include "pp_common.cuh"

namespace p3m {

// two-float accumulator (hi + lo) with Knuth's TwoSum
struct Acc2 {
  float hi, lo;
  __device__ __forceinline__ void add(float v) {
    const float s = hi + v;
    const float bp = s - hi;
    const float err = (hi - (s - bp)) + (v - bp);
    hi = s;
    lo += err;
  }
  __device__ __forceinline__ float value() const { return hi + lo; }
};

// One 32-byte record (hi and lo float4) in a single 256-bit load through the read-only path.
// The records array is 32-byte aligned and not written while the short range runs.
__device__ __forceinline__ void load_rec32(const float4* p, float4& h, float4& l) {
  asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=f"(h.x), "=f"(h.y), "=f"(h.z), "=f"(h.w), "=f"(l.x), "=f"(l.y), "=f"(l.z), "=f"(l.w)
      : "l"(p));
}

__device__ __forceinline__ void red_add_v4(float4* dst, float a, float b, float c, float d) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(dst), "f"(a), "f"(b),
               "f"(c), "f"(d)
               : "memory");
}

// predicated form: the reduction happens only where p holds (no branch around it)
__device__ __forceinline__ void red_add_v4_if(bool p, float4* dst, float a, float b, float c,
                                              float d) {
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %5, 0;\n\t"
      "@q red.global.add.v4.f32 [%0], {%1, %2, %3, %4};\n\t}" ::"l"(dst),
      "f"(a), "f"(b), "f"(c), "f"(d), "r"(static_cast<int>(p))
      : "memory");
}

// Error-free split of a short-range force component about the grid of multiples of
// kSplitQ = 2^-6 (the kernel's force unit is the pair force at a cutoff length's scale, so the
// terms are O(1) and a particle's sums stay far below 2^24 kSplitQ even with tens of thousands
// of neighbours): v = c + f exactly, with c a multiple of kSplitQ and |f| <= kSplitQ / 2.
// Adding kSplitC = 1.5 * 2^23 * kSplitQ rounds v to that grid (the sum's last mantissa bit is
// worth kSplitQ); subtracting it again is exact (Sterbenz), and so is v - c. The coarse parts c
// of one particle's terms are multiples of kSplitQ, so their FP32 atomic sum is exact, and
// independent of the order, while it stays below 2^24 kSplitQ in magnitude; only the small
// parts f are rounded when summed.
constexpr float kSplitQ = 0.015625f;
constexpr float kSplitC = 1.5f * 8388608.f * kSplitQ;
// A term of magnitude 2^21 kSplitQ or more (a pair closer than about 0.006 cutoff lengths)
// would take the coarse sum out of its exact range: it goes whole to a third array (big), where
// a particle rarely has more than one term.
constexpr float kBigTerm = 2097152.f * kSplitQ;
// (in PTX, so that no compiler pass folds (v + C) - C into v)
__device__ __forceinline__ void split_q(float v, float& c, float& f) {
  float t;
  asm("add.rn.f32 %0, %1, %2;" : "=f"(t) : "f"(v), "f"(kSplitC));
  asm("sub.rn.f32 %0, %1, %2;" : "=f"(c) : "f"(t), "f"(kSplitC));
  asm("sub.rn.f32 %0, %1, %2;" : "=f"(f) : "f"(v), "f"(c));
}

__device__ __forceinline__ bool big_term(float a, float b, float c) {
  return fmaf(a, a, fmaf(b, b, c * c)) >= kBigTerm * kBigTerm;
}

// 2-wide reduction (the fine x and y parts)
__device__ __forceinline__ void red_add_v2_if(bool p, float2* dst, float a, float b) {
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %3, 0;\n\t"
      "@q red.global.add.v2.f32 [%0], {%1, %2};\n\t}" ::"l"(dst),
      "f"(a), "f"(b), "r"(static_cast<int>(p))
      : "memory");
}

// One particle's short-range force held in three arrays: co (float4: the coarse x, y, z parts and
// the fine z part), fi (float2: the fine x and y parts) and bg (float4: big terms). Each added
// term is split; the coarse parts and the fine z part go out in one 4-wide reduction into co, the
// fine x and y parts in one 2-wide reduction into fi (24 bytes a term; the fourth coarse slot
// would otherwise carry a zero), or, if the term is big, it is reduced whole into bg. The result
// is the exact sum up to the rounding of the fine sums, whose terms are at most kSplitQ / 2, and
// of the (rare) big terms. `big` may be set for terms below kBigTerm too (a cheaper test that
// never misses a big term).
__device__ __forceinline__ void split_add_v4_if(bool p, bool big, float4* co, float2* fi,
                                                float4* bg, float a, float b, float c) {
  // x and y split on the two-wide FP32 instructions, z on the scalar ones (the same steps)
  const float2 ab = make_float2(a, b);
  const float2 abc = __fadd2_rn(__fadd2_rn(ab, make_float2(kSplitC, kSplitC)),
                                make_float2(-kSplitC, -kSplitC));
  const float2 abf = __fadd2_rn(ab, make_float2(-abc.x, -abc.y));
  float cc, cf;
  split_q(c, cc, cf);
  red_add_v4_if(p && !big, co, abc.x, abc.y, cc, cf);
  red_add_v2_if(p && !big, fi, abf.x, abf.y);
  if (p && big) red_add_v4(bg, abc.x + abf.x, abc.y + abf.y, cc + cf, 0.f);  // (a, b, c); rare
}
// the same for a compensated sum hi + lo (lo far below hi): hi is split, lo joins the fine part
__device__ __forceinline__ void split_add_v4(float4* co, float2* fi, float4* bg, float a, float b,
                                             float c, float la, float lb, float lc) {
  if (big_term(a, b, c)) {
    red_add_v4(bg, a, b, c, 0.f);
    red_add_v4(co, 0.f, 0.f, 0.f, lc);
    red_add_v2_if(true, fi, la, lb);
    return;
  }
  float ac, af, bc, bf, cc, cf;
  split_q(a, ac, af);
  split_q(b, bc, bf);
  split_q(c, cc, cf);
  red_add_v4(co, ac, bc, cc, __fadd_rn(cf, lc));
  red_add_v2_if(true, fi, __fadd_rn(af, la), __fadd_rn(bf, lb));
}

__device__ __forceinline__ float rsqrt_ftz(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ float ex2_ftz(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ float rcp_ftz(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// R(x) = erfc(x) e^{x^2}, x = kappa rho, as t P(u): t = 1 / (1 + p kappa rho), u = t - t_c
template <int kDeg, bool kHw>
__device__ __forceinline__ float erfcx_poly(const PairPoly& P, float rho) {
  const float t = kHw ? rcp_ftz(fmaf(P.pk, rho, 1.f)) : 1.f / fmaf(P.pk, rho, 1.f);
  const float u = t - P.tc;
  float R = P.c[kDeg];
#pragma unroll
  for (int m = kDeg - 1; m >= 0; --m) R = fmaf(R, u, P.c[m]);
  return R * t;
}

// Whether the tiles of pp_dense.cu hold the pair of sorted particles i, i + 1 (i even). A word per
// stretch of 64 particles: bits 0 and 1 for its first and its second piece, the end of the first
// (bits 8..15) and the beginning of the second (bits 16..23).
__device__ __forceinline__ bool in_dense_tile(const uint32_t* __restrict__ flags, uint32_t i) {
  const uint32_t f = flags[i >> 6], k = i & 63u;
  return ((f & 1u) && k < ((f >> 8) & 0xffu)) || ((f & 2u) && k >= ((f >> 16) & 0xffu));
}

// Calls visit(j0, j1) for every neighbour row of the query point (px, py, pz) (cutoff units)
// that can hold particles within distance 1, with [j0, j1) the sorted range of its cells whose
// x-extent meets (px - w, px + w), w = sqrt(1 - d^2) + slack, d the point's distance to the
// row's (y, z) rectangle less the slack. The slack (Geom::slack) exceeds every rounding in where
// the sort placed a particle, so no particle within distance 1 is left out.
template <typename T, typename V>
__device__ __forceinline__ void for_rows(const Geom& g, const uint32_t* __restrict__ starts, T px,
                                         T py, T pz, int part, int parts, V&& visit) {
  const T slack = static_cast<T>(g.slack);
  const T cwy = static_cast<T>(g.cw[1]), cwz = static_cast<T>(g.cw[2]);
  const T iwx = static_cast<T>(g.inv_cw[0]), iwy = static_cast<T>(g.inv_cw[1]),
          iwz = static_cast<T>(g.inv_cw[2]);
  const int y0 = max(static_cast<int>(floor((py - T(1) - slack) * iwy)), 0);
  const int y1 = min(static_cast<int>(floor((py + T(1) + slack) * iwy)), g.nc[1] - 1);
  const int z0 = max(static_cast<int>(floor((pz - T(1) - slack) * iwz)), 0);
  const int z1 = min(static_cast<int>(floor((pz + T(1) + slack) * iwz)), g.nc[2] - 1);
  int turn = 0;
  for (int rz = z0; rz <= z1; ++rz) {
    const T zl = static_cast<T>(rz) * cwz, zh = zl + cwz;
    const T dz = max((pz < zl ? zl - pz : (pz > zh ? pz - zh : T(0))) - slack, T(0));
    for (int ry = y0; ry <= y1; ++ry) {
      if ((turn++ & (parts - 1)) != part) continue;
      const T yl = static_cast<T>(ry) * cwy, yh = yl + cwy;
      const T dy = max((py < yl ? yl - py : (py > yh ? py - yh : T(0))) - slack, T(0));
      const T d2 = dy * dy + dz * dz;
      if (d2 >= T(1)) continue;
      const T w = sqrt(T(1) - d2) + slack;
      const int c0 = max(static_cast<int>(floor((px - w) * iwx)), 0);
      const int c1 = min(static_cast<int>(floor((px + w) * iwx)), g.nc[0] - 1);
      if (c0 > c1) continue;
      const uint32_t base = (static_cast<uint32_t>(rz) * g.nc[1] + ry) * g.nc[0];
      visit(starts[base + c0], starts[base + c1 + 1]);
    }
  }
}

// First cell of the sort's order above the z rows that hold the particles less than r_c above the
// cathode (pp_bc): those are the sorted particles before starts[near_cathode_cell].
inline uint32_t near_cathode_cell(const p3m_ctx* c) {
  const double top = (0.5 * c->g.img_c + 1.0 + c->g.slack) * c->g.inv_cw[2];
  const int rows = std::max(0, std::min(c->g.nc[2], static_cast<int>(std::floor(top)) + 1));
  return static_cast<uint32_t>(rows) * c->g.nc[1] * c->g.nc[0];
}

}  // namespace p3m
