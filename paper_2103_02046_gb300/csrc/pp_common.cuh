// Pieces shared by the FP32 and the FP64 short range: the geometry of the neighbour rows and the
// warp and block reductions.
#pragma once

#include "p3m_internal.cuh"

namespace p3m {

// Row geometry for kRows cell rows per cutoff length in y and z (Geom::rows, 1, 2 or 3): the
// neighbour rows of a particle's row are the (2 kRows + 1)^2 rows around it, numbered y fastest;
// the particle's own row is number `first`, and the half shell walked by the short range is
// rows first .. last - 1 (5 of 9, 13 of 25 or 25 of 49 rows).
template <int kRows>
struct Rows {
  static constexpr int reach = kRows;
  static constexpr int span = 2 * kRows + 1;
  static constexpr int first = span * span / 2;
  static constexpr int last = span * span;
  static constexpr int half = last - first;
};

template <int kBlk>
__device__ __forceinline__ void block_reduce_add(double v, double* dst) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  __shared__ double ws[kBlk / 32];
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    double s = threadIdx.x < kBlk / 32 ? ws[threadIdx.x] : 0.0;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) atomicAdd(dst, s);
  }
}

__device__ __forceinline__ void warp_add_u64(unsigned long long v, unsigned long long* dst) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0 && v) atomicAdd(dst, v);
}

// Sorted range [j0, j1) of neighbour row r (y fastest, Rows::first = the particle's own row
// (cy, cz)) that can hold particles within distance 1 of (px, py, pz); empty if none can. The
// rectangle distance and the x half-width carry the search slack, as in for_rows.
template <int kRows>
__device__ __forceinline__ void row_range(const Geom& g, const uint32_t* __restrict__ starts,
                                          float px, float py, float pz, int cy, int cz, int r,
                                          uint32_t& j0, uint32_t& j1) {
  using R = Rows<kRows>;
  j0 = j1 = 0;
  const int ry = cy + (r % R::span) - R::reach, rz = cz + (r / R::span) - R::reach;
  if (ry < 0 || ry >= g.nc[1] || rz < 0 || rz >= g.nc[2]) return;
  const float slack = g.slack_f;
  const float cwy = g.cw_f[1], cwz = g.cw_f[2];
  const float yl = ry * cwy, yh = yl + cwy, zl = rz * cwz, zh = zl + cwz;
  const float dy = fmaxf((py < yl ? yl - py : (py > yh ? py - yh : 0.f)) - slack, 0.f);
  const float dz = fmaxf((pz < zl ? zl - pz : (pz > zh ? pz - zh : 0.f)) - slack, 0.f);
  const float d2 = dy * dy + dz * dz;
  if (d2 >= 1.f) return;
  const float w = sqrtf(1.f - d2) + slack;
  const float iwx = g.inv_cw_f[0];
  const int c0 = max(static_cast<int>(floorf((px - w) * iwx)), 0);
  const int c1 = min(static_cast<int>(floorf((px + w) * iwx)), g.nc[0] - 1);
  if (c0 > c1) return;
  const uint32_t base = (static_cast<uint32_t>(rz) * g.nc[1] + ry) * g.nc[0];
  j0 = starts[base + c0];
  j1 = starts[base + c1 + 1];
}

}  // namespace p3m
