// FP32 short range of dense regions: tiles of 64 particles against groups of 32, each unordered
// pair once.
//
// The walk (pp.cu) sends every pair's reaction to the L2 by vector reductions, which is what bounds
// it where a particle has thousands of neighbours (L2 72% busy, issue 48%). Here a warp holds 64
// consecutive sorted particles of one cell row, two a lane, and takes the later particles of its
// half shell in groups of 32, staged in shared memory. It turns the group through its lanes: at
// turn r lane l meets particle (l + r) mod 32, whose reaction sum travels with it (three shuffles
// a turn), so a group's reactions go out once per 2048 pairs. Groups farther than r_c from the tile
// (bounding boxes of both) are skipped. The rest of a turn is the walk's pair arithmetic: exact
// separations, the fitted erfc, plain FP32 sums over one group (32 terms for a tile particle, 64
// for a group particle), then the compensated sums and the exact split of pp_f32.cuh.
//
// A tile pays where its boxes are small against r_c: of the pairs met about 0.43 are within r_c at
// 36,000 neighbours a particle (rows r_c/3 wide), fewer at lower densities, while the walk's runs
// per particle keep 0.59 to 0.37. k_dense_tiles therefore hands a stretch of 64 particles to the
// tiles only if its row holds enough of them (kDenseNeighboursMin), and the walk takes the others:
// every pair belongs to its earlier particle in sorted order, so the two can be mixed freely.
//
// Measured, short range: 1,048,576-particle Gaussian 97.1 -> 38.7 ms, 4,194,304-particle core and
// halo 121.6 -> 62.5 ms, 131,072 dense particles 2.57 -> 1.15 ms. It issues 75 to 89% of the slots
// (scalar pair arithmetic: 89% and 40.8 ms on the Gaussian; the two-wide instructions cut the
// instructions by a quarter and the FMA pipe, at 62%, takes twice as long for each). Blocks per SM
// 3, 4, 5, 6: 39.9, 38.9, 38.7, 39.9 ms; turns unrolled 1, 2, 4, 8: 41.1, 38.7, 39.8, 40.1 ms.
#include <algorithm>

#include "pp_f32.cuh"

namespace p3m {
namespace {

constexpr int kThreads = 128;
constexpr int kWarps = kThreads / 32;
constexpr int kBlocksPerSm = 5;
constexpr uint32_t kTile = 64;
// A region goes to the tiles if its particles have 2000 neighbours, or 300 and four times the mean
// over the mesh's volume. At a uniform density the walk is ahead up to about 2000 (a sphere with
// r_c = 3h, tiles against the walk: 131,072 particles of 1200 neighbours 918, 819 us; 1,300,003 of 1400
// 6.6, 5.3 ms; 16,777,216, of whose 226 neighbours chance makes 300 here and there, 23.4, 17.8 ms), while
// a bunch with a core is best served by tiles throughout (all of more than 300, 1000, 2000 neighbours:
// four steps of 131,072 dense particles 6.2, 7.3, 8.7 ms; a Gaussian of 150,000 1.01, 1.24, 1.49 ms). The
// sphere's density is 2.4 times its mesh's mean.
constexpr float kDenseNeighboursMin = 300.f, kDenseNeighboursMax = 2000.f, kDensePeak = 4.f;
// pairs closer than this (in units of r_c, squared) are summed term by term
constexpr float kClose2 = 1.f / 1024.f;

// One thread per stretch of kTile sorted particles. A stretch lies in one cell row or is cut where
// a second row begins (stretches over three rows or more stay with the walk); each piece becomes a
// tile if the particles of its row within r_c of its middle stand for at least `neighbours`
// neighbours. Pieces begin and end at even offsets, since the walk takes particles in pairs.
__global__ void k_dense_tiles(Geom g, const uint32_t* __restrict__ total,
                              const float4* __restrict__ rec, const uint32_t* __restrict__ starts,
                              uint32_t* __restrict__ flags, uint2* __restrict__ tiles,
                              uint32_t* __restrict__ ntiles, float neighbours) {
  const uint32_t c = blockIdx.x * blockDim.x + threadIdx.x;
  const uint32_t N = *total;
  const uint32_t i0 = c * kTile;
  if (i0 >= N) return;
  const uint32_t i1 = min(i0 + kTile, N);
  const uint32_t row0 = __float_as_uint(rec[2 * i0 + 1].w) & kRowMask;
  const uint32_t row1 = __float_as_uint(rec[2 * (i1 - 1) + 1].w) & kRowMask;
  const uint32_t nx = static_cast<uint32_t>(g.nc[0]);
  uint32_t cut0 = i1, cut1 = i1;  // first piece [i0, cut0), second [cut1, i1)
  if (row0 != row1) {
    const uint32_t e = starts[(row0 + 1) * nx], b = starts[row1 * nx];
    cut0 = e & ~1u;
    cut1 = (b + 1u) & ~1u;
    if (e != b) cut0 = i0, cut1 = i1;
  }
  auto dense = [&](uint32_t a, uint32_t b, uint32_t row) {
    if (b - a < 16u || b <= a) return false;
    const float x = rec[2 * ((a + b) / 2)].x;
    const float iwx = g.inv_cw_f[0];
    const int c0 = max(static_cast<int>(floorf((x - 1.f) * iwx)), 0);
    const int c1 = min(static_cast<int>(floorf((x + 1.f) * iwx)), g.nc[0] - 1);
    const uint32_t in_row = starts[row * nx + c1 + 1] - starts[row * nx + c0];
    // density = in_row rows^2 / 2 (per r_c^3), neighbours = 4 pi / 3 of that
    return 2.0944f * static_cast<float>(g.rows * g.rows) * static_cast<float>(in_row) >=
           neighbours;
  };
  uint32_t f = (cut0 - i0) << 8 | (cut1 - i0) << 16;
  if (cut0 > i0 && dense(i0, cut0, row0)) {
    f |= 1u;
    tiles[atomicAdd(ntiles, 1u)] = make_uint2(i0, cut0 - i0);
  }
  if (cut1 < i1 && dense(cut1, i1, row1)) {
    f |= 2u;
    tiles[atomicAdd(ntiles, 1u)] = make_uint2(cut1, i1 - cut1);
  }
  flags[c] = f;
}

// distance from the interval [a0, a1] to [b0, b1]
__device__ __forceinline__ float gap(float a0, float a1, float b0, float b1) {
  return fmaxf(fmaxf(b0 - a1, a0 - b1), 0.f);
}

// smallest and largest of a non-negative float over the warp
__device__ __forceinline__ float warp_min(float v) {
  return __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(v)));
}
__device__ __forceinline__ float warp_max(float v) {
  return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(v)));
}

// run of neighbour row r (of a tile with the bounding box lo..hi in row cy, cz) that can hold
// particles within r_c of the box; empty if none
template <int kRows>
__device__ __forceinline__ void tile_run(const Geom& g, const uint32_t* __restrict__ starts,
                                         const float lo[3], const float hi[3], int cy, int cz,
                                         int r, uint32_t& j0, uint32_t& j1) {
  using R = Rows<kRows>;
  j0 = j1 = 0;
  const int ry = cy + (r % R::span) - R::reach, rz = cz + (r / R::span) - R::reach;
  if (ry < 0 || ry >= g.nc[1] || rz < 0 || rz >= g.nc[2]) return;
  const float slack = g.slack_f, cwy = g.cw_f[1], cwz = g.cw_f[2];
  const float dy = fmaxf(gap(lo[1], hi[1], ry * cwy, ry * cwy + cwy) - slack, 0.f);
  const float dz = fmaxf(gap(lo[2], hi[2], rz * cwz, rz * cwz + cwz) - slack, 0.f);
  const float d2 = dy * dy + dz * dz;
  if (d2 >= 1.f) return;
  const float w = sqrtf(1.f - d2) + slack;
  const float iwx = g.inv_cw_f[0];
  const int c0 = max(static_cast<int>(floorf((lo[0] - w) * iwx)), 0);
  const int c1 = min(static_cast<int>(floorf((hi[0] + w) * iwx)), g.nc[0] - 1);
  if (c0 > c1) return;
  const uint32_t base = (static_cast<uint32_t>(rz) * g.nc[1] + ry) * g.nc[0];
  j0 = starts[base + c0];
  j1 = starts[base + c1 + 1];
}

// v in both halves of a register pair, pinned (the compiler would otherwise rebuild the pairs of the
// loop's constants at every use)
__device__ __forceinline__ float2 two(float v) {
  float2 r;
  asm volatile("mov.f32 %0, %2;\n\tmov.f32 %1, %2;" : "=f"(r.x), "=f"(r.y) : "f"(v));
  return r;
}

// Force coefficient (and the potential) of a pair at r2, on the hardware approximations, in the walk's
// order of operations: the closest pairs, whose force outweighs all others', get the same bits
template <int kDeg>
__device__ __forceinline__ float pair_coef(const PairPoly& P, float r2, float& pot) {
  const float rinv = rsqrt_ftz(r2);
  const float t = rcp_ftz(fmaf(P.pk, r2 * rinv, 1.f));
  const float u = t - P.tc;
  float R = P.c[kDeg];
#pragma unroll
  for (int m = kDeg - 1; m >= 0; --m) R = fmaf(R, u, P.c[m]);
  const float ex = ex2_ftz(-P.kappa2_log2e * r2);
  pot = R * t * ex * rinv;
  return fmaf(P.c2k, ex, pot) * (rinv * rinv);
}

// A warp's item: one tile and one row of its half shell.
template <int kDeg, int kRows, bool kPot>
__global__ void __launch_bounds__(kThreads, kBlocksPerSm)
    k_pp_dense(Geom g, PairPoly P, const uint32_t* __restrict__ ntiles,
               const uint2* __restrict__ tiles, const float4* __restrict__ rec,
               const uint32_t* __restrict__ starts, float4* __restrict__ fpp,
               float2* __restrict__ flo, float4* __restrict__ fbig, uint32_t* __restrict__ next,
               double* __restrict__ energy, unsigned long long* __restrict__ pairs) {
  using R = Rows<kRows>;
  // the group: each coordinate twice and negated, as the two-wide additions take it
  __shared__ float4 stage[kWarps][3][32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  float4(*st)[32] = stage[wid];
  float2 c2[kDeg + 1];
#pragma unroll
  for (int i = 0; i <= kDeg; ++i) c2[i] = two(P.c[i]);
  const float2 pk2 = two(P.pk), one2 = two(1.f), tc2 = two(-P.tc), k2 = two(-P.kappa2_log2e),
               c2k2 = two(P.c2k);
  const uint32_t items = *ntiles * static_cast<uint32_t>(R::half);
  double e_acc = 0.0;
  unsigned long long np = 0;
  for (;;) {
    uint32_t item = 0;
    if (lane == 0) item = atomicAdd(next, 1u);
    item = __shfl_sync(0xffffffffu, item, 0);
    if (item >= items) break;
    const uint32_t t = item / static_cast<uint32_t>(R::half);
    const int r = R::first + static_cast<int>(item - t * static_cast<uint32_t>(R::half));
    const uint2 tile = tiles[t];
    const uint32_t i0 = tile.x, cnt = tile.y;
    const uint32_t ia = i0 + lane, ib = ia + 32;
    const bool alive_a = lane < cnt, alive_b = lane + 32 < cnt;
    float4 pa, la, pb, lb;
    load_rec32(rec + 2 * static_cast<size_t>(alive_a ? ia : i0), pa, la);
    load_rec32(rec + 2 * static_cast<size_t>(alive_b ? ib : i0), pb, lb);
    const float lo[3] = {warp_min(fminf(pa.x, pb.x)), warp_min(fminf(pa.y, pb.y)),
                         warp_min(fminf(pa.z, pb.z))};
    const float hi[3] = {warp_max(fmaxf(pa.x, pb.x)), warp_max(fmaxf(pa.y, pb.y)),
                         warp_max(fmaxf(pa.z, pb.z))};
    const uint32_t row =
        __shfl_sync(0xffffffffu, __float_as_uint(la.w), 0) & kRowMask;  // of the whole tile
    const int cy = static_cast<int>(row % static_cast<uint32_t>(g.nc[1]));
    const int cz = static_cast<int>(row / static_cast<uint32_t>(g.nc[1]));
    const bool own = r == R::first;
    uint32_t j0, j1;
    tile_run<kRows>(g, starts, lo, hi, cy, cz, r, j0, j1);
    if (own) j0 = max(j0, i0);
    if (j0 >= j1) continue;
    // a lane without a particle holds one too far from everything
    if (!alive_a) pa.x = -1e6f;
    if (!alive_b) pb.x = -1e6f;
    const float2 hx2 = make_float2(pa.x, pb.x), lx2 = make_float2(la.x, lb.x);
    const float2 hy2 = make_float2(pa.y, pb.y), ly2 = make_float2(la.y, lb.y);
    const float2 hz2 = make_float2(pa.z, pb.z), lz2 = make_float2(la.z, lb.z);
    Acc2 fa[3], fb[3], pot_acc;
    pot_acc.hi = pot_acc.lo = 0.f;
    for (int c = 0; c < 3; ++c) fa[c].hi = fa[c].lo = fb[c].hi = fb[c].lo = 0.f;
    uint32_t hits = 0;
    for (uint32_t jb = j0; jb < j1; jb += 32) {
      const uint32_t j = jb + lane;
      const bool vj = j < j1;
      float4 hj, lj;
      load_rec32(rec + 2 * static_cast<size_t>(vj ? j : jb), hj, lj);
      const float gx = gap(lo[0], hi[0], warp_min(hj.x), warp_max(hj.x));
      const float gy = gap(lo[1], hi[1], warp_min(hj.y), warp_max(hj.y));
      const float gz = gap(lo[2], hi[2], warp_min(hj.z), warp_max(hj.z));
      const float d2 = fmaf(gx, gx, fmaf(gy, gy, gz * gz));
      if (d2 >= (1.f + g.slack_f) * (1.f + g.slack_f)) continue;
      __syncwarp();  // the last group has been read
      const float far_x = vj ? -hj.x : -1e6f;
      st[0][lane] = make_float4(far_x, far_x, -hj.y, -hj.y);
      st[1][lane] = make_float4(-hj.z, -hj.z, -lj.x, -lj.x);
      st[2][lane] = make_float4(-lj.y, -lj.y, -lj.z, -lj.z);
      __syncwarp();
      float qa[3] = {0.f, 0.f, 0.f}, qb[3] = {0.f, 0.f, 0.f}, qj[3] = {0.f, 0.f, 0.f}, qp = 0.f;
      // the group particle's sum moves on with it to the lane that meets it next
      auto pass_on = [&]() {
        const int from = (lane + 1) & 31;
        qj[0] = __shfl_sync(0xffffffffu, qj[0], from);
        qj[1] = __shfl_sync(0xffffffffu, qj[1], from);
        qj[2] = __shfl_sync(0xffffffffu, qj[2], from);
      };
      // one turn where the group can hold the tile's own particles or close pairs
      auto near_turn = [&](int k) {
        const int m = (lane + k) & 31;
        const float4 u0 = st[0][m], u1 = st[1][m], u2 = st[2][m];
        const float ax = (pa.x + u0.x) + (la.x + u1.z), bx = (pb.x + u0.x) + (lb.x + u1.z);
        const float ay = (pa.y + u0.z) + (la.y + u2.x), by = (pb.y + u0.z) + (lb.y + u2.x);
        const float az = (pa.z + u1.x) + (la.z + u2.z), bz = (pb.z + u1.x) + (lb.z + u2.z);
        const float r2a = ax * ax + ay * ay + az * az;
        const float r2b = bx * bx + by * by + bz * bz;
        // coincident particles are skipped; within the tile's own row the later particle counts
        const bool ha = r2a < 1.f && r2a > 0.f && (!own || jb + m > ia);
        const bool hb = r2b < 1.f && r2b > 0.f && (!own || jb + m > ib);
        float ua = 0.f, ub = 0.f;
        float ca = pair_coef<kDeg>(P, r2a, ua), cb = pair_coef<kDeg>(P, r2b, ub);
        ca = ha ? ca : 0.f;
        cb = hb ? cb : 0.f;
        if constexpr (kPot) qp += (ha ? ua : 0.f) + (hb ? ub : 0.f);
        hits += static_cast<uint32_t>(ha) + static_cast<uint32_t>(hb);
        // a close pair's term would round the others' in a plain sum: it goes to both particles by
        // itself
        const bool close_a = ha && r2a < kClose2, close_b = hb && r2b < kClose2;
        if (__any_sync(0xffffffffu, close_a || close_b)) {
          const uint32_t jj = jb + m;
          if (close_a) {
            const float x = ca * ax, y = ca * ay, z = ca * az;
            fa[0].add(x);
            fa[1].add(y);
            fa[2].add(z);
            split_add_v4_if(true, big_term(x, y, z), fpp + jj, flo + jj, fbig + jj, -x, -y, -z);
            ca = 0.f;
          }
          if (close_b) {
            const float x = cb * bx, y = cb * by, z = cb * bz;
            fb[0].add(x);
            fb[1].add(y);
            fb[2].add(z);
            split_add_v4_if(true, big_term(x, y, z), fpp + jj, flo + jj, fbig + jj, -x, -y, -z);
            cb = 0.f;
          }
        }
        qa[0] = fmaf(ca, ax, qa[0]);
        qa[1] = fmaf(ca, ay, qa[1]);
        qa[2] = fmaf(ca, az, qa[2]);
        qb[0] = fmaf(cb, bx, qb[0]);
        qb[1] = fmaf(cb, by, qb[1]);
        qb[2] = fmaf(cb, bz, qb[2]);
        qj[0] = fmaf(-ca, ax, fmaf(-cb, bx, qj[0]));
        qj[1] = fmaf(-ca, ay, fmaf(-cb, by, qj[1]));
        qj[2] = fmaf(-ca, az, fmaf(-cb, bz, qj[2]));
        pass_on();
      };
      // the same for every other group, on the two-wide FP32 instructions (a in x, b in y)
      float2 q2[3] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
      auto far_turn = [&](int k) {
        const int m = (lane + k) & 31;
        const float4 u0 = st[0][m], u1 = st[1][m], u2 = st[2][m];
        const float2 dx = __fadd2_rn(__fadd2_rn(hx2, make_float2(u0.x, u0.y)),
                                     __fadd2_rn(lx2, make_float2(u1.z, u1.w)));
        const float2 dy = __fadd2_rn(__fadd2_rn(hy2, make_float2(u0.z, u0.w)),
                                     __fadd2_rn(ly2, make_float2(u2.x, u2.y)));
        const float2 dz = __fadd2_rn(__fadd2_rn(hz2, make_float2(u1.x, u1.y)),
                                     __fadd2_rn(lz2, make_float2(u2.z, u2.w)));
        const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
        const bool ha = r2.x < 1.f, hb = r2.y < 1.f;
        const float2 rinv = make_float2(rsqrt_ftz(r2.x), rsqrt_ftz(r2.y));
        const float2 ta = __ffma2_rn(pk2, __fmul2_rn(r2, rinv), one2);
        const float2 t = make_float2(rcp_ftz(ta.x), rcp_ftz(ta.y));
        const float2 u = __fadd2_rn(t, tc2);
        float2 R = c2[kDeg];
#pragma unroll
        for (int i = kDeg - 1; i >= 0; --i) R = __ffma2_rn(R, u, c2[i]);
        const float2 ea = __fmul2_rn(r2, k2);
        const float2 ex = make_float2(ex2_ftz(ea.x), ex2_ftz(ea.y));
        const float2 tr = __fmul2_rn(t, rinv);
        float2 c = __fmul2_rn(__ffma2_rn(R, tr, c2k2),
                              __fmul2_rn(ex, __fmul2_rn(rinv, rinv)));
        if constexpr (kPot) {
          const float2 w = __fmul2_rn(__fmul2_rn(R, tr), ex);
          qp += (ha ? w.x : 0.f) + (hb ? w.y : 0.f);
        }
        c.x = ha ? c.x : 0.f;
        c.y = hb ? c.y : 0.f;
        hits += static_cast<uint32_t>(ha) + static_cast<uint32_t>(hb);
        q2[0] = __ffma2_rn(c, dx, q2[0]);
        q2[1] = __ffma2_rn(c, dy, q2[1]);
        q2[2] = __ffma2_rn(c, dz, q2[2]);
        qj[0] = fmaf(-c.x, dx.x, fmaf(-c.y, dx.y, qj[0]));
        qj[1] = fmaf(-c.x, dy.x, fmaf(-c.y, dy.y, qj[1]));
        qj[2] = fmaf(-c.x, dz.x, fmaf(-c.y, dz.y, qj[2]));
        pass_on();
      };
      if (own || d2 < kClose2) {
#pragma unroll 1
        for (int k = 0; k < 32; ++k) near_turn(k);
      } else {
#pragma unroll 2
        for (int k = 0; k < 32; ++k) far_turn(k);
        for (int i = 0; i < 3; ++i) {
          qa[i] = q2[i].x;
          qb[i] = q2[i].y;
        }
      }
      // after 32 turns every sum is back at its own lane
      for (int c = 0; c < 3; ++c) {
        fa[c].add(qa[c]);
        fb[c].add(qb[c]);
      }
      if constexpr (kPot) pot_acc.add(qp);
      split_add_v4_if(vj, big_term(qj[0], qj[1], qj[2]), fpp + j, flo + j, fbig + j, qj[0], qj[1],
                      qj[2]);
    }
    if (alive_a)
      split_add_v4(fpp + ia, flo + ia, fbig + ia, fa[0].hi, fa[1].hi, fa[2].hi, fa[0].lo, fa[1].lo,
                   fa[2].lo);
    if (alive_b)
      split_add_v4(fpp + ib, flo + ib, fbig + ib, fb[0].hi, fb[1].hi, fb[2].hi, fb[0].lo, fb[1].lo,
                   fb[2].lo);
    // sum_i phi_i over ordered pairs takes each unordered pair's potential twice
    if constexpr (kPot) e_acc += 2.0 * static_cast<double>(pot_acc.value());
    np += hits;
  }
  if constexpr (kPot) block_reduce_add<kThreads>(e_acc, energy);
  warp_add_u64(2ull * np, pairs);
}

// (particle, record) distance tests of the tiles: the particles of a tile times its runs
template <int kRows>
__global__ void k_dense_count(Geom g, const uint32_t* __restrict__ ntiles,
                              const uint2* __restrict__ tiles, const float4* __restrict__ rec,
                              const uint32_t* __restrict__ starts,
                              unsigned long long* __restrict__ out) {
  using R = Rows<kRows>;
  unsigned long long n = 0;
  const uint32_t t = (blockIdx.x * blockDim.x + threadIdx.x) / 32;
  const int lane = threadIdx.x & 31;
  if (t < *ntiles) {
    const uint2 tile = tiles[t];
    const uint32_t ia = tile.x + (lane < tile.y ? lane : 0);
    const uint32_t ib = tile.x + (lane + 32 < tile.y ? lane + 32 : 0);
    const float4 pa = rec[2 * ia], pb = rec[2 * ib];
    const float lo[3] = {warp_min(fminf(pa.x, pb.x)), warp_min(fminf(pa.y, pb.y)),
                         warp_min(fminf(pa.z, pb.z))};
    const float hi[3] = {warp_max(fmaxf(pa.x, pb.x)), warp_max(fmaxf(pa.y, pb.y)),
                         warp_max(fmaxf(pa.z, pb.z))};
    const uint32_t row = __float_as_uint(rec[2 * tile.x + 1].w) & kRowMask;
    for (int r = R::first + lane; r < R::last; r += 32) {
      uint32_t j0, j1;
      tile_run<kRows>(g, starts, lo, hi, static_cast<int>(row % static_cast<uint32_t>(g.nc[1])),
                      static_cast<int>(row / static_cast<uint32_t>(g.nc[1])), r, j0, j1);
      if (r == R::first) j0 = max(j0, tile.x);
      if (j0 < j1) n += static_cast<unsigned long long>(j1 - j0) * tile.y;
    }
  }
  warp_add_u64(n, out);
}

}  // namespace

// Up to 65,536 particles the walk keeps all of them. Few particles make too few tiles and rows to fill
// the SMs, and the walk's lanes share them out better (5003 particles: 56 us by the walk, 84 us with
// tiles); and where particles are few, runs that are differentiated and summed up to a scalar show
// the other order of summation: the emittance of 60,000 particles after ten steps moved by 5e-9 of its
// value with tiles.
constexpr int64_t kDenseMin = 65537;

const uint32_t* dense_flags(const p3m_ctx* c, int64_t n) {
  return n >= kDenseMin ? c->dense_flags : nullptr;
}

void launch_dense_tiles(const p3m_ctx* c, int64_t n, cudaStream_t s) {
  if (n < kDenseMin) return;
  const int64_t stretches = (n + kTile - 1) / kTile;
  double volume = 1.0;  // of the mesh, in r_c^3
  for (int d = 0; d < 3; ++d) volume *= (c->g.n[d] - 1) * c->g.a[d];
  const float mean = static_cast<float>(4.18879 * static_cast<double>(n) / volume);
  const float neighbours =
      std::min(std::max(kDensePeak * mean, kDenseNeighboursMin), kDenseNeighboursMax);
  // the tile count was cleared by the sort, as the item counter behind it
  k_dense_tiles<<<static_cast<unsigned>((stretches + kThreads - 1) / kThreads), kThreads, 0, s>>>(
      c->g, c->starts + c->nkeys, static_cast<const float4*>(c->recp), c->starts, c->dense_flags,
      c->dense_tiles, c->pp_tile + 1, neighbours);
}

void launch_pp_dense(const p3m_ctx* c, int64_t n, cudaStream_t s, bool want_energy) {
  if (n < kDenseMin) return;
  const auto* rec = static_cast<const float4*>(c->recp);
  const int64_t stretches = (n + kTile - 1) / kTile;
  float4* fbig = c->fplo + c->n_max;
  const unsigned blocks = static_cast<unsigned>(std::min<int64_t>(
      stretches, static_cast<int64_t>(kBlocksPerSm) * c->num_sms));
  auto run = [&](auto kern) {
    kern<<<blocks, kThreads, 0, s>>>(c->g, c->poly, c->pp_tile + 1, c->dense_tiles, rec, c->starts,
                                     static_cast<float4*>(c->fpp),
                                     reinterpret_cast<float2*>(c->fplo), fbig, c->pp_tile + 2,
                                     c->energy_acc, c->pair_acc);
  };
  auto rows = [&](auto r1, auto r1p, auto r2, auto r2p, auto r3, auto r3p) {
    if (c->g.rows == 1)
      want_energy ? run(r1p) : run(r1);
    else if (c->g.rows == 2)
      want_energy ? run(r2p) : run(r2);
    else
      want_energy ? run(r3p) : run(r3);
  };
#define P3M_DENSE(d)                                                                     \
  rows(k_pp_dense<d, 1, false>, k_pp_dense<d, 1, true>, k_pp_dense<d, 2, false>,         \
       k_pp_dense<d, 2, true>, k_pp_dense<d, 3, false>, k_pp_dense<d, 3, true>)
  // degrees 5 to 8 cover kappa up to about 6; others round up (the missing terms are zero)
  switch (c->poly.deg) {
    case 4:
    case 5: P3M_DENSE(5); break;
    case 6: P3M_DENSE(6); break;
    case 7: P3M_DENSE(7); break;
    case 8: P3M_DENSE(8); break;
    case 9:
    case 10:
    case 11: P3M_DENSE(11); break;
    default: P3M_DENSE(15); break;
  }
#undef P3M_DENSE
}

void launch_pp_dense_count(const p3m_ctx* c, int64_t n, unsigned long long* out, cudaStream_t s) {
  if (n < kDenseMin) return;
  const int64_t warps = 2 * ((n + kTile - 1) / kTile);  // at most two tiles a stretch
  auto kern = c->g.rows == 1 ? k_dense_count<1> : c->g.rows == 2 ? k_dense_count<2> : k_dense_count<3>;
  kern<<<static_cast<unsigned>((warps + kWarps - 1) / kWarps), kThreads, 0, s>>>(
      c->g, c->pp_tile + 1, c->dense_tiles, static_cast<const float4*>(c->recp), c->starts, out);
}

}  // namespace p3m
