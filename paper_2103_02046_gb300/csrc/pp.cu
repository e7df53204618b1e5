// Short-range (particle-particle) half of P3M, eq. (summation_short) with the screened kernel
// G^S(r) = erfc(a r)/r of eq. (ewald_split); the self term is omitted. For r = |xi_i - xi_j|
// below the cutoff r_c the force on i is
//   k_e q^2 [erfc(a r)/r + (2a/sqrt(pi)) e^{-a^2 r^2}] (xi_i - xi_j) / r^2.
// With pp_bc = 1 the cathode also enters the short range (Sec. 3.1.1): each particle j has an
// image of charge -q at S(xi_j) (its own image included) that acts through the same kernel.
//
// Work is in cutoff units (rho = r / r_c, kappa = a r_c): the force is
// (k_e q^2 / r_c^2) [erfc(kappa rho)/rho + (2 kappa/sqrt(pi)) e^{-kappa^2 rho^2}] rho_vec / rho^2.
//
// Search: cells are rows along x (r_c / R wide in y and z, R = Geom::rows = 2, or 1 at low
// density; r_c / nsub in x; keys x-fastest). For particle i and each of the (2R + 1)^2
// neighbour rows, the distance d from i to the row's (y, z) rectangle bounds |dx| < sqrt(1 - d^2),
// which selects one contiguous run of sorted particles; rows with d >= 1 are skipped. With R = 2
// this visits about 8 r_c^3 of volume per particle (the cutoff sphere is 4.19 r_c^3) instead of
// the 27 r_c^3 of a plain 27-cell stencil.
//
// FP32: every candidate's separation is (hi_i - hi_j) + (lo_i - lo_j) of the cutoff-unit
// positions, exact to FP32 relative rounding at any distance. Partial sums are folded into a
// two-float (TwoSum) accumulator every few steps, so the per-particle sum is compensated at a
// small fraction of an addition per pair.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "pp_f32.cuh"

namespace p3m {
namespace {

constexpr int kThreads = 128;

// ------------------------------------------------------------------------------------------
// FP32 short range: each unordered pair once (Newton's third law), each lane holding two
// particles and walking their candidate lists in lockstep with the other lanes.
//
// Pairs: particle i takes the pairs (i, j) with j > i in sorted order. Sorted order is row-major
// over (z row, y row, x cell), so these are the later part of i's own row and the neighbour
// rows after it (dz > 0, or dz = 0 and dy > 0) -- 13 of 25 rows, or 5 of 9. i's row is the one
// the sort put it in (stored with the record), so every pair is taken by exactly one of its
// particles.
//
// Lanes: lane l of a tile holds the sorted particles a = 2l and b = 2l + 1 (adjacent in sorted
// order, so nearly always in the same row and a quarter cutoff apart or less). Per neighbour row
// the lane walks the hull of the two particles' runs and tests every loaded record against
// both: one 256-bit load serves two particles, which halves the record traffic of the short
// range (the L1 data pipe bounds this kernel). Each pair is still taken exactly once: a pair
// (i, j) counts only when j > i and |xi_i - xi_j| < r_c, and the hull holds no record twice.
// When a and b lie in different rows (a row boundary) the lane keeps both run lists, each
// tested against its own particle only.
//
// The force on a and b accumulates in registers; the reaction on j (both particles' share) goes
// to j by one predicated vector reduction (red.global.add.v4.f32) into the zeroed result array,
// and a's and b's own sums are added the same way at the end.
//
// Walk: each lane first writes its non-empty runs (at most 13, or 26 across a row boundary) to
// shared memory, then the warp steps through them together, two records per lane per step; a
// lane moves on to its next run as soon as one ends. Lanes with nothing left re-read record 0
// with every result masked. The step is straight-line code: the pair function runs for every
// lane and candidate and its results are selected by the hit predicate, since with 64 lane
// candidates per step some lane nearly always holds a pair. Separations are exact to FP32
// relative rounding ((hi_i - hi_j) + (lo_i - lo_j)). FP32 partial sums are folded into a
// two-float (TwoSum) accumulator every 16 steps.
// The pair function uses one ex2 for both e^{-kappa^2 rho^2} terms and the fitted form
// R(x) = erfc(x) e^{x^2} = t P(u), t = 1 / (1 + p x): erfc(kappa rho) = R * e^{-kappa^2 rho^2};
// rsqrt, rcp and ex2 are the hardware approximations (flush-to-zero: every argument here is a
// normal number).
// ------------------------------------------------------------------------------------------
constexpr int kPpThreads = 128;     // threads per block of the FP32 short range
constexpr int kPpBlocksPerSm = 6;    // resident blocks per SM of the short range (80 registers)
// Lanes that share a pair of particles and split its half-shell rows: 1, doubled (to 16 at most)
// while the lanes would not fill the resident blocks. Short range with 1, 2, 4, 8, 16 lanes:
// 5003 particles 308, 183, 126, 89, 73 us; 131,072 (dense) 3.57, 2.70, 1.88, 1.95, 2.00 ms;
// 261,121 (sphere) 184, 155, 156, 175, 214 us; 2,097,152 748 us (1), 846, 949 (2, 4).
constexpr int kPpMaxLogParts = 4;

// pair_poly on the hardware approximations; r2 in (0, 1]
template <int kDeg>
__device__ __forceinline__ void pair_poly_hw(const PairPoly& P, float r2, float& fco,
                                             float& pot) {
  const float rinv = rsqrt_ftz(r2);
  const float rho = r2 * rinv;
  const float R = erfcx_poly<kDeg, true>(P, rho);
  const float ex = ex2_ftz(-P.kappa2_log2e * r2);
  pot = R * ex * rinv;
  fco = fmaf(P.c2k, ex, pot) * (rinv * rinv);
}

template <int kDeg>
__device__ __forceinline__ void pair_poly(const PairPoly& P, float r2, float& fco, float& pot) {
  const float rinv = rsqrtf(r2);
  const float rho = r2 * rinv;
  const float R = erfcx_poly<kDeg, false>(P, rho);
  const float ex = exp2f(-P.kappa2_log2e * r2);
  pot = R * ex * rinv;
  fco = fmaf(P.c2k, ex, pot) * (rinv * rinv);
}

// b's own runs (particle ib in row row_b), for a lane whose two particles sit in different rows
template <int kRows, typename Emit>
__device__ __forceinline__ void b_runs(const Geom& g, const uint32_t* __restrict__ starts,
                                       const float4& pb, const float4& lb, uint32_t ib, int part,
                                       int parts, Emit&& emit) {
  constexpr int kFirst = Rows<kRows>::first, kLast = Rows<kRows>::last;  // half shell
  const uint32_t row_b = __float_as_uint(lb.w) & kRowMask;
  const int cyb = static_cast<int>(row_b % static_cast<uint32_t>(g.nc[1]));
  const int czb = static_cast<int>(row_b / static_cast<uint32_t>(g.nc[1]));
#pragma unroll 1
  for (int r = kFirst + part; r < kLast; r += parts) {
    uint32_t j0, j1;
    row_range<kRows>(g, starts, pb.x, pb.y, pb.z, cyb, czb, r, j0, j1);
    j0 = max(j0, ib + 1);
    if (j0 < j1) emit(j0, j1);
  }
}

// The runs of the lane holding sorted particles a = ia and b = ia + 1 (b only if alive_b),
// in walk order: emit(j0, j1) for each non-empty run. With a and b in one row (same) each run is
// the hull of the two particles' runs in one neighbour row and is tested against both;
// otherwise a's runs come first (split of them) and are tested against a only, then b's
// (unless kOnlyA: the caller then takes b's runs later, from b_runs). Of the half shell's rows the
// lane takes every parts-th from row number part on (lanes that share a pair split its rows).
template <int kRows, bool kOnlyA = false, typename Emit>
__device__ __forceinline__ void pair_runs(const Geom& g, const uint32_t* __restrict__ starts,
                                          const float4& pa, const float4& la, const float4& pb,
                                          const float4& lb, uint32_t ia, bool alive_b, int part,
                                          int parts, bool& same, int& split, Emit&& emit) {
  constexpr int kFirst = Rows<kRows>::first, kLast = Rows<kRows>::last;  // half shell
  const uint32_t ib = ia + 1;
  const uint32_t row_a = __float_as_uint(la.w) & kRowMask;
  const uint32_t row_b = __float_as_uint(lb.w) & kRowMask;
  same = !alive_b || row_a == row_b;
  const int cya = static_cast<int>(row_a % static_cast<uint32_t>(g.nc[1]));
  const int cza = static_cast<int>(row_a / static_cast<uint32_t>(g.nc[1]));
  int n = 0;
#pragma unroll 1
  for (int r = kFirst + part; r < kLast; r += parts) {
    uint32_t j0, j1;
    row_range<kRows>(g, starts, pa.x, pa.y, pa.z, cya, cza, r, j0, j1);
    j0 = max(j0, ia + 1);  // own row: only the particles after a (a no-op for later rows)
    if (same && alive_b) {
      uint32_t k0, k1;
      row_range<kRows>(g, starts, pb.x, pb.y, pb.z, cya, cza, r, k0, k1);
      k0 = max(k0, ib + 1);
      if (k0 < k1) {
        j0 = j0 < j1 ? min(j0, k0) : k0;
        j1 = max(j1, k1);
      }
    }
    if (j0 < j1) {
      emit(j0, j1);
      ++n;
    }
  }
  split = n;
  if (!kOnlyA && !same) b_runs<kRows>(g, starts, pb, lb, ib, part, parts, emit);
}

// Run slots per lane of k_pp_f32: a's and b's runs, up to twice the half shell when their rows
// differ. With 3 rows per cutoff (25 half-shell rows) that would not fit beside 6 blocks per
// SM: a lane whose particles sit in different rows then walks a's runs first and b's after
// them, in the same slots.
__host__ __device__ constexpr int pp_pair_runs(int rows) {
  return (rows >= 3 ? 1 : 2) * ((2 * rows + 1) * (2 * rows + 1) - (2 * rows + 1) * (2 * rows + 1) / 2);
}
inline size_t pp_run_bytes(int rows) {
  return 2 * sizeof(uint32_t) * static_cast<size_t>(pp_pair_runs(rows)) * kPpThreads;
}

// Work stealing inside a warp: once at least kStealMin lanes have walked all their runs, each
// of them takes work from a lane that still has some: that lane's last unstarted run, or else
// the back half of its current run if at least 2 kStealRecs records are left of it. The thief
// first sends the sums of the pair it held to their force arrays, then adopts the donor's pair
// (positions, index, which of the two the run is tested against) with zeroed sums, which it
// sends out in turn when it is done or steals again; the reduction targets are shared, so the
// owner's force is the sum of its holders' parts. This takes the warp's step count from the
// maximum of its lanes' walks towards their mean.
constexpr int kStealMin = 8;
constexpr uint32_t kStealRecs = 4;

__device__ __forceinline__ float4 shfl_f4(float4 v, int src) {
  v.x = __shfl_sync(0xffffffffu, v.x, src);
  v.y = __shfl_sync(0xffffffffu, v.y, src);
  v.z = __shfl_sync(0xffffffffu, v.z, src);
  v.w = __shfl_sync(0xffffffffu, v.w, src);
  return v;
}

// Pairs with images (pp_bc), for the particles less than r_c above the cathode: image pairs act on
// the particle only. A kernel of its own, since inside k_pp_f32 its registers would spill those of
// the walk (0 -> 20 bytes; 801 -> 820 us on the 2M sphere). The sort is z-major, so these particles
// are among the first `near` sorted ones; kImgLanes lanes share one and split the rows around its
// image point.
constexpr int kImgLanes = 8;

template <int kDeg>
__global__ void __launch_bounds__(kThreads)
    k_pp_images(Geom g, PairPoly P, uint32_t near_cell, const float4* __restrict__ rec,
                const uint32_t* __restrict__ starts, float4* __restrict__ fpp,
                float2* __restrict__ flo, float4* __restrict__ fbig, double* __restrict__ energy,
                unsigned long long* __restrict__ pairs) {
  const uint32_t near = starts[near_cell];
  const int part = threadIdx.x & (kImgLanes - 1);
  const float ch = static_cast<float>(g.img_c);
  const float cl = static_cast<float>(g.img_c - static_cast<double>(ch));
  double e_acc = 0.0;
  unsigned long long ni = 0;
  for (uint32_t i = (blockIdx.x * kThreads + threadIdx.x) / kImgLanes; i < near;
       i += gridDim.x * (kThreads / kImgLanes)) {
    const float4 p = rec[2 * i], l = rec[2 * i + 1];
    const double zi = static_cast<double>(p.z) + static_cast<double>(l.z);
    if (zi - 0.5 * g.img_c >= 1.0) continue;
    const float mz = static_cast<float>(g.img_c - zi);
    Acc2 sum[3];
    for (int c = 0; c < 3; ++c) sum[c].hi = sum[c].lo = 0.f;
    for_rows<float>(g, starts, p.x, p.y, mz, part, kImgLanes, [&](uint32_t ja, uint32_t jb) {
      float rowv[4] = {0.f, 0.f, 0.f, 0.f};
      for (uint32_t jj = ja; jj < jb; ++jj) {
        const float4 hj = rec[2 * jj], lj = rec[2 * jj + 1];
        const float ax = (p.x - hj.x) + (l.x - lj.x);
        const float ay = (p.y - hj.y) + (l.y - lj.y);
        const float s = p.z + hj.z;
        const float bp = s - p.z;
        const float e = (p.z - (s - bp)) + (hj.z - bp);
        const float az = ((s - ch) + e) + ((l.z + lj.z) - cl);
        const float r2 = ax * ax + ay * ay + az * az;
        if (r2 < 1.f && r2 > 0.f) {
          float fco, pot;
          pair_poly<kDeg>(P, r2, fco, pot);
          rowv[0] -= fco * ax;
          rowv[1] -= fco * ay;
          rowv[2] -= fco * az;
          rowv[3] -= pot;
          ++ni;
        }
      }
      for (int c = 0; c < 3; ++c) sum[c].add(rowv[c]);
      e_acc += static_cast<double>(rowv[3]);
    });
    split_add_v4(fpp + i, flo + i, fbig + i, sum[0].hi, sum[1].hi, sum[2].hi, sum[0].lo, sum[1].lo,
                 sum[2].lo);
  }
  block_reduce_add<kThreads>(e_acc, energy);
  warp_add_u64(ni, pairs + 1);
}

template <int kDeg, int kRows>
__global__ void __launch_bounds__(kPpThreads, kPpBlocksPerSm)
    k_pp_f32(Geom g, PairPoly P, const uint32_t* __restrict__ total,
             const float4* __restrict__ rec, const uint32_t* __restrict__ starts,
             float4* __restrict__ fpp, float2* __restrict__ flo, float4* __restrict__ fbig,
             uint32_t* __restrict__ next_tile, int log_parts,
             const uint32_t* __restrict__ dense,
             double* __restrict__ energy, unsigned long long* __restrict__ pairs) {
  // particles per tile: two a lane, or two for the 2^log_parts lanes that share a pair's rows
  const uint32_t kTile = (2 * kPpThreads) >> log_parts;
  const int parts = 1 << log_parts, part = threadIdx.x & (parts - 1);
  constexpr bool kPhased = kRows >= 3;
  constexpr int kPairRuns = pp_pair_runs(kRows);
  static_assert(kPairRuns == (kPhased ? 1 : 2) * Rows<kRows>::half, "run slots");
  // the lanes' runs, [kPairRuns][kPpThreads] each, in dynamic shared memory
  extern __shared__ uint32_t pp_runs[];
  uint32_t(*run_j0)[kPpThreads] = reinterpret_cast<uint32_t(*)[kPpThreads]>(pp_runs);
  uint32_t(*run_j1)[kPpThreads] = run_j0 + kPairRuns;
  __shared__ uint8_t donor_s[kPpThreads / 32][32];
  __shared__ uint32_t tile_s;
  const int tid = threadIdx.x;
  const int lane = tid & 31;
  const uint32_t N = *total;
  double e_acc = 0.0;
  unsigned long long np = 0;
  // persistent blocks: each takes the next tile of kTile sorted particles until none is left
  // (the block's four warps work on adjacent particles, which share most of their neighbours
  // in L1)
  for (;;) {
    if (tid == 0) tile_s = atomicAdd(next_tile, 1u);
    __syncthreads();
    const uint32_t tile = tile_s;
    __syncthreads();
    if (static_cast<uint64_t>(tile) * kTile >= N) break;
    // the pair the lane holds: a = ia, b = ia + 1 (a thief adopts another lane's pair)
    uint32_t ia = tile * kTile + 2 * (tid >> log_parts);
    bool alive_a = ia < N, alive_b = ia + 1 < N;
    if (dense && alive_a && in_dense_tile(dense, ia)) alive_a = alive_b = false;
    // lanes past the last particle read record 0 (in bounds) and take part in the lockstep
    // loop with every result masked out
    const uint32_t ea = alive_a ? ia : 0u, eb = alive_b ? ia + 1 : ea;
    float4 pa = rec[2 * ea], la = rec[2 * ea + 1];
    float4 pb = rec[2 * eb], lb = rec[2 * eb + 1];
    // runs: with a and b in one row, the hull of their two runs per neighbour row (tested
    // against both); otherwise a's runs [0, split) and b's runs [split, cnt) (kPhased: a's
    // runs, then b's in their place once they are walked, while pending_b)
    int cnt = 0, split = 0;
    bool same = true;
    auto emit = [&](uint32_t j0, uint32_t j1) {
      run_j0[cnt][tid] = j0;
      run_j1[cnt][tid] = j1;
      ++cnt;
    };
    if (alive_a)
      pair_runs<kRows, kPhased>(g, starts, pa, la, pb, lb, ia, alive_b, part, parts, same, split,
                                emit);
    bool pending_b = kPhased && alive_a && !same;
    uint32_t ptr = 0, end = 0;
    int k = 0;
    if (cnt > 0) {
      ptr = run_j0[0][tid];
      end = run_j1[0][tid];
    }
    bool ta = same || split > 0;                               // the current run is tested against a
    bool tb = alive_b && (same || (!kPhased && split == 0));   // ... and against b
    Acc2 sa[4], sb[4];
    for (int c = 0; c < 4; ++c) sa[c].hi = sa[c].lo = sb[c].hi = sb[c].lo = 0.f;
    float qa[4] = {0.f, 0.f, 0.f, 0.f}, qb[4] = {0.f, 0.f, 0.f, 0.f};
    uint32_t np_part = 0;
    // the held pair's sums (hi + lo of the compensated accumulators) to its force arrays, split
    // like the reactions, and zeroed; sum_i phi_i over ordered pairs takes each unordered
    // pair's potential twice
    auto flush = [&]() {
      for (int c = 0; c < 4; ++c) {
        sa[c].add(qa[c]);
        sb[c].add(qb[c]);
        qa[c] = qb[c] = 0.f;
      }
      if (alive_a) {
        split_add_v4(fpp + ia, flo + ia, fbig + ia, sa[0].hi, sa[1].hi, sa[2].hi, sa[0].lo,
                     sa[1].lo, sa[2].lo);
        e_acc += 2.0 * static_cast<double>(sa[3].value());
      }
      if (alive_b) {
        split_add_v4(fpp + ia + 1, flo + ia + 1, fbig + ia + 1, sb[0].hi, sb[1].hi, sb[2].hi,
                     sb[0].lo, sb[1].lo, sb[2].lo);
        e_acc += 2.0 * static_cast<double>(sb[3].value());
      }
      for (int c = 0; c < 4; ++c) sa[c].hi = sa[c].lo = sb[c].hi = sb[c].lo = 0.f;
    };
    // one candidate record j (hj, lj) against a and b
    auto cand = [&](bool v, uint32_t j, const float4& hj, const float4& lj) {
      const float ax = (pa.x - hj.x) + (la.x - lj.x);
      const float ay = (pa.y - hj.y) + (la.y - lj.y);
      const float az = (pa.z - hj.z) + (la.z - lj.z);
      const float bx = (pb.x - hj.x) + (lb.x - lj.x);
      const float by = (pb.y - hj.y) + (lb.y - lj.y);
      const float bz = (pb.z - hj.z) + (lb.z - lj.z);
      const float r2a = ax * ax + ay * ay + az * az;
      const float r2b = bx * bx + by * by + bz * bz;
      // coincident particles (r2 == 0) are skipped
      const bool ha = v && ta && r2a < 1.f && r2a > 0.f;
      const bool hb = v && tb && r2b < 1.f && r2b > 0.f;
      float fa, ua, fb, ub;
      pair_poly_hw<kDeg>(P, ha ? r2a : 0.5f, fa, ua);
      pair_poly_hw<kDeg>(P, hb ? r2b : 0.5f, fb, ub);
      fa = ha ? fa : 0.f;
      ua = ha ? ua : 0.f;
      fb = hb ? fb : 0.f;
      ub = hb ? ub : 0.f;
      const float fax = fa * ax, fay = fa * ay, faz = fa * az;
      const float fbx = fb * bx, fby = fb * by, fbz = fb * bz;
      qa[0] += fax;
      qa[1] += fay;
      qa[2] += faz;
      qa[3] += ua;
      qb[0] += fbx;
      qb[1] += fby;
      qb[2] += fbz;
      qb[3] += ub;
      np_part += static_cast<uint32_t>(ha) + static_cast<uint32_t>(hb);
      // the reaction on j, split into coarse and fine parts (j's potential is summed on the
      // owner side only); it is big only if fa + fb is, as separations are below 1
      split_add_v4_if(ha || hb, fa + fb >= kBigTerm, fpp + j, flo + j, fbig + j, -(fax + fbx),
                      -(fay + fby), -(faz + fbz));
    };
    int step = 0;
    while (__any_sync(0xffffffffu, ptr < end || pending_b)) {
      // a lane without a candidate reads record 0, as every such lane does, so that the load
      // costs the warp one extra sector at most; its results are masked out
      const bool va = ptr < end, vb = ptr + 1 < end;
      const uint32_t ja = va ? ptr : 0u, jb = vb ? ptr + 1 : 0u;
      float4 h0, l0, h1, l1;  // both loads in flight before either record is used
      load_rec32(rec + 2 * static_cast<size_t>(ja), h0, l0);
      load_rec32(rec + 2 * static_cast<size_t>(jb), h1, l1);
      cand(va, ja, h0, l0);
      cand(vb, jb, h1, l1);
      ptr += 2;
      {
        // the next run without a branch: slot k stays in bounds (k < cnt, or k = 0)
        const bool sw = ptr >= end && k + 1 < cnt;
        k += sw ? 1 : 0;
        const uint32_t nj0 = run_j0[k][tid], nj1 = run_j1[k][tid];
        ptr = sw ? nj0 : ptr;
        end = sw ? nj1 : end;
        if constexpr (!kPhased) {
          ta = same || k < split;
          tb = alive_b && (same || k >= split);
        }
      }
      if constexpr (kPhased) {
        // a's runs walked (rare: a and b in different rows): b's runs take their slots
        const bool go = pending_b && ptr >= end;
        if (__any_sync(0xffffffffu, go)) {
          if (go) {
            cnt = 0;
            b_runs<kRows>(g, starts, pb, lb, ia + 1, part, parts, emit);
            k = 0;
            pending_b = false;
            ta = false;
            tb = true;
            ptr = cnt > 0 ? run_j0[0][tid] : 0u;
            end = cnt > 0 ? run_j1[0][tid] : 0u;
          }
        }
      }
      {
        const bool idle = ptr >= end && !pending_b;
        const unsigned im = __ballot_sync(0xffffffffu, idle);
        if (__popc(im) >= kStealMin) {
          const bool spare = k + 1 < cnt;  // an unstarted run (runs are never empty)
          const bool halve = !spare && ptr < end && end - ptr >= 2 * kStealRecs;
          const bool offer = spare || halve;
          const unsigned om = __ballot_sync(0xffffffffu, offer);
          if (om != 0u) {
            // the offered run [g0, g1) and whom it is tested against (bit 0: a, bit 1: b);
            // bit 2: b exists
            uint32_t g0 = 0, g1 = 0, gf = alive_b ? 4u : 0u;
            if (spare) {
              const int kk = cnt - 1;
              g0 = run_j0[kk][tid];
              g1 = run_j1[kk][tid];
              if constexpr (kPhased)  // all runs of the current phase are tested alike
                gf |= (ta ? 1u : 0u) | (tb ? 2u : 0u);
              else
                gf |= ((same || kk < split) ? 1u : 0u) |
                      ((alive_b && (same || kk >= split)) ? 2u : 0u);
            } else if (halve) {
              g0 = ptr + (((end - ptr) >> 1) & ~1u);  // the donor keeps an even count
              g1 = end;
              gf |= (ta ? 1u : 0u) | (tb ? 2u : 0u);
            }
            // the r-th idle lane takes from the r-th offering lane
            const unsigned lt = (1u << lane) - 1u;
            const int nt = __popc(im), no = __popc(om);
            const int orank = __popc(om & lt), trank = __popc(im & lt);
            if (offer) donor_s[tid >> 5][orank] = static_cast<uint8_t>(lane);
            __syncwarp();
            const bool take = idle && trank < no;
            const int src = take ? static_cast<int>(donor_s[tid >> 5][trank]) : lane;
            __syncwarp();
            if (offer && orank < nt) {
              if (spare)
                --cnt;
              else
                end = g0;
            }
            if (take) flush();  // the sums of the pair held so far
            // every lane takes part; a lane that takes nothing reads its own values
            pa = shfl_f4(pa, src);
            la = shfl_f4(la, src);
            pb = shfl_f4(pb, src);
            lb = shfl_f4(lb, src);
            ia = __shfl_sync(0xffffffffu, ia, src);
            g0 = __shfl_sync(0xffffffffu, g0, src);
            g1 = __shfl_sync(0xffffffffu, g1, src);
            gf = __shfl_sync(0xffffffffu, gf, src);
            if (take) {
              alive_a = true;
              alive_b = (gf & 4u) != 0u;
              ta = (gf & 1u) != 0u;
              tb = (gf & 2u) != 0u;
              // the run-switch formulas above then keep (ta, tb) for this single run (an idle
              // lane has no b runs pending)
              same = ta && tb;
              split = ta ? 1 : 0;
              k = 0;
              cnt = 0;
              ptr = g0;
              end = g1;
            }
          }
        }
      }
      // the own sums: plain FP32 over at most 32 terms (16 steps of two records), then folded
      // into the TwoSum accumulators; so the rounding of a particle's own sum is at most
      // 31 * 2^-24 times the largest 32-term partial sum, per fold, instead of growing with the
      // neighbour count
      if ((++step & 15) == 0) {
        for (int c = 0; c < 4; ++c) {
          sa[c].add(qa[c]);
          sb[c].add(qb[c]);
          qa[c] = qb[c] = 0.f;
        }
        np += np_part;
        np_part = 0;
      }
    }
    np += np_part;
    flush();
  }
  if (energy) block_reduce_add<kPpThreads>(e_acc, energy);
  warp_add_u64(2ull * np, pairs);
}

// (particle, record) distance tests k_pp_f32 makes on the current sorted records: the same
// runs, summed instead of walked (a run shared by a and b counts twice). Run on request only,
// so that the short range itself carries no counter.
template <int kRows>
__global__ void k_pp_count_f32(Geom g, const uint32_t* __restrict__ total,
                               const float4* __restrict__ rec,
                               const uint32_t* __restrict__ starts,
                               const uint32_t* __restrict__ dense,
                               unsigned long long* __restrict__ out) {
  const uint32_t N = *total;
  const uint32_t lane_pair = blockIdx.x * static_cast<uint32_t>(blockDim.x) + threadIdx.x;
  const uint32_t ia = 2 * lane_pair, ib = ia + 1;
  unsigned long long n = 0;
  if (ia < N && !(dense && in_dense_tile(dense, ia))) {
    const bool alive_b = ib < N;
    const uint32_t eb = alive_b ? ib : ia;
    const float4 pa = rec[2 * ia], la = rec[2 * ia + 1];
    const float4 pb = rec[2 * eb], lb = rec[2 * eb + 1];
    bool same = true;
    int split = 0;
    pair_runs<kRows>(g, starts, pa, la, pb, lb, ia, alive_b, 0, 1, same, split,
                     [&](uint32_t j0, uint32_t j1) { n += j1 - j0; });
    if (same && alive_b) n *= 2;
  }
  warp_add_u64(n, out);
}

}  // namespace

void launch_pp(const p3m_ctx* c, int64_t n, cudaStream_t s, bool want_energy) {
  if (n == 0) return;
  if (!c->fp32) {
    launch_pp64(c, n, s, want_energy);
    return;
  }
  const uint32_t* total = c->starts + c->nkeys;
  {
    // the kernel adds each pair's force to both particles; the result (coarse, fine and big parts)
    // and the tile counter were cleared by the sort
    float4* fbig = c->fplo + c->n_max;
    // particles with many neighbours go to the tile kernel, the others to the walk
    const uint32_t* dense = dense_flags(c, n);
    // persistent grid of a few blocks per SM: the SM resources it leaves free let the mesh
    // chain, on the other stream, run at the same time
    // lanes per pair of particles (kPpMaxLogParts)
    const int64_t full = static_cast<int64_t>(kPpBlocksPerSm) * c->num_sms * kPpThreads;
    int log_parts = 0;
    while (log_parts < kPpMaxLogParts && (((n + 1) / 2) << log_parts) < full) ++log_parts;
    const int64_t per_tile = (2 * kPpThreads) >> log_parts;
    const int64_t tiles = (n + per_tile - 1) / per_tile;
    const unsigned wblocks = static_cast<unsigned>(
        std::min<int64_t>(tiles, static_cast<int64_t>(kPpBlocksPerSm) * c->num_sms));
    // the kernel for the context's row geometry (Geom::rows cell rows per cutoff)
    auto run = [&](auto k_rows1, auto k_rows2, auto k_rows3) {
      auto kern = c->g.rows == 1 ? k_rows1 : (c->g.rows == 2 ? k_rows2 : k_rows3);
      const size_t smem = pp_run_bytes(c->g.rows);
      if (smem > 48 * 1024)
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(smem));
      kern<<<wblocks, kPpThreads, smem, s>>>(
          c->g, c->poly, total, static_cast<const float4*>(c->recp), c->starts,
          static_cast<float4*>(c->fpp), reinterpret_cast<float2*>(c->fplo), fbig, c->pp_tile,
          log_parts, dense, c->energy_acc, c->pair_acc);
    };
    if (c->g.pp_bc) {
      const uint32_t near_cell = near_cathode_cell(c);
      const unsigned iblocks = static_cast<unsigned>(std::min<int64_t>(
          (n * kImgLanes + kThreads - 1) / kThreads, static_cast<int64_t>(c->num_sms) * 8));
      auto images = [&](auto kern) {
        kern<<<iblocks, kThreads, 0, s>>>(c->g, c->poly, near_cell,
                                          static_cast<const float4*>(c->recp), c->starts,
                                          static_cast<float4*>(c->fpp),
                                          reinterpret_cast<float2*>(c->fplo), fbig,
                                          c->energy_acc, c->pair_acc);
      };
      switch (c->poly.deg) {
        case 4: images(k_pp_images<4>); break;
        case 5: images(k_pp_images<5>); break;
        case 6: images(k_pp_images<6>); break;
        case 7: images(k_pp_images<7>); break;
        case 8: images(k_pp_images<8>); break;
        case 9: images(k_pp_images<9>); break;
        case 10: images(k_pp_images<10>); break;
        case 11: images(k_pp_images<11>); break;
        case 12: images(k_pp_images<12>); break;
        case 13: images(k_pp_images<13>); break;
        case 14: images(k_pp_images<14>); break;
        default: images(k_pp_images<15>); break;
      }
    }
    switch (c->poly.deg) {
      case 4: run(k_pp_f32<4, 1>, k_pp_f32<4, 2>, k_pp_f32<4, 3>); break;
      case 5: run(k_pp_f32<5, 1>, k_pp_f32<5, 2>, k_pp_f32<5, 3>); break;
      case 6: run(k_pp_f32<6, 1>, k_pp_f32<6, 2>, k_pp_f32<6, 3>); break;
      case 7: run(k_pp_f32<7, 1>, k_pp_f32<7, 2>, k_pp_f32<7, 3>); break;
      case 8: run(k_pp_f32<8, 1>, k_pp_f32<8, 2>, k_pp_f32<8, 3>); break;
      case 9: run(k_pp_f32<9, 1>, k_pp_f32<9, 2>, k_pp_f32<9, 3>); break;
      case 10: run(k_pp_f32<10, 1>, k_pp_f32<10, 2>, k_pp_f32<10, 3>); break;
      case 11: run(k_pp_f32<11, 1>, k_pp_f32<11, 2>, k_pp_f32<11, 3>); break;
      case 12: run(k_pp_f32<12, 1>, k_pp_f32<12, 2>, k_pp_f32<12, 3>); break;
      case 13: run(k_pp_f32<13, 1>, k_pp_f32<13, 2>, k_pp_f32<13, 3>); break;
      case 14: run(k_pp_f32<14, 1>, k_pp_f32<14, 2>, k_pp_f32<14, 3>); break;
      default: run(k_pp_f32<15, 1>, k_pp_f32<15, 2>, k_pp_f32<15, 3>); break;
    }
    // (after the walk: in a sparse bunch the walk is what takes time, and it then starts at once)
    launch_pp_dense(c, n, s, want_energy);
  }
}

void launch_pp_count(const p3m_ctx* c, int64_t n, unsigned long long* out, cudaStream_t s) {
  if (!c->fp32) return;  // FP64: the short range counts as it walks
  cudaMemsetAsync(out, 0, sizeof(unsigned long long), s);
  if (n == 0) return;
  // the tiles of the last sort, whatever call it was made for
  cudaMemsetAsync(c->pp_tile + 1, 0, sizeof(uint32_t), s);
  launch_dense_tiles(c, n, s);
  const int64_t lane_pairs = (n + 1) / 2;
  auto kern = c->g.rows == 1   ? k_pp_count_f32<1>
              : c->g.rows == 2 ? k_pp_count_f32<2>
                               : k_pp_count_f32<3>;
  kern<<<static_cast<unsigned>((lane_pairs + kThreads - 1) / kThreads), kThreads, 0, s>>>(
      c->g, c->starts + c->nkeys, static_cast<const float4*>(c->recp), c->starts,
      dense_flags(c, n), out);
  launch_pp_dense_count(c, n, out, s);
}

}  // namespace p3m
