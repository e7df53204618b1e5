// Vector-Jacobian product of the FP32 short-range force map, each unordered pair once: for a pair
// (i, j), j > i, with d = xi_i - xi_j and H(d) = fco(rho) I + dfr(rho) d d^T (the pair energy's
// Hessian, even in d), i gets H(d) (w_i - w_j) and j gets its negative. The result goes to acc4
// (zeroed, cutoff units), w comes in sorted order as float4 (ws). Image pairs (pp_bc) act on i only:
// acc_i -= H(d) (w_i - S w_j), d = xi_i - S xi_j.
//
// A walk of each particle's runs in the half shell, two records per lane and step; every pair's
// reaction goes to the L2 by a vector reduction, and w_j is loaded for every pair, which bounds it
// in dense bunches. (Tiles as in pp_dense.cu take a third of the time there, but round differently:
// they moved the product of 262,144 dense particles by 8e-7, as much as its whole error.)
#include <algorithm>

#include "pp_f32.cuh"

namespace p3m {
namespace {

constexpr int kThreads = 128;
constexpr int kWalkBlocksPerSm = 10;  // resident blocks per SM of the walk (48 registers)
// Lanes that share a particle and split the rows of its half shell: 1, doubled (to 16 at most)
// while the lanes would not fill the walk's resident blocks. Whole products, one lane and the rule:
// 8000 dense particles 853 -> 284 us, 30,000 3.46 -> 1.01 ms, 120,000 4.76 -> 3.25 ms, a sphere of
// 100,000 745 -> 484 us; with images (in a kernel of their own, as in the forces) 5001 particles
// 1027 -> 350 us, a core and halo of 170,000 17.2 -> 11.1 ms.
constexpr int kMaxLogParts = 4;
constexpr int kImgLanes = 8;

template <int kDeg>
__device__ __forceinline__ void pair_hess_poly(const PairPoly& P, float r2, float& fco,
                                               float& dfr) {
  const float rinv = rsqrtf(r2);
  const float rho = r2 * rinv;
  const float R = erfcx_poly<kDeg, false>(P, rho);
  const float ex = exp2f(-P.kappa2_log2e * r2);
  const float pot = R * ex * rinv;           // erfc(kappa rho) / rho
  const float cex = P.c2k * ex;
  const float A = pot + cex;                 // rho^2 times the force coefficient
  const float rinv2 = rinv * rinv;
  fco = A * rinv2;
  // dA/drho = -c2k e/rho - erfc/rho^2 - 2 kappa^2 rho c2k e; dfr = (dA/rho^2 - 2 A/rho^3)/rho
  const float dA = -(cex + pot) * rinv - 2.f * P.kappa2 * rho * cex;
  dfr = (dA - 2.f * A * rinv) * rinv2 * rinv;
}

// The walk: persistent blocks, runs in shared memory, two records per lane per step.
template <int kDeg, int kRows>
__global__ void __launch_bounds__(kThreads, kWalkBlocksPerSm)
    k_vjp_walk(Geom g, PairPoly P, const uint32_t* __restrict__ total,
               const float4* __restrict__ rec, const uint32_t* __restrict__ starts,
               const float4* __restrict__ ws, float4* __restrict__ acc4,
               uint32_t* __restrict__ next_tile, int log_parts) {
  using R = Rows<kRows>;
  __shared__ uint32_t run_j0[R::half][kThreads], run_j1[R::half][kThreads];
  __shared__ uint32_t tile_s;
  const int tid = threadIdx.x;
  const uint32_t N = *total;
  for (;;) {
    if (tid == 0) tile_s = atomicAdd(next_tile, 1u);
    __syncthreads();
    const uint32_t tile = tile_s;
    __syncthreads();
    const uint32_t i0 = tile * (kThreads >> log_parts);
    if (i0 >= N) break;
    const uint32_t i = i0 + (tid >> log_parts);
    const int parts = 1 << log_parts, mine = tid & (parts - 1);
    const bool alive = i < N;
    const uint32_t ie = alive ? i : 0u;
    const float4 pi = rec[2 * ie], li = rec[2 * ie + 1];
    const float4 wi = ws[ie];
    int cnt = 0;
    if (alive) {
      const uint32_t row = __float_as_uint(li.w) & kRowMask;
      const int cy = static_cast<int>(row % static_cast<uint32_t>(g.nc[1]));
      const int cz = static_cast<int>(row / static_cast<uint32_t>(g.nc[1]));
      for (int r = R::first + mine; r < R::last; r += parts) {
        uint32_t j0, j1;
        row_range<kRows>(g, starts, pi.x, pi.y, pi.z, cy, cz, r, j0, j1);
        j0 = max(j0, i + 1);
        if (j0 < j1) {
          run_j0[cnt][tid] = j0;
          run_j1[cnt][tid] = j1;
          ++cnt;
        }
      }
    }
    uint32_t ptr = 0, end = 0;
    if (cnt > 0) {
      ptr = run_j0[0][tid];
      end = run_j1[0][tid];
    }
    int k = 0;
    Acc2 sum[3];
    for (int c = 0; c < 3; ++c) sum[c].hi = sum[c].lo = 0.f;
    float part[3] = {0.f, 0.f, 0.f};
    auto pair = [&](bool hit, float r2, float rx, float ry, float rz, uint32_t j) {
      float fco, dfr;
      pair_hess_poly<kDeg>(P, hit ? r2 : 0.5f, fco, dfr);
      const float4 wj = ws[hit ? j : ie];
      const float v0 = wi.x - wj.x, v1 = wi.y - wj.y, v2 = wi.z - wj.z;
      const float dv = hit ? dfr * (rx * v0 + ry * v1 + rz * v2) : 0.f;
      fco = hit ? fco : 0.f;
      const float c0 = fmaf(fco, v0, dv * rx), c1 = fmaf(fco, v1, dv * ry),
                  c2 = fmaf(fco, v2, dv * rz);
      part[0] += c0;
      part[1] += c1;
      part[2] += c2;
      if (hit) red_add_v4(acc4 + j, -c0, -c1, -c2, 0.f);
    };
    int step = 0;
    while (__any_sync(0xffffffffu, ptr < end)) {
      const bool va = ptr < end, vb = ptr + 1 < end;
      const float4* pa = va ? rec + 2 * static_cast<size_t>(ptr) : rec;
      const float4* pb = vb ? rec + 2 * static_cast<size_t>(ptr + 1) : rec;
      float4 ha, la, hb, lb;
      load_rec32(pa, ha, la);
      load_rec32(pb, hb, lb);
      const float ax = (pi.x - ha.x) + (li.x - la.x), ay = (pi.y - ha.y) + (li.y - la.y),
                  az = (pi.z - ha.z) + (li.z - la.z);
      const float bx = (pi.x - hb.x) + (li.x - lb.x), by = (pi.y - hb.y) + (li.y - lb.y),
                  bz = (pi.z - hb.z) + (li.z - lb.z);
      const float ra = ax * ax + ay * ay + az * az, rb = bx * bx + by * by + bz * bz;
      const bool hita = va && ra < 1.f && ra > 0.f;
      const bool hitb = vb && rb < 1.f && rb > 0.f;
      if (__any_sync(0xffffffffu, hita)) pair(hita, ra, ax, ay, az, ptr);
      if (__any_sync(0xffffffffu, hitb)) pair(hitb, rb, bx, by, bz, ptr + 1);
      ptr += 2;
      {
        // the next run without a branch: slot k stays in bounds (k < cnt, or k = 0)
        const bool sw = ptr >= end && k + 1 < cnt;
        k += sw ? 1 : 0;
        const uint32_t nj0 = run_j0[k][tid], nj1 = run_j1[k][tid];
        ptr = sw ? nj0 : ptr;
        end = sw ? nj1 : end;
      }
      if ((++step & 7) == 0) {
        for (int c = 0; c < 3; ++c) {
          sum[c].add(part[c]);
          part[c] = 0.f;
        }
      }
    }
    for (int c = 0; c < 3; ++c) sum[c].add(part[c]);
    if (alive) red_add_v4(acc4 + i, sum[0].value(), sum[1].value(), sum[2].value(), 0.f);
  }
}

// Pairs with images, for the particles less than r_c above the cathode (the first ones in sorted
// order); kImgLanes lanes share one and split the rows around its image point.
template <int kDeg>
__global__ void __launch_bounds__(kThreads)
    k_vjp_images(Geom g, PairPoly P, uint32_t near_cell, const float4* __restrict__ rec,
                 const uint32_t* __restrict__ starts, const float4* __restrict__ ws,
                 float4* __restrict__ acc4) {
  const uint32_t near = starts[near_cell];
  const int part = threadIdx.x & (kImgLanes - 1);
  const float ch = static_cast<float>(g.img_c);
  const float cl = static_cast<float>(g.img_c - static_cast<double>(ch));
  for (uint32_t i = (blockIdx.x * kThreads + threadIdx.x) / kImgLanes; i < near;
       i += gridDim.x * (kThreads / kImgLanes)) {
    const float4 pi = rec[2 * i], li = rec[2 * i + 1], wi = ws[i];
    const double zi = static_cast<double>(pi.z) + static_cast<double>(li.z);
    if (zi - 0.5 * g.img_c >= 1.0) continue;
    const float mz = static_cast<float>(g.img_c - zi);
    Acc2 sum[3];
    for (int c = 0; c < 3; ++c) sum[c].hi = sum[c].lo = 0.f;
    for_rows<float>(g, starts, pi.x, pi.y, mz, part, kImgLanes, [&](uint32_t ja, uint32_t jb) {
      float rowv[3] = {0.f, 0.f, 0.f};
      for (uint32_t jj = ja; jj < jb; ++jj) {
        const float4 hj = rec[2 * jj], lj = rec[2 * jj + 1];
        const float ax = (pi.x - hj.x) + (li.x - lj.x);
        const float ay = (pi.y - hj.y) + (li.y - lj.y);
        const float s = pi.z + hj.z;
        const float bp = s - pi.z;
        const float e = (pi.z - (s - bp)) + (hj.z - bp);
        const float az = ((s - ch) + e) + ((li.z + lj.z) - cl);
        const float r2 = ax * ax + ay * ay + az * az;
        if (r2 < 1.f && r2 > 0.f) {
          float fco, dfr;
          pair_hess_poly<kDeg>(P, r2, fco, dfr);
          const float4 wj = ws[jj];
          const float v0 = wi.x - wj.x, v1 = wi.y - wj.y, v2 = wi.z + wj.z;  // w_i - S w_j
          const float dv = dfr * (ax * v0 + ay * v1 + az * v2);
          rowv[0] -= fmaf(fco, v0, dv * ax);
          rowv[1] -= fmaf(fco, v1, dv * ay);
          rowv[2] -= fmaf(fco, v2, dv * az);
        }
      }
      for (int c = 0; c < 3; ++c) sum[c].add(rowv[c]);
    });
    red_add_v4(acc4 + i, sum[0].value(), sum[1].value(), sum[2].value(), 0.f);
  }
}

// w (input order, FP64) -> ws (sorted order, float4); the result cleared (entry i, coalesced).
__global__ void k_gather_w(const uint32_t* __restrict__ total, int64_t n,
                           const float4* __restrict__ rec, const double* __restrict__ w,
                           float4* __restrict__ ws, float4* __restrict__ acc4) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) acc4[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  if (i >= *total) return;
  const long long idx = __float_as_int(rec[2 * i].w);
  ws[i] = make_float4(static_cast<float>(w[3 * idx]), static_cast<float>(w[3 * idx + 1]),
                      static_cast<float>(w[3 * idx + 2]), 0.f);
}

template <int kDeg>
void launch_vjp(const p3m_ctx* c, int64_t n, const float4* ws, cudaStream_t s) {
  const uint32_t* total = c->starts + c->nkeys;
  const auto* rec = static_cast<const float4*>(c->recp);
  auto* acc4 = static_cast<float4*>(c->fpp);
  if (c->g.pp_bc) {
    const unsigned blocks = static_cast<unsigned>(std::min<int64_t>(
        (n * kImgLanes + kThreads - 1) / kThreads, static_cast<int64_t>(c->num_sms) * 8));
    k_vjp_images<kDeg><<<blocks, kThreads, 0, s>>>(c->g, c->poly, near_cathode_cell(c), rec,
                                                   c->starts, ws, acc4);
  }
  const int64_t resident = static_cast<int64_t>(kWalkBlocksPerSm) * c->num_sms;
  int log_parts = 0;
  while (log_parts < kMaxLogParts && (n << log_parts) < resident * kThreads) ++log_parts;
  const int64_t blocks = ((n << log_parts) + kThreads - 1) / kThreads;
  auto walk = c->g.rows == 1   ? k_vjp_walk<kDeg, 1>
              : c->g.rows == 2 ? k_vjp_walk<kDeg, 2>
                               : k_vjp_walk<kDeg, 3>;
  walk<<<static_cast<unsigned>(std::min(blocks, resident)), kThreads, 0, s>>>(
      c->g, c->poly, total, rec, c->starts, ws, acc4, c->pp_tile, log_parts);
}

}  // namespace

void launch_pp_vjp(const p3m_ctx* c, int64_t n, const double* w, cudaStream_t s) {
  if (n == 0) return;
  if (!c->fp32) {
    launch_pp64_vjp(c, n, w, s);
    return;
  }
  // weights in sorted order (in the memory of the force's fine parts, not in use here), result in
  // fpp (cutoff units; the mesh gather scales it); the counters were cleared by the sort
  float4* ws = c->fplo;
  k_gather_w<<<static_cast<unsigned>((n + kThreads - 1) / kThreads), kThreads, 0, s>>>(
      c->starts + c->nkeys, n, static_cast<const float4*>(c->recp), w, ws,
      static_cast<float4*>(c->fpp));
  switch (c->poly.deg) {
    case 4: launch_vjp<4>(c, n, ws, s); break;
    case 5: launch_vjp<5>(c, n, ws, s); break;
    case 6: launch_vjp<6>(c, n, ws, s); break;
    case 7: launch_vjp<7>(c, n, ws, s); break;
    case 8: launch_vjp<8>(c, n, ws, s); break;
    case 9: launch_vjp<9>(c, n, ws, s); break;
    case 10: launch_vjp<10>(c, n, ws, s); break;
    case 11: launch_vjp<11>(c, n, ws, s); break;
    case 12: launch_vjp<12>(c, n, ws, s); break;
    case 13: launch_vjp<13>(c, n, ws, s); break;
    case 14: launch_vjp<14>(c, n, ws, s); break;
    default: launch_vjp<15>(c, n, ws, s); break;
  }
}

}  // namespace p3m
