// FP64 short range, eq. (summation_short) with the screened kernel of eq. (ewald_split), and the
// vector-Jacobian product of the same force map.
//
// What bounds it: this part has two FP64 lanes per clock and SM (64 cycles an instruction and
// scheduler), 1/64 of its FP32 rate, and a vectorless FP64 reduction costs the L2 one sector
// operation per component. So nothing here is FP64 but the sums of the partial sums:
//   * positions are 56-bit fixed-point numbers held as three FP32-exact pieces (24 + 24 + 8 bits,
//     k_scatter), whose differences are exact, so a separation is a double-float number good to
//     2^-48 and never less exact than the difference of FP64 coordinates;
//   * r^2, the pair function (pair_table.cuh) and the products are double-float;
//   * every ordered pair is evaluated by its own particle, so there are no reactions to reduce
//     (three FP64 reductions per pair cost more L2 time than the second evaluation costs issue
//     slots), no result array to clear, and the sums have a fixed order for fixed sorted records.
//
// Work split: S lanes (4, 8, 16 or 32) share a particle. They compute its neighbour rows' runs
// together, then walk each run 2 S records at a time (adjacent lanes read adjacent 16-byte records)
// and test the distance in FP32 on the leading 24 bits (inside the search slack). What passes is
// queued per group in shared memory and evaluated S at a time by all lanes, so the expensive part
// runs nearly full whatever the density. S = 4 for large counts; more lanes per particle when the
// particles alone would not fill the SMs.
//
// Measured against one lane a particle with FP64 separations, sums and reactions: 4096-particle
// Gaussian 2812 -> 58 us (S = 32; S = 4, 8, 16: 312, 169, 101 us), 2,097,152-particle sphere
// 4.34 -> 2.21 ms (S = 4; S = 8, 16, 32: 3.1, 4.6, 7.8 ms). There it issues 62% of the slots
// (1.86e9 instructions, about half of them the evaluation of 1.5e8 ordered pairs, half the search
// and the walk) and waits on L1 latency for most of the rest.
#include <algorithm>
#include <memory>

#include "pair_table.cuh"
#include "pp_common.cuh"

namespace p3m {
namespace {

using dfm::F2;

// One block per SM, of 24 warps for the force (80 registers) and 20 where a second table takes the
// shared memory: one copy of a table serves them all, and the L1 keeps room for the records that
// neighbouring particles share. On the 2,097,152-particle sphere 16, 20, 24 and 28 warps take
// 2.78, 2.42, 2.24 and 2.36 ms (blocks of 4 warps with a table each: 2.55 ms).
template <int kMode>
__host__ __device__ constexpr int threads64() {
  return kMode == 0 ? 768 : 640;
}
constexpr int kRing = 8;   // queued candidates per lane of a group (4: 6% slower; 16: the same)
constexpr int kFold = 32;  // evaluations between folds of the double-float sums into FP64

enum Mode64 { kForce = 0, kForcePot = 1, kVjp = 2 };

struct Args64 {
  const uint32_t* total;
  const float4* ph;   // {x, y, z leading 24 bits, row}
  const float4* pml;  // {x, y, z next 24 bits, trailing 8 bits of each axis}
  const uint32_t* starts;
  const dfm::PairTab* tab;
  const dfm::PairDF* df;
  const float4* w;    // kVjp: {w hi, .} {w lo, .} per sorted particle
  D4* out;            // kForce, kForcePot
  double* acc;        // kVjp: [3 n]
  double scale;       // kVjp
  const unsigned long long* wbound;  // kVjp: bits of the largest |w|
  double* energy;
  unsigned long long* pairs;
  uint32_t* next;
  int log_s;
};

// The pair function where there is no table (kappa above 6.5): double-float from the fit, or FP64
// where that does not reach either. f: force coefficient; g: the potential (hess = false) or the
// Hessian term.
struct PairFG {
  F2 f, g;
};
__device__ __noinline__ PairFG pair_no_table(const dfm::PairDF* df, double kappa, F2 s, bool hess) {
  PairFG o;
  if (df) {
    if (hess) {
      dfm::pair_hess_df(df->k, df->coef, s, o.f, o.g);
    } else {
      const dfm::PairOut p = dfm::pair_df(df->k, df->coef, s);
      o.f = p.fco;
      o.g = p.pot;
    }
    return o;
  }
  const double r2 = static_cast<double>(s.hi) + static_cast<double>(s.lo);
  const double r = sqrt(r2), x = kappa * r;
  const double c2k = 2.0 * kappa * 0.56418958354775628695;
  const double ex = c2k * exp(-x * x), pot = erfc(x) / r, A = pot + ex;
  o.f = dfm::split_double_fp64(A / r2);
  if (hess) {
    const double dA = -A / r - 2.0 * kappa * kappa * r * ex;
    o.g = dfm::split_double_fp64((dA / r2 - 2.0 * A / (r2 * r)) / r);
  } else {
    o.g = dfm::split_double_fp64(pot);
  }
  return o;
}

__device__ __forceinline__ F2 tab_lookup(const dfm::TabFn* t, int row, float u, float ul,
                                         float c5 = 0.f) {
  const float4 q = reinterpret_cast<const float4*>(t->a)[row];
  const float4 r = reinterpret_cast<const float4*>(t->b)[row];
  const float a[4] = {q.x, q.y, q.z, q.w}, b[4] = {r.x, r.y, r.z, r.w};
  return dfm::tab_eval(a, b, u, ul, c5);
}

// shared memory of the tables a mode reads
template <int kMode, bool kTab>
__host__ __device__ constexpr size_t tab_bytes() {
  return !kTab ? 0
               : sizeof(dfm::TabFn) * (kMode == kForce ? 1 : 2) +
                     (kMode == kVjp ? sizeof(float) * dfm::kTabRows : 0);
}

// byte k of v as the float 2^23 + byte
__device__ __forceinline__ float byte_float(uint32_t v, int k) {
  return __uint_as_float(__byte_perm(v, 0x4B000000u, 0x7540u | static_cast<uint32_t>(k)));
}

// one axis of a separation: exact differences of the pieces, as hi + lo
__device__ __forceinline__ F2 sep(float hi, float hj, float mi, float mj, float bi, float bj,
                                  float ls) {
  const float H = __fsub_rn(hi, hj), M = __fsub_rn(mi, mj);
  const float s = __fadd_rn(H, M);  // H is 0 or at least the largest |M|
  const float e = __fsub_rn(M, __fsub_rn(s, H));
  return F2{s, __fmaf_rn(__fsub_rn(bi, bj), ls, e)};
}

// a b as p + e (not renormalised)
__device__ __forceinline__ F2 prod(F2 a, F2 b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);
  e = __fmaf_rn(a.hi, b.lo, e);
  e = __fmaf_rn(a.lo, b.hi, e);
  return F2{p, e};
}

// running double-float sum
__device__ __forceinline__ void accumulate(F2& a, F2 v) {
  const F2 s = dfm::two_sum(a.hi, v.hi);
  a.hi = s.hi;
  a.lo = __fadd_rn(a.lo, __fadd_rn(s.lo, v.lo));
}

// x^2 + y^2 + z^2 of double-float components
__device__ __forceinline__ F2 norm2(const F2 d[3]) {
  F2 q[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const float p = __fmul_rn(d[c].hi, d[c].hi);
    q[c] = F2{p, __fmaf_rn(__fadd_rn(d[c].hi, d[c].hi), d[c].lo, __fmaf_rn(d[c].hi, d[c].hi, -p))};
  }
  const F2 a = dfm::two_sum(q[0].hi, q[1].hi);
  const F2 b = dfm::two_sum(a.hi, q[2].hi);
  const float lo = __fadd_rn(__fadd_rn(a.lo, b.lo), __fadd_rn(q[0].lo, __fadd_rn(q[1].lo, q[2].lo)));
  return dfm::fast_two_sum(b.hi, lo);
}

template <int kMode, int kRows, bool kTab>
__global__ void __launch_bounds__(threads64<kMode>(), 1) k_pp64(Geom g, Args64 a) {
  constexpr int kThreads64 = threads64<kMode>(), kWarps64 = kThreads64 / 32;
  using R = Rows<kRows>;
  constexpr int kTabQuads = tab_bytes<kMode, kTab>() / sizeof(float4);
  extern __shared__ float4 tab_s[];  // the tables, then each warp's runs, then its queues
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  if constexpr (kTab) {
    constexpr int kQuads = sizeof(dfm::TabFn) / sizeof(float4);
    const float4* src = reinterpret_cast<const float4*>(&a.tab->fco);
    for (int t = tid; t < kQuads; t += kThreads64) tab_s[t] = src[t];
    if constexpr (kMode != kForce) {
      src = reinterpret_cast<const float4*>(kMode == kVjp ? &a.tab->dfr : &a.tab->pot);
      for (int t = tid; t < kQuads; t += kThreads64) tab_s[kQuads + t] = src[t];
    }
    if constexpr (kMode == kVjp) {
      float* c5 = reinterpret_cast<float*>(tab_s + 2 * kQuads);
      for (int t = tid; t < dfm::kTabRows; t += kThreads64) c5[t] = a.tab->dfr5[t];
    }
    __syncthreads();
  }
  const dfm::TabFn* tab0 = reinterpret_cast<const dfm::TabFn*>(tab_s);
  const dfm::TabFn* tab1 = tab0 + 1;
  const float* tab5 = reinterpret_cast<const float*>(tab0 + 2);
  const int S = 1 << a.log_s;
  const int group = lane >> a.log_s, part = lane & (S - 1), gbase = group << a.log_s;
  const uint32_t gmask = (S == 32 ? 0xffffffffu : ((1u << S) - 1u)) << gbase;
  const uint32_t below = gmask & ((1u << lane) - 1u);  // the group's lanes before this one
  const int cap = S * kRing;
  uint2(*runs)[8] = reinterpret_cast<uint2(*)[8]>(tab_s + kTabQuads) + wid * R::last;  // 8 groups
  uint32_t* ring = reinterpret_cast<uint32_t*>(reinterpret_cast<uint2(*)[8]>(tab_s + kTabQuads) +
                                               kWarps64 * R::last) +
                   wid * (32 * kRing) + group * cap;
  const uint32_t N = *a.total;
  const float thr = (1.f + g.slack_f) * (1.f + g.slack_f);
  const uint32_t per_warp = 32u >> a.log_s;
  double e_acc = 0.0;
  unsigned long long np = 0, ni = 0, ncand = 0;
  for (;;) {
    uint32_t tile = 0;
    if (lane == 0) tile = atomicAdd(a.next, 1u);
    tile = __shfl_sync(0xffffffffu, tile, 0);
    if (static_cast<uint64_t>(tile) * per_warp >= N) break;
    const uint32_t i = tile * per_warp + group;
    const bool alive = i < N;
    const uint32_t ie = alive ? i : 0u;
    float4 hi = a.ph[ie], mi = a.pml[ie];
    const uint32_t lb = __float_as_uint(mi.w);
    float b0 = byte_float(lb, 0), b1 = byte_float(lb, 1), b2 = byte_float(lb, 2);
    const uint32_t row = __float_as_uint(hi.w);
    const int cy = static_cast<int>(row % static_cast<uint32_t>(g.nc[1]));
    int cz = static_cast<int>(row / static_cast<uint32_t>(g.nc[1]));
    F2 wi[3];
    if constexpr (kMode == kVjp) {
      const float4 wh = a.w[2 * ie], wl = a.w[2 * ie + 1];
      wi[0] = F2{wh.x, wl.x};
      wi[1] = F2{wh.y, wl.y};
      wi[2] = F2{wh.z, wl.z};
    }
    double F[3] = {0.0, 0.0, 0.0}, phi = 0.0;
    // phase 1 (pp_bc): the pairs with images, as the pairs of the particle's own image point
    // y = S xi_i with the particles: |xi_i - S xi_j| = |y - xi_j|, and the image's charge and the
    // mirror map give the signs (-, -, +)
    bool on = alive;
    for (int phase = 0; phase < 2; ++phase) {
      if (phase == 1) {
        if (!g.pp_bc) break;
        const double z = static_cast<double>(hi.z) + static_cast<double>(mi.z) +
                         (static_cast<double>(b2) - 8388608.0) * static_cast<double>(g.pos_ls);
        on = alive && z - 0.5 * g.img_c < 1.0;
        if (!__any_sync(0xffffffffu, on)) break;
        const long long q = __double2ll_rn((g.img_c - z) * g.pos_scale);
        hi.z = static_cast<float>(static_cast<int>(q >> 32)) * g.pos_hs;
        mi.z = static_cast<float>(static_cast<int>((q >> 8) & 0xffffff)) * g.pos_ms;
        b2 = 8388608.f + static_cast<float>(static_cast<int>(q & 0xff));
        cz = static_cast<int>(floorf(hi.z * g.inv_cw_f[2]));
        if constexpr (kMode == kVjp) wi[2] = dfm::neg(wi[2]);
      }
      __syncwarp();  // the last phase's runs and queue are done with
      int nr = 0;
      uint32_t steps = 0;  // walk steps of the group, then of the warp
      for (int r0 = 0; r0 < R::last; r0 += S) {
        uint32_t j0 = 0, j1 = 0;
        if (on && r0 + part < R::last)
          row_range<kRows>(g, a.starts, hi.x, hi.y, hi.z, cy, cz, r0 + part, j0, j1);
        const bool some = j0 < j1;
        const uint32_t b = __ballot_sync(0xffffffffu, some);
        if (some) runs[nr + __popc(b & below)][group] = make_uint2(j0, j1);
        nr += __popc(b & gmask);
        if (some) {
          steps += (j1 - j0 + 2 * S - 1) >> (a.log_s + 1);
          if (phase == 0) ncand += j1 - j0;
        }
      }
      for (int o = 1; o < S; o <<= 1) steps += __shfl_xor_sync(0xffffffffu, steps, o);
      steps = __reduce_max_sync(0xffffffffu, steps);
      __syncwarp();
      uint32_t ptr = 0, end = 0;
      if (nr > 0) {
        const uint2 t = runs[0][group];
        ptr = t.x;
        end = t.y;
      }
      int k = 0, head = 0, cnt = 0, evals = 0;
      uint32_t hits = 0;
      F2 acc[3], pa = F2{0.f, 0.f};
#pragma unroll
      for (int c = 0; c < 3; ++c) acc[c] = F2{0.f, 0.f};
      const double sign = phase == 0 ? 1.0 : -1.0;
      auto fold = [&]() {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          F[c] += (c == 2 ? 1.0 : sign) *
                  (static_cast<double>(acc[c].hi) + static_cast<double>(acc[c].lo));
          acc[c] = F2{0.f, 0.f};
        }
        if constexpr (kMode == kForcePot) {
          phi += sign * (static_cast<double>(pa.hi) + static_cast<double>(pa.lo));
          pa = F2{0.f, 0.f};
        }
      };
      // in phase 0 a particle is not its own neighbour; in phase 1 its own image counts
      const uint32_t self = phase == 0 ? i : 0xffffffffu;
      for (;;) {
        // walk while every group's queue has room for a step's candidates
        if (steps > 0 && !__any_sync(0xffffffffu, cnt > cap - 2 * S)) {
          --steps;
          const uint32_t ja = ptr + part, jb = ja + S;
          const bool va = ja < end, vb = jb < end;
          const float4 pa4 = a.ph[va ? ja : ie], pb4 = a.ph[vb ? jb : ie];
          const float ax = hi.x - pa4.x, ay = hi.y - pa4.y, az = hi.z - pa4.z;
          const float bx = hi.x - pb4.x, by = hi.y - pb4.y, bz = hi.z - pb4.z;
          const bool ha = va && ja != self && fmaf(ax, ax, fmaf(ay, ay, az * az)) < thr;
          const bool hb = vb && jb != self && fmaf(bx, bx, fmaf(by, by, bz * bz)) < thr;
          const uint32_t ma = __ballot_sync(0xffffffffu, ha), mb = __ballot_sync(0xffffffffu, hb);
          const int na = __popc(ma & gmask);
          if (ha) ring[(head + cnt + __popc(ma & below)) & (cap - 1)] = ja;
          if (hb) ring[(head + cnt + na + __popc(mb & below)) & (cap - 1)] = jb;
          cnt += na + __popc(mb & gmask);
          ptr += 2 * S;
          if (ptr >= end && k + 1 < nr) {
            ++k;
            const uint2 t = runs[k][group];
            ptr = t.x;
            end = t.y;
          }
          continue;
        }
        if (!__any_sync(0xffffffffu, cnt > 0)) break;
        // evaluate up to S queued candidates of each group
        __syncwarp();
        const bool has = part < cnt;
        const uint32_t j = has ? ring[(head + part) & (cap - 1)] : ie;
        const float4 hj = a.ph[j], mj = a.pml[j];
        const uint32_t lj = __float_as_uint(mj.w);
        F2 d[3];
        d[0] = sep(hi.x, hj.x, mi.x, mj.x, b0, byte_float(lj, 0), g.pos_ls);
        d[1] = sep(hi.y, hj.y, mi.y, mj.y, b1, byte_float(lj, 1), g.pos_ls);
        d[2] = sep(hi.z, hj.z, mi.z, mj.z, b2, byte_float(lj, 2), g.pos_ls);
        F2 s = norm2(d);
        // in the cutoff; coincident particles are skipped
        const bool hit = has && (s.hi < 1.f || (s.hi == 1.f && s.lo < 0.f)) && s.hi > 0.f;
        F2 f, h = F2{0.f, 0.f};
        if constexpr (kTab) {
          float centre;
          const int tr = dfm::tab_row(s.hi, centre);  // (a valid row also where nothing is hit)
          const float u = __fsub_rn(s.hi, centre);
          f = tab_lookup(tab0, tr, u, s.lo);
          if constexpr (kMode == kForcePot) h = tab_lookup(tab1, tr, u, s.lo);
          if constexpr (kMode == kVjp) h = tab_lookup(tab1, tr, u, s.lo, tab5[tr]);
          if (hit && s.hi < dfm::kTabMin) dfm::pair_close(a.tab->close, s, kMode == kVjp, f, h);
        } else {
          if (!hit) s = F2{0.5f, 0.f};
          const PairFG o = pair_no_table(a.df, g.kappa_eff, s, kMode == kVjp);
          f = o.f;
          h = o.g;
        }
        f.hi = hit ? f.hi : 0.f;
        f.lo = hit ? f.lo : 0.f;
        if constexpr (kMode == kVjp) {
          h.hi = hit ? h.hi : 0.f;
          h.lo = hit ? h.lo : 0.f;
          const float4 wh = a.w[2 * j], wl = a.w[2 * j + 1];
          const F2 wj[3] = {F2{wh.x, wl.x}, F2{wh.y, wl.y}, F2{wh.z, wl.z}};
          F2 v[3], t[3];
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            v[c] = dfm::two_sum(wi[c].hi, -wj[c].hi);
            v[c] = dfm::fast_two_sum(v[c].hi, __fadd_rn(v[c].lo, __fsub_rn(wi[c].lo, wj[c].lo)));
            t[c] = prod(d[c], v[c]);
          }
          const F2 q0 = dfm::two_sum(t[0].hi, t[1].hi), q1 = dfm::two_sum(q0.hi, t[2].hi);
          F2 dv = dfm::fast_two_sum(
              q1.hi, __fadd_rn(__fadd_rn(q0.lo, q1.lo),
                               __fadd_rn(t[0].lo, __fadd_rn(t[1].lo, t[2].lo))));
          dv = prod(h, dv);
          dv = dfm::fast_two_sum(dv.hi, dv.lo);
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            accumulate(acc[c], prod(f, v[c]));
            accumulate(acc[c], prod(dv, d[c]));
          }
        } else {
#pragma unroll
          for (int c = 0; c < 3; ++c) accumulate(acc[c], prod(f, d[c]));
          if constexpr (kMode == kForcePot)
            accumulate(pa, F2{hit ? h.hi : 0.f, hit ? h.lo : 0.f});
        }
        hits += hit ? 1u : 0u;
        const int took = min(cnt, S);
        head += took;
        cnt -= took;
        if (++evals % kFold == 0) fold();
      }
      fold();
      if (phase == 0)
        np += hits;
      else
        ni += hits;
    }
    // the group's lanes in a fixed tree
    for (int o = 1; o < S; o <<= 1) {
      for (int c = 0; c < 3; ++c) F[c] += __shfl_xor_sync(0xffffffffu, F[c], o);
      if constexpr (kMode == kForcePot) phi += __shfl_xor_sync(0xffffffffu, phi, o);
    }
    if (alive && part == 0) {
      if constexpr (kMode == kVjp) {
        const double sc = a.scale * w_unscale(*a.wbound);
        for (int c = 0; c < 3; ++c) a.acc[3 * static_cast<size_t>(i) + c] = sc * F[c];
      } else {
        a.out[i] = D4{F[0], F[1], F[2], phi};
        e_acc += phi;
      }
    }
  }
  if (kMode == kForcePot && a.energy) block_reduce_add<kThreads64>(e_acc, a.energy);
  if constexpr (kMode != kVjp) {
    warp_add_u64(np, a.pairs);
    warp_add_u64(ni, a.pairs + 1);
    warp_add_u64(ncand, a.pairs + 2);
  }
}

// largest |w| (non-negative doubles order as their bits)
__global__ void k_w_bound(const double* __restrict__ w, int64_t n3,
                          unsigned long long* __restrict__ bound) {
  double b = 0.0;
  for (int64_t t = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; t < n3;
       t += static_cast<int64_t>(gridDim.x) * blockDim.x)
    b = fmax(b, fabs(w[t]));
  for (int o = 16; o > 0; o >>= 1) b = fmax(b, __shfl_xor_sync(0xffffffffu, b, o));
  if ((threadIdx.x & 31) == 0 && b > 0.0)
    atomicMax(bound, static_cast<unsigned long long>(__double_as_longlong(b)));
}

// w in sorted order as double-float, scaled by the power of two that brings the largest |w| to
// [1, 2) (any FP64 magnitude then fits FP32's exponents)
__global__ void k_gather_w64(const uint32_t* __restrict__ total, const Rec64* __restrict__ recm,
                             const double* __restrict__ w,
                             const unsigned long long* __restrict__ bound,
                             float4* __restrict__ ws) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= *total) return;
  const long long idx = rec_index(recm[i]);
  const double sc = w_scale(*bound);
  F2 v[3];
  for (int c = 0; c < 3; ++c) v[c] = dfm::split_double_fp64(w[3 * idx + c] * sc);
  ws[2 * static_cast<size_t>(i)] = make_float4(v[0].hi, v[1].hi, v[2].hi, 0.f);
  ws[2 * static_cast<size_t>(i) + 1] = make_float4(v[0].lo, v[1].lo, v[2].lo, 0.f);
}

// Lanes per particle: 4, doubled while that leaves fewer than two warps per scheduler slot of
// the resident blocks.
int lanes_log2(const p3m_ctx* c, int64_t n) {
  int ls = 2;
  const int64_t want = static_cast<int64_t>(c->num_sms) * 32 * 32;  // 32 warps an SM
  while (ls < 5 && (n << ls) < want) ++ls;
  return ls;
}

template <int kMode, int kRows, bool kTab>
void run64(const p3m_ctx* c, int64_t n, Args64 a, cudaStream_t s) {
  constexpr int kThreads64 = threads64<kMode>(), kWarps64 = kThreads64 / 32;
  constexpr size_t smem =
      tab_bytes<kMode, kTab>() +
      kWarps64 * (sizeof(uint2) * Rows<kRows>::last * 8 + sizeof(uint32_t) * 32 * kRing);
  static_assert(smem + 1024 <= 227 * 1024, "shared memory of one SM");
  auto kern = k_pp64<kMode, kRows, kTab>;
  cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  a.log_s = lanes_log2(c, n);
  const int64_t warps = ((n << a.log_s) + 31) / 32;
  const unsigned blocks = static_cast<unsigned>(
      std::min<int64_t>((warps + kWarps64 - 1) / kWarps64, c->num_sms));
  kern<<<blocks, kThreads64, smem, s>>>(c->g, a);
}

template <int kMode>
void dispatch64(const p3m_ctx* c, int64_t n, const Args64& a, cudaStream_t s) {
  const bool tab = c->ptab != nullptr;
  if (c->g.rows == 1)
    tab ? run64<kMode, 1, true>(c, n, a, s) : run64<kMode, 1, false>(c, n, a, s);
  else if (c->g.rows == 2)
    tab ? run64<kMode, 2, true>(c, n, a, s) : run64<kMode, 2, false>(c, n, a, s);
  else
    tab ? run64<kMode, 3, true>(c, n, a, s) : run64<kMode, 3, false>(c, n, a, s);
}

Args64 args64(const p3m_ctx* c) {
  Args64 a{};
  a.total = c->starts + c->nkeys;
  a.ph = static_cast<const float4*>(c->recp);
  a.pml = a.ph + c->n_max;
  a.starts = c->starts;
  a.tab = c->ptab;
  a.df = c->pdf;
  a.next = c->pp_tile;
  a.pairs = c->pair_acc;
  return a;
}

}  // namespace

cudaError_t pair_table_setup(p3m_ctx* c) {
  std::unique_ptr<dfm::PairTab> tab(new dfm::PairTab());
  if (!dfm::fit_pair_tab(c->g.kappa_eff, *tab)) return cudaSuccess;
  cudaError_t e = cudaMalloc(&c->ptab, sizeof(dfm::PairTab));
  if (e == cudaSuccess)
    e = cudaMemcpy(c->ptab, tab.get(), sizeof(dfm::PairTab), cudaMemcpyHostToDevice);
  return e;
}

void launch_pp64(const p3m_ctx* c, int64_t n, cudaStream_t s, bool want_energy) {
  if (n == 0) return;
  Args64 a = args64(c);
  a.out = static_cast<D4*>(c->fpp);
  // the pair potentials are summed for the energy or the deterministic mode's fixed-order sum
  const bool pot = c->det || want_energy;
  a.energy = pot && !c->det ? c->energy_acc : nullptr;
  if (pot)
    dispatch64<kForcePot>(c, n, a, s);
  else
    dispatch64<kForce>(c, n, a, s);
  if (c->det) launch_det_sum_pp(c, n, s);
}

void launch_pp64_vjp(const p3m_ctx* c, int64_t n, const double* w, cudaStream_t s) {
  if (n == 0) return;
  Args64 a = args64(c);
  float4* ws = static_cast<float4*>(c->fpp);  // the short-range result's memory, not in use here
  a.w = ws;
  a.acc = c->acc;
  a.wbound = c->wbound;
  // d/dxi of (k_e q^2 / r_c^2) f(rho): one more factor 1/r_c
  a.scale = c->g.ke * c->g.q * c->g.q / (c->g.rc * c->g.rc * c->g.rc);
  cudaMemsetAsync(c->wbound, 0, sizeof(unsigned long long), s);
  const int64_t n3 = 3 * n;
  k_w_bound<<<static_cast<unsigned>(std::min<int64_t>((n3 + 255) / 256, 1216)), 256, 0, s>>>(
      w, n3, c->wbound);
  k_gather_w64<<<static_cast<unsigned>((n + 255) / 256), 256, 0, s>>>(
      a.total, static_cast<const Rec64*>(c->recm), w, c->wbound, ws);
  dispatch64<kVjp>(c, n, a, s);
}

}  // namespace p3m
