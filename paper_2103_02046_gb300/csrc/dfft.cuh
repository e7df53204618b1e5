// Complex arithmetic and column transforms for the FP64 path's mesh solve, in double-float (CD) and
// in FP64 (CZ). Double-float: every real is an unevaluated sum hi + lo of two FP32 numbers (about 48
// significant bits), so the butterflies run on GB300's FP32 pipes instead of its scarce FP64 units.
//
// Transforms: power-of-two lengths in [16, 2048], radix-8 Stockham autosort passes (then one
// radix-4 or radix-2 pass when the length's logarithm is not a multiple of 3) in shared memory;
// twiddles from tables computed on the host in extended precision.
#pragma once

#include "df_math.cuh"
#include "p3m_internal.cuh"

namespace p3m {

using dfm::F2;

// complex double-float
struct alignas(16) CD {
  F2 x, y;
};

// Double-float sum with one error-free transformation of the leading parts: its error is
// bounded by a few units of 2^-48 times |a| + |b| (a normwise bound, which is what a transform's
// error analysis uses), at half the cost of the fully renormalised sum.
__device__ __forceinline__ F2 dadd(F2 a, F2 b) {
  const F2 s = dfm::two_sum(a.hi, b.hi);
  return dfm::fast_two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo)));
}
__device__ __forceinline__ F2 dsub(F2 a, F2 b) { return dadd(a, dfm::neg(b)); }

__device__ __forceinline__ CD cd_add(CD a, CD b) { return CD{dadd(a.x, b.x), dadd(a.y, b.y)}; }
__device__ __forceinline__ CD cd_sub(CD a, CD b) { return CD{dsub(a.x, b.x), dsub(a.y, b.y)}; }
__device__ __forceinline__ CD cd_mul(CD a, CD b) {
  return CD{dsub(dfm::mul(a.x, b.x), dfm::mul(a.y, b.y)),
            dadd(dfm::mul(a.x, b.y), dfm::mul(a.y, b.x))};
}
// a * (s i), s = +-1 (exact)
__device__ __forceinline__ CD cd_mul_si(CD a, float s) {
  return s > 0.f ? CD{dfm::neg(a.y), a.x} : CD{a.y, dfm::neg(a.x)};
}

// the same in FP64
struct alignas(16) CZ {
  double x, y;
};
__device__ __forceinline__ CZ cd_add(CZ a, CZ b) { return CZ{a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ CZ cd_sub(CZ a, CZ b) { return CZ{a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ CZ cd_mul(CZ a, CZ b) {
  return CZ{fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x)};
}
__device__ __forceinline__ CZ cd_mul_si(CZ a, float s) {
  return s > 0.f ? CZ{-a.y, a.x} : CZ{a.y, -a.x};
}
constexpr double kHalfSqrt2 = 0.70710678118654752440;
__device__ __forceinline__ CZ w8_1(CZ a, float s) {
  return s > 0.f ? CZ{kHalfSqrt2 * (a.x - a.y), kHalfSqrt2 * (a.y + a.x)}
                 : CZ{kHalfSqrt2 * (a.x + a.y), kHalfSqrt2 * (a.y - a.x)};
}
__device__ __forceinline__ CZ w8_3(CZ a, float s) {
  return s > 0.f ? CZ{-kHalfSqrt2 * (a.x + a.y), kHalfSqrt2 * (a.x - a.y)}
                 : CZ{kHalfSqrt2 * (a.y - a.x), -kHalfSqrt2 * (a.y + a.x)};
}
__device__ __forceinline__ CZ conj_of(CZ a) { return CZ{a.x, -a.y}; }
__device__ __forceinline__ CD conj_of(CD a) { return CD{a.x, dfm::neg(a.y)}; }
template <typename E>
__device__ __forceinline__ E c_zero() {
  return E{};
}

__device__ __forceinline__ CD cd_zero() { return CD{F2{0.f, 0.f}, F2{0.f, 0.f}}; }
__device__ __forceinline__ double d_of(F2 a) {
  return static_cast<double>(a.hi) + static_cast<double>(a.lo);
}
__device__ __forceinline__ double2 cd_to(CD a) { return make_double2(d_of(a.x), d_of(a.y)); }
// the charge spectrum's doubles, split without FP64 instructions
__device__ __forceinline__ CD cd_split(double2 v) {
  return CD{dfm::split_double(v.x), dfm::split_double(v.y)};
}

// sqrt(1/2) in double-float
__device__ __forceinline__ F2 half_sqrt2() {
  return F2{0.70710677f, 1.21016175e-08f};  // the leading 24 bits and the next 24
}

// (a.x - s a.y, a.y + s a.x) sqrt(1/2): a times the eighth root h (1 + s i)
__device__ __forceinline__ CD w8_1(CD a, float s) {
  const F2 h = half_sqrt2();
  const F2 re = s > 0.f ? dsub(a.x, a.y) : dadd(a.x, a.y);
  const F2 im = s > 0.f ? dadd(a.y, a.x) : dsub(a.y, a.x);
  return CD{dfm::mul(re, h), dfm::mul(im, h)};
}
// (-a.x - s a.y, -a.y + s a.x) sqrt(1/2): a times h (-1 + s i)
__device__ __forceinline__ CD w8_3(CD a, float s) {
  const F2 h = half_sqrt2();
  const F2 re = s > 0.f ? dfm::neg(dadd(a.x, a.y)) : dsub(a.y, a.x);
  const F2 im = s > 0.f ? dsub(a.x, a.y) : dfm::neg(dadd(a.y, a.x));
  return CD{dfm::mul(re, h), dfm::mul(im, h)};
}

// R-point DFTs in registers: u_s <- sum_r u_r e^{sign 2 pi i r s / R}.
template <typename E>
__device__ __forceinline__ void ddft2(E& a, E& b) {
  const E t = a;
  a = cd_add(t, b);
  b = cd_sub(t, b);
}

template <typename E>
__device__ __forceinline__ void ddft4(E& u0, E& u1, E& u2, E& u3, float sign) {
  const E t0 = cd_add(u0, u2), t1 = cd_sub(u0, u2);
  const E t2 = cd_add(u1, u3), t3 = cd_mul_si(cd_sub(u1, u3), sign);
  u0 = cd_add(t0, t2);
  u2 = cd_sub(t0, t2);
  u1 = cd_add(t1, t3);
  u3 = cd_sub(t1, t3);
}

// even and odd halves as two 4-point DFTs, joined with the eighth roots of unity
template <typename E>
__device__ __forceinline__ void ddft8_join(E (&u)[8], E e0, E e1, E e2, E e3, E o0, E o1, E o2,
                                           E o3, float sign) {
  o1 = w8_1(o1, sign);
  o2 = cd_mul_si(o2, sign);
  o3 = w8_3(o3, sign);
  u[0] = cd_add(e0, o0);
  u[4] = cd_sub(e0, o0);
  u[1] = cd_add(e1, o1);
  u[5] = cd_sub(e1, o1);
  u[2] = cd_add(e2, o2);
  u[6] = cd_sub(e2, o2);
  u[3] = cd_add(e3, o3);
  u[7] = cd_sub(e3, o3);
}

template <typename E>
__device__ __forceinline__ void ddft8(E (&u)[8], float sign) {
  E e0 = u[0], e1 = u[2], e2 = u[4], e3 = u[6];
  E o0 = u[1], o1 = u[3], o2 = u[5], o3 = u[7];
  ddft4(e0, e1, e2, e3, sign);
  ddft4(o0, o1, o2, o3, sign);
  ddft8_join(u, e0, e1, e2, e3, o0, o1, o2, o3, sign);
}

// ddft8 for u_4 .. u_7 = 0: the even and odd 4-point DFTs each have two non-zero inputs
template <typename E>
__device__ __forceinline__ void ddft8_lower_inputs(E (&u)[8], float sign) {
  const E x0 = u[0], x1 = u[1], x2 = u[2], x3 = u[3];
  const E x2s = cd_mul_si(x2, sign), x3s = cd_mul_si(x3, sign);
  ddft8_join(u, cd_add(x0, x2), cd_add(x0, x2s), cd_sub(x0, x2), cd_sub(x0, x2s), cd_add(x1, x3),
             cd_add(x1, x3s), cd_sub(x1, x3), cd_sub(x1, x3s), sign);
}

// shared-memory index with one pad element per 16
__host__ __device__ __forceinline__ int dpad(int i) { return i + (i >> 4); }
// elements from one column to the next: odd, so that 16-byte accesses across columns (the global
// loads and stores run over consecutive columns) fall in different banks
__host__ __device__ __forceinline__ int dcolumn(int N) { return dpad(N) | 1; }

enum DPassKind { kDGeneral = 0, kDFirstHalf = 1, kDLastLower = 2 };

// One Stockham pass of radix R on one column of length N = 2^logN after passes whose radices
// multiply to p = 2^logp: butterfly i (of N / R) reads u_r = x[i + r N/R], applies the twiddles
// e^{sign 2 pi i r k / (p R)}, k = i mod p, takes the R-point DFT and writes
// y[(i - k) R + k + r p]. Each thread does 8 / R butterflies; reads and writes are separated by
// a barrier, so the pass runs in place. kDFirstHalf: inputs r >= R/2 are zero (and p = 1);
// kDLastLower: only outputs r < R/2 are kept.
template <int R, int kKind, typename E>
__device__ __forceinline__ void dpass(E* a, int logN, int logp, int i0, int tpc, float sign,
                                      const E* __restrict__ tw) {
  constexpr int kB = 8 / R;
  constexpr int kLogR = R == 8 ? 3 : (R == 4 ? 2 : 1);
  constexpr int kIn = kKind == kDFirstHalf ? R / 2 : R;
  constexpr int kOut = kKind == kDLastLower ? R / 2 : R;
  const int T = (1 << logN) >> kLogR;
  E u[kB][R];
#pragma unroll
  for (int q = 0; q < kB; ++q)
#pragma unroll
    for (int r = 0; r < R; ++r) u[q][r] = r < kIn ? a[dpad(i0 + q * tpc + r * T)] : c_zero<E>();
  __syncthreads();
  const int p = 1 << logp;
  const int tshift = logN - logp - kLogR;  // twiddle table step N / (p R)
#pragma unroll
  for (int q = 0; q < kB; ++q) {
    const int i = i0 + q * tpc;
    const int k = i & (p - 1);
    if (kKind != kDFirstHalf && logp > 0) {
#pragma unroll
      for (int r = 1; r < R; ++r) {
        E w = tw[(r * k) << tshift];             // e^{-2 pi i r k / (p R)}
        if (sign > 0.f) w = conj_of(w);          // for the inverse
        u[q][r] = cd_mul(u[q][r], w);
      }
    }
    if constexpr (R == 8) {
      if constexpr (kKind == kDFirstHalf)
        ddft8_lower_inputs(u[q], sign);
      else
        ddft8(u[q], sign);
    } else if constexpr (R == 4) {
      ddft4(u[q][0], u[q][1], u[q][2], u[q][3], sign);
    } else {
      ddft2(u[q][0], u[q][1]);
    }
    const int j = ((i - k) << kLogR) + k;
#pragma unroll
    for (int r = 0; r < kOut; ++r) a[dpad(j + r * p)] = u[q][r];
  }
  __syncthreads();
}

template <int kKind, typename E>
__device__ __forceinline__ void drun_pass(int R, E* a, int logN, int logp, int i0, int tpc,
                                          float sign, const E* __restrict__ tw) {
  if (R == 8)
    dpass<8, kKind>(a, logN, logp, i0, tpc, sign, tw);
  else if (R == 4)
    dpass<4, kKind>(a, logN, logp, i0, tpc, sign, tw);
  else
    dpass<2, kKind>(a, logN, logp, i0, tpc, sign, tw);
}

// Forward transform (sign -1) of a column that is zero in its upper half, or inverse transform
// (sign +1) of which only the lower half is kept; unnormalised, length 2^logN >= 16.
template <bool kForward, typename E>
__device__ void dcolumn_fft(E* a, int logN, int i0, int tpc, const E* __restrict__ tw) {
  const float sign = kForward ? -1.f : 1.f;
  const int npass = (logN + 2) / 3;
  for (int q = 0, logp = 0; q < npass; ++q) {
    const int logR = (logN - logp) >= 3 ? 3 : logN - logp;
    const int R = 1 << logR;
    if (kForward && q == 0)
      drun_pass<kDFirstHalf>(R, a, logN, logp, i0, tpc, sign, tw);
    else if (!kForward && q == npass - 1)
      drun_pass<kDLastLower>(R, a, logN, logp, i0, tpc, sign, tw);
    else
      drun_pass<kDGeneral>(R, a, logN, logp, i0, tpc, sign, tw);
    logp += logR;
  }
}

}  // namespace p3m
