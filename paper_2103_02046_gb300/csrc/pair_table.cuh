// Interval table of the short-range pair function for the FP64 path.
//
// In cutoff units the force coefficient, the potential and the adjoint's Hessian term of a pair
// depend on s = rho^2 alone. Each is tabulated on [2^-8, 1): every octave of s is cut into 256
// intervals (numbered by the leading 8 mantissa bits of s), and on each interval the function is a
// polynomial of degree 4 in u = s - c, c the interval's centre, |u| <= s / 512. Each degree then
// adds a factor of about 2^-8, so degrees 3 and 4 are evaluated in FP32 (together they are below
// 2^-25 of the value) and degrees 0 to 2 in double-float (Horner with one error-free product and
// sum per degree). That is about 30 FP32 operations and two 16-byte loads for a value, in place of
// the reciprocal square root, the fitted erfc(x) e^{x^2} of degree 12 and the exponential of
// df_math.cuh (about 700 operations). Pairs closer than r_c / 16 (s < 2^-8; 2.4e-4 of uniformly
// spread neighbours) take the series of the same functions about s = 0.
//
// Written so that it compiles as host code too (the host evaluation backs a CPU test).
#pragma once

#include <cmath>
#include <cstdint>

#include "df_math.cuh"

namespace dfm {

constexpr int kTabOctaves = 8;
constexpr int kTabPerOctave = 256;
constexpr int kTabRows = kTabOctaves * kTabPerOctave;
constexpr uint32_t kTabShift = 15;             // 23 mantissa bits less the 8 that number the row
constexpr uint32_t kTabBase = 0x3b800000u >> kTabShift;  // 2^-8
constexpr float kTabMin = 0.00390625f;         // 2^-8
constexpr double kTabMaxKappa = 6.5;
// accepted error of a table, relative to the unscreened pair term (a pair's screened term is a
// small fraction of it near the cutoff, where the neighbours within dominate the sum)
constexpr double kTabTol = 2e-14;

struct alignas(16) Quad {
  float c[4];
};
// One function's rows: {c0 hi, c0 lo, c1 hi, c1 lo} and {c2 hi, c2 lo, c3, c4}, in two arrays so
// that 16-byte reads of different rows spread over all shared-memory banks.
struct TabFn {
  Quad a[kTabRows], b[kTabRows];
};
// Close pairs: with x = kappa rho, erfc(x) = 1 - erf(x), and erf(x) / rho and the Gaussian term are
// even power series in rho, so fco = s^{-3/2} - P(s), pot = s^{-1/2} - Q(s) and
// dfr = -3 s^{-5/2} - 2 P'(s). The correction is below 2^-4 of the first term at s = 2^-8 (kappa
// up to 6.5), and its terms fall by x^2 <= 0.166 and their factorials.
constexpr int kCloseTerms = 9;
struct CloseSeries {
  F2 p[kCloseTerms], q[kCloseTerms];
};
struct PairTab {
  TabFn fco, pot, dfr;
  float dfr5[kTabRows];  // c5 of dfr, whose terms fall more slowly
  CloseSeries close;
};

DFM_HD uint32_t bits_of_f(float v) {
#if defined(__CUDA_ARCH__)
  return __float_as_uint(v);
#else
  uint32_t b;
  memcpy(&b, &v, sizeof b);
  return b;
#endif
}

// Row of s and its centre, s in [2^-8, 1). Any other s takes the last row (a finite value, which
// the caller discards or replaces).
DFM_HD int tab_row(float s, float& centre) {
  uint32_t r = (bits_of_f(s) >> kTabShift) - kTabBase;
  r = r < static_cast<uint32_t>(kTabRows) ? r : static_cast<uint32_t>(kTabRows - 1);
  centre = float_of(((r + kTabBase) << kTabShift) | (1u << (kTabShift - 1)));
  return static_cast<int>(r);
}

// one Horner step in double-float: c + (u + ul) R, |c| > |u R|
DFM_HD F2 tab_step(F2 R, float u, float ul, float ch, float cl) {
  const float p = mul_rn(u, R.hi);
  float e = fma_rn(u, R.hi, -p);
  e = fma_rn(u, R.lo, e);
  e = fma_rn(ul, R.hi, e);
  const float h = add_rn(ch, p);
  const float err = sub_rn(p, sub_rn(h, ch));
  return F2{h, add_rn(err, add_rn(cl, e))};
}

// the polynomial of one row at u + ul (u = s.hi - c exactly, ul = s.lo); c5 of dfr, else 0
DFM_HD F2 tab_eval(const float* a, const float* b, float u, float ul, float c5 = 0.f) {
  F2 R = F2{fma_rn(fma_rn(c5, u, b[3]), u, b[2]), 0.f};
  R = tab_step(R, u, ul, b[0], b[1]);
  R = tab_step(R, u, ul, a[2], a[3]);
  return tab_step(R, u, ul, a[0], a[1]);
}

// fco and (hess ? dfr : pot) for 0 < s < 2^-8
DFM_HD void pair_close(const CloseSeries& C, F2 s, bool hess, F2& f, F2& g) {
  const F2 rinv = rsqrt_df(s);
  const F2 r2inv = mul(rinv, rinv), r3inv = mul(r2inv, rinv);
  F2 p = C.p[kCloseTerms - 1];
  for (int k = kCloseTerms - 2; k >= 0; --k) p = add(mul(p, s), C.p[k]);
  f = sub(r3inv, p);
  if (hess) {
    F2 d = mul_f(C.p[kCloseTerms - 1], static_cast<float>(kCloseTerms - 1));
    for (int k = kCloseTerms - 2; k >= 1; --k) d = add(mul(d, s), mul_f(C.p[k], static_cast<float>(k)));
    g = neg(add(mul_f(mul(r3inv, r2inv), 3.f), mul_f(d, 2.f)));
  } else {
    F2 q = C.q[kCloseTerms - 1];
    for (int k = kCloseTerms - 2; k >= 0; --k) q = add(mul(q, s), C.q[k]);
    g = sub(rinv, q);
  }
}

// ---- host side: the fit ----
// Fills the table for kappa = alpha r_c in (0, 6.5]; false if some row misses kTabTol.
inline bool fit_pair_tab(double kappa, PairTab& T) {
  if (!(kappa > 0.0) || kappa > kTabMaxKappa) return false;
  constexpr int N = 6;  // coefficients (dfr; the others one less)
  const double pi = 3.14159265358979323846;
  const double c2k = 2.0 * kappa / std::sqrt(pi);
  auto split = [](double v) {
    const float h = static_cast<float>(v);
    return F2{h, static_cast<float>(v - static_cast<double>(h))};
  };
  // erf(x) = (2/sqrt(pi)) sum (-1)^k x^{2k+1} / (k! (2k+1)); with e^{-x^2} = sum (-1)^k x^{2k} / k!:
  //   Q_k = c2k (-1)^k kappa^{2k} / (k! (2k+1)),
  //   s P(s) = Q(s) - c2k e^{-kappa^2 s}: P_k = Q_{k+1} - c2k (-1)^{k+1} kappa^{2k+2} / (k+1)!
  {
    double t = c2k;  // c2k (-1)^k kappa^{2k} / k!
    for (int k = 0; k <= kCloseTerms; ++k) {
      const double q = t / (2 * k + 1);
      if (k < kCloseTerms) T.close.q[k] = split(q);
      if (k > 0) T.close.p[k - 1] = split(q - t);
      t *= -kappa * kappa / (k + 1);
    }
  }
  // the functions at s (0 fco, 1 pot, 2 dfr)
  auto value = [&](double s, double out[3]) {
    const double r = std::sqrt(s), x = kappa * r;
    const double ex = c2k * std::exp(-x * x), pot = std::erfc(x) / r, A = pot + ex;
    out[0] = A / s;
    out[1] = pot;
    // A' = -A / r - 2 kappa^2 r ex; dfr = (A'/s - 2 A/(s r)) / r
    out[2] = (-A / r - 2.0 * kappa * kappa * r * ex - 2.0 * A / r) / (s * r);
  };
  double node[2][N], cosk[2][N][N];  // [0]: 5 coefficients, [1]: 6
  for (int t = 0; t < 2; ++t)
    for (int j = 0; j < N - 1 + t; ++j) {
      node[t][j] = std::cos(pi * (j + 0.5) / (N - 1 + t));
      for (int k = 0; k < N - 1 + t; ++k) cosk[t][k][j] = std::cos(k * pi * (j + 0.5) / (N - 1 + t));
    }
  TabFn* fn[3] = {&T.fco, &T.pot, &T.dfr};
  for (int r = 0; r < kTabRows; ++r) {
    const double c = float_of(((static_cast<uint32_t>(r) + kTabBase) << kTabShift) |
                              (1u << (kTabShift - 1)));
    const double hw = c - float_of((static_cast<uint32_t>(r) + kTabBase) << kTabShift);
    double v[2][N][3];
    for (int t = 0; t < 2; ++t)
      for (int j = 0; j < N - 1 + t; ++j) value(c + hw * node[t][j], v[t][j]);
    for (int f = 0; f < 3; ++f) {
      // Chebyshev coefficients, then monomials in u / hw (T_{k+1} = 2 t T_k - T_{k-1})
      const int t = f == 2 ? 1 : 0, n = N - 1 + t;
      double mono[N] = {}, tm[N] = {}, tk[N] = {}, tp[N];
      tm[0] = 1.0;
      tk[1] = 1.0;
      for (int k = 0; k < n; ++k) {
        double ch = 0.0;
        for (int j = 0; j < n; ++j) ch += v[t][j][f] * cosk[t][k][j];
        ch *= (k == 0 ? 1.0 : 2.0) / n;
        for (int m = 0; m < N; ++m) mono[m] += ch * tm[m];
        for (int m = 0; m < N; ++m) tp[m] = (m > 0 ? 2.0 * tk[m - 1] : 0.0) - tm[m];
        for (int m = 0; m < N; ++m) tm[m] = tk[m], tk[m] = tp[m];
      }
      const F2 c0 = split(mono[0]), c1 = split(mono[1] / hw), c2 = split(mono[2] / (hw * hw));
      fn[f]->a[r] = Quad{{c0.hi, c0.lo, c1.hi, c1.lo}};
      fn[f]->b[r] = Quad{{c2.hi, c2.lo, static_cast<float>(mono[3] / (hw * hw * hw)),
                          static_cast<float>(mono[4] / (hw * hw * hw * hw))}};
      if (f == 2) T.dfr5[r] = static_cast<float>(mono[5] / (hw * hw * hw * hw * hw));
    }
    // the rows' error at the ends and between, against the unscreened terms 1/rho^3, 1/rho, 3/rho^5
    for (int q = -2; q <= 2; ++q) {
      const double u = 0.5 * q * hw * (1.0 - 1e-7), s = c + u;
      const double top[3] = {1.0 / (s * std::sqrt(s)), 1.0 / std::sqrt(s),
                             3.0 / (s * s * std::sqrt(s))};
      double ref[3];
      value(s, ref);
      for (int f = 0; f < 3; ++f) {
        const float *a = fn[f]->a[r].c, *b = fn[f]->b[r].c;
        auto two = [](const float* h) { return static_cast<double>(h[0]) + static_cast<double>(h[1]); };
        const double c5 = f == 2 ? T.dfr5[r] : 0.0;
        const double y = ((((c5 * u + b[3]) * u + b[2]) * u + two(b)) * u + two(a + 2)) * u + two(a);
        if (!(std::fabs(y - ref[f]) <= kTabTol * top[f])) return false;
      }
    }
  }
  return true;
}

}  // namespace dfm
