// Host check of the FP64 path's pair-function table (csrc/pair_table.cuh) against long-double erfc
// and exp, for kappa = alpha r_c given on the command line: over pairs spread uniformly in the
// cutoff sphere (rho = cbrt(u)) the error of the force coefficient, the potential and the Hessian
// term, weighted with the pair force (rho fco, pot, rho^2 dfr) and relative to its root mean
// square, of the table and of the double-float functions of df_math.cuh; the largest error at the
// rows' edges relative to the unscreened terms; and the largest relative error of the close-pair
// series. One JSON line.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <memory>

#include "pair_table.cuh"

int main(int argc, char** argv) {
  const double kappa = argc > 1 ? std::atof(argv[1]) : 3.0;
  std::unique_ptr<dfm::PairTab> T(new dfm::PairTab());
  std::unique_ptr<dfm::PairDF> P(new dfm::PairDF());
  const bool fit = dfm::fit_pair_tab(kappa, *T) && dfm::fit_pair_df(kappa, *P);
  const long double pi = 3.14159265358979323846264338327950288L;
  double tab[3] = {}, df[3] = {}, norm[3] = {}, edge[3] = {};
  auto exact = [&](long double s, long double out[3]) {
    const long double r = sqrtl(s), x = kappa * r, ex = 2.0L * kappa / sqrtl(pi) * expl(-x * x);
    const long double pot = erfcl(x) / r, A = pot + ex;
    out[0] = A / s;
    out[1] = pot;
    out[2] = (-A / r - 2.0L * kappa * kappa * r * ex - 2.0L * A / r) / (s * r);
  };
  auto lookup = [&](dfm::F2 s, dfm::F2 out[3]) {
    float c;
    const int row = dfm::tab_row(s.hi, c);
    const float u = dfm::sub_rn(s.hi, c);
    out[0] = dfm::tab_eval(T->fco.a[row].c, T->fco.b[row].c, u, s.lo);
    out[1] = dfm::tab_eval(T->pot.a[row].c, T->pot.b[row].c, u, s.lo);
    out[2] = dfm::tab_eval(T->dfr.a[row].c, T->dfr.b[row].c, u, s.lo, T->dfr5[row]);
  };
  for (int k = 0; fit && k < 100000; ++k) {
    const double rho = std::cbrt((k + 0.5) / 100000.0), sv = rho * rho;
    if (sv < dfm::kTabMin) continue;
    const dfm::F2 s = dfm::split_double_fp64(sv);
    const long double sl = static_cast<long double>(s.hi) + s.lo;
    long double ref[3];
    exact(sl, ref);
    dfm::F2 t[3], d[3];
    lookup(s, t);
    const dfm::PairOut o = dfm::pair_df(P->k, P->coef, s);
    dfm::pair_hess_df(P->k, P->coef, s, d[0], d[2]);
    d[0] = o.fco;
    d[1] = o.pot;
    const double w[3] = {rho, 1.0, sv};
    for (int f = 0; f < 3; ++f) {
      const double a = w[f] * static_cast<double>(static_cast<long double>(t[f].hi) + t[f].lo - ref[f]);
      const double b = w[f] * static_cast<double>(static_cast<long double>(d[f].hi) + d[f].lo - ref[f]);
      const double c = w[f] * static_cast<double>(ref[f]);
      tab[f] += a * a;
      df[f] += b * b;
      norm[f] += c * c;
    }
  }
  // both ends of every row, one float inside
  for (int r = 0; fit && r < dfm::kTabRows; ++r)
    for (int side = 0; side < 2; ++side) {
      const uint32_t b = (static_cast<uint32_t>(r) + dfm::kTabBase) << dfm::kTabShift;
      const dfm::F2 s{dfm::float_of(side ? b + (1u << dfm::kTabShift) - 1u : b), 0.f};
      long double ref[3];
      exact(s.hi, ref);
      dfm::F2 t[3];
      lookup(s, t);
      const double top[3] = {std::pow(s.hi, -1.5), std::pow(s.hi, -0.5), 3.0 * std::pow(s.hi, -2.5)};
      for (int f = 0; f < 3; ++f)
        edge[f] = std::fmax(edge[f], std::fabs(static_cast<double>(
                                         static_cast<long double>(t[f].hi) + t[f].lo - ref[f])) / top[f]);
    }
  // close pairs: the series on (0, 2^-8), relative errors
  double close[3] = {};
  for (int k = 1; fit && k <= 20000; ++k) {
    const double sv = dfm::kTabMin * std::pow(k / 20001.0, 4.0);
    const dfm::F2 s = dfm::split_double_fp64(sv);
    long double ref[3];
    exact(static_cast<long double>(s.hi) + s.lo, ref);
    dfm::F2 t[3], f2;
    dfm::pair_close(T->close, s, false, t[0], t[1]);
    dfm::pair_close(T->close, s, true, f2, t[2]);
    for (int f = 0; f < 3; ++f)
      close[f] = std::fmax(close[f], std::fabs(static_cast<double>(
                                         (static_cast<long double>(t[f].hi) + t[f].lo) / ref[f] - 1.0L)));
  }
  std::printf("{\"fit\": %s, \"close\": [%.3e, %.3e, %.3e]", fit ? "true" : "false", close[0],
              close[1], close[2]);
  const char* name[3] = {"fco", "pot", "dfr"};
  for (int f = 0; f < 3; ++f)
    std::printf(", \"%s\": [%.3e, %.3e, %.3e]", name[f], std::sqrt(tab[f] / norm[f]),
                std::sqrt(df[f] / norm[f]), edge[f]);
  std::printf("}\n");
  return 0;
}
