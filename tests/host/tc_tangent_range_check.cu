// Host program that runs source_tangents (the FP32 dual-number derivatives of the FP64 Newton's
// Jacobian) over the whole range of states (not part of libtc_gb300.so; built and run by
// tests/test_tangent_range.py with the library's csrc/ on the include path).
//
// Prints one JSON object: states, states with a value or derivative that is not finite, and the
// largest error of the derivatives of H/K, C_H2 and C_H+ along ln T against central differences of
// the FP64 terms, over the difference's magnitude and that of the terms (1e99 once one is NaN).
#include <cmath>
#include <cstdio>

#include "tc_kernels.cuh"

using namespace tcg;

namespace {
struct Eval {
  double f[3], terms[3], xe, td;
};
Eval eval(const CellC<double>& c, double T, double x2, double xp) {
  const ChemT<double> b = chem_T(c, T, 0u);
  const CoolT<double> k = cool_T(c, b, 0u);
  const Equil<double> q = equilibrium(c, b, x2, xp, -1.0);
  const Src<double> s = source(c, b, k, x2, xp, 1.0 - 2.0 * x2 - xp, q, -1.0, -1.0);
  const double hk = 1.0 / (c.muH * KB * 1.5);
  return Eval{{(s.G - c.n * s.L) * hk, s.CH2, s.CHp},
              {(s.G + c.n * std::fabs(s.L)) * hk, s.form + s.dest, s.ion + s.rec},
              q.xe,
              s.Td};
}
}  // namespace

int main() {
  DevParams p{1.0, 2.73, 1.0, 1.0, 1.0 / 3.0, 0.1, 1e-3, 1e-12, 1e-6, 1.0, 50, 1000000, 0};
  const double ns[] = {1e-4, 1e-2, 1, 100, 1e4, 1e6}, x2s[] = {0, 1e-30, 1e-12, 1e-3, 0.4999},
               xps[] = {0, 1e-45, 1e-30, 1e-6, 0.5, 1.0 - 1e-9}, xis[] = {0, 2e-16, 1e-13}, Fs[] = {0, 1e9},
               Zs[] = {1e-3, 1, 3}, chis[] = {0, 1e-3, 1, 1e4};
  long long total = 0, bad = 0;
  double worst[3] = {0, 0, 0};
  for (int i = 0; i <= 36; ++i)
    for (double n : ns)
      for (double x2 : x2s)
        for (double xp : xps)
          for (double xi : xis)
            for (double F : Fs)
              for (double Z : Zs)
                for (double chi : chis) {
                  if (2.0 * x2 + xp > 1.0) continue;
                  const double T = std::pow(10.0, 0.25 * i) * ((i == 0) ? 1.0 : 0.93);  // off the clamps at 10 and 1e4 K
                  const CellC<double> c = make_cell(n, chi, chi, 0.5, 1.0, F, xi, Z, Z, p);
                  const CellC<float> cf = cast_cell<float>(c);
                  const Eval e = eval(c, T, x2, xp);
                  const float hk = float(1.0 / (c.muH * KB * 1.5));
                  bool fine = true;
                  float df[3][3], dq[3][3];
                  Tan32 v;
                  for (int pass = 0; pass < 2; ++pass) {
                    source_tangents(cf, 0u, hk, float(T), float(x2), float(xp), float(1.0 - 2.0 * x2 - xp), float(e.xe),
                                    float(e.td), df, dq, 0, 3, (pass == 0) ? &v : nullptr);
                    for (int r = 0; r < 3; ++r)
                      for (int j = 0; j < 3; ++j) fine = fine && std::isfinite(df[r][j]) && std::isfinite(dq[r][j]);
                  }
                  for (int r = 0; r < 3; ++r) fine = fine && std::isfinite(v.f[r]) && std::isfinite(v.dtd[r]);
                  fine = fine && std::isfinite(v.xe) && std::isfinite(v.td);
                  ++total;
                  if (!fine) ++bad;
                  const Eval a = eval(c, T * std::exp(1e-5), x2, xp), b = eval(c, T * std::exp(-1e-5), x2, xp);
                  for (int r = 0; r < 3; ++r) {
                    const double d = (a.f[r] - b.f[r]) / 2e-5;
                    const double err = std::fabs(df[r][0] - d) / (std::fabs(d) + e.terms[r] + 1e-36);
                    if (!std::isnan(worst[r]) && !(err <= worst[r])) worst[r] = err;
                  }
                }
  for (double& w : worst)
    if (std::isnan(w)) w = 1e99;
  printf("{\"states\": %lld, \"bad\": %lld, \"H\": %.3e, \"CH2\": %.3e, \"CHp\": %.3e}\n", total, bad, worst[0], worst[1],
         worst[2]);
  return 0;
}
