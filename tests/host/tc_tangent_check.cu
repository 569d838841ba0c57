// Host program that checks source_tangents (the FP32 dual-number derivatives of the
// source terms and of the C/O/e equilibrium, the FP64 Newton's Jacobian) against central
// differences of the FP64 evaluation (not part of libtc_gb300.so; built and run by
// tests/test_tangent.py with the library's csrc/ on the include path).
//
// Usage: tc_tangent_check IN
//   IN: n as int64, then 12 arrays of n doubles (n, chi_pe, chi_lw, f_shld_H2, f_shld_C,
//       F_LyC, xi, Z'_g, Z'_d, T, x_H2, x_H+), then dt as a double (unused).
// Prints one JSON object: per derivative, the largest |dual - difference| over the sum of
// the difference's magnitude and that of the terms it is a difference of.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <vector>

#include "tc_kernels.cuh"

using namespace tcg;

namespace {
struct Eval {
  double f[3], q[3], terms[3], qterms[3], xe, td;
};
Eval eval(const CellC<double>& c, unsigned flags, double T, double x2, double xp) {
  const ChemT<double> b = chem_T(c, T, flags);
  const CoolT<double> k = cool_T(c, b, flags);
  const Equil<double> q = equilibrium(c, b, x2, xp, -1.0);
  const Src<double> s = source(c, b, k, x2, xp, 1.0 - 2.0 * x2 - xp, q, -1.0, -1.0);
  const double hk = 1.0 / (c.muH * KB * 1.5);
  Eval e;
  e.f[0] = (s.G - c.n * s.L) * hk; e.f[1] = s.CH2; e.f[2] = s.CHp;
  e.q[0] = q.xe; e.q[1] = q.xCp; e.q[2] = q.xCO;
  e.terms[0] = (s.G + c.n * std::fabs(s.L)) * hk;
  e.terms[1] = s.form + s.dest;
  e.terms[2] = s.ion + s.rec;
  e.qterms[0] = q.xe;
  e.qterms[1] = q.xCp;
  e.qterms[2] = 2.0 * c.xCtot * x2 / (1.0 + c.rCO2);  // of x_CO = 2 x_C x_H2 (1 - f) / (1 + r)
  e.xe = q.xe;
  e.td = s.Td;
  return e;
}
}  // namespace

int main(int argc, char** argv) {
  if (argc != 2) return 2;
  FILE* fh = fopen(argv[1], "rb");
  if (!fh) return 3;
  int64_t n = 0;
  if (fread(&n, 8, 1, fh) != 1 || n <= 0) return 4;
  std::vector<double> in(12 * (size_t)n);
  if (fread(in.data(), 8, in.size(), fh) != in.size()) return 5;
  fclose(fh);
  auto col = [&](int k) { return in.data() + (size_t)k * n; };
  DevParams p{1.0, 2.73, 1.0, 1.0, 1.0 / 3.0, 0.1, 1e-3, 1e-12, 1e-6, 1.0, 50, 1000000, 0};
  const unsigned flag_sets[2] = {0u, FL_CONST_KGR | FL_NO_ROVIB | FL_NO_CIE};
  double worst_f[3][3] = {{0}}, worst_q[3][3] = {{0}};
  for (int64_t i = 0; i < n; ++i) {
    const CellC<double> c = make_cell(col(0)[i], col(1)[i], col(2)[i], col(3)[i], col(4)[i], col(5)[i], col(6)[i],
                                      col(7)[i], col(8)[i], p);
    const CellC<float> cf = cast_cell<float>(c);
    const double T = col(9)[i], x2 = col(10)[i], xp = col(11)[i];
    for (unsigned flags : flag_sets) {
      const Eval e = eval(c, flags, T, x2, xp);
      float df[3][3], dq[3][3];
      source_tangents(cf, flags, float(1.0 / (c.muH * KB * 1.5)), float(T), float(x2), float(xp),
                      float(1.0 - 2.0 * x2 - xp), float(e.xe), float(e.td), df, dq);
      // central differences over a relative 2e-5 of each unknown; the scale of a
      // derivative along an abundance is its unknown's
      const double u[3] = {1.0, x2, xp};
      for (int j = 0; j < 3; ++j) {
        const double h = 1e-5 * u[j];
        if (!(h > 1e-12)) continue;  // the difference would be rounding
        const Eval a = eval(c, flags, (j == 0) ? T * std::exp(h) : T, x2 + (j == 1) * h, xp + (j == 2) * h);
        const Eval b = eval(c, flags, (j == 0) ? T * std::exp(-h) : T, x2 - (j == 1) * h, xp - (j == 2) * h);
        for (int r = 0; r < 3; ++r) {
          const double d = (a.f[r] - b.f[r]) / (2.0 * h), dd = (a.q[r] - b.q[r]) / (2.0 * h);
          const double ef = std::fabs(df[r][j] - d) / (std::fabs(d) + e.terms[r] / u[j]);
          const double eq = std::fabs(dq[r][j] - dd) / (std::fabs(dd) + e.qterms[r] / u[j] + 1e-30);
          if (!(ef <= worst_f[r][j])) worst_f[r][j] = ef;
          if (!(eq <= worst_q[r][j])) worst_q[r][j] = eq;
        }
      }
    }
  }
  const char* fn[3] = {"H", "CH2", "CHp"};
  const char* qn[3] = {"xe", "xCp", "xCO"};
  const char* un[3] = {"lnT", "xH2", "xHp"};
  printf("{");
  for (int r = 0; r < 3; ++r)
    for (int j = 0; j < 3; ++j)
      printf("%s\"%s_%s\": %.3e, \"%s_%s\": %.3e", (r || j) ? ", " : "", fn[r], un[j], worst_f[r][j], qn[r], un[j],
             worst_q[r][j]);
  printf("}\n");
  return 0;
}
