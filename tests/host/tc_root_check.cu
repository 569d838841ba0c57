// Host program that compares the roots of the FP64 Newton solve with roots in long double, a
// substep at a time (not part of libtc_gb300.so; built and run by tests/test_root.py with the
// library's csrc/ on the include path).
//
// Usage: tc_root_check IN
//   IN: n as int64, then 12 arrays of n doubles (n, chi_pe, chi_lw, f_shld_H2, f_shld_C,
//       F_LyC, xi, Z'_g, Z'_d, T, x_H2, x_H+), then dt as a double.
// Prints one JSON object: substeps, those that newton_tangent left to the plain iteration (and
// of these, those that do not count its iterations), those without a long double root, and the
// largest relative error of T_mu, x_H2 and x_H+ (the abundances where above 1e-20) after it.
#include <math.h>

// long double forms of the functions the physics templates call (declared ahead of them)
#define HD __host__ __device__ inline
namespace tcg {
HD long double m_exp(long double x) { return expl(x); }
HD long double m_log(long double x) { return logl(x); }
HD long double m_sqrt(long double x) { return sqrtl(x); }
HD long double m_max(long double a, long double b) { return a < b ? b : a; }
HD long double m_min(long double a, long double b) { return b < a ? b : a; }
HD long double m_abs(long double a) { return fabsl(a); }
}  // namespace tcg

#include <cstdint>
#include <cstdio>
#include <vector>

#include "tc_kernels.cuh"

using namespace tcg;
typedef long double LD;
namespace tcg {
template <> struct Prec<LD> {
  static constexpr double root_tol = 1e-18;
  static constexpr bool fp32_range = false;
  static constexpr int cls = 0;
};
}  // namespace tcg

namespace {
struct Problem {
  CellC<LD> c;
  unsigned flags;
  LD mu, Kinv, dts;
  LD yn[3];
  void f(const LD* y, LD* r) const {
    const ChemT<LD> b = chem_T(c, mu * y[0], flags);
    const CoolT<LD> k = cool_T(c, b, flags);
    const Equil<LD> q = equilibrium(c, b, y[1], y[2], LD(-1));
    const Src<LD> s = source(c, b, k, y[1], y[2], 1 - 2 * y[1] - y[2], q, LD(-1), LD(-1));
    r[0] = y[0] - yn[0] - dts * (c.n * s.G - c.n * c.n * s.L) * Kinv;
    r[1] = y[1] - yn[1] - dts * s.CH2;
    r[2] = y[2] - yn[2] - dts * s.CHp;
  }
  // Newton from y, in unknowns scaled by their values
  bool root(LD* y) const {
    for (int it = 0; it < 40; ++it) {
      LD r[3], J[3][3], d[3], s[3];
      f(y, r);
      for (int j = 0; j < 3; ++j) s[j] = m_max(m_abs(y[j]), LD(1e-30));
      for (int j = 0; j < 3; ++j) {
        LD z[3] = {y[0], y[1], y[2]}, q[3];
        const LD h = 1e-9L * s[j];
        z[j] += h;
        f(z, q);
        for (int i = 0; i < 3; ++i) J[i][j] = (q[i] - r[i]) / h * s[j] / s[i];
      }
      for (int i = 0; i < 3; ++i) r[i] = -r[i] / s[i];
      if (!solve3<LD>(J, r, d)) return false;
      LD m = 0;
      for (int i = 0; i < 3; ++i) {
        y[i] += d[i] * s[i];
        m = m_max(m, m_abs(d[i]));
      }
      if (!(m < 1)) return false;
      if (m < 1e-15L) return true;
    }
    return false;
  }
};
}  // namespace

int main(int argc, char** argv) {
  if (argc != 2) return 2;
  FILE* fh = fopen(argv[1], "rb");
  if (!fh) return 3;
  int64_t n = 0;
  if (fread(&n, 8, 1, fh) != 1 || n <= 0) return 4;
  std::vector<double> in(12 * (size_t)n);
  double dt = 0;
  if (fread(in.data(), 8, in.size(), fh) != in.size() || fread(&dt, 8, 1, fh) != 1) return 5;
  fclose(fh);
  auto col = [&](int k) { return in.data() + (size_t)k * n; };
  DevParams p{1.0, 2.73, 1.0, 1.0, 1.0 / 3.0, 0.1, 1e-3, 1e-12, 1e-6, 1.0, 50, 1000000, 0};
  DevFields f{};
  f.n = col(0); f.chi_pe = col(1); f.chi_lw = col(2); f.fh2 = col(3); f.fc = col(4);
  f.Flyc = col(5); f.xi = col(6); f.Zg = col(7); f.Zd = col(8);
  f.T = col(9); f.xH2 = col(10); f.xHp = col(11);
  long long nsub = 0, left = 0, miscounted = 0, noroot = 0;
  double worst[3] = {0, 0, 0};
  for (int64_t i = 0; i < n; ++i) {
    CellC<double> c;
    double T0, x20, xp0;
    load_cell(f, i, p, c, T0, x20, xp0);
    const CellC<float> cf = cast_cell<float>(c);
    LaneState s;
    s.t = 0.0; s.xH2 = x20; s.xHp = xp0; s.Td = -1.0; s.nsub = 0; s.status = 0; s.iters = 0;
    ChemT<double> b0 = chem_T(c, T0, p.flags);
    Equil<double> q0 = equilibrium(c, b0, x20, xp0, -1.0);
    s.xe = q0.xe; s.xCp = q0.xCp; s.xCO = q0.xCO;
    double xe_g = s.xe, td_g = -1.0;
    s.mu = c.muH / (1.1 + s.xe - x20);
    s.Tmu = T0 / s.mu;
    while (s.t < dt && !(s.status & ST_NONFIN)) {
      bool last;
      const double dts = substep_start64<1>(c, p, dt, s, td_g, last);
      const double yn[3] = {s.Tmu, s.xH2, s.xHp};
      double y[3] = {yn[0], yn[1], yn[2]}, xg = xe_g, tg = td_g;
      Equil<double> q;
      int spent = 0;
      ++nsub;
      if (newton_tangent<1>(c, cf, p, s.mu, 1.0 / c.K, yn, dts, y, xg, tg, &q, &spent) < 0) {
        ++left;
        LaneState a = s, b = s;  // with the abandoned iterations, and by the plain iteration alone
        double xa = xe_g, ta = td_g, xb = xe_g, tb = td_g;
        solve_substep64<1>(c, p, dt, dts, last, a, xa, ta, nullptr, &cf, true);
        solve_substep64<1>(c, p, dt, dts, last, b, xb, tb);
        if (a.iters != b.iters + spent || a.Tmu != b.Tmu) ++miscounted;
      } else {
        Problem P{cast_cell<LD>(c), p.flags, s.mu, 1 / LD(c.K), dts, {yn[0], yn[1], yn[2]}};
        LD z[3] = {y[0], y[1], y[2]};
        if (!P.root(z)) {
          ++noroot;
        } else {
          for (int j = 0; j < 3; ++j) {
            if (j > 0 && !(z[j] > 1e-20L)) continue;
            const double e = double(m_abs(y[j] - z[j]) / z[j]);
            if (!(e <= worst[j]) && !isnan(worst[j])) worst[j] = e;
          }
        }
      }
      solve_substep64<1>(c, p, dt, dts, last, s, xe_g, td_g, nullptr, &cf, true);
    }
  }
  printf("{\"substeps\": %lld, \"left\": %lld, \"miscounted\": %lld, \"noroot\": %lld, \"T\": %.3e, \"xH2\": %.3e, \"xHp\": %.3e}\n", nsub,
         left, miscounted, noroot, worst[0], worst[1], worst[2]);
  return 0;
}
