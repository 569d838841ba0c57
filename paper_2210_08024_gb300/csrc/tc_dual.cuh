// Dual numbers in FP32: a value and its derivative along one direction, the scalar type
// that differentiates the source terms (forward-mode differentiation, Wengert 1964) for
// the Newton iteration's Jacobian.
//
// A derivative from dual numbers carries FP32's rounding (~1e-6 relative to its largest
// term) and no truncation error, where a forward difference of FP32 values is good to
// ~1e-3 and one of FP64 values costs three more FP64 evaluations of the source terms: a
// GB300 issues 32 FP32 warp instructions or more in the time of one FP64 one.
// The Jacobian only steers the iteration; residuals, updates and roots stay in FP64.
//
// On the device the elementary functions are the approximate FP32 ones (errors of a few
// 1e-7, growing as 1e-7 |x| in the exponential).  Literal constants and the cell's
// constants stay plain FP32 values.  Comparisons look at the value alone.
#pragma once
#include "tc_phys.cuh"

namespace tcg {

struct dualf {
  float v, d;
  dualf() = default;
  TCG_FN constexpr dualf(double x) : v(float(x)), d(0.0f) {}  // a constant
  TCG_FN static dualf make(float v, float d) {
    dualf r;
    r.v = v;
    r.d = d;
    return r;
  }
};
template <> struct Prec<dualf> {
  static constexpr double root_tol = 1e-7;
  static constexpr bool fp32_range = true;
  static constexpr int cls = 3;
};

template <> struct ConstOf<dualf> { using type = float; };

// One MUFU instruction each on the device (with a scaling multiply for exp and log), by PTX:
// the intrinsics of a build without fast math wrap them in range handling.  Subnormal
// arguments and results flush to zero.
TCG_FN float dual_rcp(float x) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
#else
  return 1.0f / x;
#endif
}
TCG_FN float dual_exp(float x) {
#ifdef __CUDA_ARCH__
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x * 1.44269504f));
  return r;
#else
  return expf(x);
#endif
}
TCG_FN float dual_log(float x) {
#ifdef __CUDA_ARCH__
  float r;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r * 0.693147181f;
#else
  return logf(x);
#endif
}
TCG_FN float dual_sqrt(float x) {
#ifdef __CUDA_ARCH__
  float r;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
#else
  return sqrtf(x);
#endif
}

TCG_FN dualf operator+(dualf a, dualf b) { return dualf::make(a.v + b.v, a.d + b.d); }
TCG_FN dualf operator+(float a, dualf b) { return dualf::make(a + b.v, b.d); }
TCG_FN dualf operator+(dualf a, float b) { return dualf::make(a.v + b, a.d); }
TCG_FN dualf operator-(dualf a, dualf b) { return dualf::make(a.v - b.v, a.d - b.d); }
TCG_FN dualf operator-(float a, dualf b) { return dualf::make(a - b.v, -b.d); }
TCG_FN dualf operator-(dualf a, float b) { return dualf::make(a.v - b, a.d); }
TCG_FN dualf operator-(dualf a) { return dualf::make(-a.v, -a.d); }
TCG_FN dualf operator*(dualf a, dualf b) { return dualf::make(a.v * b.v, fmaf(a.v, b.d, a.d * b.v)); }
TCG_FN dualf operator*(float a, dualf b) { return dualf::make(a * b.v, a * b.d); }
TCG_FN dualf operator*(dualf a, float b) { return dualf::make(a.v * b, a.d * b); }
TCG_FN dualf operator/(dualf a, dualf b) {
  const float r = dual_rcp(b.v), q = a.v * r;
  return dualf::make(q, (a.d - q * b.d) * r);
}
TCG_FN dualf operator/(float a, dualf b) {
  const float r = dual_rcp(b.v), q = a * r;
  return dualf::make(q, -(q * b.d) * r);
}
TCG_FN dualf operator/(dualf a, float b) {
  const float r = dual_rcp(b);
  return dualf::make(a.v * r, a.d * r);
}
TCG_FN dualf& operator+=(dualf& a, dualf b) { a = a + b; return a; }
TCG_FN bool operator<(dualf a, dualf b) { return a.v < b.v; }
TCG_FN bool operator>(dualf a, dualf b) { return a.v > b.v; }
TCG_FN bool operator<=(dualf a, dualf b) { return a.v <= b.v; }
TCG_FN bool operator>=(dualf a, dualf b) { return a.v >= b.v; }
TCG_FN bool operator==(dualf a, dualf b) { return a.v == b.v; }

TCG_FN dualf m_exp(dualf x) {
  const float e = dual_exp(x.v);
  return dualf::make(e, e * x.d);
}
TCG_FN dualf m_log(dualf x) { return dualf::make(dual_log(x.v), x.d * dual_rcp(x.v)); }
TCG_FN dualf m_sqrt(dualf x) {
  const float s = dual_sqrt(x.v);
  return dualf::make(s, 0.5f * x.d * dual_rcp(s));
}
TCG_FN dualf m_max(dualf a, dualf b) { return (a.v < b.v) ? b : a; }
TCG_FN dualf m_min(dualf a, dualf b) { return (b.v < a.v) ? b : a; }
TCG_FN dualf m_max(dualf a, float b) { return (a.v < b) ? dualf::make(b, 0.0f) : a; }
TCG_FN dualf m_min(dualf a, float b) { return (b < a.v) ? dualf::make(b, 0.0f) : a; }
TCG_FN dualf m_abs(dualf a) { return (a.v < 0.0f) ? -a : a; }

// The C/O/e equilibrium along one direction at x_e.  With g(x; y) the electron balance's
// residual, dx_e = -(dg/dy) / (dg/dx): one evaluation of x_C+ at the fixed x_e, its
// derivative along y by duals and along x by the formula of equilibrium().  With `refine`,
// x_e is an estimate: it takes one Newton step, and x_C+ and ln psi move with it to first
// order.
TCG_FN Equil<dualf> equil_tangent(const CellC<float>& c, const ChemT<dualf>& b, dualf xH2, dualf xHp, float xe,
                                  bool refine) {
  TCG_COUNT_T(equil, dualf);
  Equil<dualf> q;
  const dualf w = 1.0f - b.S;
  q.xOp = c.xOtot * xHp;
  q.xMHp = (2.0f * c.xMH_pref) * xH2 * b.xMH_T;
  const dualf a0 = w * (xHp + q.xOp + q.xMHp) + b.S * (xHp + b.xe_hot);
  const dualf src = (c.zpiC_rad + c.zcrC) + (1040.0f * c.xi) * xH2;
  const dualf sink0 = src + c.n * (b.kCpH2 * xH2);
  const bool coupled = w.v * c.xCtot > 0.0f && src.v > 0.0f;
  if (refine) xe = coupled ? fminf(fmaxf(xe, a0.v), a0.v + w.v * c.xCtot) : a0.v;
  const float ne = fmaxf(xe * c.n, 1e-30f);
  const dualf psi = (c.G0 * dual_rcp(ne)) * b.sqT + 50.0f;
  const dualf lp = m_log(psi);
  const dualf pa = m_exp(float(WDC2) * lp);
  const dualf pb = b.wdC3T * m_exp(b.wdCex * lp);
  const dualf D = 1.0f + float(WDC1) * pa * (1.0f + pb);
  const dualf agr = (float(1e-14 * WDC0) * c.Zd) / D;
  const dualf den = sink0 + c.n * (agr + b.arrC * xe);
  const dualf r = (c.xCtot * src) / den;
  // along x_e at fixed y
  const float dlp = (xe * c.n > 1e-30f) ? (50.0f - psi.v) * dual_rcp(psi.v * xe) : 0.0f;
  const float dD = float(WDC1) * (float(WDC2) * pa.v * (1.0f + pb.v) + pa.v * b.wdCex.v * pb.v) * dlp;
  const float dagr = -agr.v * dual_rcp(D.v) * dD;
  const float dr = -r.v * dual_rcp(den.v) * ((dagr + b.arrC.v) * c.n);
  const float igp = dual_rcp(1.0f - w.v * dr);
  const float dxe = coupled ? (a0.d + w.d * r.v + w.v * r.d) * igp : a0.d;
  const float sx = (refine && coupled) ? (a0.v + w.v * r.v - xe) * igp : 0.0f;
  q.xe = dualf::make(xe + sx, dxe);
  q.xCp = dualf::make(fminf(fmaxf(r.v + dr * sx, 0.0f), c.xCtot), r.d + dr * dxe);
  q.lpsi = dualf::make(lp.v + dlp * sx, lp.d + dlp * dxe);
  const dualf fr = m_max((c.xCtot > 0.0f) ? q.xCp / c.xCtot : dualf(0.0), xHp);
  q.xCO = (2.0f * c.xCtot) * xH2 * (1.0f - fr) / (1.0f + c.rCO2);
  q.xC = c.xCtot - q.xCp - q.xCO;
  q.xO = c.xOtot - q.xCO - q.xOp;
  return q;
}

// The dust temperature along one direction at td (the energy balance of dust_T
// differentiated); with `refine`, td takes one Newton step first.
TCG_FN dualf dust_tangent(const CellC<float>& c, const ChemT<dualf>& b, float td, bool refine) {
  if (!(c.Zd > 0.0f)) return b.T;
  const dualf C = c.Cgd * b.sqT;
  float y2 = td * td;
  float dh = c.Bd * td * (6.0f * y2 * y2 - 2.0f * c.Tc4) + C.v;
  if (refine) {
    td -= (c.Bd * y2 * (y2 * y2 - c.Tc4) - c.Gd - C.v * (b.T.v - td)) * dual_rcp(dh);
    y2 = td * td;
    dh = c.Bd * td * (6.0f * y2 * y2 - 2.0f * c.Tc4) + C.v;
  }
  return dualf::make(td, (C.d * (b.T.v - td) + C.v * b.T.d) * dual_rcp(dh));
}

// f = (H/K, C_H2, C_H+) in FP32 with the estimates of x_e and T_d refined, and T_d's
// derivatives (the outputs of source_tangents beyond the Jacobian).
struct Tan32 {
  float f[3], xe, td, dtd[3];
};

// Derivatives of f and of (x_e, x_C+, x_CO) along ln T, x_H2 and x_H+ at one state, given
// its x_e and dust temperature: df[i][j] and dq[i][j], j the direction, for the directions
// j0 <= j < j1.  The temperature blocks are differentiated once; the two abundance
// directions run on them with their derivatives cleared.  `hk` is 1 / (mu_H k_B / (gamma -
// 1)): H/K = (Gamma - n Lambda) hk stays in FP32's range at any density.  With `val`, x_e and
// td are estimates (one Newton step each) and the values are returned too.
TCG_BIG inline void source_tangents(const CellC<float>& c, unsigned flags, float hk, float T, float x2, float xp,
                                    float xH, float xe, float td, float (*df)[3], float (*dq)[3], int j0 = 0,
                                    int j1 = 3, Tan32* val = nullptr) {
  ChemT<dualf> b = chem_T(c, dualf::make(T, (j0 == 0) ? T : 0.0f), flags);
  CoolT<dualf> k = cool_T(c, b, flags);
#pragma unroll 1
  for (int j = j0; j < j1; ++j) {
    if (j == 1 && j0 == 0) {
      dualf* pb = reinterpret_cast<dualf*>(&b);
      dualf* pk = reinterpret_cast<dualf*>(&k);
      for (int i = 0; i < int(sizeof(b) / sizeof(dualf)); ++i) pb[i].d = 0.0f;
      for (int i = 0; i < int(sizeof(k) / sizeof(dualf)); ++i) pk[i].d = 0.0f;
    }
    const dualf X2 = dualf::make(x2, (j == 1) ? 1.0f : 0.0f), XP = dualf::make(xp, (j == 2) ? 1.0f : 0.0f);
    const dualf XH = dualf::make(xH, (j == 0) ? 0.0f : (j == 1) ? -2.0f : -1.0f);
    const Equil<dualf> q = equil_tangent(c, b, X2, XP, xe, val != nullptr);
    const Src<dualf> s = source(c, b, k, X2, XP, XH, q, dust_tangent(c, b, td, val != nullptr), dualf(-1.0));
    df[0][j] = (s.G.d - c.n * s.L.d) * hk;
    df[1][j] = s.CH2.d;
    df[2][j] = s.CHp.d;
    dq[0][j] = q.xe.d;
    dq[1][j] = q.xCp.d;
    dq[2][j] = q.xCO.d;
    if (val) {
      val->f[0] = (s.G.v - c.n * s.L.v) * hk;
      val->f[1] = s.CH2.v;
      val->f[2] = s.CHp.v;
      val->xe = q.xe.v;
      val->td = s.Td.v;
      val->dtd[j] = s.Td.d;
    }
  }
}

}  // namespace tcg
