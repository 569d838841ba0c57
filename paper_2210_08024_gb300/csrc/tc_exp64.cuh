// FP64 exponential and logarithm by tables, for the step's FP64 physics and the six-ray
// fields: about 50 of either a source evaluation, and a GB300 issues one FP64 warp
// instruction per 19 cycles and SM, so their FP64 operations decide (one step: 128^3 slab by
// FP64 Newton 88.2 -> 75.5 ms, 96^3 by the paper's scheme at 3e3 yr 15.5 -> 13.1 ms).  Both follow Tang's
// table-driven method (ACM TOMS 15, 144, 1989; 16, 378, 1990), with tables long enough for
// short polynomials; integer instructions, table loads and selections run beside the FP64
// pipe.
//
//   exp64: x = (512 m + j) ln2/512 + r, |r| <= ln2/1024; e^x = 2^m 2^(j/512) (1 + p(r)) with
//          p of degree 4 (truncation below 2e-19: the cubic coefficient takes 0.87 a^2/120, a =
//          ln2/1024, of the next term) and 2^(j/512) in two parts.  10 FP64 instructions (16
//          FMA slots measured for exp()); error below 0.51 ulp.
//          The last stretches of the range, with subnormal results (-745.5 to -708) and
//          around overflow (709 to 709.9), go to exp().
//   log64: x = 2^m z, z in [0.7, 1.41), j the bin of z, c_j ~ 1/z, r = z c_j - 1, |r| <=
//          2^-8; log x = m ln2 - log c_j + log(1 + r) to r^7, m ln2 and -log c_j in two
//          parts; the bin around 1 has c = 1 and keeps the relative accuracy there.  20
//          FP64 instructions (30 slots for log()); error below 0.52 ulp.  Arguments that are
//          not positive, normal and finite go to log().
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include "tc_exp64_table.inc"

#ifndef TCG_FN
#define TCG_FN __host__ __device__ __forceinline__
#endif

namespace tcg {

struct alignas(16) ExpEntry {  // loaded as one double2
  double h, l;
};
struct LogEntry {
  double c, h, l;
};
static __device__ const ExpEntry kExp64Dev[512] = {TCG_EXP64_TABLE};
static __device__ const LogEntry kLog64Dev[128] = {TCG_LOG64_TABLE};
static const ExpEntry kExp64Host[512] = {TCG_EXP64_TABLE};
static const LogEntry kLog64Host[128] = {TCG_LOG64_TABLE};

TCG_FN int hi_word(double x) {
#ifdef __CUDA_ARCH__
  return __double2hiint(x);
#else
  uint64_t u;
  memcpy(&u, &x, 8);
  return (int)(u >> 32);
#endif
}
TCG_FN int lo_word(double x) {
#ifdef __CUDA_ARCH__
  return __double2loint(x);
#else
  uint64_t u;
  memcpy(&u, &x, 8);
  return (int)(uint32_t)u;
#endif
}
TCG_FN double from_words(int hi, int lo) {
#ifdef __CUDA_ARCH__
  return __hiloint2double(hi, lo);
#else
  const uint64_t u = ((uint64_t)(uint32_t)hi << 32) | (uint32_t)lo;
  double x;
  memcpy(&x, &u, 8);
  return x;
#endif
}

// The reduced exponential: y + lo = 2^(j/512) (1 + p(r)) and k, with e^x = 2^(k >> 9) (y + lo).
TCG_FN double exp64_parts(double x, int& k, double& lo) {
  constexpr double MAGIC = 6755399441055744.0;  // 1.5 2^52: adding it rounds to an integer
  const double t = fma(x, 0x1.71547652b82fep+9, MAGIC);  // 512 / ln 2
  k = lo_word(t);
  const double kd = t - MAGIC;
  double r = fma(kd, -0x1.62e42fefa3800p-10, x);  // exact: k C1 and x lie on the grid 2^-52
  r = fma(kd, -0x1.ef35793c76730p-54, r);
#ifdef __CUDA_ARCH__
  const double2 e = __ldg(reinterpret_cast<const double2*>(kExp64Dev) + (k & 511));
  const double th = e.x, tl = e.y;
#else
  const double th = kExp64Host[k & 511].h, tl = kExp64Host[k & 511].l;
#endif
  double q = fma(r, 1.0 / 24.0, 0x1.555555c7793d8p-3);
  q = fma(q, r, 0.5);
  const double p = fma(q, r * r, r);
  const double w = fma(th, p, tl);
  const double y = th + w;  // in [1, 2]
  lo = (th - y) + w;
  return y;
}
TCG_FN double times_pow2(double y, int m) { return from_words(hi_word(y) + (int)((unsigned)m << 20), lo_word(y)); }

TCG_FN double exp64(double x) {
  int k;
  double lo;
  const double y = exp64_parts(x, k, lo);
  const double s = times_pow2(y, k >> 9);
  // the ends of the range, by the high word: |x| >= 708, infinities and NaN
  const int hx = hi_word(x), ax = hx & 0x7fffffff;
  if (ax < 0x40862000) return s;
  if (ax > 0x7ff00000 || (ax == 0x7ff00000 && lo_word(x) != 0)) return x;  // NaN
  if (ax < ((hx < 0) ? 0x40874c00 : 0x40862f00)) return exp(x);
  return (hx < 0) ? 0.0 : from_words(0x7ff00000, 0);
}

TCG_FN double log64(double x) {
  const int hx = hi_word(x);
  if ((unsigned)(hx - 0x00100000) >= 0x7fe00000u) return log(x);  // not positive, normal and finite
  const int d = hx - 0x3fe69000;  // z in [0.7051, 1.4102): the bin around 1 is [1 - 2^-9, 1 + 2^-8)
  const int m = d >> 20, j = (d >> 13) & 127;
  const double z = from_words(hx - (int)((unsigned)m << 20), lo_word(x));
#ifdef __CUDA_ARCH__
  const LogEntry* e = kLog64Dev + j;
  const double c = __ldg(&e->c), h = __ldg(&e->h), l = __ldg(&e->l);
#else
  const double c = kLog64Host[j].c, h = kLog64Host[j].h, l = kLog64Host[j].l;
#endif
  const double md = from_words(0x43300000, m + 2048) - 4503599627372544.0;  // (2^52 + m + 2048) - (2^52 + 2048)
  const double zc = z * c, r = zc - 1.0, rl = fma(z, c, -zc);  // z c - 1 = r + rl exactly
  const double w = fma(md, 0x1.62e42fefa3800p-1, h);  // exact: both on the grid 2^-42
  double q = fma(r, 1.0 / 7.0, -1.0 / 6.0);
  q = fma(q, r, 0.2);
  q = fma(q, r, -0.25);
  q = fma(q, r, 1.0 / 3.0);
  q = fma(q, r, -0.5);
  double u = fma(md, 0x1.ef35793c76730p-45, fma(rl, 1.0 - r, l));  // d log(1 + r) = dr (1 - r + ...)
  u = fma(q, r * r, u);
  const double v = w + r;  // |w| > |r| or w = 0: the sum's error is exact in (w - v) + r
  return v + (((w - v) + r) + u);
}

}  // namespace tcg
