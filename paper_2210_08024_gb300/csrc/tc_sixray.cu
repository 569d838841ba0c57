// Six-ray radiation fields, H2 self-shielding and CR attenuation (Secs. 5.2, 5.3;
// include/tc_sixray.h).
//
// Three passes, one per axis; each adds the two rays along its axis to per-cell
// accumulators held in the output arrays and the last one turns them into the fields:
//   acc.Nmin (in xi_cr)      smallest ray column seen so far
//   acc.Spe  (in chi_pe)     sum of exp(-sigma_PE (N_ray - Nmin))
//   acc.Slw  (in chi_lw)     sum of exp(-sigma_LW (N_ray - Nmin))
//   acc.Sh2  (in f_shld_h2)  sum of exp(-sigma_LW (N_ray - Nmin)) f_shld,H2(N_H2,ray)
// A ray's column is the sum of n over the cells between its entry face and the cell (the
// cell size is applied where a column is used), accumulated from that face (exclusive scans
// in both directions; a line total minus a prefix would cancel to rounding noise near the
// far face, which the H2 self-shielding factor resolves in its Doppler-core regime).
//
// All three passes run one kernel.  The lines of an axis are flattened over both other axes,
// so that no lane idles at an odd extent; a block holds LINES = 4 of them (one 32-byte
// sector of neighbours along x) cut into 8 to 32 segments, one a thread, whose sums are
// combined in shared memory (a two-level scan).  Small blocks spread an FP64-bound grid
// evenly over the SMs: 32 lines a block put a 45 x 70 x 33 grid's y pass on 47 of them.  Each
// segment is swept forwards (the ray entering at the low face) and backwards (the ray
// entering at the high face); the last pass converts the accumulators in its second sweep.
// Along x the lanes read whole rows: sectors are reused from L1 over the next cells, and the
// pass stays bound by FP64 like the others.
//
// What bounds it: FP64 instructions, 85% pipe busy before and after.  Per cell and ray: the
// self-shielding factor (a reciprocal square root, a reciprocal and an exponential, the first
// two from FP32 seeds) and the weight (one exponential of half the exponent, squared and
// cubed for the two bands; one formula whether the ray or the smallest column so far is the
// smaller).  862 -> 420 FP64 instructions a cell against exp(), sqrt(), four divisions and a
// branch with its own exp() and sqrt(); 128^3: 3.73 -> 1.80 ms, 45 x 70 x 33: 353 -> 145 us.
// Against an 80-bit reference (64 x 48 x 56) the 2-norm errors went from 1.49e-16 to
// 1.32e-16 (chi_PE, chi_LW) and stayed at 2.0e-16 (f_shld,H2) and 1.7e-16 (N_eff).
#include <cuda_runtime.h>
#include <math.h>

#include "../../include/tc_sixray.h"
#include "tc_exp64.cuh"

namespace tcg {
namespace {

constexpr double N0_CRATT = 9.35e20;  // Eq. e:cratt
constexpr int LINES = 4;      // lines per block
constexpr int SEG_MAX = 32;   // segments per line, at most

struct SrConst {
  double dx, spe, slw, inv_spe, chi0, xi0;
  double half_tau;   // sigma_PE dx / 2
  double tpe, tpe_lo, tlw, tlw_lo;  // sigma dx of the two bands, each with its rounding error
  double x5, x15;    // dx / 5e14 cm^-2 and a third of it
};

// FP32 value near a normal double of FP32's range (truncated), and the double of an FP32
// value, by their bits: conversions would run on the FP64 pipe.
__device__ __forceinline__ float near_float(double x) {
  return __int_as_float(((__double2hiint(x) - 0x38000000) << 3) | (int)((unsigned)__double2loint(x) >> 29));
}
__device__ __forceinline__ double widen(float x) {
  const int b = __float_as_int(x);
  return __hiloint2double((b >> 3) + 0x38000000, b << 29);
}

// Eq. e:fshld_H2_DB with b_5 = 3 and x = N_H2 / 5e14 cm^-2: a = 1 + x, q = 1 + x/3.  1/sqrt(a)
// by one third-order step from the FP32 value (error 2^-22 -> 2^-65), sqrt(a) from it with
// one correction, 1/q^2 by one third-order step.  Columns where FP32 could not hold 1/q^2
// (none is) take the plain functions.
__device__ __forceinline__ double f_shld_db(double a, double q) {
  if (!((unsigned)(__double2hiint(a) - 0x3fe00000) < 0x03c00000u)) {  // not in [2^-1, 2^59)
    const double s = sqrt(a);
    return 0.965 / (q * q) + 0.035 / s * exp(-8.5e-4 * s);
  }
  const double y0 = widen(rsqrtf(near_float(a)));
  const double e = fma(-a * y0, y0, 1.0);
  const double rs = fma(y0, e * fma(e, 0.375, 0.5), y0);
  double s = a * rs;
  s = fma(fma(-s, s, a), 0.5 * rs, s);
  const float rf = __frcp_rn(near_float(q));
  const double r0 = widen(rf * rf), q2 = q * q;
  const double g = fma(-q2, r0, 1.0);
  const double rq2 = fma(r0, fma(g, g, g), r0);
  return fma(0.965, rq2, 0.035 * rs * exp64(-8.5e-4 * s));
}

// (1 - e^-t)/t, the cell average of e^-s over optical depth t: below 1 (all but the densest
// cells) the series to t^18 (the rest below 1e-18, 19 FMAs and no division), which rounds
// once near the end where expm1() and a division round three times.
__device__ __forceinline__ double cell_average(double t) {
  if (!(t <= 1.0)) return -expm1(-t) / t;
  constexpr double c[19] = {1.0, -1.0 / 2, 1.0 / 6, -1.0 / 24, 1.0 / 120, -1.0 / 720, 1.0 / 5040, -1.0 / 40320,
                            1.0 / 362880, -1.0 / 3628800, 1.0 / 39916800, -1.0 / 479001600, 1.0 / 6227020800.0,
                            -1.0 / 87178291200.0, 1.0 / 1307674368000.0, -1.0 / 20922789888000.0,
                            1.0 / 355687428096000.0, -1.0 / 6402373705728000.0, 1.0 / 121645100408832000.0};
  double g = c[18];
#pragma unroll
  for (int i = 17; i >= 0; --i) g = fma(g, t, c[i]);
  return g;
}

struct Acc {
  double Nmin, Spe, Slw, Sh2;
};

// p = e^2x and q = e^3x for x <= 0 from one exponential y + lo: p = y^2 + 2 y lo, q = p y + p lo.
__device__ __forceinline__ void weights(double x, double& p, double& q) {
  int e;
  double lo;
  const double y = exp64_parts(x, e, lo);
  const int m = e >> 9;
  p = fma(y, y, 2.0 * (y * lo));
  q = fma(p, y, p * lo);
  if (!(x >= -236.0)) {  // a product may leave the normal range; NaN, whose bits are no exponent's
    const double h = exp64(x);
    p = h * h;
    q = p * h;
    return;
  }
  p = times_pow2(p, 2 * m);
  q = times_pow2(q, 3 * m);
}

// Adds one ray with dust column N and H2 column NH2 to the cell centre (in units of the
// cell size).  With h = exp(-sigma_PE |N - Nmin| / 2), either the ray's weights are h^2 and
// h^3 (sigma_LW / sigma_PE = 1.5), or the ray is the new smallest column and the sums so far
// shrink by them.  h's own rounding error goes into both, which then round once or twice.
__device__ __forceinline__ void add_ray(Acc& a, const SrConst& k, double N, double NH2, bool first) {
  const double f = f_shld_db(fma(NH2, k.x5, 1.0), fma(NH2, k.x15, 1.0));
  if (first) {
    a = Acc{N, 1.0, 1.0, f};
    return;
  }
  const double d = N - a.Nmin;
  double p, q;
  weights(-k.half_tau * fabs(d), p, q);
  const bool less = d < 0.0;
  a.Nmin = less ? N : a.Nmin;
  a.Spe = fma(a.Spe, less ? p : 1.0, less ? 1.0 : p);
  const double keep = less ? q : 1.0, add = less ? 1.0 : q;
  a.Slw = fma(a.Slw, keep, add);
  a.Sh2 = fma(a.Sh2, keep, add * f);
}

__device__ __forceinline__ Acc load_acc(const double* chi_pe, const double* chi_lw, const double* fh2,
                                        const double* xi, long long c) {
  return Acc{xi[c], chi_pe[c], chi_lw[c], fh2[c]};
}

__device__ __forceinline__ void store_acc(double* chi_pe, double* chi_lw, double* fh2, double* xi, long long c,
                                          const Acc& a) {
  xi[c] = a.Nmin;
  chi_pe[c] = a.Spe;
  chi_lw[c] = a.Slw;
  fh2[c] = a.Sh2;
}

// The rays along one axis.  Line i starts at (i % inner) s0 + (i / inner) s1 and steps by
// lstride, len cells long; a block holds LINES of them in blockDim.y segments.  FIRST: the
// accumulators start empty; LAST: they become the fields.
template <bool FIRST, bool LAST>
__global__ void __launch_bounds__(LINES * SEG_MAX) k_sr_lines(long long nlines, long long inner, long long s0, long long s1,
                                                   long long len, long long lstride, SrConst k,
                                                   const double* __restrict__ n, const double* __restrict__ xh2,
                                                   double* chi_pe, double* chi_lw, double* fh2, double* xi,
                                                   double* Neff) {
  __shared__ double sN[SEG_MAX][LINES], sH[SEG_MAX][LINES];
  const int lane = threadIdx.x, seg = threadIdx.y, nseg = blockDim.y;
  const long long i = blockIdx.x * (long long)LINES + lane;
  const bool live = i < nlines;
  const long long base = (i % inner) * s0 + (i / inner) * s1;
  const long long c0 = len * seg / nseg, c1 = len * (seg + 1) / nseg;
  double sn = 0.0, sh = 0.0;
  if (live)
    for (long long c = c0; c < c1; ++c) {
      const long long e = base + c * lstride;
      sn += n[e];
      sh = fma(xh2[e], n[e], sh);
    }
  sN[seg][lane] = sn;
  sH[seg][lane] = sh;
  __syncthreads();
  // columns of the segments before this one (from the low face) and after it (from the
  // high face)
  double fN = 0.0, fH = 0.0, bN = 0.0, bH = 0.0;
  for (int s = 0; s < seg; ++s) { fN += sN[s][lane]; fH += sH[s][lane]; }
  for (int s = nseg - 1; s > seg; --s) { bN += sN[s][lane]; bH += sH[s][lane]; }
  if (!live) return;
  for (long long c = c0; c < c1; ++c) {
    const long long e = base + c * lstride;
    const double nn = n[e], nh = xh2[e] * nn;
    Acc a = Acc{0.0, 0.0, 0.0, 0.0};
    if (!FIRST) a = load_acc(chi_pe, chi_lw, fh2, xi, e);
    add_ray(a, k, fN, fma(0.5, nh, fH), FIRST);
    store_acc(chi_pe, chi_lw, fh2, xi, e, a);
    fN += nn;
    fH += nh;
  }
  for (long long c = c1 - 1; c >= c0; --c) {
    const long long e = base + c * lstride;
    const double nn = n[e], nh = xh2[e] * nn;
    Acc a = load_acc(chi_pe, chi_lw, fh2, xi, e);
    add_ray(a, k, bN, fma(0.5, nh, bH), false);
    bN += nn;
    bH += nh;
    if (!LAST) {
      store_acc(chi_pe, chi_lw, fh2, xi, e, a);
    } else {
      const double gpe = cell_average(k.tpe * nn);
      const double glw = cell_average(k.tlw * nn);
      chi_pe[e] = k.chi0 / 6.0 * exp64(-fma(k.tpe, a.Nmin, k.tpe_lo * a.Nmin)) * a.Spe * gpe;
      chi_lw[e] = k.chi0 / 6.0 * exp64(-fma(k.tlw, a.Nmin, k.tlw_lo * a.Nmin)) * a.Slw * glw;
      fh2[e] = a.Sh2 / a.Slw;
      double ne = 0.0;
      if (k.spe > 0.0) ne = fma(-log64(a.Spe * gpe * (1.0 / 6.0)), k.inv_spe, a.Nmin * k.dx);
      xi[e] = (ne <= N0_CRATT) ? k.xi0 : k.xi0 * N0_CRATT / ne;
      if (Neff) Neff[e] = ne;
    }
  }
}

// Segments per line: 8 (long segments spend less on the scan), and more, of two cells at
// least, where the grid is too small to give every SM partition two warps.
int segments(long long nlines, long long len, int num_sms) {
  int s = 8;
  while (s < SEG_MAX && 4LL * s <= len && nlines * s < 256LL * num_sms) s *= 2;
  return s;
}

bool al8(const void* p) { return (((unsigned long long)p) & 7ull) == 0; }

}  // namespace
}  // namespace tcg

extern "C" int tc_sixray(const tc_sixray_grid* g, const double* n, const double* x_h2, double* chi_pe,
                         double* chi_lw, double* f_shld_h2, double* xi_cr, double* N_eff, void* stream) {
  using namespace tcg;
  if (!g || g->nx < 1 || g->ny < 1 || g->nz < 1) return TC_EINVAL;
  if (!(g->dx_cm > 0.0) || !isfinite(g->dx_cm) || !(g->chi0 >= 0.0) || !(g->xi0 >= 0.0) || !(g->Zd >= 0.0) ||
      !isfinite(g->chi0) || !isfinite(g->xi0) || !isfinite(g->Zd))
    return TC_EINVAL;
  const double ncell_d = (double)g->nx * (double)g->ny * (double)g->nz;
  if (ncell_d > 4.0e12) return TC_EINVAL;
  const void* ptrs[] = {n, x_h2, chi_pe, chi_lw, f_shld_h2, xi_cr};
  for (const void* p : ptrs)
    if (!p || !al8(p)) return TC_EINVAL;
  if (N_eff && !al8(N_eff)) return TC_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  SrConst k;
  k.dx = g->dx_cm;
  k.spe = 1.0e-21 * g->Zd;
  k.slw = 1.5e-21 * g->Zd;
  k.inv_spe = (k.spe > 0.0) ? 1.0 / k.spe : 0.0;
  k.half_tau = 0.5 * k.spe * k.dx;
  k.tpe = k.spe * k.dx;
  k.tpe_lo = fma(k.spe, k.dx, -k.tpe);
  k.tlw = k.slw * k.dx;
  k.tlw_lo = fma(k.slw, k.dx, -k.tlw);
  k.x5 = k.dx / 5e14;
  k.x15 = k.dx / 1.5e15;
  k.chi0 = g->chi0;
  k.xi0 = g->xi0;
  int dev = 0, num_sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return TC_ECUDA;
  const long long nx = g->nx, ny = g->ny, nz = g->nz;
  // lines along z start at x + nx y, along y at x + nx ny z, along x at nx (y + ny z)
  const long long nl[3] = {nx * ny, nx * nz, ny * nz};
  for (long long m : nl)
    if ((m + LINES - 1) / LINES > 2147483647LL) return TC_EINVAL;
  const dim3 bz(LINES, segments(nl[0], nz, num_sms)), by(LINES, segments(nl[1], ny, num_sms)),
      bx(LINES, segments(nl[2], nx, num_sms));
  auto blocks = [](long long lines) { return (unsigned)((lines + LINES - 1) / LINES); };
  k_sr_lines<true, false><<<blocks(nl[0]), bz, 0, st>>>(nl[0], nl[0], 1, 0, nz, nx * ny, k, n, x_h2,
                                                                        chi_pe, chi_lw, f_shld_h2, xi_cr, nullptr);
  if (cudaGetLastError() != cudaSuccess) return TC_ECUDA;
  k_sr_lines<false, false><<<blocks(nl[1]), by, 0, st>>>(nl[1], nx, 1, nx * ny, ny, nx, k, n, x_h2,
                                                                         chi_pe, chi_lw, f_shld_h2, xi_cr, nullptr);
  if (cudaGetLastError() != cudaSuccess) return TC_ECUDA;
  k_sr_lines<false, true><<<blocks(nl[2]), bx, 0, st>>>(nl[2], nl[2], nx, 0, nx, 1, k, n, x_h2, chi_pe,
                                                                        chi_lw, f_shld_h2, xi_cr, N_eff);
  if (cudaGetLastError() != cudaSuccess) return TC_ECUDA;
  return TC_OK;
}
