// Program that checks the device's FP64 quotient, exponential and logarithm (m_div of
// csrc/tc_phys.cuh; exp64 and log64 of csrc/tc_exp64.cuh) on the GPU (not part of
// libtc_gb300.so; built and run by tests/test_gpu_div64.py).
//
// 2^20 threads draw 16 pairs each.  The quotient's error comes from its exact residual,
// |a - q b| / (|b| ulp(q)); exp64 and log64 must equal the host's same-named functions bit
// for bit (the same operations), checked on the first 2^16 arguments.  Prints one JSON object.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <vector>

#include "tc_phys.cuh"

using namespace tcg;

__host__ __device__ inline unsigned long long mix(unsigned long long z) {  // splitmix64 (Steele, Lea & Flood 2014)
  z += 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
// A double with a uniform mantissa and an exponent in [lo, lo + n).
__host__ __device__ inline double draw(unsigned long long s, int lo, int n) {
  const unsigned long long r = mix(s);
  const int e = lo + (int)(mix(r) % (unsigned)n);
  const double m = 1.0 + (double)(r >> 12) * 0x1p-52;
  return ldexp((r & 1) ? m : -m, e);
}

constexpr int kThreads = 1 << 20, kDraws = 16, kCheck = 1 << 16;

__global__ void check(unsigned long long* worst, double* ex, double* lg) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= kThreads) return;
  double w = 0.0;
  for (int i = 0; i < kDraws; ++i) {
    const unsigned long long s = (unsigned long long)t * kDraws + i;
    const double a = draw(2 * s, -150, 300), b = draw(2 * s + 1, -150, 300);
    const double q = m_div(a, b);
    int e;
    frexp(q, &e);
    w = fmax(w, fabs(fma(-q, b, a)) / (fabs(b) * ldexp(1.0, e - 53)));
  }
  atomicMax(worst, (unsigned long long)__double_as_longlong(w));
  if (t < kCheck) {
    ex[t] = exp64(draw(7ull * t, -20, 29));
    lg[t] = log64(fabs(draw(11ull * t, -300, 600)));
  }
}

// special operands: what the plain division gives
__global__ void special(double* out) {
  const double v[8] = {0.0, -0.0, 1.0, -3.0, INFINITY, -INFINITY, 1e-310, 1e300};
  const int i = threadIdx.x >> 3, j = threadIdx.x & 7;
  out[threadIdx.x] = m_div(v[i], v[j]);
}

int main() {
  unsigned long long* worst;
  double *ex, *lg, *sp;
  if (cudaMalloc(&worst, 8) || cudaMemset(worst, 0, 8) || cudaMalloc(&ex, kCheck * 8) || cudaMalloc(&lg, kCheck * 8) ||
      cudaMalloc(&sp, 64 * 8))
    return 2;
  check<<<kThreads / 256, 256>>>(worst, ex, lg);
  special<<<1, 64>>>(sp);
  unsigned long long w;
  std::vector<double> hex(kCheck), hlg(kCheck), hsp(64);
  if (cudaMemcpy(&w, worst, 8, cudaMemcpyDeviceToHost) || cudaMemcpy(hex.data(), ex, kCheck * 8, cudaMemcpyDeviceToHost) ||
      cudaMemcpy(hlg.data(), lg, kCheck * 8, cudaMemcpyDeviceToHost) || cudaMemcpy(hsp.data(), sp, 512, cudaMemcpyDeviceToHost))
    return 3;
  double ulp;
  memcpy(&ulp, &w, 8);
  int bad_exp = 0, bad_log = 0, bad_special = 0;
  for (int t = 0; t < kCheck; ++t) {
    const double x = draw(7ull * t, -20, 29), y = fabs(draw(11ull * t, -300, 600));
    bad_exp += (std::fabs(x) < 708.0) && exp64(x) != hex[t];
    bad_log += log64(y) != hlg[t];
  }
  const double v[8] = {0.0, -0.0, 1.0, -3.0, INFINITY, -INFINITY, 1e-310, 1e300};
  for (int k = 0; k < 64; ++k) {
    const double want = v[k >> 3] / v[k & 7];
    bad_special += !(hsp[k] == want || (want != want && hsp[k] != hsp[k]));
  }
  printf("{\"div_ulp\": %.4f, \"exp_differs\": %d, \"log_differs\": %d, \"special_differs\": %d}\n", ulp, bad_exp, bad_log,
         bad_special);
  return 0;
}
