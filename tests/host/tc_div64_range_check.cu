// Program that compares the device's FP64 quotient (m_div of csrc/tc_phys.cuh) with the correctly
// rounded division over all exponents, on the GPU (not part of libtc_gb300.so; built and run by
// tests/test_gpu_div64_range.py).
//
// Random pairs with exponents from -1074 to 1023, and every pair of 2^e (1 + m 2^-52) for e at and
// beside the edges of the range that m_div takes.  Prints one JSON object: pairs, the largest
// difference in units of the last place, and the pairs that are not finite on one side alone.
#include <cmath>
#include <cstdio>

#include "tc_phys.cuh"

using namespace tcg;

__device__ inline unsigned long long mix(unsigned long long z) {  // splitmix64 (Steele, Lea & Flood 2014)
  z += 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
__device__ inline long long ordered(double x) {  // counts doubles upwards, both zeros as 0
  const long long v = __double_as_longlong(x);
  return (v < 0) ? (long long)(0x8000000000000000ull) - v : v;
}
__device__ inline void compare(double a, double b, unsigned long long* out) {
  const double q = m_div(a, b), w = __ddiv_rn(a, b);
  if (isfinite(q) && isfinite(w)) {
    const long long d = llabs(ordered(q) - ordered(w));
    atomicMax(out, (unsigned long long)d);
  } else if (!(q == w || (isnan(q) && isnan(w)))) {
    atomicAdd(out + 1, 1ull);
  }
}
__global__ void random_pairs(unsigned long long* out) {
  const unsigned long long t = blockIdx.x * blockDim.x + threadIdx.x;
  for (int i = 0; i < 16; ++i) {
    const unsigned long long r = mix(32 * t + 2 * i), s = mix(32 * t + 2 * i + 1);
    const double a = ldexp(1.0 + (double)(r >> 12) * 0x1p-52, (int)(mix(r) % 2098u) - 1074);
    const double b = ldexp(1.0 + (double)(s >> 12) * 0x1p-52, (int)(mix(s) % 2098u) - 1074);
    compare((r & 1) ? a : -a, (s & 1) ? b : -b, out);
  }
}
__device__ const int kEdges[] = {-1074, -1022, -768, -767, -664, -512, -511, -510, -1, 0, 510, 511, 512, 513, 664, 768, 769, 1023};
__global__ void edge_pairs(unsigned long long* out) {
  const int n = sizeof(kEdges) / sizeof(int);
  const int i = blockIdx.x, j = threadIdx.x;
  if (i >= n || j >= n) return;
  for (int m = 0; m < 9; ++m) {
    const double v[3] = {0x1p0, 0x1.8p0 + 0x1p-52, 0x1.fffffffffffffp0};
    compare(ldexp(v[m / 3], kEdges[i]), ldexp(v[m % 3], kEdges[j]), out);
  }
}

int main() {
  unsigned long long* out;
  unsigned long long r[2];
  if (cudaMalloc(&out, 16) || cudaMemset(out, 0, 16)) return 2;
  random_pairs<<<4096, 256>>>(out);
  edge_pairs<<<18, 32>>>(out);
  if (cudaMemcpy(r, out, 16, cudaMemcpyDeviceToHost)) return 3;
  printf("{\"pairs\": %lld, \"units\": %llu, \"not_finite\": %llu}\n", 4096LL * 256 * 16 + 18 * 18 * 9, r[0], r[1]);
  return 0;
}
