// Training of the seed network on the GPU (declared in include/tc_mlp.h).
//
// Parameters live on the device as one FP32 master vector in the order
//   W1[64][13], b1[64], W2[64][64], b2[64], W3[64][64], b3[64], W4[3][64], b4[3]
// (weights [out][in]).  The forward and backward passes use the weights rounded to
// BF16, as the step kernel's inference does, and accumulate in FP32.  The weight
// gradient of the BF16 network is applied to the FP32 masters by Adam.
//
// Forward and backward pass are one kernel: a block takes tiles of 64 samples through all
// layers and back with the weights and the tile's activations in shared memory, and keeps
// its share of the weight gradients in registers until its last tile.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <new>
#include <vector>

#include "../../include/tc.h"
#include "../../include/tc_mlp.h"
#include "tc_mlp.cuh"
#include "tc_mlp_mma.cuh"

namespace tcg {
namespace {
// One block of 256 threads: the [out][in] copy of the blob's transposed weights that
// the tensor-core inference reads as B fragments (tc_mlp_mma.cuh).
__global__ void k_mlp_mma_layout(const MlpDev* __restrict__ w, MlpMma* __restrict__ m) {
  for (int i = threadIdx.x; i < MLP_INP; i += blockDim.x) {
    m->mean[i] = w->in_mean[i];
    m->inv_std[i] = w->in_inv_std[i];
  }
  for (int i = threadIdx.x; i < MLP_HID; i += blockDim.x) {
    m->b1[i] = w->b1[i];
    m->b2[i] = w->b2[i];
    m->b3[i] = w->b3[i];
  }
  for (int i = threadIdx.x; i < 8; i += blockDim.x) m->b4[i] = (i < MLP_OUT) ? w->b4[i] : 0.f;
  for (int i = threadIdx.x; i < MLP_HID * MLP_INP; i += blockDim.x) {
    const int o = i / MLP_INP, k = i % MLP_INP;
    m->W1[i] = w->W1t[k * MLP_HID + o];
  }
  for (int i = threadIdx.x; i < MLP_HID * MLP_HID; i += blockDim.x) {
    const int o = i / MLP_HID, k = i % MLP_HID;
    m->W2[i] = w->W2t[k * MLP_HID + o];
    m->W3[i] = w->W3t[k * MLP_HID + o];
  }
  for (int i = threadIdx.x; i < 8 * MLP_HID; i += blockDim.x) {
    const int o = i / MLP_HID, k = i % MLP_HID;
    m->W4[i] = (o < MLP_OUT) ? w->W4t[k * 4 + o] : __float2bfloat16_rn(0.f);
  }
}
}  // namespace

cudaError_t mlp_mma_layout(const MlpDev* w, MlpMma* m, cudaStream_t st) {
  k_mlp_mma_layout<<<1, 256, 0, st>>>(w, m);
  return cudaGetLastError();
}
}  // namespace tcg

namespace {

using tcg::MLP_HID;
using tcg::MLP_IN;
using tcg::MLP_OUT;

constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + 64 * MLP_IN, OFF_W2 = OFF_B1 + 64, OFF_B2 = OFF_W2 + 64 * 64,
              OFF_W3 = OFF_B2 + 64, OFF_B3 = OFF_W3 + 64 * 64, OFF_W4 = OFF_B3 + 64, OFF_B4 = OFF_W4 + 3 * 64,
              NPARAM = OFF_B4 + 3;

__device__ __forceinline__ float bf(float w) { return __bfloat162float(__float2bfloat16_rn(w)); }
__device__ __forceinline__ float silu_d(float z) {
  const float s = 1.0f / (1.0f + __expf(-z));
  return s * (1.0f + z * (1.0f - s));
}

// ------------------------------------------------------------------ the fused pass
// What bounds it: FP32 FMAs from shared memory (6 x 9411 a sample, 0.46 GFLOP for a batch of
// 8192: 6 us at the FP32 rate), and for one tile the chain of its seven small products.  As
// separate kernels per layer (one thread an output, weights read with a 256-byte stride,
// the weight gradients by a few thousand threads) the same batch took 430 us on the device.
// Layout: activations are [unit][sample] with rows of TS + 4 floats (16-byte loads; rows
// read side by side fall into different banks), hidden weights are held in both
// orientations so that either product reads four neighbouring values at once.  A thread owns
// 4 units x 4 samples of a layer, or 4 x 4 weights of a gradient: eight 16-byte loads for 64
// FMAs there.  64 samples: 180 KB of shared memory, and a batch of 8192 is one tile on each of
// 128 SMs.
constexpr int TS = 64;          // samples per tile
constexpr int LD = TS + 4;      // row length of an activation
constexpr int NT = 256;         // threads per block (eight warps)
constexpr int HID = MLP_HID;
static_assert(HID == 64 && MLP_OUT == 3 && MLP_IN <= 16, "thread maps below");

struct Smem {
  float W1t[MLP_IN * LD], W2t[HID * LD], W3t[HID * LD];  // [in][out], rows of LD
  float W2[HID * HID], W3[HID * HID];                    // [out][in]
  float W4[MLP_OUT * HID];
  float b1[HID], b2[HID], b3[HID], b4[4];
  float A0[MLP_IN * LD];
  float H1[HID * LD], H2[HID * LD], H3[HID * LD];
  float Z1[HID * LD], Z2[HID * LD], Z3[HID * LD];  // pre-activations, then the gradients to them
  float G[MLP_OUT * LD];
};

// Z[n][s] = b[n] + sum_k Wt[k][n] A[k][s] in the order of k; H = silu(Z).
template <int K>
__device__ __forceinline__ void layer_fwd(const float* __restrict__ A, const float* __restrict__ Wt,
                                          const float* __restrict__ bias, float* __restrict__ Z,
                                          float* __restrict__ H) {
  const int s0 = 4 * (threadIdx.x & 15), n0 = 4 * (threadIdx.x >> 4);
  float acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = bias[n0 + i];
#pragma unroll 8
  for (int k = 0; k < K; ++k) {
    const float4 a = *reinterpret_cast<const float4*>(A + k * LD + s0);
    const float4 w = *reinterpret_cast<const float4*>(Wt + k * LD + n0);
    const float av[4] = {a.x, a.y, a.z, a.w}, wv[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(wv[i], av[j], acc[i][j]);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float4 z = {acc[i][0], acc[i][1], acc[i][2], acc[i][3]};
    float4 h = {tcg::mlp_silu(z.x), tcg::mlp_silu(z.y), tcg::mlp_silu(z.z), tcg::mlp_silu(z.w)};
    *reinterpret_cast<float4*>(Z + (n0 + i) * LD + s0) = z;
    *reinterpret_cast<float4*>(H + (n0 + i) * LD + s0) = h;
  }
}

// Z[k][s] <- (sum_n G[n][s] W[n][k]) silu'(Z[k][s]): each thread replaces its own values.
template <int N>
__device__ __forceinline__ void layer_bwd(const float* __restrict__ G, const float* __restrict__ W,
                                          float* __restrict__ Z) {
  const int s0 = 4 * (threadIdx.x & 15), k0 = 4 * (threadIdx.x >> 4);
  float acc[4][4] = {};
#pragma unroll 8
  for (int n = 0; n < N; ++n) {
    const float4 g = *reinterpret_cast<const float4*>(G + n * LD + s0);
    const float4 w = *reinterpret_cast<const float4*>(W + n * HID + k0);
    const float gv[4] = {g.x, g.y, g.z, g.w}, wv[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(gv[j], wv[i], acc[i][j]);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float4* zp = reinterpret_cast<float4*>(Z + (k0 + i) * LD + s0);
    const float4 z = *zp;
    *zp = float4{acc[i][0] * silu_d(z.x), acc[i][1] * silu_d(z.y), acc[i][2] * silu_d(z.z), acc[i][3] * silu_d(z.w)};
  }
}

__device__ __forceinline__ float dot4(float4 a, float4 b, float acc) {
  return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, acc))));
}

// dW[n][k] += sum_s G[n][s] A[k][s] for n = 4 (t / 16) + i, k = t % 16 + 16 j; db[n] += sum_s G[n][s].
__device__ __forceinline__ void layer_dw(const float* __restrict__ G, const float* __restrict__ A, float (&dw)[4][4],
                                         float (&db)[4]) {
  const int kx = threadIdx.x & 15, n0 = 4 * (threadIdx.x >> 4);
#pragma unroll 4
  for (int s = 0; s < TS; s += 4) {
    float4 g[4], a[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) g[i] = *reinterpret_cast<const float4*>(G + (n0 + i) * LD + s);
#pragma unroll
    for (int j = 0; j < 4; ++j) a[j] = *reinterpret_cast<const float4*>(A + (kx + 16 * j) * LD + s);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      db[i] += (g[i].x + g[i].y) + (g[i].z + g[i].w);
#pragma unroll
      for (int j = 0; j < 4; ++j) dw[i][j] = dot4(g[i], a[j], dw[i][j]);
    }
  }
}

// The forward pass of B rows of X (out, when given, receives the outputs), and with TRAIN
// the loss sum_b sum_m w_m (O - Y)^2 / B, and its gradient added to what grad holds.  The loss
// of the blocks is summed in FP64 (acc, zero at the start) and written by the last one: FP32
// additions of the 768 warps' sums to one word left it up to 1.6e-6 off.
struct LossAcc {
  double sum;
  unsigned blocks;
};
template <bool TRAIN>
__global__ void __launch_bounds__(NT) k_pass(const float* __restrict__ theta, const float* __restrict__ norm,
                                             const float* __restrict__ X, const float* __restrict__ Y, int B, float w0,
                                             float w1, float w2, float* __restrict__ out, float* __restrict__ grad,
                                             LossAcc* __restrict__ acc, float* __restrict__ loss) {
  extern __shared__ float4 smem_raw[];
  Smem& m = *reinterpret_cast<Smem*>(smem_raw);
  const int t = threadIdx.x;
  for (int i = t; i < HID * MLP_IN; i += NT) m.W1t[(i % MLP_IN) * LD + i / MLP_IN] = bf(theta[OFF_W1 + i]);
  for (int i = t; i < HID * HID; i += NT) {
    const int o = i / HID, k = i % HID;
    const float v2 = bf(theta[OFF_W2 + i]), v3 = bf(theta[OFF_W3 + i]);
    m.W2t[k * LD + o] = v2;
    m.W3t[k * LD + o] = v3;
    if (TRAIN) {
      m.W2[i] = v2;
      m.W3[i] = v3;
    }
  }
  for (int i = t; i < MLP_OUT * HID; i += NT) m.W4[i] = bf(theta[OFF_W4 + i]);
  if (t < HID) {
    m.b1[t] = theta[OFF_B1 + t];
    m.b2[t] = theta[OFF_B2 + t];
    m.b3[t] = theta[OFF_B3 + t];
  }
  if (t < MLP_OUT) m.b4[t] = theta[OFF_B4 + t];
  float dw1[4] = {}, db1 = 0.f, dw2[4][4] = {}, db2[4] = {}, dw3[4][4] = {}, db3[4] = {}, dw4 = 0.f, db4 = 0.f;
  float lsum = 0.f;
  for (long long b0 = (long long)blockIdx.x * TS; b0 < B; b0 += (long long)gridDim.x * TS) {
    const int live = (B - b0 < TS) ? int(B - b0) : TS;
    __syncthreads();  // the last tile's gradients are done with the activations
    for (int i = t; i < TS * MLP_IN; i += NT) {
      const int s = i / MLP_IN, k = i % MLP_IN;
      m.A0[k * LD + s] = (s < live) ? (X[b0 * MLP_IN + i] - norm[k]) * norm[MLP_IN + k] : 0.f;
    }
    __syncthreads();
    layer_fwd<MLP_IN>(m.A0, m.W1t, m.b1, m.Z1, m.H1);
    __syncthreads();
    layer_fwd<HID>(m.H1, m.W2t, m.b2, m.Z2, m.H2);
    __syncthreads();
    layer_fwd<HID>(m.H2, m.W3t, m.b3, m.Z3, m.H3);
    __syncthreads();
    if (t < MLP_OUT * TS) {  // the output layer: one output of one sample a thread
      const int o = t / TS, s = t % TS;
      float acc = m.b4[o];
#pragma unroll 8
      for (int k = 0; k < HID; ++k) acc = fmaf(m.W4[o * HID + k], m.H3[k * LD + s], acc);
      const long long r = (b0 + s) * MLP_OUT + o;
      if (out && s < live) out[r] = acc;
      if (TRAIN) {
        const float w = (o == 0) ? w0 : (o == 1) ? w1 : w2;
        const float d = (s < live) ? acc - Y[r] : 0.f;
        m.G[o * LD + s] = 2.f * w * d / (float)B;
        lsum += w * d * d / (float)B;
      }
    }
    if (!TRAIN) continue;
    __syncthreads();
    if (t < MLP_OUT * HID) {
      const int o = t / HID, k = t % HID;
#pragma unroll 4
      for (int s = 0; s < TS; s += 4) {
        const float4 g = *reinterpret_cast<const float4*>(m.G + o * LD + s);
        dw4 = dot4(g, *reinterpret_cast<const float4*>(m.H3 + k * LD + s), dw4);
        db4 += (g.x + g.y) + (g.z + g.w);
      }
    }
    layer_bwd<MLP_OUT>(m.G, m.W4, m.Z3);
    __syncthreads();
    layer_dw(m.Z3, m.H2, dw3, db3);
    layer_bwd<HID>(m.Z3, m.W3, m.Z2);
    __syncthreads();
    layer_dw(m.Z2, m.H1, dw2, db2);
    layer_bwd<HID>(m.Z2, m.W2, m.Z1);
    __syncthreads();
    {  // first layer: unit t / 4, inputs t % 4 + 4 j
      const int n = t >> 2, k0 = t & 3;
#pragma unroll 4
      for (int s = 0; s < TS; s += 4) {
        const float4 g = *reinterpret_cast<const float4*>(m.Z1 + n * LD + s);
        db1 += (g.x + g.y) + (g.z + g.w);
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (k0 + 4 * j < MLP_IN)
            dw1[j] = dot4(g, *reinterpret_cast<const float4*>(m.A0 + (k0 + 4 * j) * LD + s), dw1[j]);
      }
    }
  }
  if (!TRAIN) return;
  __shared__ float ws[NT / 32];
  for (int o = 16; o > 0; o >>= 1) lsum += __shfl_down_sync(0xffffffffu, lsum, o);
  if ((t & 31) == 0) ws[t >> 5] = lsum;
  __syncthreads();
  if (t == 0) {
    atomicAdd(&acc->sum, (double)(((ws[0] + ws[1]) + (ws[2] + ws[3])) + ((ws[4] + ws[5]) + (ws[6] + ws[7]))));
    __threadfence();
    if (loss && atomicAdd(&acc->blocks, 1u) == gridDim.x - 1) {
      __threadfence();
      *loss = (float)atomicAdd(&acc->sum, 0.0);
    }
  }
  {
    const int kx = t & 15, n0 = 4 * (t >> 4);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        atomicAdd(grad + OFF_W2 + (n0 + i) * HID + kx + 16 * j, dw2[i][j]);
        atomicAdd(grad + OFF_W3 + (n0 + i) * HID + kx + 16 * j, dw3[i][j]);
      }
      if (kx == 0) {
        atomicAdd(grad + OFF_B2 + n0 + i, db2[i]);
        atomicAdd(grad + OFF_B3 + n0 + i, db3[i]);
      }
    }
    if (t < MLP_OUT * HID) {
      atomicAdd(grad + OFF_W4 + t, dw4);
      if (t % HID == 0) atomicAdd(grad + OFF_B4 + t / HID, db4);
    }
    const int n = t >> 2, k0 = t & 3;
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (k0 + 4 * j < MLP_IN) atomicAdd(grad + OFF_W1 + n * MLP_IN + k0 + 4 * j, dw1[j]);
    if (k0 == 0) atomicAdd(grad + OFF_B1 + n, db1);
  }
}

__global__ void k_adam(float* __restrict__ theta, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, int n, float lr, float b1, float b2, float eps, float c1, float c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float gi = g[i];
  const float mi = b1 * m[i] + (1.f - b1) * gi;
  const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  theta[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

inline int blocks(long long n, int t) { return (int)((n + t - 1) / t); }

}  // namespace

struct tc_mlp {
  float* theta = nullptr;  // NPARAM masters
  float* grad = nullptr;
  float* m = nullptr;
  float* v = nullptr;
  float* norm = nullptr;   // mean[MLP_IN], inv_std[MLP_IN]
  LossAcc* acc = nullptr;
  int num_sms = 1;
  long long t = 0;         // Adam step count
  float h_mean[MLP_IN], h_inv_std[MLP_IN];
};

namespace {

int pass_grid(const tc_mlp* h, int B) {
  const long long tiles = ((long long)B + TS - 1) / TS;
  return (int)(tiles < h->num_sms ? tiles : h->num_sms);
}

// Whether n floats at a and m floats at b share memory.  The fused pass writes while other blocks
// still read, so results that lie in their inputs go through a buffer.
bool overlap(const float* a, size_t n, const float* b, size_t m) {
  const uintptr_t x = (uintptr_t)a, y = (uintptr_t)b;
  return x < y + m * sizeof(float) && y < x + n * sizeof(float);
}

// splitmix64 (Steele, Lea & Flood 2014) for a reproducible weight initialisation.
uint64_t splitmix64(uint64_t& s) {
  uint64_t z = (s += 0x9E3779B97F4A7C15ull);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

}  // namespace

extern "C" {

int tc_mlp_n_params(void) { return NPARAM; }

int tc_mlp_create(unsigned long long seed, tc_mlp** out) {
  if (!out) return TC_EINVAL;
  tc_mlp* h = new (std::nothrow) tc_mlp();
  if (!h) return TC_ENOMEM;
  bool ok = cudaMalloc(&h->theta, NPARAM * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&h->grad, NPARAM * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&h->m, NPARAM * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&h->v, NPARAM * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&h->norm, 2 * MLP_IN * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&h->acc, sizeof(LossAcc)) == cudaSuccess;
  int dev = 0;
  ok = ok && cudaGetDevice(&dev) == cudaSuccess &&
       cudaDeviceGetAttribute(&h->num_sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
       cudaFuncSetAttribute(k_pass<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem)) ==
           cudaSuccess &&
       cudaFuncSetAttribute(k_pass<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem)) ==
           cudaSuccess;
  if (!ok) {
    tc_mlp_destroy(h);
    return TC_ENOMEM;
  }
  // Uniform initialisation with bound sqrt(6 / fan_in) (He et al. 2015), zero biases.
  std::vector<float> th(NPARAM, 0.f);
  uint64_t s = seed;
  auto fill = [&](int off, int nout, int nin) {
    const double bound = sqrt(6.0 / nin);
    for (int i = 0; i < nout * nin; ++i) {
      const double u = (double)(splitmix64(s) >> 11) * (1.0 / 9007199254740992.0);
      th[off + i] = (float)((2.0 * u - 1.0) * bound);
    }
  };
  fill(OFF_W1, 64, MLP_IN);
  fill(OFF_W2, 64, 64);
  fill(OFF_W3, 64, 64);
  fill(OFF_W4, 3, 64);
  for (int i = OFF_W4; i < OFF_W4 + 3 * 64; ++i) th[i] *= 0.1f;  // small initial outputs
  for (int k = 0; k < MLP_IN; ++k) { h->h_mean[k] = 0.f; h->h_inv_std[k] = 1.f; }
  float nrm[2 * MLP_IN];
  for (int k = 0; k < MLP_IN; ++k) { nrm[k] = 0.f; nrm[MLP_IN + k] = 1.f; }
  ok = cudaMemcpy(h->theta, th.data(), NPARAM * sizeof(float), cudaMemcpyHostToDevice) == cudaSuccess &&
       cudaMemset(h->m, 0, NPARAM * sizeof(float)) == cudaSuccess &&
       cudaMemset(h->v, 0, NPARAM * sizeof(float)) == cudaSuccess &&
       cudaMemcpy(h->norm, nrm, sizeof(nrm), cudaMemcpyHostToDevice) == cudaSuccess;
  if (!ok) {
    tc_mlp_destroy(h);
    return TC_ECUDA;
  }
  *out = h;
  return TC_OK;
}

void tc_mlp_destroy(tc_mlp* h) {
  if (!h) return;
  cudaFree(h->theta);
  cudaFree(h->grad);
  cudaFree(h->m);
  cudaFree(h->v);
  cudaFree(h->norm);
  cudaFree(h->acc);
  delete h;
}

int tc_mlp_set_norm(tc_mlp* h, const float* mean, const float* stdev) {
  if (!h || !mean || !stdev) return TC_EINVAL;
  float nrm[2 * MLP_IN];
  for (int k = 0; k < MLP_IN; ++k) {
    if (!(stdev[k] > 0.f) || !isfinite(mean[k])) return TC_EINVAL;
    h->h_mean[k] = mean[k];
    h->h_inv_std[k] = 1.f / stdev[k];
    nrm[k] = h->h_mean[k];
    nrm[MLP_IN + k] = h->h_inv_std[k];
  }
  return cudaMemcpy(h->norm, nrm, sizeof(nrm), cudaMemcpyHostToDevice) == cudaSuccess ? TC_OK : TC_ECUDA;
}

int tc_mlp_set_params(tc_mlp* h, const float* theta) {
  if (!h || !theta) return TC_EINVAL;
  return cudaMemcpy(h->theta, theta, NPARAM * sizeof(float), cudaMemcpyHostToDevice) == cudaSuccess ? TC_OK
                                                                                                      : TC_ECUDA;
}

int tc_mlp_get_params(const tc_mlp* h, float* theta) {
  if (!h || !theta) return TC_EINVAL;
  return cudaMemcpy(theta, h->theta, NPARAM * sizeof(float), cudaMemcpyDeviceToHost) == cudaSuccess ? TC_OK
                                                                                                      : TC_ECUDA;
}

int tc_mlp_predict(tc_mlp* h, const float* X, int B, float* out, void* stream) {
  if (!h || B < 0 || (B > 0 && (!X || !out))) return TC_EINVAL;
  if (B == 0) return TC_OK;
  cudaStream_t st = (cudaStream_t)stream;
  const size_t n = (size_t)B * MLP_OUT;
  float* o = out;
  if (overlap(out, n, X, (size_t)B * MLP_IN) && cudaMallocAsync(&o, n * sizeof(float), st) != cudaSuccess) return TC_ENOMEM;
  k_pass<false><<<pass_grid(h, B), NT, sizeof(Smem), st>>>(h->theta, h->norm, X, nullptr, B, 0.f, 0.f, 0.f, o, nullptr,
                                                           nullptr, nullptr);
  bool ok = cudaGetLastError() == cudaSuccess;
  if (o != out) {
    ok = cudaMemcpyAsync(out, o, n * sizeof(float), cudaMemcpyDeviceToDevice, st) == cudaSuccess && ok;
    ok = cudaFreeAsync(o, st) == cudaSuccess && ok;
  }
  return ok ? TC_OK : TC_ECUDA;
}

int tc_mlp_grad(tc_mlp* h, const float* X, const float* Y, int B, const float* w3, float* grad, float* loss,
                void* stream) {
  if (!h || B < 1 || !X || !Y) return TC_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  const bool apart = grad && !overlap(grad, NPARAM, X, (size_t)B * MLP_IN) && !overlap(grad, NPARAM, Y, (size_t)B * MLP_OUT);
  float* g = apart ? grad : h->grad;
  if (cudaMemsetAsync(g, 0, NPARAM * sizeof(float), st) != cudaSuccess) return TC_ECUDA;
  if (cudaMemsetAsync(h->acc, 0, sizeof(LossAcc), st) != cudaSuccess) return TC_ECUDA;
  const float w0 = w3 ? w3[0] : 1.f, w1 = w3 ? w3[1] : 1.f, w2 = w3 ? w3[2] : 1.f;
  k_pass<true><<<pass_grid(h, B), NT, sizeof(Smem), st>>>(h->theta, h->norm, X, Y, B, w0, w1, w2, nullptr, g, h->acc, loss);
  if (cudaGetLastError() != cudaSuccess) return TC_ECUDA;
  if (grad && !apart && cudaMemcpyAsync(grad, g, NPARAM * sizeof(float), cudaMemcpyDeviceToDevice, st) != cudaSuccess)
    return TC_ECUDA;
  return TC_OK;
}

int tc_mlp_train_step(tc_mlp* h, const float* X, const float* Y, int B, const float* w3, float lr, float* loss,
                      void* stream) {
  int rc = tc_mlp_grad(h, X, Y, B, w3, nullptr, loss, stream);
  if (rc != TC_OK) return rc;
  h->t += 1;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - (float)pow(b1, (double)h->t), c2 = 1.f - (float)pow(b2, (double)h->t);
  k_adam<<<blocks(NPARAM, 256), 256, 0, (cudaStream_t)stream>>>(h->theta, h->grad, h->m, h->v, NPARAM, lr, b1, b2,
                                                                 1e-8f, c1, c2);
  return cudaGetLastError() == cudaSuccess ? TC_OK : TC_ECUDA;
}

size_t tc_mlp_blob_bytes(void) { return sizeof(tcg::MlpDev); }

int tc_mlp_export(const tc_mlp* h, void* blob, size_t cap) {
  if (!h || !blob || cap < sizeof(tcg::MlpDev)) return TC_EINVAL;
  std::vector<float> th(NPARAM);
  if (cudaMemcpy(th.data(), h->theta, NPARAM * sizeof(float), cudaMemcpyDeviceToHost) != cudaSuccess) return TC_ECUDA;
  tcg::MlpDev d;
  memset(&d, 0, sizeof(d));
  d.magic = tcg::MLP_MAGIC;
  d.version = tcg::MLP_VERSION;
  d.n_in = MLP_IN;
  d.n_hid = MLP_HID;
  d.n_out = MLP_OUT;
  d.bytes = (uint32_t)sizeof(tcg::MlpDev);
  for (int k = 0; k < tcg::MLP_INP; ++k) {
    d.in_mean[k] = (k < MLP_IN) ? h->h_mean[k] : 0.f;
    d.in_inv_std[k] = (k < MLP_IN) ? h->h_inv_std[k] : 0.f;
  }
  const __nv_bfloat16 zero = __float2bfloat16_rn(0.f);
  for (int i = 0; i < tcg::MLP_INP * MLP_HID; ++i) d.W1t[i] = zero;
  for (int i = 0; i < MLP_HID * 4; ++i) d.W4t[i] = zero;
  for (int j = 0; j < MLP_HID; ++j) {
    for (int k = 0; k < MLP_IN; ++k) d.W1t[k * MLP_HID + j] = __float2bfloat16_rn(th[OFF_W1 + j * MLP_IN + k]);
    for (int k = 0; k < MLP_HID; ++k) {
      d.W2t[k * MLP_HID + j] = __float2bfloat16_rn(th[OFF_W2 + j * MLP_HID + k]);
      d.W3t[k * MLP_HID + j] = __float2bfloat16_rn(th[OFF_W3 + j * MLP_HID + k]);
    }
    d.b1[j] = th[OFF_B1 + j];
    d.b2[j] = th[OFF_B2 + j];
    d.b3[j] = th[OFF_B3 + j];
  }
  for (int m = 0; m < MLP_OUT; ++m) {
    for (int k = 0; k < MLP_HID; ++k) d.W4t[k * 4 + m] = __float2bfloat16_rn(th[OFF_W4 + m * MLP_HID + k]);
    d.b4[m] = th[OFF_B4 + m];
  }
  d.b4[3] = 0.f;
  memcpy(blob, &d, sizeof(d));
  return TC_OK;
}

}  // extern "C"
