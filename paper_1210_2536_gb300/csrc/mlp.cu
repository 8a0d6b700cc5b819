// Learned format selector: a 12 -> 64 -> 64 -> 8 MLP over the feature
// parameters.  It takes the place of the paper's C5.0 ruleset classifier
// f(x, TH) -> {DIA, ELL, CSR, COO} (arXiv 1210.2536, Sec. 5, Eq. "mapping"),
// predicting one of the eight GPU kernel variants, and its softmax maximum
// plays the role of the rule confidence checked against a threshold (Sec. 6).
//
// Inference and training run in these kernels: a CTA holds the whole network
// (5512 FP32 parameters) in shared memory and processes 32 samples.
// Gradients are reduced per CTA and then across CTAs in a fixed order, so a
// training step is deterministic.
//
// A step of the training driver (128 samples) is 2 MFLOP in 4 CTAs: bound by
// the latency of loading the parameters and of the chain of layers, not by any
// throughput.  So a layer must not wait on shared memory: weight rows are
// padded to 68 floats (lanes that each read a 16-byte piece of their own row
// then cover all banks; unpadded, 64 floats apart, they met in the same ones),
// and a thread computes one output of four samples (or eight rows of one
// column of a weight gradient), so that 16 multiply-adds share five loads.
// mlp_loss_grad at 128 samples: 43.3 us before, 13.3 us now (ncu, cold caches);
// mlp_forward of one sample 25.8 -> 5.4 us; a training step 53 -> 35 to 41 us, now
// the host's time to issue its launches.
#include <algorithm>
#include <atomic>
#include <cmath>

#include "smat_internal.h"
#include "spmv_device.cuh"

namespace smat {
namespace {

constexpr int IN = 12, H = 64, OUT = 8, S = 32, NT = 512;
constexpr int OW1 = 0, OB1 = OW1 + H * IN, OW2 = OB1 + H, OB2 = OW2 + H * H, OW3 = OB2 + H,
              OB3 = OW3 + OUT * H, NP = OB3 + OUT;
static_assert(NP == SMAT_MLP_PARAMS, "parameter layout");

// shared layout (floats; every array starts on 16 bytes), rows of H padded to HP
constexpr int HP = H + 4;
constexpr int SW1 = 0, SB1 = SW1 + H * IN, SW2 = SB1 + H, SB2 = SW2 + H * HP, SW3 = SB2 + H, SB3 = SW3 + OUT * HP,
              SX = SB3 + OUT, SH1 = SX + S * IN, SH2 = SH1 + S * HP, SZ = SH2 + S * HP, SDZ = SZ + S * OUT,
              SDH2 = SDZ + S * OUT, SDH1 = SDH2 + S * HP, SFWD = SDZ, STOT = SDH1 + S * HP;

// Where parameter p sits in shared memory.
__device__ __forceinline__ int param_slot(int p) {
  if (p < OW2) return p;  // W1 and b1 as they are
  if (p < OB2) return SW2 + (p - OW2) / H * HP + (p - OW2) % H;
  if (p < OW3) return SB2 + p - OB2;
  if (p < OB3) return SW3 + (p - OW3) / H * HP + (p - OW3) % H;
  return SB3 + p - OB3;
}

__device__ __forceinline__ float dot4(float4 a, float4 b, float acc) {
  return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, acc))));
}
__device__ __forceinline__ float4 at4(const float *p) { return *reinterpret_cast<const float4 *>(p); }

// Thread t of a layer of H outputs: output t % H of the samples 4 * (t / H) ..
// + 3, so the samples are the same for a whole warp.
__device__ __forceinline__ int unit() { return threadIdx.x % H; }
__device__ __forceinline__ int sample0() { return threadIdx.x / H * 4; }
static_assert(NT / H * 4 == S, "a pass covers the CTA's samples");

__device__ void block_forward(float *sm, const float *__restrict__ params, const float *__restrict__ X, int s0,
                              int ns) {
#pragma unroll
  for (int k = 0; k < (NP + NT - 1) / NT; ++k) {
    const int p = threadIdx.x + k * NT;
    if (p < NP) sm[param_slot(p)] = params[p];
  }
  for (int q = threadIdx.x; q < S * IN; q += NT) sm[SX + q] = q / IN < ns ? X[(long long)s0 * IN + q] : 0.0f;
  __syncthreads();
  const int j = unit(), sa = sample0();
  if (sa < ns) {
    float a[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) a[u] = sm[SB1 + j];
#pragma unroll
    for (int i = 0; i < IN; i += 4) {
      const float4 w = at4(sm + SW1 + j * IN + i);
#pragma unroll
      for (int u = 0; u < 4; ++u) a[u] = dot4(w, at4(sm + SX + (sa + u) * IN + i), a[u]);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) sm[SH1 + (sa + u) * HP + j] = a[u] > 0.0f ? a[u] : 0.0f;
  }
  __syncthreads();
  if (sa < ns) {
    float a[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) a[u] = sm[SB2 + j];
#pragma unroll
    for (int i = 0; i < H; i += 4) {
      const float4 w = at4(sm + SW2 + j * HP + i);
#pragma unroll
      for (int u = 0; u < 4; ++u) a[u] = dot4(w, at4(sm + SH1 + (sa + u) * HP + i), a[u]);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) sm[SH2 + (sa + u) * HP + j] = a[u] > 0.0f ? a[u] : 0.0f;
  }
  __syncthreads();
  if (threadIdx.x < S * OUT && (int)threadIdx.x / OUT < ns) {
    const int s = threadIdx.x / OUT, c = threadIdx.x % OUT;
    float a = sm[SB3 + c];
#pragma unroll
    for (int i = 0; i < H; i += 4) a = dot4(at4(sm + SW3 + c * HP + i), at4(sm + SH2 + s * HP + i), a);
    sm[SZ + threadIdx.x] = a;
  }
  __syncthreads();
}

__global__ void __launch_bounds__(NT) mlp_forward_kernel(const float *__restrict__ params,
                                                         const float *__restrict__ X, int B,
                                                         float *__restrict__ logits) {
  griddep_wait();
  extern __shared__ __align__(16) float sm[];
  const int s0 = blockIdx.x * S, ns = min(S, B - s0);
  block_forward(sm, params, X, s0, ns);
  for (int q = threadIdx.x; q < ns * OUT; q += NT) logits[(long long)s0 * OUT + q] = sm[SZ + q];
}

// Soft-target cross-entropy and backpropagation for one CTA's samples; the
// CTA's gradient sums go to work[blockIdx.x][0..NP) and its loss sum to
// work[blockIdx.x][NP].
__global__ void __launch_bounds__(NT) mlp_loss_grad_kernel(const float *__restrict__ params,
                                                           const float *__restrict__ X,
                                                           const float *__restrict__ T, int B,
                                                           float *__restrict__ work) {
  griddep_wait();
  extern __shared__ __align__(16) float sm[];
  const int s0 = blockIdx.x * S, ns = min(S, B - s0);
  block_forward(sm, params, X, s0, ns);
  __shared__ float s_loss[S];
  const float invB = 1.0f / (float)B;
  if (threadIdx.x < S * OUT) {  // a thread per sample and class, eight lanes of a warp per sample
    const int s = threadIdx.x / OUT;
    const bool on = s < ns;
    const float z = on ? sm[SZ + threadIdx.x] : 0.0f, t = on ? T[(long long)s0 * OUT + threadIdx.x] : 0.0f;
    float zmax = z;
#pragma unroll
    for (int o = OUT / 2; o > 0; o >>= 1) zmax = fmaxf(zmax, __shfl_xor_sync(0xffffffffu, zmax, o));
    float se = expf(z - zmax), tsum = t;
#pragma unroll
    for (int o = OUT / 2; o > 0; o >>= 1) {
      se += __shfl_xor_sync(0xffffffffu, se, o);
      tsum += __shfl_xor_sync(0xffffffffu, tsum, o);
    }
    const float lse = zmax + logf(se);
    float lossv = -t * (z - lse);
#pragma unroll
    for (int o = OUT / 2; o > 0; o >>= 1) lossv += __shfl_xor_sync(0xffffffffu, lossv, o);
    sm[SDZ + threadIdx.x] = on ? (tsum * expf(z - lse) - t) * invB : 0.0f;
    if (threadIdx.x % OUT == 0) s_loss[s] = lossv;
  }
  __syncthreads();
  float *out = work + (long long)blockIdx.x * (NP + 1);
  const int j = unit(), sa = sample0();
  // derivative at the second hidden layer
  {
    float a[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int c = 0; c < OUT; c += 4) {
      const float *w = sm + SW3 + c * HP + j;
      const float4 w4 = make_float4(w[0], w[HP], w[2 * HP], w[3 * HP]);
#pragma unroll
      for (int u = 0; u < 4; ++u) a[u] = dot4(w4, at4(sm + SDZ + (sa + u) * OUT + c), a[u]);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int q = (sa + u) * HP + j;
      sm[SDH2 + q] = sm[SH2 + q] > 0.0f ? a[u] : 0.0f;
    }
  }
  // layer 3: one weight per thread
  static_assert(OUT * H == NT, "one third-layer weight per thread");
  {
    const int c = threadIdx.x / H;
    float g = 0.0f;
#pragma unroll 8
    for (int s = 0; s < ns; ++s) g = fmaf(sm[SDZ + s * OUT + c], sm[SH2 + s * HP + j], g);
    out[OW3 + threadIdx.x] = g;
  }
  if (threadIdx.x < OUT) {
    float g = 0.0f;
#pragma unroll 8
    for (int s = 0; s < ns; ++s) g += sm[SDZ + s * OUT + threadIdx.x];
    out[OB3 + threadIdx.x] = g;
  }
  __syncthreads();
  // derivative at the first hidden layer
  {
    float a[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 4
    for (int k = 0; k < H; k += 4) {
      const float *w = sm + SW2 + k * HP + j;
      const float4 w4 = make_float4(w[0], w[HP], w[2 * HP], w[3 * HP]);
#pragma unroll
      for (int u = 0; u < 4; ++u) a[u] = dot4(w4, at4(sm + SDH2 + (sa + u) * HP + k), a[u]);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int q = (sa + u) * HP + j;
      sm[SDH1 + q] = sm[SH1 + q] > 0.0f ? a[u] : 0.0f;
    }
  }
  // layer 2: weights of the eight units k0 .. k0 + 7 from input j
  {
    const int k0 = threadIdx.x / H * 8;
    float g[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) g[k] = 0.0f;
#pragma unroll 4
    for (int s = 0; s < ns; ++s) {
      const float h = sm[SH1 + s * HP + j];
      const float4 a = at4(sm + SDH2 + s * HP + k0), b = at4(sm + SDH2 + s * HP + k0 + 4);
      g[0] = fmaf(a.x, h, g[0]); g[1] = fmaf(a.y, h, g[1]); g[2] = fmaf(a.z, h, g[2]); g[3] = fmaf(a.w, h, g[3]);
      g[4] = fmaf(b.x, h, g[4]); g[5] = fmaf(b.y, h, g[5]); g[6] = fmaf(b.z, h, g[6]); g[7] = fmaf(b.w, h, g[7]);
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) out[OW2 + (k0 + k) * H + j] = g[k];
  }
  if (threadIdx.x < H) {
    float g = 0.0f;
#pragma unroll 8
    for (int s = 0; s < ns; ++s) g += sm[SDH2 + s * HP + threadIdx.x];
    out[OB2 + threadIdx.x] = g;
  }
  __syncthreads();
  // layer 1
  for (int q = threadIdx.x; q < H * IN; q += NT) {
    const int k = q / IN, i = q % IN;
    float g = 0.0f;
#pragma unroll 8
    for (int s = 0; s < ns; ++s) g = fmaf(sm[SDH1 + s * HP + k], sm[SX + s * IN + i], g);
    out[OW1 + q] = g;
  }
  if (threadIdx.x < H) {
    float g = 0.0f;
#pragma unroll 8
    for (int s = 0; s < ns; ++s) g += sm[SDH1 + s * HP + threadIdx.x];
    out[OB1 + threadIdx.x] = g;
  }
  if (threadIdx.x == NT - 1) {
    float l = 0.0f;
    for (int s = 0; s < ns; ++s) l += s_loss[s];
    out[NP] = l;
  }
}

// grad[p] = sum over CTAs in index order; loss = (sum of CTA losses) / B.
__global__ void __launch_bounds__(128) mlp_reduce_kernel(const float *__restrict__ work, int nblk, int B,
                                                         float *__restrict__ grad, float *__restrict__ loss) {
  griddep_wait();
  const int p = blockIdx.x * 128 + threadIdx.x;
  if (p > NP) return;
  float a = 0.0f;
#pragma unroll 8
  for (int c = 0; c < nblk; ++c) a += work[(long long)c * (NP + 1) + p];
  if (p < NP) grad[p] = a;
  else *loss = a / (float)B;
}

__global__ void __launch_bounds__(128) adam_kernel(float *__restrict__ p, const float *__restrict__ g,
                                                   float *__restrict__ m, float *__restrict__ v, long long n, float lr,
                                                   float b1, float b2, float eps, float c1, float c2) {
  griddep_wait();
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    float gi = g[i];
    float mi = b1 * m[i] + (1.0f - b1) * gi;
    float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

static_assert(SFWD * sizeof(float) <= 48 * 1024, "the forward kernel needs no larger shared memory limit");

// mlp_loss_grad_kernel's shared memory is above the default limit, which is
// raised per device.
cudaError_t raise_smem_limit() {
  static std::atomic<bool> raised[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || (dev < 64 && raised[dev].load())) return e;
  e = cudaFuncSetAttribute(mlp_loss_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(STOT * sizeof(float)));
  if (e == cudaSuccess && dev < 64) raised[dev] = true;
  return e;
}

}  // namespace

cudaError_t launch_mlp_forward(const float *params, const float *X, int B, float *logits, cudaStream_t s) {
  if (B <= 0) return cudaSuccess;
  return launch_pdl(mlp_forward_kernel, dim3((B + S - 1) / S), dim3(NT), SFWD * sizeof(float), s, params, X, (int)B,
                    logits);
}

}  // namespace smat

using namespace smat;

extern "C" {

smat_status_t smat_mlp_forward(const float *params, const float *X, int32_t B, float *logits, void *stream) {
  if (B < 0 || (B > 0 && (!params || !X || !logits))) return SMAT_ERR_INVALID_ARG;
  return launch_mlp_forward(params, X, B, logits, (cudaStream_t)stream) == cudaSuccess ? SMAT_OK : SMAT_ERR_CUDA;
}

int64_t smat_mlp_work_floats(int32_t B) { return (int64_t)((B + S - 1) / S) * (NP + 1); }

smat_status_t smat_mlp_loss_grad(const float *params, const float *X, const float *T, int32_t B, float *grad,
                                 float *loss, float *work, void *stream) {
  if (B <= 0 || !params || !X || !T || !grad || !loss || !work) return SMAT_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  if (raise_smem_limit() != cudaSuccess) return SMAT_ERR_CUDA;
  int nblk = (B + S - 1) / S;
  cudaError_t e = launch_pdl(mlp_loss_grad_kernel, dim3(nblk), dim3(NT), STOT * sizeof(float), s, params, X, T, (int)B,
                             work);
  if (e == cudaSuccess)
    e = launch_pdl(mlp_reduce_kernel, dim3((NP + 1 + 127) / 128), dim3(128), 0, s, (const float *)work, nblk, (int)B,
                   grad, loss);
  return e == cudaSuccess ? SMAT_OK : SMAT_ERR_CUDA;
}

smat_status_t smat_mlp_adam(float *p, const float *g, float *m, float *v, int64_t n, int32_t t, float lr,
                            float beta1, float beta2, float eps, void *stream) {
  if (n < 0 || t < 1 || (n > 0 && (!p || !g || !m || !v))) return SMAT_ERR_INVALID_ARG;
  if (n == 0) return SMAT_OK;
  float c1 = (float)(1.0 - std::pow((double)beta1, (double)t));
  float c2 = (float)(1.0 - std::pow((double)beta2, (double)t));
  const int blocks = (int)std::min<long long>((n + 127) / 128, 8192);
  return launch_pdl(adam_kernel, dim3(blocks), dim3(128), 0, (cudaStream_t)stream, p, g, m, v, (long long)n, lr, beta1,
                    beta2, eps, c1, c2) == cudaSuccess ? SMAT_OK : SMAT_ERR_CUDA;
}

}  // extern "C"
