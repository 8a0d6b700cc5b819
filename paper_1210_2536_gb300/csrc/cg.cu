// Mixed-precision conjugate gradients around the adaptive SpMV.
//
// The paper reports SpMV in single and double precision (Sec. 7.2) and
// motivates the library by iterative solvers that call SpMV hundreds of times
// (Sec. 1, Sec. 7.3).  This solver keeps FP64 only where accuracy is decided:
// the outer loop forms r = b - A x with an FP64 handle and updates x in FP64
// (iterative refinement); the inner loop runs CG in FP32 on A d = r / ||r||
// through an FP32 (or BF16-valued) handle, whose products move half (or a
// third) of the bytes.
//
// Inner iterations keep every scalar on the device: an iteration is the
// product and one cooperative kernel (cg_vector_kernel) that does both dot
// products and all vector updates, with no host round trip, and chunks of
// iterations are replayed from a CUDA graph.  Every sum is taken in a fixed
// order, so a solve is reproducible.  The host reads the residual only between
// chunks.
#include <cuda.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstring>

#include "smat_internal.h"
#include "spmv_device.cuh"

namespace smat {
namespace {

constexpr int CG_NT = 256;
constexpr int CG_BLOCKS = 152 * 4;
// Threads of a cg_vector_kernel CTA, one CTA per SM: with the vectors in
// registers, and streaming them with CV_U float4s of each vector in flight per
// thread (us on 2^24 rows, 40 bytes a row: 512 x 4 105.7, 768 x 3 96.0,
// 768 x 4 97.4, 1024 x 3 95.9 with spills, 512 x 8 98.9; 2^21 rows 11.6-13.1).
constexpr int CV_RESIDENT_NT = 1024, CV_STREAM_NT = 768, CV_U = 3;

// A grid barrier's wait, in SM clocks: about two seconds, and half a millisecond
// once a barrier of the solve has given up (passing one takes a few us; the
// streaming passes before it, up to 100 us on 2^24 rows).
constexpr long long CV_WAIT = 4000000000ll, CV_WAIT_STALLED = 1ll << 20;
struct GridWait {
  long long limit;
  int never;  // test hook: no barrier is passed
};

// Device-side scalars of one solve.
struct CgScalars {
  float rho, rho0;
  int stalled;  // a grid barrier ran out of its limit: the iteration is not valid
  unsigned int arrived;  // CTAs that reached a grid barrier, over all barriers of the inner solve
  double dot64;
  unsigned int counter[2];
};

template <typename T>
__device__ __forceinline__ T block_sum(T v) {
  __shared__ T sh[CG_NT / 32];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  T r = 0;
  if (threadIdx.x < 32) {
    r = threadIdx.x < CG_NT / 32 ? sh[threadIdx.x] : (T)0;
    for (int o = 16; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
  }
  return r;  // valid in thread 0
}

// Last block to finish sums the per-block partials in block order (fixed,
// hence deterministic) and returns true in its thread 0 with *total set.
template <typename T>
__device__ __forceinline__ bool finish_reduce(T part, T *partials, unsigned int *counter, T *total) {
  __shared__ bool last;
  if (threadIdx.x == 0) {
    partials[blockIdx.x] = part;
    __threadfence();
    last = atomicAdd(counter, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return false;
  T s = 0;
  if (threadIdx.x < 32) {
    // lane l sums partials l, l+32, ... in order; then a fixed shuffle tree
    for (unsigned b = threadIdx.x; b < gridDim.x; b += 32) s += ((volatile T *)partials)[b];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  }
  if (threadIdx.x == 0) {
    *total = s;
    *counter = 0;  // ready for the next launch
  }
  return threadIdx.x == 0;
}

// FP64 dot product a.b -> sc->dot64.  Four elements of each array in flight
// per thread: one at a time (37.4 us for 2 x 134 MB) left the memory idle
// between loads.  The caller's vectors are only 8-byte aligned.
__global__ void __launch_bounds__(CG_NT) dot64_kernel(const double *__restrict__ a, const double *__restrict__ b,
                                                      long long n, double *partials, CgScalars *sc) {
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  const long long step = (long long)gridDim.x * CG_NT;
  for (long long i = (long long)blockIdx.x * CG_NT + threadIdx.x; i < n; i += 4 * step) {
    double u[4], v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const bool on = i + k * step < n;
      u[k] = on ? a[i + k * step] : 0.0;
      v[k] = on ? b[i + k * step] : 0.0;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) acc[k] = fma(u[k], v[k], acc[k]);
  }
  double part = block_sum((acc[0] + acc[1]) + (acc[2] + acc[3]));
  double tot;
  if (finish_reduce(part, partials, &sc->counter[0], &tot)) sc->dot64 = tot;
}

// r32 = (float)(r * inv_scale); d = 0; p = r32; rho = r32.r32, rho0 = rho.
__global__ void __launch_bounds__(CG_NT) inner_init_kernel(const double *__restrict__ r, double inv_scale, long long n,
                                                           float *__restrict__ res, float *__restrict__ p,
                                                           float *__restrict__ d, float *partials, CgScalars *sc) {
  float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  const long long step = (long long)gridDim.x * CG_NT;
  for (long long i = (long long)blockIdx.x * CG_NT + threadIdx.x; i < n; i += 4 * step) {
    float v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = i + k * step < n ? (float)(r[i + k * step] * inv_scale) : 0.0f;
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (i + k * step < n) {
        res[i + k * step] = v[k];
        p[i + k * step] = v[k];
        d[i + k * step] = 0.0f;
        acc[k] = fmaf(v[k], v[k], acc[k]);
      }
  }
  float part = block_sum((acc[0] + acc[1]) + (acc[2] + acc[3]));
  float tot;
  if (finish_reduce(part, partials, &sc->counter[1], &tot)) {
    sc->rho = tot;
    sc->rho0 = tot;
    sc->arrived = 0;  // the grid barriers count from here
  }
}

// One thread of each CTA: waits until every CTA of the grid (all resident: a
// cooperative launch) has arrived.  The wait is bounded: a grid that gives up
// sets sc->stalled, which the host reads with the residual, and every CTA still
// runs to its end, arriving at each barrier.  The iterations queued behind it are
// invalid too, so from then on a barrier that is not passed soon is left: the
// host looks only after a chunk, whose every barrier would otherwise wait for
// the whole limit.
__device__ __forceinline__ void grid_arrive_wait(CgScalars *sc, const GridWait &wait) {
  __threadfence();
  const unsigned ticket = atomicAdd(&sc->arrived, 1u);
  const unsigned target = ticket - ticket % gridDim.x + gridDim.x;
  const long long t0 = clock64();
  for (;;) {
    unsigned now;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(now) : "l"(&sc->arrived) : "memory");
    if ((int)(now - target) >= 0 && !wait.never) break;
    const long long waited = clock64() - t0;
    if (waited > wait.limit || (waited > CV_WAIT_STALLED && *(volatile int *)&sc->stalled)) {
      sc->stalled = 1;
      break;
    }
  }
}

__device__ __forceinline__ float warp_total(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sum over all threads of the grid, in every thread: per CTA, then the CTAs'
// partials in the same order in every CTA.  CLUSTER: the grid is one
// thread-block cluster (or one CTA), whose hardware barrier takes the place of
// the counter in memory.  One warp per CTA reads the partials: with all of
// them reading (24 K requests for the same lines) a sum over 147 CTAs took
// 7 us instead of 2.
template <bool CLUSTER, int NT>
__device__ __forceinline__ float grid_sum(float v, float *partials, CgScalars *sc, const GridWait &wait) {
  __shared__ float sh[NT / 32], total;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  v = warp_total(v);
  if (lane == 0) sh[w] = v;
  __syncthreads();
  if (w == 0) {
    v = warp_total(lane < NT / 32 ? sh[lane] : 0.0f);
    if (lane == 0) {
      if (CLUSTER && gridDim.x == 1) {
        total = v;
      } else {
        partials[blockIdx.x] = v;
        if (!CLUSTER) grid_arrive_wait(sc, wait);
      }
    }
    __syncwarp();
  }
  if (CLUSTER && gridDim.x == 1) {
    __syncthreads();
    return total;
  }
  if (CLUSTER)
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  if (w == 0) {
    v = 0.0f;
    for (unsigned b = lane; b < gridDim.x; b += 32) v += __ldcg(partials + b);
    v = warp_total(v);
    if (lane == 0) total = v;
  }
  __syncthreads();
  return total;
}

__device__ __forceinline__ float4 fma4(float a, float4 x, float4 y) {
  return make_float4(fmaf(a, x.x, y.x), fmaf(a, x.y, y.y), fmaf(a, x.z, y.z), fmaf(a, x.w, y.w));
}
__device__ __forceinline__ float dot4(float4 x, float4 y, float acc) {
  return fmaf(x.w, y.w, fmaf(x.z, y.z, fmaf(x.y, y.y, fmaf(x.x, y.x, acc))));
}

__device__ __forceinline__ float sum_of(const float (&a)[CV_U]) {
  float v = a[0];
#pragma unroll
  for (int k = 1; k < CV_U; ++k) v += a[k];
  return v;
}

// The vector part of one CG iteration after q = A p, in one launch of at most
// one CTA per SM, all resident:
//   alpha = rho / p.q (0 on breakdown);  res -= alpha q;  rho' = res.res;
//   beta = rho'/rho;  d += alpha p;  p = res + beta p;  rho = rho'.
//
// RESIDENT (a thread holds one float4 of each vector): everything is read
// once, kept in registers across the two sums and written once.  Bound by the
// latency of the reads and of the two grid-wide sums.
//
// Otherwise bound by memory: p and q are read, then q and res read and res
// written, then d, res and p read and d and p written: 40 bytes per row (d
// moves with p's last use).  A thread handles the same float4s in every pass,
// and the passes run in turn up and down the vectors, so that each starts on
// what the one before left in L1 and L2.
//
// It took the place of three kernels that moved one float per load (p.q; d,
// res and the new residual; p), 208 us for 2^24 rows (44 bytes a row) and
// three launches an iteration; this one takes 96 us there (7.0 TB/s), 12.1 us
// for 2^21 rows and 2.7-8.3 us with the vectors in registers.  Solves of 160
// iterations: 256^3 grid 52.7 -> 31.9 ms, 101^3 5.7 -> 3.5 ms, 16^3 2.2 -> 1.4.
template <bool CLUSTER, bool RESIDENT, int NT = RESIDENT ? CV_RESIDENT_NT : CV_STREAM_NT>
__global__ void __launch_bounds__(NT, 1) cg_vector_kernel(float *__restrict__ p, const float *__restrict__ q,
                                                          float *__restrict__ d, float *__restrict__ res, int n,
                                                          float *partials, CgScalars *sc, GridWait wait) {
  griddep_wait();
  const float rho = __ldcg(&sc->rho);  // CTA 0 writes the new one after the last sum
  const int n4 = n / 4, step = gridDim.x * NT, first = blockIdx.x * NT + threadIdx.x;
  const bool tail = blockIdx.x == 0 && (int)threadIdx.x < n - 4 * n4;  // the last n % 4 elements
  const int it = 4 * n4 + threadIdx.x;
  float4 *p4 = reinterpret_cast<float4 *>(p), *d4 = reinterpret_cast<float4 *>(d), *r4 = reinterpret_cast<float4 *>(res);
  const float4 *q4 = reinterpret_cast<const float4 *>(q);
  const float4 zero = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  if (RESIDENT) {
    const bool on = first < n4;
    const float4 P = on ? p4[first] : zero, Q = on ? q4[first] : zero, D = on ? d4[first] : zero;
    float4 R = on ? r4[first] : zero;
    const float tp = tail ? p[it] : 0.0f, tq = tail ? q[it] : 0.0f, td = tail ? d[it] : 0.0f;
    float tr = tail ? res[it] : 0.0f;
    const float pq = grid_sum<CLUSTER, NT>(dot4(P, Q, tp * tq), partials, sc, wait);
    const float alpha = (pq > 0.0f && rho > 0.0f) ? rho / pq : 0.0f;
    R = fma4(-alpha, Q, R);
    tr = fmaf(-alpha, tq, tr);
    const float rho1 = grid_sum<CLUSTER, NT>(dot4(R, R, tr * tr), partials + gridDim.x, sc, wait);
    const float beta = rho > 0.0f ? rho1 / rho : 0.0f;
    if (blockIdx.x == 0 && threadIdx.x == 0) sc->rho = rho1;
    if (on) {
      r4[first] = R;
      d4[first] = fma4(alpha, P, D);
      p4[first] = fma4(beta, P, R);
    }
    if (tail) {
      res[it] = tr;
      d[it] = fmaf(alpha, tp, td);
      p[it] = fmaf(beta, tp, tr);
    }
    return;
  }
  const int rounds = (n4 + CV_U * step - 1) / (CV_U * step);
  float acc[CV_U];
#pragma unroll
  for (int k = 0; k < CV_U; ++k) acc[k] = 0.0f;
  for (int t = rounds - 1; t >= 0; --t) {
    float4 a[CV_U], b[CV_U];
#pragma unroll
    for (int k = 0; k < CV_U; ++k) {
      const int i = first + (t * CV_U + k) * step;
      a[k] = i < n4 ? p4[i] : zero;
      b[k] = i < n4 ? q4[i] : zero;
    }
#pragma unroll
    for (int k = 0; k < CV_U; ++k) acc[k] = dot4(a[k], b[k], acc[k]);
  }
  if (tail) acc[0] = fmaf(p[it], q[it], acc[0]);
  const float pq = grid_sum<CLUSTER, NT>(sum_of(acc), partials, sc, wait);
  const float alpha = (pq > 0.0f && rho > 0.0f) ? rho / pq : 0.0f;
#pragma unroll
  for (int k = 0; k < CV_U; ++k) acc[k] = 0.0f;
  for (int t = 0; t < rounds; ++t) {
    float4 a[CV_U], b[CV_U];
#pragma unroll
    for (int k = 0; k < CV_U; ++k) {
      const int i = first + (t * CV_U + k) * step;
      a[k] = i < n4 ? q4[i] : zero;
      b[k] = i < n4 ? r4[i] : zero;
    }
#pragma unroll
    for (int k = 0; k < CV_U; ++k) {
      const int i = first + (t * CV_U + k) * step;
      b[k] = fma4(-alpha, a[k], b[k]);
      if (i < n4) r4[i] = b[k];
      acc[k] = dot4(b[k], b[k], acc[k]);
    }
  }
  if (tail) {
    const float v = fmaf(-alpha, q[it], res[it]);
    res[it] = v;
    acc[0] = fmaf(v, v, acc[0]);
  }
  const float rho1 = grid_sum<CLUSTER, NT>(sum_of(acc), partials + gridDim.x, sc, wait);
  const float beta = rho > 0.0f ? rho1 / rho : 0.0f;
  if (blockIdx.x == 0 && threadIdx.x == 0) sc->rho = rho1;
  for (int t = rounds - 1; t >= 0; --t) {
    float4 a[CV_U], b[CV_U], c[CV_U];
#pragma unroll
    for (int k = 0; k < CV_U; ++k) {
      const int i = first + (t * CV_U + k) * step;
      a[k] = i < n4 ? p4[i] : zero;
      b[k] = i < n4 ? r4[i] : zero;
      c[k] = i < n4 ? d4[i] : zero;
    }
#pragma unroll
    for (int k = 0; k < CV_U; ++k) {
      const int i = first + (t * CV_U + k) * step;
      if (i < n4) {
        d4[i] = fma4(alpha, a[k], c[k]);
        p4[i] = fma4(beta, a[k], b[k]);
      }
    }
  }
  if (tail) {
    d[it] = fmaf(alpha, p[it], d[it]);
    p[it] = fmaf(beta, p[it], res[it]);
  }
}

// x += scale * (double) d.
__global__ void __launch_bounds__(CG_NT) refine_kernel(double *__restrict__ x, const float *__restrict__ d,
                                                       double scale, long long n) {
  const long long step = (long long)gridDim.x * CG_NT;
  for (long long i = (long long)blockIdx.x * CG_NT + threadIdx.x; i < n; i += 4 * step) {
    double u[4];
    float v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const bool on = i + k * step < n;
      u[k] = on ? x[i + k * step] : 0.0;
      v[k] = on ? d[i + k * step] : 0.0f;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (i + k * step < n) x[i + k * step] = fma(scale, (double)v[k], u[k]);
  }
}

int blocks_for(long long n) {
  long long b = (n + CG_NT - 1) / CG_NT;
  return (int)(b < CG_BLOCKS ? (b < 1 ? 1 : b) : CG_BLOCKS);
}

// The launch shape of cg_vector_kernel for n rows.
struct VectorShape {
  int ctas;
  bool cluster, resident;
};

// The device's SMs, and those that the current context may use: a green
// context holds some of them only, and CTAs beyond its own are never resident
// together.
template <typename F>
F driver_function(const char *name, unsigned version) {
  void *p = nullptr;
  cudaDriverEntryPointQueryResult r;
  if (cudaGetDriverEntryPointByVersion(name, &p, version, cudaEnableDefault, &r) != cudaSuccess ||
      r != cudaDriverEntryPointSuccess)
    p = nullptr;
  return (F)p;
}

void count_sms(int *device, int *context) {
  static const auto current = driver_function<CUresult (*)(CUcontext *)>("cuCtxGetCurrent", 4000);
  static const auto resource =
      driver_function<CUresult (*)(CUcontext, CUdevResource *, CUdevResourceType)>("cuCtxGetDevResource", 12040);
  int dev = 0;
  *device = 1;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(device, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    *device = 1;
  *context = *device;
  CUcontext ctx = nullptr;
  CUdevResource res;
  if (current && resource && current(&ctx) == CUDA_SUCCESS && ctx &&
      resource(ctx, &res, CU_DEV_RESOURCE_TYPE_SM) == CUDA_SUCCESS && res.sm.smCount > 0)
    *context = std::min(*device, (int)res.sm.smCount);
}

VectorShape vector_shape(long long n) {
  int device, sms;
  count_sms(&device, &sms);
  // CTAs of one float4 per thread
  const long long want = std::max((n + 4 * CV_RESIDENT_NT - 1) / (4 * CV_RESIDENT_NT), 1ll);
  // one cluster of the portable size; a context with part of the SMs may not
  // have as many next to each other
  if (want <= 8 && sms == device) {
    int c = 1;
    while (c < want) c *= 2;
    return {c, true, true};
  }
  const int most = std::min(sms, CG_BLOCKS);
  return {(int)std::min<long long>(most, want), false, want <= most};
}

cudaError_t launch_cg_vector(const VectorShape &v, float *p, const float *q, float *d, float *res, long long n,
                             float *partials, CgScalars *sc, const GridWait &wait, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)v.ctas);
  cfg.blockDim = dim3(v.resident ? CV_RESIDENT_NT : CV_STREAM_NT);
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  cfg.attrs = at;
  if (v.cluster) {
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)v.ctas;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, cg_vector_kernel<true, true>, p, q, d, res, (int)n, partials, sc, wait);
  }
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, v.resident ? cg_vector_kernel<false, true> : cg_vector_kernel<false, false>, p, q, d,
                            res, (int)n, partials, sc, wait);
}

struct Workspace {
  void *mem = nullptr;
  ~Workspace() { dev_free(mem); }
};

}  // namespace
}  // namespace smat

using namespace smat;

extern "C" void smat_cg_opts_default(smat_cg_opts_t *o) {
  if (!o) return;
  std::memset(o, 0, sizeof(*o));
  o->rtol = 1e-10;
  o->max_outer = 50;
  o->max_inner = 500;
  o->inner_rtol = 1e-4f;
  o->max_total_inner = 0;
  o->check_every = 10;
  o->use_graph = 1;
}

extern "C" smat_status_t smat_cg_mixed(smat_handle_t a64, smat_handle_t a32, const double *b, double *x,
                                       const smat_cg_opts_t *opts_in, smat_cg_info_t *info, void *stream) {
  if (!a64 || !a32 || !b || !x) return SMAT_ERR_INVALID_ARG;
  if (a64->dtype != SMAT_F64 || a32->dtype == SMAT_F64) return SMAT_ERR_INVALID_ARG;
  if (a64->m != a64->n || a32->m != a64->m || a32->n != a64->n) return SMAT_ERR_INVALID_ARG;
  smat_cg_opts_t o;
  if (opts_in) o = *opts_in; else smat_cg_opts_default(&o);
  if (o.check_every < 1) o.check_every = 1;
  const long long n = a64->n;
  smat_cg_info_t inf{};
  if (n == 0) {
    inf.converged = 1;
    if (info) *info = inf;
    return SMAT_OK;
  }
  cudaStream_t user = (cudaStream_t)stream;
  // workspace: r (f64), partials (f64, CG_BLOCKS), res/p/q/d (f32), scalars;
  // every array starts on 256 bytes, whatever n: the ELL and DIA products take
  // p and q with 16-byte accesses and would fall back to CSR-scalar otherwise
  const auto up = [](size_t bytes) { return (bytes + 255) / 256 * 256; };
  const size_t off_r = 0, off_part = off_r + up((size_t)n * 8), off_res = off_part + up((size_t)CG_BLOCKS * 8);
  const size_t off_p = off_res + up((size_t)n * 4), off_q = off_p + up((size_t)n * 4), off_d = off_q + up((size_t)n * 4);
  const size_t off_sc = off_d + up((size_t)n * 4), total = off_sc + sizeof(CgScalars);
  Workspace ws;
  cudaError_t e = dev_alloc(&ws.mem, total);
  if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? SMAT_ERR_ALLOC : SMAT_ERR_CUDA;
  char *base = (char *)ws.mem;
  double *r = (double *)(base + off_r), *part64 = (double *)(base + off_part);
  float *part32 = (float *)(base + off_part);
  float *res = (float *)(base + off_res), *p = (float *)(base + off_p), *q = (float *)(base + off_q),
        *d = (float *)(base + off_d);
  CgScalars *sc = (CgScalars *)(base + off_sc);
  // a private stream (capturable), ordered after the caller's stream
  cudaStream_t s = nullptr;
  cudaEvent_t ev = nullptr;
  cudaGraphExec_t gexec = nullptr;
  cudaGraph_t graph = nullptr;
  smat_status_t status = SMAT_OK;
  const int gb = blocks_for(n);
  const VectorShape gv = vector_shape(n);
  GridWait wait{CV_WAIT, 0};
  long long stall_cycles = 0;
  if (stall_waits(&stall_cycles)) wait = {stall_cycles > 0 ? stall_cycles : CV_WAIT, 1};
  const double one = 1.0, mone = -1.0;
  const float onef = 1.0f, zerof = 0.0f;
  double nb = 0.0, nr = 0.0;
  auto chk = [&](cudaError_t ce) {
    if (ce != cudaSuccess && status == SMAT_OK) status = ce == cudaErrorMemoryAllocation ? SMAT_ERR_ALLOC : SMAT_ERR_CUDA;
    return ce == cudaSuccess;
  };
  auto spmv32 = [&]() -> bool {
    smat_status_t st = smat_spmv(a32, &onef, p, &zerof, q, s);
    if (st != SMAT_OK && status == SMAT_OK) status = st;
    return st == SMAT_OK;
  };
  auto inner_iteration = [&]() -> bool {
    if (!spmv32()) return false;
    return chk(launch_cg_vector(gv, p, q, d, res, n, part32, sc, wait, s));
  };
  auto residual_norm = [&](double *out) -> bool {
    // r = b - A64 x in FP64, then ||r||
    if (!chk(cudaMemcpyAsync(r, b, (size_t)n * 8, cudaMemcpyDeviceToDevice, s))) return false;
    smat_status_t st = smat_spmv(a64, &mone, x, &one, r, s);
    if (st != SMAT_OK) { if (status == SMAT_OK) status = st; return false; }
    dot64_kernel<<<gb, CG_NT, 0, s>>>(r, r, n, part64, sc);
    double v = 0.0;
    if (!chk(cudaMemcpyAsync(&v, &sc->dot64, 8, cudaMemcpyDeviceToHost, s))) return false;
    if (!chk(cudaStreamSynchronize(s))) return false;
    *out = std::sqrt(v);
    return true;
  };
  const auto t0 = std::chrono::steady_clock::now();
  do {
    if (!chk(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking))) break;
    if (!chk(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming))) break;
    if (!chk(cudaEventRecord(ev, user)) || !chk(cudaStreamWaitEvent(s, ev, 0))) break;
    // the inner products' carries on s, which cannot be allocated while it
    // captures: other streams may hold the handle's own
    Scratch carries;
    if (needs_scratch(a32, a32->variant) && !chk(stream_scratch(a32, s, &carries))) break;
    if (!chk(cudaMemsetAsync(sc, 0, sizeof(CgScalars), s))) break;
    dot64_kernel<<<gb, CG_NT, 0, s>>>(b, b, n, part64, sc);
    double bb = 0.0;
    if (!chk(cudaMemcpyAsync(&bb, &sc->dot64, 8, cudaMemcpyDeviceToHost, s)) || !chk(cudaStreamSynchronize(s))) break;
    nb = std::sqrt(bb);
    if (nb == 0.0) {  // b = 0: x = 0 is the solution
      chk(cudaMemsetAsync(x, 0, (size_t)n * 8, s));
      nr = 0.0;
      inf.converged = 1;
      break;
    }
    if (!residual_norm(&nr)) break;
    const int chunk = o.check_every;
    while (nr / nb > o.rtol && inf.outer < o.max_outer &&
           (o.max_total_inner <= 0 || inf.inner_total < o.max_total_inner)) {
      inner_init_kernel<<<gb, CG_NT, 0, s>>>(r, 1.0 / nr, n, res, p, d, part32, sc);
      if (!chk(cudaGetLastError())) break;
      int it = 0;
      const float stop2 = o.inner_rtol * o.inner_rtol;
      bool ok = true;
      while (it < o.max_inner && (o.max_total_inner <= 0 || inf.inner_total + it < o.max_total_inner)) {
        int k = std::min(chunk, o.max_inner - it);
        if (o.max_total_inner > 0) k = std::min(k, o.max_total_inner - inf.inner_total - it);
        if (o.use_graph && k == chunk) {
          if (!gexec) {  // capture one chunk of iterations once, replay it afterwards
            std::shared_lock<std::shared_mutex> capturing(capture_mu());
            if (!chk(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal))) { ok = false; break; }
            bool cap_ok = true;
            for (int j = 0; j < chunk && cap_ok; ++j) cap_ok = inner_iteration();
            cudaError_t ce = cudaStreamEndCapture(s, &graph);
            capturing.unlock();
            if (!cap_ok || !chk(ce)) { ok = false; break; }
            if (!chk(cudaGraphInstantiate(&gexec, graph, 0))) { ok = false; break; }
          }
          if (!chk(cudaGraphLaunch(gexec, s))) { ok = false; break; }
        } else {
          for (int j = 0; j < k && ok; ++j) ok = inner_iteration();
          if (!ok) break;
        }
        it += k;
        CgScalars now;
        if (!chk(cudaMemcpyAsync(&now, sc, sizeof(now), cudaMemcpyDeviceToHost, s)) ||
            !chk(cudaStreamSynchronize(s))) { ok = false; break; }
        if (now.stalled) {
          chk(cudaErrorLaunchTimeout);
          ok = false;
          break;
        }
        const float rho = now.rho, rho0 = now.rho0;
        if (!(rho <= stop2 * rho0) && std::isfinite(rho) && rho > 0.0f) continue;
        break;
      }
      if (!ok) break;
      inf.inner_total += it;
      refine_kernel<<<gb, CG_NT, 0, s>>>(x, d, nr, n);
      if (!chk(cudaGetLastError())) break;
      ++inf.outer;
      if (!residual_norm(&nr)) break;
    }
  } while (false);
  if (s) cudaStreamSynchronize(s);
  // the caller's stream continues after the solve
  if (ev && s && status == SMAT_OK) {
    chk(cudaEventRecord(ev, s));
    chk(cudaStreamWaitEvent(user, ev, 0));
  }
  if (gexec) cudaGraphExecDestroy(gexec);
  if (graph) cudaGraphDestroy(graph);
  if (ev) cudaEventDestroy(ev);
  if (s) {
    release_stream_scratch(a64, s);
    release_stream_scratch(a32, s);
    cudaStreamDestroy(s);
  }
  inf.relres = nb > 0.0 ? nr / nb : 0.0;
  if (nb > 0.0 && inf.relres <= o.rtol) inf.converged = 1;
  inf.seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
  if (info) *info = inf;
  if (status != SMAT_OK) return status;
  return inf.converged ? SMAT_OK : SMAT_ERR_NOT_CONVERGED;
}
