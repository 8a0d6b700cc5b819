// Building blocks of the kernels whose unit of work is a warp with eight
// consecutive stored entries per lane (COO and SPLIT tiles, csr_flat.cu).
#pragma once

#include "spmv_device.cuh"

namespace smat {
namespace {

constexpr unsigned FULL = 0xffffffffu;

// 32-byte streaming loads (sm_100 and later): one L1 request per 32-byte
// sector.  Two 16-byte loads of one sector by the same thread are two
// requests, and on a kernel bound by the rate of sector requests the second
// one costs as much as the first (and comes back from L2 when the streamed
// line was evicted in between).  p must be 32-byte aligned.
__device__ __forceinline__ void ld32_i32(const int32_t *p, int *o) {
  asm("ld.global.cs.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=r"(o[0]), "=r"(o[1]), "=r"(o[2]), "=r"(o[3]), "=r"(o[4]), "=r"(o[5]), "=r"(o[6]), "=r"(o[7])
      : "l"(p));
}
__device__ __forceinline__ void ld32_f32(const float *p, float *o) {
  asm("ld.global.cs.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=f"(o[0]), "=f"(o[1]), "=f"(o[2]), "=f"(o[3]), "=f"(o[4]), "=f"(o[5]), "=f"(o[6]), "=f"(o[7])
      : "l"(p));
}
__device__ __forceinline__ void ld32_f64(const double *p, double *o) {
  asm("ld.global.cs.v4.f64 {%0, %1, %2, %3}, [%4];" : "=d"(o[0]), "=d"(o[1]), "=d"(o[2]), "=d"(o[3]) : "l"(p));
}
__device__ __forceinline__ bool aligned32(const void *p) { return ((uintptr_t)p & 31u) == 0; }

// IPT consecutive int32 from p (16-byte aligned when `full`; 32-byte loads
// when 32-byte aligned, uniform over a tile since runs start at multiples of 8).
template <int IPT>
__device__ __forceinline__ void load_i32_run(const int32_t *__restrict__ p, bool full, int valid, int (&o)[IPT],
                                             int fill) {
  if (full && IPT % 8 == 0 && aligned32(p)) {
#pragma unroll
    for (int q = 0; q < IPT / 8; ++q) ld32_i32(p + 8 * q, o + 8 * q);
  } else if (full) {
#pragma unroll
    for (int q = 0; q < IPT / 4; ++q) {
      int4 v = __ldcs(reinterpret_cast<const int4 *>(p) + q);
      o[4 * q] = v.x; o[4 * q + 1] = v.y; o[4 * q + 2] = v.z; o[4 * q + 3] = v.w;
    }
  } else {
#pragma unroll
    for (int q = 0; q < IPT; ++q) o[q] = q < valid ? ld_idx(p + q) : fill;
  }
}

template <typename V, int IPT>
__device__ __forceinline__ void load_val_run(const V *__restrict__ p, bool full, int valid,
                                             typename Compute<V>::T (&o)[IPT]) {
  constexpr int R = 16 / (int)sizeof(V);
  if constexpr (sizeof(V) == 8 && IPT % 4 == 0) {
    if (full && aligned32(p)) {
#pragma unroll
      for (int q = 0; q < IPT / 4; ++q) ld32_f64(reinterpret_cast<const double *>(p) + 4 * q, o + 4 * q);
      return;
    }
  } else if constexpr (sizeof(V) == 4 && IPT % 8 == 0) {
    if (full && aligned32(p)) {
#pragma unroll
      for (int q = 0; q < IPT / 8; ++q) ld32_f32(reinterpret_cast<const float *>(p) + 8 * q, o + 8 * q);
      return;
    }
  }
  if (full) {
#pragma unroll
    for (int q = 0; q < IPT / R; ++q) {
      typename Compute<V>::T t[R];
      load_vals<V, R>(p + q * R, t);
#pragma unroll
      for (int r = 0; r < R; ++r) o[q * R + r] = t[r];
    }
  } else {
#pragma unroll
    for (int q = 0; q < IPT; ++q) o[q] = q < valid ? (typename Compute<V>::T)ld_val(p + q) : 0;
  }
}

// Within one warp whose 32 lanes' chunks form a tile: the inclusive
// segmented sum of the lanes' open partial sums c, segments starting at the
// lanes where a row ended (their c opens the next row).  A lane with a row
// end gets the sum at the lane before it: the partials of the row its first
// row end closes.  *open is the sum at lane 31, the row left open at the
// tile's end.  Shuffles only; fixed order.
// Doubling steps that no lane needs any more (a row ended within reach of
// every lane) are left out: in FP64 one step of a warp holds the SM's FP64 pipe
// for 16 clocks, as long as one of the tile's eight multiply-adds.
template <typename T>
__device__ __forceinline__ T warp_carries(bool h, T c, T *open) {
  const int lane = threadIdx.x & 31;
  unsigned reach = ~__ballot_sync(FULL, h);  // lanes that no row end in the last o lanes stops
  T v = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    if (reach == 0) break;
    const T vu = __shfl_up_sync(FULL, v, o);
    if (lane >= o && ((reach >> lane) & 1u)) v = vu + v;
    reach &= reach << o;
  }
  *open = __shfl_sync(FULL, v, 31);
  const T prev = __shfl_up_sync(FULL, v, 1);
  return lane == 0 ? (T)0 : prev;
}

// y[r] += alpha * (sum of the carries of row r), r = rows[carry_row] (rows
// nullptr: carry_row itself); the carries of one row are consecutive.  A warp
// takes the 32 carries at c0 and adds up the runs that start among them (a
// segmented scan); a run that reaches past them is followed by the whole warp,
// 128 carries at a time, so that a row of millions of entries does not wait for
// one thread.
template <typename T, int MODE>
__device__ __forceinline__ void add_carries(long long c0, const int32_t *__restrict__ rows,
                                            const int32_t *__restrict__ carry_row, const T *__restrict__ carry_val,
                                            long long ntiles, const Epi<T, MODE> &ep, T *__restrict__ y) {
  const int lane = threadIdx.x & 31;
  const long long c = c0 + lane;
  const int row = c < ntiles ? carry_row[c] : -1;
  T v = c < ntiles ? carry_val[c] : (T)0;
  int prev = __shfl_up_sync(FULL, row, 1);
  if (lane == 0) prev = c0 > 0 ? carry_row[c0 - 1] : -1;
  const bool head = row >= 0 && row != prev;
  // each head's sum over its run: the lanes after it with the same row
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const T up = __shfl_down_sync(FULL, v, o);
    const int ur = __shfl_down_sync(FULL, row, o);
    if (lane + o < 32 && ur == row) v = add_rn(v, up);
  }
  // the run of the last head, when it goes on past these 32
  const int last = __shfl_sync(FULL, row, 31);
  const unsigned heads = __ballot_sync(FULL, head && row == last);
  if (last >= 0 && heads) {
    T more = 0;
    for (long long q0 = c0 + 32; q0 < ntiles; q0 += 128) {
      int rr[4];
      T vv[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const long long q = q0 + 32 * k + lane;
        rr[k] = q < ntiles ? carry_row[q] : -1;
        vv[k] = q < ntiles ? carry_val[q] : (T)0;
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) more = rr[k] == last ? add_rn(more, vv[k]) : more;
      if (__shfl_sync(FULL, rr[3], 31) != last) break;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) more = add_rn(more, __shfl_xor_sync(FULL, more, o));
    if (lane == __ffs(heads) - 1) v = add_rn(v, more);
  }
  if (head) {
    const long long r = rows ? rows[row] : row;
    y[r] = add_rn(y[r], MODE == EPI_COPY ? v : mul_rn(ep.alpha, v));
  }
}

template <typename T, int MODE>
__global__ void __launch_bounds__(256) carry_kernel(const int32_t *__restrict__ rows,
                                                    const int32_t *__restrict__ carry_row,
                                                    const T *__restrict__ carry_val, long long ntiles, Epi<T, MODE> ep,
                                                    T *__restrict__ y) {
  griddep_wait();
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long c0 = (long long)blockIdx.x * blockDim.x + (threadIdx.x & ~31u); c0 < ntiles; c0 += stride)
    add_carries<T, MODE>(c0, rows, carry_row, carry_val, ntiles, ep, y);
}

}  // namespace
}  // namespace smat
