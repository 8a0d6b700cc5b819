// CSR validation and feature extraction on the GPU (arXiv 1210.2536, Sec. 4,
// Table "Feature parameters of a sparse matrix").
//
// Everything here is integer work over rowptr and colidx, so the results are
// exact and independent of scheduling:
//   row_stats   : max_RD, min_RD, sum rd^2, empty rows and the row-degree
//                 histogram h[k]                             (one read of rowptr)
//   diag_count  : the count of stored entries on every diagonal d = j - i
//                                                            (one read of colidx)
//   diag_reduce : Ndiags, number of "true" diagonals and the occupied offsets
// The floating-point features are finished on the host from these integers.
#include <algorithm>
#include <climits>

#include "smat_internal.h"
#include "warp_tile.cuh"

namespace smat {
namespace {

__device__ __forceinline__ int warp_max(int v) {
  for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(FULL, v, o));
  return v;
}
__device__ __forceinline__ int warp_min(int v) {
  for (int o = 16; o > 0; o >>= 1) v = min(v, __shfl_xor_sync(FULL, v, o));
  return v;
}
template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
  return v;
}

// Row containing flattened nonzero k, given each lane's row start (lanes past
// the group hold UINT_MAX): the largest lane L with start_L <= k.
__device__ __forceinline__ int row_lane_of(unsigned start_of_my_row, unsigned k) {
  int L = 0;
#pragma unroll
  for (int step = 16; step > 0; step >>= 1) {
    int cand = L + step;
    unsigned sc = __shfl_sync(FULL, start_of_my_row, cand & 31);
    if (cand < 32 && sc <= k) L = cand;
  }
  return L;
}

// ---------------------------------------------------------------------------
// K1: validation, in two balanced passes.  Per row: the row pointer must not
// fall, and the row's first entry is marked in a bitmap over the stored
// entries.  Per entry (8 per thread, one 32-byte load; the next thread's first
// column by a shuffle): the column must lie in [0, n), and must be below the
// next entry's unless a row starts there.  Work is spread by rows and by
// entries, so a few very long rows do not hold one warp while the others idle.
// Every index read is clamped into the arrays, so malformed input cannot send
// either pass out of bounds.  28.7 M entries: 11 + 40 us (columns 45 us with 4
// entries per thread, 44 with two groups of 8 in flight).
// ---------------------------------------------------------------------------
__global__ void validate_rows_kernel(const int32_t *__restrict__ rowptr, long long m, long long nnz,
                                     unsigned *__restrict__ starts, int *flag) {
  int err = 0;
  if (blockIdx.x == 0 && threadIdx.x == 0 && (rowptr[0] != 0 || (long long)rowptr[m] != nnz)) err |= ERRF_ROWPTR;
  for (long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x; r < m;
       r += (long long)gridDim.x * blockDim.x) {
    const long long s = rowptr[r], e = rowptr[r + 1];
    if (e < s) err |= ERRF_ROWPTR;
    if (s >= 0 && s < nnz) atomicOr(&starts[s >> 5], 1u << (s & 31));
  }
  err = __reduce_or_sync(FULL, err);
  if ((threadIdx.x & 31) == 0 && err) atomicOr(flag, err);
}

__global__ void __launch_bounds__(256) validate_cols_kernel(const int32_t *__restrict__ col, long long nnz, long long n,
                                                            const unsigned *__restrict__ starts, int *flag) {
  int err = 0;
  const int lane = threadIdx.x & 31;
  const long long groups = (nnz + 7) / 8, stride = (long long)gridDim.x * blockDim.x;
  for (long long t0 = (long long)blockIdx.x * blockDim.x + threadIdx.x - lane; t0 < groups; t0 += stride) {
    const long long k0 = 8 * (t0 + lane);
    const int valid = (int)max(0ll, min(8ll, nnz - k0));
    int c[8];
    load_i32_run<8>(col + k0, valid == 8, valid, c, 0);
    // bits of entries k0 + 1 .. k0 + 8: k0 + 8 may sit in the next word
    unsigned marks = 0;
    if (valid > 0) {
      marks = __ldg(starts + (k0 >> 5)) >> (k0 & 31) >> 1;
      if (((k0 + 8) & 31) == 0) marks |= (__ldg(starts + ((k0 + 8) >> 5)) & 1u) << 7;
    }
    int next = __shfl_down_sync(FULL, c[0], 1);
    if (lane == 31) next = k0 + 8 < nnz ? __ldg(col + k0 + 8) : 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int after = i < 7 ? c[i < 7 ? i + 1 : 7] : next;
      if (i < valid && (c[i] < 0 || (long long)c[i] >= n)) err |= ERRF_COL_RANGE;
      if (i < valid && k0 + i + 1 < nnz && !((marks >> i) & 1u) && after <= c[i]) err |= ERRF_COL_ORDER;
    }
  }
  err = __reduce_or_sync(FULL, err);
  if (lane == 0 && err) atomicOr(flag, err);
}

// ---------------------------------------------------------------------------
// K2: integer statistics and histogram of the row degrees in one pass over the
// row pointers.  Degrees below HIST_LEN are counted in shared memory (equal ones
// of a warp at once); longer rows are few (at most NNZ / HIST_LEN) and listed.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) row_stats_kernel(const int32_t *__restrict__ rowptr, long long m,
                                                        FeatureHead *out, int32_t *__restrict__ long_rows) {
  __shared__ int sh_hist[HIST_LEN];
  for (int t = threadIdx.x; t < HIST_LEN; t += blockDim.x) sh_hist[t] = 0;
  __syncthreads();
  unsigned long long s2 = 0;
  int mx = 0, mn = INT_MAX, emp = 0;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (long long r0 = (long long)blockIdx.x * blockDim.x + threadIdx.x - lane; r0 < m;
       r0 += (long long)gridDim.x * blockDim.x) {
    const int rd = r0 + lane < m ? rowptr[r0 + lane + 1] - rowptr[r0 + lane] : -1;
    if (rd >= 0) {
      s2 += (unsigned long long)rd * (unsigned long long)rd;
      mx = max(mx, rd);
      mn = min(mn, rd);
      emp += (rd == 0);
      if (rd >= HIST_LEN) long_rows[atomicAdd(&out->nlong, 1)] = rd;
    }
    const unsigned peers = __match_any_sync(FULL, rd);
    if (rd >= 0 && rd < HIST_LEN && lane == __ffs(peers) - 1) atomicAdd(&sh_hist[rd], __popc(peers));
  }
  s2 = warp_sum(s2);
  mx = warp_max(mx);
  mn = warp_min(mn);
  emp = warp_sum(emp);
  __shared__ unsigned long long sh_s2[8];
  __shared__ int sh_mx[8], sh_mn[8], sh_emp[8];
  if (lane == 0) { sh_s2[w] = s2; sh_mx[w] = mx; sh_mn[w] = mn; sh_emp[w] = emp; }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 1; k < 8; ++k) {
      s2 += sh_s2[k];
      mx = max(mx, sh_mx[k]);
      mn = min(mn, sh_mn[k]);
      emp += sh_emp[k];
    }
    if (s2) atomicAdd(&out->s2, s2);
    atomicMax(&out->max_rd, mx);
    atomicMax(&out->below_max, INT_MAX - mn);  // the smallest degree, kept so that it starts at zero
    if (emp) atomicAdd(&out->empty_rows, emp);
  }
  for (int t = threadIdx.x; t < HIST_LEN; t += blockDim.x)
    if (sh_hist[t]) atomicAdd(&out->hist[t], sh_hist[t]);
}

// ---------------------------------------------------------------------------
// K3: stored entries per diagonal.  A warp owns an equal share of the entries,
// whatever the rows' lengths: with 32 rows per warp, the warps of a power-law
// matrix that held rows of 10^4 entries ran on alone (2e6 rows, 28.7 M entries:
// 918 us, now 226; uniform 1e6, 16 M: 105 and 129).  The row of its first entry comes from a 32-way search; the rows of
// the following entries from 32 row pointers held by the lanes.  Counts are
// aggregated first across the warp (__match_any_sync), then in a per-CTA shared
// hash table whose final entries reach global memory, so that a banded matrix
// issues a handful of global atomics per CTA; once HT_MOST slots are taken
// (random columns, very wide stencils) the entries count in global memory
// directly, at most about 200 G/s (142 us for the power-law matrix).  A table
// that was kept until its probes failed cost wide box stencils most of their
// time: all features of the radius-6 one on 20^3 took 2761 us, now 204; radius 3
// on 40^3 540 and 312.
// ---------------------------------------------------------------------------
constexpr int HT = 2048;           // hash slots per CTA
constexpr int HT_PROBES = 4;
constexpr int HT_MOST = 512;      // slots taken when the table is given up
constexpr int EMPTY_KEY = INT_MIN;

// Adds c to diagonal d's count in the CTA's table, or to the global count when
// its probes find no slot.  A table with HT_MOST slots taken is given up (random
// columns): the CTA's later entries go to the global counts directly.
__device__ __forceinline__ void ht_add(int *keys, int *cnts, int *g_cnt, long long m, int d, int c, int *used) {
  unsigned h = ((unsigned)d * 2654435761u) >> (32 - 11);
#pragma unroll 1
  for (int p = 0; p < HT_PROBES; ++p) {
    int prev = atomicCAS(&keys[h], EMPTY_KEY, d);
    if (prev == EMPTY_KEY) atomicAdd(used, 1);
    if (prev == EMPTY_KEY || prev == d) {
      atomicAdd(&cnts[h], c);
      return;
    }
    h = (h + 1) & (HT - 1);
  }
  atomicAdd(&g_cnt[(long long)d + m - 1], c);
}

// The row that holds entry k (0 <= k < nnz): the last r with rowptr[r] <= k.
// The whole warp searches, 32 row pointers at a time.
__device__ __forceinline__ long long warp_row_of(const int32_t *__restrict__ rowptr, long long lo, long long m,
                                                 long long k) {
  const int lane = threadIdx.x & 31;
  long long hi = m;  // rowptr[lo] <= k < rowptr[hi]
  while (hi - lo > 1) {
    const long long step = (hi - lo + 31) / 32, p = lo + (lane + 1) * step;
    const bool below = p < hi && (long long)__ldg(rowptr + p) <= k;
    const int c = __popc(__ballot_sync(FULL, below));
    hi = min(lo + (c + 1) * step, hi);
    lo += c * step;
  }
  return lo;
}

__global__ void __launch_bounds__(256, 8) diag_count_kernel(const int32_t *__restrict__ rowptr,
                                                            const int32_t *__restrict__ col, long long m, unsigned nnz,
                                                            unsigned share, int *g_cnt) {
  __shared__ int keys[HT], cnts[HT];
  __shared__ int used;  // slots taken
  if (threadIdx.x == 0) used = 0;
  for (int t = threadIdx.x; t < HT; t += blockDim.x) { keys[t] = EMPTY_KEY; cnts[t] = 0; }
  __syncthreads();
  constexpr int U = 4;  // steps of 32 entries whose columns are loaded together
  const int lane = threadIdx.x & 31;
  const unsigned upto = 0xffffffffu >> (31 - lane);  // lanes 0 .. lane
  const unsigned long long k0 = (unsigned long long)(blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5)) * share;
  int *const count0 = g_cnt + (m - 1);
  if (k0 < nnz) {
    const unsigned k1 = min((unsigned)k0 + share, nnz);
    long long w = warp_row_of(rowptr, 0, m, (long long)k0);  // the lanes hold the pointers of rows w .. w + 31
    unsigned start = 0, wend = 0;                            // rowptr[w + lane], rowptr[w + 32]
    bool simple = false;                                     // none of those rows is empty
    auto hold = [&]() {
      start = w + lane <= m ? (unsigned)__ldg(rowptr + w + lane) : UINT_MAX;
      wend = w + 32 <= m ? (unsigned)__ldg(rowptr + w + 32) : UINT_MAX;
      unsigned next = __shfl_down_sync(FULL, start, 1);
      if (lane == 31) next = wend;
      simple = __all_sync(FULL, start < next || w + lane >= m);
    };
    hold();
    for (unsigned base = (unsigned)k0; base < k1; base += 32 * U) {
      int c[U];
#pragma unroll
      for (int u = 0; u < U; ++u) c[u] = base + 32 * u + lane < k1 ? __ldg(col + base + 32 * u + lane) : 0;
      const bool full = __shfl_sync(FULL, *(volatile int *)&used, 0) > HT_MOST;  // one decision for the warp
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const unsigned b = base + 32 * u, k = b + lane;
        const bool active = k < k1;
        int row = 0;
        bool open = active;
        for (;;) {
          int L;
          if (simple) {
            // rows that start before the step, then those that start at or before this lane
            const unsigned rel = start - b;
            const unsigned heads = __reduce_or_sync(FULL, rel < 32 ? 1u << rel : 0u);
            L = __popc(__ballot_sync(FULL, start < b)) - 1 + __popc(heads & upto);
          } else {
            L = row_lane_of(start, k);
          }
          if (open && k < wend) {
            row = (int)w + L;
            open = false;
          }
          const unsigned left = __ballot_sync(FULL, open);
          if (left == 0) break;
          const unsigned next = __shfl_sync(FULL, k, __ffs(left) - 1);
          w += 32;
          hold();
          if (wend <= next) {  // a run of empty rows
            w = warp_row_of(rowptr, w, m, next);
            hold();
          }
        }
        const int d = c[u] - row;
        if (full) {
          if (active) atomicAdd(count0 + d, 1);
        } else {
          const unsigned act = __ballot_sync(FULL, active);
          if (active) {
            const unsigned peers = __match_any_sync(act, d);
            if (lane == __ffs(peers) - 1) ht_add(keys, cnts, g_cnt, m, d, __popc(peers), &used);
          }
        }
      }
    }
  }
  __syncthreads();
  for (int t = threadIdx.x; t < HT; t += blockDim.x)
    if (keys[t] != EMPTY_KEY) atomicAdd(count0 + keys[t], cnts[t]);
}

// ---------------------------------------------------------------------------
// K3b: occupied / "true" diagonals, plus the occupied offsets (unordered; the
// host sorts them) up to `cap` of them.  counts = {Ndiags, Ntrue}.  A thread
// remembers which of up to 32 diagonals are occupied; a CTA then takes the
// places of all of its offsets with one atomic (an atomic or a look at the
// counter per warp and step took longer than reading the counts: 4 M diagonals
// 72 us, now 15).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) diag_reduce_kernel(const int *__restrict__ cnt, long long m, long long n,
                                                          int tau_num, int tau_den, unsigned long long *counts,
                                                          int32_t *offsets, long long cap) {
  __shared__ unsigned s_occ[8], s_tru[8];
  __shared__ unsigned long long s_first;
  const long long nd = m + n - 1, stride = (long long)gridDim.x * blockDim.x;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (long long base = (long long)blockIdx.x * blockDim.x; base < nd; base += 32 * stride) {
    unsigned bits = 0, tru = 0;
#pragma unroll 8
    for (int u = 0; u < 32; ++u) {
      const long long t = base + u * stride + threadIdx.x;
      const int c = t < nd ? __ldcs(cnt + t) : 0;
      if (c > 0) {
        const long long d = t - (m - 1), len = d >= 0 ? min(m, n - d) : min(m + d, n);
        bits |= 1u << u;
        if ((long long)tau_den * c > (long long)tau_num * len) ++tru;
      }
    }
    const unsigned occ = __popc(bits);
    unsigned before = occ;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned p = __shfl_up_sync(FULL, before, o);
      if (lane >= o) before += p;
    }
    tru = __reduce_add_sync(FULL, tru);
    if (lane == 31) { s_occ[w] = before; s_tru[w] = tru; }
    __syncthreads();
    if (threadIdx.x == 0) {
      unsigned o = 0, t = 0;
      for (int k = 0; k < 8; ++k) {
        const unsigned here = s_occ[k];
        s_occ[k] = o;
        o += here;
        t += s_tru[k];
      }
      s_first = o ? atomicAdd(&counts[0], (unsigned long long)o) : 0;
      if (t) atomicAdd(&counts[1], (unsigned long long)t);
    }
    __syncthreads();
    long long at = (long long)s_first + s_occ[w] + before - occ;
    for (; bits && at < cap; bits &= bits - 1, ++at)
      offsets[at] = (int32_t)(base + (__ffs(bits) - 1) * stride + threadIdx.x - (m - 1));
    __syncthreads();  // s_occ and s_first are free again
  }
}

int grid_for(long long work, int block, int max_blocks) {
  long long g = (work + block - 1) / block;
  if (g < 1) g = 1;
  if (g > max_blocks) g = max_blocks;
  return (int)g;
}

}  // namespace

size_t validate_starts_words(int64_t nnz) { return (size_t)(nnz / 32 + 2); }

cudaError_t launch_validate(const smat_s *h, int *d_flag, unsigned *d_starts, cudaStream_t s) {
  validate_rows_kernel<<<grid_for(std::max<int64_t>(h->m, 1), 256, 152 * 16), 256, 0, s>>>(h->rowptr, h->m, h->nnz,
                                                                                          d_starts, d_flag);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || h->nnz == 0) return e;
  validate_cols_kernel<<<grid_for((h->nnz + 7) / 8, 256, 152 * 16), 256, 0, s>>>(h->colidx, h->nnz, h->n, d_starts,
                                                                               d_flag);
  return cudaGetLastError();
}

cudaError_t launch_row_stats(const int32_t *rowptr, int64_t m, FeatureHead *head, int32_t *long_rows, cudaStream_t s) {
  if (m <= 0) return cudaSuccess;
  row_stats_kernel<<<grid_for(m, 256, 152 * 4), 256, 0, s>>>(rowptr, m, head, long_rows);
  return cudaGetLastError();
}

cudaError_t launch_diag_count(const int32_t *rowptr, const int32_t *colidx, int64_t m, int64_t nnz, int *d_diag_cnt,
                              cudaStream_t s) {
  if (m <= 0 || nnz <= 0) return cudaSuccess;
  // at most 8 CTAs per SM, at least 256 entries per warp
  const int g = grid_for((nnz + 7) / 8, 256, 152 * 8);
  const long long share = ((nnz + g * 8ll - 1) / (g * 8ll) + 31) / 32 * 32;
  diag_count_kernel<<<g, 256, 0, s>>>(rowptr, colidx, m, (unsigned)nnz, (unsigned)share, d_diag_cnt);
  return cudaGetLastError();
}

cudaError_t launch_diag_reduce(const int *d_diag_cnt, int64_t m, int64_t n, int tau_num, int tau_den,
                               unsigned long long *d_counts, int32_t *d_offsets, int64_t cap,
                               cudaStream_t s) {
  if (m + n - 1 <= 0) return cudaSuccess;
  int g = grid_for(m + n - 1, 256, 152 * 8);
  diag_reduce_kernel<<<g, 256, 0, s>>>(d_diag_cnt, m, n, tau_num, tau_den, d_counts, d_offsets, cap);
  return cudaGetLastError();
}

}  // namespace smat
