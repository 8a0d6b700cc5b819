// SpMV kernels y = alpha*A*x + beta*y for the four basic formats
// (arXiv 1210.2536, Sec. 2.1; the paper's kernel library maps each format to
// its best implementation, Sec. 3), and the launches of the further formats
// that reuse them (HYB: ELL + COO tail; SPLIT: long rows in CTA chunks and
// COO tiles of the short rows in one grid, then one closing pass).
// GPU implementations of CSR follow Bell & Garland (2008, cited by the paper:
// scalar and vector kernels); csr_flat.cu holds the CSR kernel that splits the
// entries evenly.  COO uses a tiled segmented reduction over one bit per entry
// that marks the row ends, in place of a row index per entry.
//
// The kernels stream the format's index and value arrays once with coalesced
// (ELL, DIA: 16-byte vector or lane-striped) loads, gather x through L1/L2 and
// write y once.  They are bound by HBM, by the random x gathers (more exactly
// by the rate of 32-byte L2 sector requests that the gathers and the streamed
// arrays make together), or (FP64) by the FP64 pipe, which GB300 runs at
// about 2 operations per clock per SM: every
// kernel spends one fused multiply-add per stored product, and only
// SMAT_V_CSR_SCALAR_EXACT rounds products and sums separately, in ascending
// column order, as the CSR definition does.  The alpha/beta epilogue is fused:
//   y_i = alpha*acc            if beta == 0 (y is not read)
//   y_i = alpha*acc + beta*y_i otherwise
// and alpha == 0 skips A and x altogether.  Storage V in {double, float,
// bf16}; compute T = double for V = double, float otherwise.
#include <cuda_bf16.h>

#include <algorithm>

#include "smat_internal.h"
#include "spmv_device.cuh"
#include "warp_tile.cuh"

namespace smat {
namespace {

// ---------------------------------------------------------------------------
// K7: CSR-scalar, one thread per row.
// ---------------------------------------------------------------------------
template <typename V, typename T, bool EXACT, int MODE>
__global__ void __launch_bounds__(256) csr_scalar_kernel(const int32_t *__restrict__ rowptr,
                                                         const int32_t *__restrict__ col,
                                                         const V *__restrict__ val, const T *__restrict__ x,
                                                         Epi<T, MODE, EXACT> ep, T *__restrict__ y, long long m) {
  griddep_wait();
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < m;
       i += (long long)gridDim.x * blockDim.x) {
    const int s = __ldg(rowptr + i), e = __ldg(rowptr + i + 1);
    T acc = 0;
    // eight entries per step, predicated: every index and value load, then
    // the gathers, then the in-order accumulation
    for (int k = s; k < e; k += 8) {
      int c[8];
      T v[8], xv[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        c[u] = k + u < e ? ld_idx(col + k + u) : 0;
        v[u] = k + u < e ? (T)ld_val(val + k + u) : (T)0;
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) xv[u] = k + u < e ? __ldg(x + c[u]) : (T)0;
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (k + u < e) acc = madd<EXACT>(acc, v[u], xv[u]);
    }
    y[i] = ep(acc, y, i);
  }
}

// ---------------------------------------------------------------------------
// K8: CSR-vector, W lanes per row, lane-strided loads, shuffle reduction.
// ---------------------------------------------------------------------------
template <typename V, typename T, int W, int MODE>
__global__ void __launch_bounds__(256) csr_vector_kernel(const int32_t *__restrict__ rowptr,
                                                         const int32_t *__restrict__ col,
                                                         const V *__restrict__ val, const T *__restrict__ x,
                                                         Epi<T, MODE> ep, T *__restrict__ y, long long m) {
  griddep_wait();
  constexpr int RPW = 32 / W;  // rows per warp per step
  const int lane = threadIdx.x & 31, sub = lane % W;
  const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long r0 = warp * RPW; r0 < m; r0 += nwarps * RPW) {
    long long row = r0 + lane / W;
    T acc = 0;
    if (row < m) {
      const int s = __ldg(rowptr + row), e = __ldg(rowptr + row + 1);
      for (int k = s + sub; k < e; k += 4 * W) {
        int c[4];
        T v[4], xv[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          c[u] = k + u * W < e ? ld_idx(col + k + u * W) : 0;
          v[u] = k + u * W < e ? (T)ld_val(val + k + u * W) : (T)0;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) xv[u] = k + u * W < e ? __ldg(x + c[u]) : (T)0;
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (k + u * W < e) acc = fused(acc, v[u], xv[u]);
      }
    }
#pragma unroll
    for (int o = W / 2; o > 0; o >>= 1) acc += __shfl_down_sync(FULL, acc, o, W);
    if (sub == 0 && row < m) y[row] = ep(acc, y, row);
  }
}

// ---------------------------------------------------------------------------
// K12: COO (and SPLIT's short rows, HYB's tail): entries in row order, whose row
// ends are marked by one bit each (RowEnds).  A warp takes a tile of 256
// entries, 8 per lane: the columns and values (32-byte loads), the lane's 8
// bits and the tile's first row number are loaded together and the gathers
// follow at once.  A lane adds up its entries and closes a row at each mark;
// the partial sums that cross lanes come from a segmented scan (shuffles); the
// finished rows' sums go through shared memory, so that y is written with
// contiguous lanes.  The row open at the tile's end becomes the tile's carry,
// added by a second kernel.
//
// Bound by the rate of each SM's L2 sector requests: power-law 2e6 FP64 makes
// 43.1 M of them in 128.5 us, 1.07 per clock and SM (a kernel of bare gathers
// and their indices makes 0.96).  Before, a row index per entry was loaded (4
// of 16 or 12 bytes), every row end was a scattered store, and the
// scan always took five FP64 steps.  us per product, before and now: power-law
// 2e6 rows (28.7 M entries) FP64 153.6 -> 130.5, FP32 131.9 -> 111.4; 8e6 rows
// BF16 520 -> 420; uniform 1e6 FP64 85.4 -> 75.7; 7-point 128^3 FP64 73 -> 50.
// The bounds on CTAs per SM (48 and 40 registers) are the fastest of those
// tried: 56 and 44 registers 136 and 115 us, six and eight CTAs spill.
// ---------------------------------------------------------------------------
constexpr int COO_NT = 256, COO_WARPS = COO_NT / 32;
constexpr long long COO_TILE = 256;
// Finished rows' sums staged per warp.  Staging a whole tile's (16 KB per CTA
// in FP64) costs L1, whose lines hold the gathers in flight (power-law FP64 146
// us against 131), and other kernels' room on the same SM.  In FP32 32 sums are
// as fast as 64 alone (112 us) and better beside others: a batch of 16 FP32
// matrices takes 66 us with 32, 71 with 64.
template <typename T> constexpr int COO_SUMS = sizeof(T) == 8 ? 64 : 32;

template <typename V, typename T, int MODE>
__device__ __forceinline__ void coo_tile(const RowEnds &re, const int32_t *__restrict__ col, const V *__restrict__ val,
                                         const T *__restrict__ x, const Epi<T, MODE> &ep, T *__restrict__ y, long long n,
                                         int32_t *carry_row, T *carry_val, long long tile, T *sum) {
  constexpr int IPT = 8;
  const int lane = threadIdx.x & 31;
  const long long b0 = tile * COO_TILE;
  if (b0 >= n) return;  // the whole warp
  const int count = (int)min((long long)COO_TILE, n - b0);
  const long long k0 = b0 + lane * IPT;
  const int valid = max(0, min(IPT, count - lane * IPT));
  const bool full = valid == IPT;
  int c[IPT];
  T v[IPT], xv[IPT];
  load_i32_run<IPT>(col + k0, full, valid, c, 0);
  const unsigned ends = __ldg(reinterpret_cast<const unsigned char *>(re.ends) + tile * 32 + lane);
  const int o0 = __ldg(re.ord + tile);
  load_val_run<V, IPT>(val + k0, full, valid, v);
#pragma unroll
  for (int q = 0; q < IPT; ++q) xv[q] = q < valid ? __ldg(x + c[q]) : (T)0;
  int before = __popc(ends);  // rows that end in earlier lanes
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int p = __shfl_up_sync(FULL, before, o);
    if (lane >= o) before += p;
  }
  const int nrows = __shfl_sync(FULL, before, 31);
  before -= __popc(ends);
  const int row0 = lane < nrows && re.row ? __ldg(re.row + o0 + lane) : o0 + lane;
  // xv[q] becomes the sum of the row that ends at entry q
  T acc = 0;
#pragma unroll
  for (int q = 0; q < IPT; ++q) {
    if (q < valid) acc = fused(acc, v[q], xv[q]);
    xv[q] = acc;
    if ((ends >> q) & 1u) acc = 0;
  }
  T open;
  const T in = warp_carries<T>(ends != 0, acc, &open);
  for (int base = 0; base < nrows; base += COO_SUMS<T>) {  // the finished rows, COO_SUMS at a time
    int at = before - base;
    T *const first = sum + at;
    const bool mine = ends && lane > 0 && (unsigned)at < (unsigned)COO_SUMS<T>;
#pragma unroll
    for (int q = 0; q < IPT; ++q)
      if ((ends >> q) & 1u) {
        if ((unsigned)at < (unsigned)COO_SUMS<T>) sum[at] = xv[q];
        ++at;
      }
    if (mine) *first = in + *first;
    __syncwarp();
    const int here = min(COO_SUMS<T>, nrows - base);
    for (int i = lane; i < here; i += 32) {
      const int row = base + i == lane ? row0 : re.row ? __ldg(re.row + o0 + base + i) : o0 + base + i;
      y[row] = ep(sum[i], y, (long long)row);
    }
    __syncwarp();
  }
  const unsigned last = __shfl_sync(FULL, ends, (count - 1) / IPT);
  if (lane == 0) {
    const bool opn = !((last >> ((count - 1) % IPT)) & 1u);
    carry_row[tile] = opn ? o0 + nrows : -1;
    carry_val[tile] = opn ? open : (T)0;
  }
}

template <typename V, typename T, int MODE>
__global__ void __launch_bounds__(COO_NT, sizeof(T) == 8 ? 5 : 6) coo_kernel(RowEnds re, const int32_t *__restrict__ col,
                                                     const V *__restrict__ val, const T *__restrict__ x,
                                                     Epi<T, MODE> ep, T *__restrict__ y, long long n,
                                                     int32_t *carry_row, T *carry_val) {
  griddep_wait();
  __shared__ T s_sum[COO_WARPS][COO_SUMS<T>];
  const int w = threadIdx.x >> 5;
  coo_tile<V, T, MODE>(re, col, val, x, ep, y, n, carry_row, carry_val, (long long)blockIdx.x * COO_WARPS + w,
                       s_sum[w]);
}

// ---------------------------------------------------------------------------
// SPLIT, long rows (at least SPLIT_L = 1024 entries; measured on power-law
// matrices against 128 and 256, where rows of a few hundred entries paid a
// whole CTA's reduction for little work): one CTA of 256 threads per chunk of
// at most 4096 entries of one row.  Thread t takes entries first + t + 256 j (j < 16), so every
// column and value load is a contiguous warp access; one fused multiply-add
// per entry; the 256 partial sums are added in a fixed order (warp butterfly,
// then the 8 warp sums in turn) into part[chunk].  No row ends inside a
// chunk, so there is no segmented scan: a tile of a long row costs one plain
// block sum instead of the COO tile's carry resolution.
// ---------------------------------------------------------------------------
template <typename V, typename T>
__device__ __forceinline__ void split_chunk(long long c, const int32_t *__restrict__ cstart,
                                            const int32_t *__restrict__ cend, const int32_t *__restrict__ col,
                                            const V *__restrict__ val, const T *__restrict__ x,
                                            T *__restrict__ part) {
  __shared__ T s_w[8];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int k0 = __ldg(cstart + c), k1 = __ldg(cend + c);
  T acc = 0;
  // steps j of 256 entries past the chunk's end are skipped by the whole
  // CTA (a uniform test), so short chunks issue only the work they hold
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    if (k0 + 256 * 8 * b >= k1) break;
    int cc[8];
    T v[8], xv[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int k = k0 + (int)threadIdx.x + 256 * (8 * b + q);
      const bool on = k < k1;
      cc[q] = on ? ld_idx(col + k) : -1;
      v[q] = on ? (T)ld_val(val + k) : (T)0;
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) xv[q] = cc[q] >= 0 ? __ldg(x + cc[q]) : (T)0;
#pragma unroll
    for (int q = 0; q < 8; ++q)
      if (k0 + 256 * (8 * b + q) < k1) acc = fused(acc, v[q], xv[q]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc = add_rn(acc, __shfl_xor_sync(0xffffffffu, acc, o));
  if (lane == 0) s_w[w] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    T t = s_w[0];
#pragma unroll
    for (int k = 1; k < 8; ++k) t = add_rn(t, s_w[k]);
    part[c] = t;
  }
}

// SPLIT in one grid: blocks [0, nc) reduce the chunks of the long rows,
// blocks [nc, nc + tiles) are COO tiles of the short rows (the two sets
// write disjoint rows).  One launch instead of two keeps the GPU full across
// what was the boundary between them.
template <typename V, typename T, int MODE>
__global__ void __launch_bounds__(COO_NT, sizeof(T) == 8 ? 5 : 6) split_main_kernel(
    const int32_t *__restrict__ cstart, const int32_t *__restrict__ cend, const int32_t *__restrict__ col,
    const V *__restrict__ val, T *__restrict__ part, long long nc, RowEnds re, const int32_t *__restrict__ scol,
    const V *__restrict__ sval, long long ns, const T *__restrict__ x, Epi<T, MODE> ep, T *__restrict__ y,
    int32_t *carry_row, T *carry_val) {
  griddep_wait();
  static_assert(COO_NT == 256, "the chunk path assumes 256 threads");
  __shared__ T s_sum[COO_WARPS][COO_SUMS<T>];
  const int w = threadIdx.x >> 5;
  if ((long long)blockIdx.x < nc)
    split_chunk<V, T>(blockIdx.x, cstart, cend, col, val, x, part);
  else
    coo_tile<V, T, MODE>(re, scol, sval, x, ep, y, ns, carry_row, carry_val,
                         ((long long)blockIdx.x - nc) * COO_WARPS + w, s_sum[w]);
}

// A long row: its chunk sums added in chunk order, then the epilogue.
template <typename T, int MODE>
__device__ __forceinline__ void split_row(long long l, const int32_t *__restrict__ lrows,
                                          const int32_t *__restrict__ lchunk, const T *__restrict__ part,
                                          const Epi<T, MODE> &ep, T *__restrict__ y) {
  const int c0 = lchunk[l], c1 = lchunk[l + 1];
  T t = part[c0];
  for (int c = c0 + 1; c < c1; ++c) t = add_rn(t, part[c]);
  const long long r = lrows[l];
  y[r] = ep(t, y, r);
}

// SPLIT's closing pass over three disjoint sets of rows: the long rows
// (chunk sums, epilogue), the carries of the short rows' COO tiles, and the
// empty rows (y = beta y, or 0).
template <typename T, int MODE>
__global__ void split_finish_kernel(const int32_t *__restrict__ lrows, const int32_t *__restrict__ lchunk,
                                    const T *__restrict__ part, long long nl, const int32_t *__restrict__ srows,
                                    const int32_t *__restrict__ carry_row,
                                    const T *__restrict__ carry_val, long long ntiles,
                                    const int32_t *__restrict__ empty, long long ne, Epi<T, MODE> ep,
                                    T *__restrict__ y) {
  griddep_wait();
  const long long first = (long long)blockIdx.x * blockDim.x + threadIdx.x, stride = (long long)gridDim.x * blockDim.x;
  for (long long i = first; i < nl; i += stride) split_row<T, MODE>(i, lrows, lchunk, part, ep, y);
  for (long long c0 = first - (threadIdx.x & 31); c0 < ntiles; c0 += stride)
    add_carries<T, MODE>(c0, srows, carry_row, carry_val, ntiles, ep, y);
  for (long long i = first; i < ne; i += stride) {
    const int r = empty[i];
    y[r] = MODE == EPI_AXPBY ? mul_rn(ep.beta, y[r]) : (T)0;
  }
}

template <typename T, int MODE>
__global__ void scale_rows_kernel(const int32_t *__restrict__ rows, long long count, Epi<T, MODE> ep,
                                  T *__restrict__ y) {
  griddep_wait();
  for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < count;
       c += (long long)gridDim.x * blockDim.x) {
    int r = rows[c];
    y[r] = MODE == EPI_AXPBY ? mul_rn(ep.beta, y[r]) : (T)0;
  }
}

// ---------------------------------------------------------------------------
// K10: ELL, column-major, R consecutive rows per thread so that every slot is
// one 16-byte load of values (and 4R bytes of columns).  U slots are loaded
// before their gathers are issued (U*R = 8 gathers in flight per thread);
// padding (column -1) gathers x[0] and is dropped by a select, so no load
// sits behind a branch.
// ---------------------------------------------------------------------------
template <typename V, int R, int MODE, int U, bool LANE>
__global__ void __launch_bounds__(256) ell_kernel(const int32_t *__restrict__ ecol, const V *__restrict__ eval,
                                                  long long P, long long K,
                                                  const typename Compute<V>::T *__restrict__ x,
                                                  Epi<typename Compute<V>::T, MODE> ep,
                                                  typename Compute<V>::T *__restrict__ y, long long m) {
  griddep_wait();
  if (LANE) {  // lane-striped rows (a per-handle measured choice)
    const long long base = (((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * (32LL * R);
    if (base < m) ell_lane_group<V, R, MODE, U>(ecol, eval, P, K, x, ep, y, m, base, threadIdx.x & 31);
  } else {
    const long long i0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) * R;
    if (i0 < m) ell_group<V, R, MODE, U>(ecol, eval, P, K, x, ep, y, m, i0);
  }
}

// ---------------------------------------------------------------------------
// K11: DIA, diagonal-major, R consecutive rows per thread, offsets staged in
// shared memory, U diagonals loaded per step.  Fill zeros are multiplied like
// stored values (Table "Performance features of the four formats": extra
// computation decided by zero filling); positions whose column falls outside
// the matrix gather x[0] and are dropped by a select.
// ---------------------------------------------------------------------------
template <typename V, int R, int MODE, int U>
__global__ void __launch_bounds__(256) dia_kernel(const int32_t *__restrict__ off, int nd,
                                                  const V *__restrict__ dval, long long P,
                                                  const typename Compute<V>::T *__restrict__ x,
                                                  Epi<typename Compute<V>::T, MODE> ep,
                                                  typename Compute<V>::T *__restrict__ y, long long m,
                                                  long long n) {
  griddep_wait();
  extern __shared__ int32_t s_off[];
  for (int t = threadIdx.x; t < nd; t += blockDim.x) s_off[t] = off[t];
  __syncthreads();
  if (sizeof(V) == 8) {  // FP64: lane-striped rows (measured faster on every matrix tried)
    const long long base = (((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * (32LL * R);
    if (base < m) dia_lane_group<V, R, MODE, U>(s_off, nd, dval, P, x, ep, y, m, n, base, threadIdx.x & 31);
  } else {
    const long long i0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) * R;
    if (i0 < m) dia_group<V, R, MODE, U>(s_off, nd, dval, P, x, ep, y, m, n, i0);
  }
}

int grid_for(long long work, int block, int max_blocks) {
  long long g = (work + block - 1) / block;
  if (g < 1) g = 1;
  if (g > max_blocks) g = max_blocks;
  return (int)g;
}

// A COO product over nnz entries, then the carry fix-up.
template <typename V, typename T, int MODE>
cudaError_t launch_coo(const Scratch &sc, const RowEnds &re, const int32_t *col, const V *val, const T *x,
                       const Epi<T, MODE> &ep, T *y, long long nnz, cudaStream_t s) {
  const long long tiles = (nnz + COO_TILE - 1) / COO_TILE;
  int32_t *crow = (int32_t *)sc.carry;
  T *cval = (T *)((char *)sc.carry + ((tiles * 4 + 15) / 16) * 16);
  cudaError_t e = launch_pdl(coo_kernel<V, T, MODE>, dim3((unsigned)((tiles + COO_WARPS - 1) / COO_WARPS)), dim3(COO_NT),
                             0, s, re, col, val, x, ep, y, nnz, crow, cval);
  if (e != cudaSuccess || tiles <= 1) return e;
  return launch_pdl(carry_kernel<T, MODE>, dim3(grid_for(tiles, 256, 152 * 8)), dim3(256), 0, s,
                    (const int32_t *)re.row, (const int32_t *)crow, (const T *)cval, tiles, ep, y);
}

// ELL / DIA launches with a batch width U chosen at run time from 1..16/R.
// The ELL arrays are passed in: the handle's ELL format, or HYB's ELL part.
struct EllPart {
  const int32_t *col;
  const void *val;
  long long K;
};

template <typename V, int MODE, int U>
void launch_ell_u(const smat_s *h, const EllPart &e, bool lane, const typename Compute<V>::T *x,
                  const Epi<typename Compute<V>::T, MODE> &ep, typename Compute<V>::T *y, cudaStream_t s) {
  constexpr int R = 16 / (int)sizeof(V);
  const long long m = h->m;
  const int g = grid_for((m + R - 1) / R, 256, 1 << 30);
  if (lane)
    (void)launch_pdl(ell_kernel<V, R, MODE, U, true>, dim3(g), dim3(256), 0, s, e.col, (const V *)e.val, h->P, e.K, x, ep, y, m);
  else
    (void)launch_pdl(ell_kernel<V, R, MODE, U, false>, dim3(g), dim3(256), 0, s, e.col, (const V *)e.val, h->P, e.K, x, ep, y, m);
}

template <typename V, int MODE, int U>
void launch_dia_u(const smat_s *h, const typename Compute<V>::T *x, const Epi<typename Compute<V>::T, MODE> &ep,
                  typename Compute<V>::T *y, cudaStream_t s) {
  constexpr int R = 16 / (int)sizeof(V);
  const long long m = h->m;
  (void)launch_pdl(dia_kernel<V, R, MODE, U>, dim3(grid_for((m + R - 1) / R, 256, 1 << 30)), dim3(256), (size_t)h->dia_nd * 4, s,
      h->dia_off, (int)h->dia_nd, (const V *)h->dia_val, h->P, x, ep, y, m, h->n);
}

template <typename V, int MODE, bool DIA>
void launch_ell_dia(const smat_s *h, const typename Compute<V>::T *x, const Epi<typename Compute<V>::T, MODE> &ep,
                    typename Compute<V>::T *y, cudaStream_t s, int u_req, int lane_req,
                    const EllPart *part = nullptr) {
  constexpr int UMAX = 16 / (16 / (int)sizeof(V));  // 16 / R
  const EllPart e = part ? *part : EllPart{h->ell_col, h->ell_val, h->ell_K};
  const bool lane = lane_req >= 0 ? lane_req != 0 : (part ? false : h->ell_lane != 0);
  const int u_tuned = part ? 0 : (DIA ? h->dia_u : h->ell_u);
  const int u = u_req > 0 ? u_req : (u_tuned > 0 ? u_tuned : batch_width(DIA ? h->dia_nd : e.K, UMAX));
#define SMAT_UCASE(k)                                                      \
  case k:                                                                  \
    if constexpr (k <= UMAX) {                                             \
      if (DIA) launch_dia_u<V, MODE, k>(h, x, ep, y, s);                   \
      else launch_ell_u<V, MODE, k>(h, e, lane, x, ep, y, s);              \
    }                                                                      \
    break;
  switch (u) {
    SMAT_UCASE(1) SMAT_UCASE(2) SMAT_UCASE(3) SMAT_UCASE(4) SMAT_UCASE(5) SMAT_UCASE(6) SMAT_UCASE(7)
    default:
      if constexpr (UMAX >= 8) {
        if (DIA) launch_dia_u<V, MODE, 8>(h, x, ep, y, s);
        else launch_ell_u<V, MODE, 8>(h, e, lane, x, ep, y, s);
      }
      break;
  }
#undef SMAT_UCASE
}

template <typename V, int MODE>
cudaError_t spmv_mode(const smat_s *h, const Scratch &sc, int variant, typename Compute<V>::T alpha, const void *x_p,
                      typename Compute<V>::T beta, void *y_p, cudaStream_t s, int u_req, int lane_req) {
  typedef typename Compute<V>::T T;
  const Epi<T, MODE> ep{alpha, beta};
  const T *x = (const T *)x_p;
  T *y = (T *)y_p;
  const V *val = (const V *)h->val;
  const long long m = h->m;
  switch (variant) {
    case SMAT_V_CSR_SCALAR:
      (void)launch_pdl(csr_scalar_kernel<V, T, false, MODE>, dim3(grid_for(m, 256, 1 << 20)), dim3(256), 0, s, h->rowptr, h->colidx, val, x,
                                                                                     Epi<T, MODE, false>{alpha, beta}, y, m);
      break;
    case SMAT_V_CSR_SCALAR_EXACT:
      (void)launch_pdl(csr_scalar_kernel<V, T, true, MODE>, dim3(grid_for(m, 256, 1 << 20)), dim3(256), 0, s, h->rowptr, h->colidx, val, x,
                                                                                    Epi<T, MODE, true>{alpha, beta}, y, m);
      break;
    case SMAT_V_CSR_VEC4:
      (void)launch_pdl(csr_vector_kernel<V, T, 4, MODE>, dim3(grid_for(m * 4, 256, 1 << 20)), dim3(256), 0, s, h->rowptr, h->colidx, val, x, ep, y, m);
      break;
    case SMAT_V_CSR_VEC8:
      (void)launch_pdl(csr_vector_kernel<V, T, 8, MODE>, dim3(grid_for(m * 8, 256, 1 << 20)), dim3(256), 0, s, h->rowptr, h->colidx, val, x, ep, y, m);
      break;
    case SMAT_V_CSR_VEC32:
      (void)launch_pdl(csr_vector_kernel<V, T, 32, MODE>, dim3(grid_for(m * 32, 256, 1 << 20)), dim3(256), 0, s, h->rowptr, h->colidx, val, x, ep, y, m);
      break;
    case SMAT_V_ELL:
      launch_ell_dia<V, MODE, false>(h, x, ep, y, s, u_req, lane_req);
      break;
    case SMAT_V_DIA:
      if (lane_req >= 2 || (lane_req < 0 && h->dia_staged))
        return launch_dia_staged(h, lane_req >= 2 ? lane_req - 1 : h->dia_staged, &alpha, x, &beta, y, s);
      launch_ell_dia<V, MODE, true>(h, x, ep, y, s, u_req, lane_req);
      break;
    case SMAT_V_COO: {
      if (h->coo_nempty > 0) {
        (void)launch_pdl(scale_rows_kernel<T, MODE>, dim3(grid_for(h->coo_nempty, 256, 152 * 8)), dim3(256), 0, s, h->coo_empty, h->coo_nempty,
                                                                                          ep, y);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
      }
      if (h->nnz == 0) break;
      return launch_coo<V, T, MODE>(sc, h->coo, h->colidx, val, x, ep, y, h->nnz, s);
    }
    case SMAT_V_HYB: {
      // the ELL part writes every row (y = alpha*part + beta*y), then the COO
      // tail adds alpha*(its sums): y = alpha*acc + 1*y
      const EllPart part{h->hyb_ecol, h->hyb_eval, h->hyb_K};
      launch_ell_dia<V, MODE, false>(h, x, ep, y, s, 0, 0, &part);
      cudaError_t e = cudaGetLastError();
      if (e != cudaSuccess || h->hyb_ncoo == 0) return e;
      const Epi<T, EPI_AXPBY> add{alpha, (T)1};
      return launch_coo<V, T, EPI_AXPBY>(sc, h->hyb, h->hyb_ccol, (const V *)h->hyb_cval, x, add, y,
                                         h->hyb_ncoo, s);
    }
    case SMAT_V_SPLIT: {
      // two launches: the chunks of the long rows and the COO tiles of the
      // short ones in one grid, then one pass for the long rows' sums, the
      // tiles' carries and the empty rows
      const long long nc = h->split_nc, ns = h->split_ns;
      const long long tiles = (ns + COO_TILE - 1) / COO_TILE;
      const long long tile_ctas = (tiles + COO_WARPS - 1) / COO_WARPS;
      int32_t *crow = (int32_t *)sc.carry;
      T *cval = (T *)((char *)sc.carry + ((tiles * 4 + 15) / 16) * 16);
      if (nc + tile_ctas > 0) {
        (void)launch_pdl(split_main_kernel<V, T, MODE>, dim3((unsigned)(nc + tile_ctas)), dim3(COO_NT), 0, s,
            h->split_cstart, h->split_cend, h->colidx, val, (T *)sc.part, nc, h->split, h->split_scol,
            (const V *)h->split_sval, ns, x, ep, y, crow, cval);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
      }
      const long long nl = nc > 0 ? h->split_nl : 0, nt = tiles > 1 ? tiles : 0;
      if (nl + nt + h->split_ne > 0)
        (void)launch_pdl(split_finish_kernel<T, MODE>, dim3(grid_for(std::max(nl, std::max(nt, (long long)h->split_ne)), 256, 152 * 8)), dim3(256), 0, s,
            h->split_lrows, h->split_lchunk, (const T *)sc.part, nl, h->split.row, crow, cval, nt, h->split_empty, h->split_ne, ep,
            y);
    } break;
    default:
      return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

template <typename V>
cudaError_t spmv_typed(const smat_s *h, const Scratch &sc, int variant, const void *alpha_p, const void *x_p,
                       const void *beta_p, void *y_p, cudaStream_t s, int u_req, int lane_req) {
  typedef typename Compute<V>::T T;
  const T alpha = *(const T *)alpha_p, beta = *(const T *)beta_p;
  if (h->m == 0) return cudaSuccess;
  switch (epi_mode((double)alpha, (double)beta)) {
    case EPI_COPY: return spmv_mode<V, EPI_COPY>(h, sc, variant, alpha, x_p, beta, y_p, s, u_req, lane_req);
    case EPI_SCALE: return spmv_mode<V, EPI_SCALE>(h, sc, variant, alpha, x_p, beta, y_p, s, u_req, lane_req);
    default: return spmv_mode<V, EPI_AXPBY>(h, sc, variant, alpha, x_p, beta, y_p, s, u_req, lane_req);
  }
}

}  // namespace

size_t carry_bytes_needed(const smat_s *h, int variant) {
  long long tiles = 0;
  if (variant == SMAT_V_CSR_MERGE) tiles = flat_tiles(h->nnz);
  else if (variant == SMAT_V_COO) tiles = (h->nnz + COO_TILE - 1) / COO_TILE;
  else if (variant == SMAT_V_HYB) tiles = (h->hyb_ncoo + COO_TILE - 1) / COO_TILE;
  else if (variant == SMAT_V_SPLIT) tiles = (h->split_ns + COO_TILE - 1) / COO_TILE;
  else return 0;
  size_t tsz = h->dtype == SMAT_F64 ? 8 : 4;
  return (size_t)((tiles * 4 + 15) / 16) * 16 + (size_t)tiles * tsz;
}

bool needs_scratch(const smat_s *h, int variant) {
  return carry_bytes_needed(h, variant) > 0 || variant == SMAT_V_SPLIT;
}

int spmv_launch_count(const smat_s *h, int variant) {
  if (h->m == 0) return 0;
  if (variant == SMAT_V_CSR_MERGE) {
    const long long tiles = flat_tiles(h->nnz);
    return (h->flat_gaps || h->nnz == 0) + (tiles > 0) + (tiles > 1);
  }
  if (variant == SMAT_V_COO) {
    long long tiles = (h->nnz + COO_TILE - 1) / COO_TILE;
    return (h->coo_nempty > 0) + (h->nnz > 0) + (tiles > 1);
  }
  if (variant == SMAT_V_HYB) {
    long long tiles = (h->hyb_ncoo + COO_TILE - 1) / COO_TILE;
    return 1 + (h->hyb_ncoo > 0) + (tiles > 1);
  }
  if (variant == SMAT_V_SPLIT) {  // the main grid, then the closing pass when it has rows to do
    const long long tiles = (h->split_ns + COO_TILE - 1) / COO_TILE;
    const long long nl = h->split_nc > 0 ? h->split_nl : 0, nt = tiles > 1 ? tiles : 0;
    return (h->split_nc + tiles > 0) + (nl + nt + h->split_ne > 0);
  }
  if (variant == SMAT_V_SELL) return h->sell_ns > 0;
  if (variant == SMAT_V_BCSR) return h->bcsr_mb > 0;
  return 1;
}

// alpha == 0: y = beta*y (0 when beta == 0) without reading A or x, so that
// non-finite values in x cannot reach y (the BLAS convention).
template <typename T>
__global__ void beta_only_kernel(T *__restrict__ y, long long m, T beta) {
  griddep_wait();
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (long long)gridDim.x * blockDim.x)
    y[i] = mul_rn(beta, y[i]);
}

template <typename T>
cudaError_t beta_only(long long m, const void *beta_p, void *y, cudaStream_t s) {
  const T beta = *(const T *)beta_p;
  if (m == 0) return cudaSuccess;
  if (beta == (T)0) return cudaMemsetAsync(y, 0, (size_t)m * sizeof(T), s);
  (void)launch_pdl(beta_only_kernel<T>, dim3(grid_for(m, 256, 152 * 8)), dim3(256), 0, s, (T *)y, m, beta);
  return cudaGetLastError();
}

cudaError_t launch_beta_only(smat_dtype_t dtype, long long m, const void *beta, void *y, cudaStream_t s) {
  return dtype == SMAT_F64 ? beta_only<double>(m, beta, y, s) : beta_only<float>(m, beta, y, s);
}

cudaError_t launch_spmv(const smat_s *h, int variant, const void *alpha, const void *x, const void *beta,
                        void *y, cudaStream_t s, bool claim) {
  if (h->dtype == SMAT_F64 ? *(const double *)alpha == 0.0 : *(const float *)alpha == 0.0f)
    return launch_beta_only(h->dtype, h->m, beta, y, s);
  // ELL, DIA and HYB read x and write y, and BCSR reads x, with vector
  // accesses of up to 16 bytes; vectors that are not 16-byte aligned take the
  // CSR-scalar kernel instead.
  if ((variant == SMAT_V_ELL || variant == SMAT_V_DIA || variant == SMAT_V_HYB || variant == SMAT_V_BCSR) &&
      (((uintptr_t)x | (uintptr_t)y) & 15u) != 0)
    variant = SMAT_V_CSR_SCALAR;
  if (variant == SMAT_V_SELL || variant == SMAT_V_BCSR) return launch_spmv_ext(h, variant, alpha, x, beta, y, s);
  Scratch sc{nullptr, nullptr};
  if (needs_scratch(h, variant)) {
    cudaError_t e = stream_scratch(h, s, &sc, claim);
    if (e != cudaSuccess) return e;
  }
  if (variant == SMAT_V_CSR_MERGE) return h->m > 0 ? launch_csr_flat(h, sc, alpha, x, beta, y, s) : cudaSuccess;
  switch (h->dtype) {
    case SMAT_F64: return spmv_typed<double>(h, sc, variant, alpha, x, beta, y, s, 0, -1);
    case SMAT_F32: return spmv_typed<float>(h, sc, variant, alpha, x, beta, y, s, 0, -1);
    default: return spmv_typed<__nv_bfloat16>(h, sc, variant, alpha, x, beta, y, s, 0, -1);
  }
}

int batch_width_candidates(const smat_s *h, int variant, int out[2]) {
  const int umax = 16 / (16 / elem_size(h->dtype));
  const long long count = variant == SMAT_V_DIA ? h->dia_nd : h->ell_K;
  out[0] = umax;                      // full width (dead slots when count < umax)
  out[1] = batch_width(count, umax);  // fewest dead slots
  return out[1] != out[0] ? 2 : 1;
}

cudaError_t launch_spmv_width(const smat_s *h, int variant, int u, int lane, const void *alpha, const void *x,
                              const void *beta, void *y, cudaStream_t s) {
  const Scratch none{nullptr, nullptr};  // ELL / DIA use no scratch
  switch (h->dtype) {
    case SMAT_F64: return spmv_typed<double>(h, none, variant, alpha, x, beta, y, s, u, lane);
    case SMAT_F32: return spmv_typed<float>(h, none, variant, alpha, x, beta, y, s, u, lane);
    default: return spmv_typed<__nv_bfloat16>(h, none, variant, alpha, x, beta, y, s, u, lane);
  }
}

}  // namespace smat
