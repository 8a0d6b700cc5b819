// SMAT_V_CSR_MERGE and the allocation-free product: CSR split evenly by stored
// entries, whatever the rows' lengths (after merge-path SpMV, Merrill & Garland
// 2016, which splits rows and entries together).
//
// A warp takes 256 consecutive stored entries (a chunk), eight per lane, read
// with 16- and 32-byte loads that need no row information, and gathers x for
// them at once.  Meanwhile it reads the row pointers of the rows that end in
// the chunk (a contiguous range: tile_row holds the row of every tile's first
// entry) and marks each row's last entry in a 256-bit map in shared memory.  A
// lane then adds up its entries, closing a row at each mark; a segmented scan
// over the lanes (shuffles) brings the partial sums of the rows that started
// in earlier lanes; the finished rows go through shared memory, so that y is
// written with contiguous lanes.  The row left open at a tile's end is its
// carry, added by a second kernel.
//
// On random columns it is bound by how many gathers its resident warps keep in
// flight (FP64: 64 registers, 32 warps per SM) against a warp's chain of
// loads, sums and scan; on regular ones by the same chain.  It took the place
// of merge-path tiles of 2048 items per CTA, whose 16-byte (value, x) pairs
// went through shared memory, eight-way bank conflicts and three block
// barriers.  us per product, before and now (x and y included):
//   power-law 2e6 rows, 28.7 M entries  FP64 378 -> 195, FP32 163 -> 132
//   uniform 1e6 rows, 16 M entries      FP64 198 -> 107
//   7-point 128^3                       FP64  83 ->  77
//   8x8 blocks, 1e6 rows                FP32  37 ->  17
// and through the allocation-free call, which also finds the tiles' rows:
//   power-law 1.5e6 FP32 137 -> 105, 2e6 FP64 461 -> 205, uniform 1e5 FP32 25 -> 14.
// Reading the first row pointers before the gathers is 7 % of the FP64
// power-law product; writing the rows 32 at a time from the lanes of their row
// pointers, with 0.3 instead of 3 KB of shared memory per warp, was slower
// (48-74 registers: FP32 143, 7-point 83).
#include <algorithm>
#include <climits>
#include <mutex>

#include "smat_internal.h"
#include "spmv_device.cuh"
#include "warp_tile.cuh"

namespace smat {
namespace {

constexpr int FLAT_NT = 256, FLAT_WARPS = FLAT_NT / 32;
constexpr int FLAT_SHIFT = 8, FLAT_CHUNK = 1 << FLAT_SHIFT;  // entries per warp and step
// Where a tile finishes more rows than this, flat_empty_kernel writes all of the
// matrix's empty rows and the tiles none (each is written once: beta must not
// be applied twice): one warp writing millions of rows would hold the product.
constexpr int FLAT_MAX_ROWS = 4096;

int grid_for(long long work, int block, int max_blocks) {
  long long g = (work + block - 1) / block;
  if (g < 1) g = 1;
  if (g > max_blocks) g = max_blocks;
  return (int)g;
}

// tile_row[t] = the row of entry t << shift (0 for t = 0, so that leading empty
// rows belong to the first tile), tile_row[ntiles] = m: a thread per row
// writes the tiles that start in it, a warp together where they are many.
// EMPTY: also y = beta*y (0) on the empty rows.
template <typename T, int MODE, bool EMPTY>
__global__ void __launch_bounds__(256) flat_rows_kernel(const int32_t *__restrict__ rowptr, long long m, int shift,
                                                        long long ntiles, int32_t *__restrict__ tile_row,
                                                        Epi<T, MODE> ep, T *__restrict__ y) {
  griddep_wait();
  const int lane = threadIdx.x & 31;
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long r0 = (long long)blockIdx.x * blockDim.x + threadIdx.x - lane; r0 < m; r0 += stride) {
    const long long r = r0 + lane;
    long long t0 = 0, t1 = 0;  // the tiles that start in row r
    if (r < m) {
      const long long s = __ldg(rowptr + r), e = __ldg(rowptr + r + 1);
      if (s < e) {
        t0 = std::max(((s - 1) >> shift) + 1, 1ll);
        t1 = ((e - 1) >> shift) + 1;
      } else if (EMPTY) {
        y[r] = ep((T)0, y, r);
      }
      if (r == 0) {
        tile_row[0] = 0;
        tile_row[ntiles] = (int32_t)m;
      }
    }
    const bool many = t1 - t0 > 8;
    if (!many)
      for (long long t = t0; t < t1; ++t) tile_row[t] = (int32_t)r;
    for (unsigned left = __ballot_sync(FULL, many); left; left &= left - 1) {
      const int src = __ffs(left) - 1;
      const long long a = __shfl_sync(FULL, t0, src), b = __shfl_sync(FULL, t1, src);
      for (long long t = a + lane; t < b; t += 32) tile_row[t] = (int32_t)(r0 + src);
    }
  }
}

// y = beta*y (0) on the empty rows.
template <typename T, int MODE>
__global__ void __launch_bounds__(256) flat_empty_kernel(const int32_t *__restrict__ rowptr, long long m,
                                                         Epi<T, MODE> ep, T *__restrict__ y) {
  griddep_wait();
  for (long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x; r < m; r += (long long)gridDim.x * blockDim.x)
    if (__ldg(rowptr + r) == __ldg(rowptr + r + 1)) y[r] = ep((T)0, y, r);
}

// *flag = 1 when a tile finishes more than FLAT_MAX_ROWS rows.
__global__ void flat_gaps_kernel(const int32_t *__restrict__ tile_row, long long ntiles, int *flag) {
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < ntiles; t += (long long)gridDim.x * blockDim.x)
    if (tile_row[t + 1] - tile_row[t] > FLAT_MAX_ROWS) *flag = 1;
}

// First row in [r, rend) that ends past entry k (rend when none does).
__device__ __forceinline__ int row_past(const int32_t *__restrict__ rowptr, int r, int rend, int k) {
  int lo = r, hi = rend;
  while (lo < hi) {
    const int mid = lo + (hi - lo) / 2;
    if (__ldg(rowptr + mid + 1) <= k) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// ALIGNED: col and val take 32-byte (bfloat16: 16-byte) loads; otherwise each
// entry is loaded by itself.  write_empty: this kernel writes the empty rows too.
template <typename V, typename T, int MODE, bool ALIGNED>
__global__ void __launch_bounds__(FLAT_NT) csr_flat_kernel(const int32_t *__restrict__ rowptr,
                                                           const int32_t *__restrict__ col, const V *__restrict__ val,
                                                           const T *__restrict__ x, Epi<T, MODE> ep,
                                                           T *__restrict__ y, long long nnz,
                                                           const int32_t *__restrict__ tile_row, long long ntiles,
                                                           int chunks, bool write_empty, int32_t *__restrict__ carry_row,
                                                           T *__restrict__ carry_val) {
  griddep_wait();
  constexpr int IPT = 8;
  __shared__ T s_sum[FLAT_WARPS][FLAT_CHUNK];
  __shared__ int s_row[FLAT_WARPS][FLAT_CHUNK];
  __shared__ unsigned s_end[FLAT_WARPS][FLAT_CHUNK / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long long tile = (long long)blockIdx.x * FLAT_WARPS + w;
  if (tile >= ntiles) return;  // the whole warp
  T *sum = s_sum[w];
  int *rows = s_row[w];
  unsigned *end = s_end[w];
  int r = __ldg(tile_row + tile);
  const int rend = __ldg(tile_row + tile + 1);
  T run = 0;  // what the row open at the end of the last chunk holds
  int last_end = 0;
  for (int ch = 0; ch < chunks; ++ch) {
    const long long b0 = (tile * chunks + ch) * FLAT_CHUNK;
    if (b0 >= nnz) break;
    const int count = (int)std::min<long long>(FLAT_CHUNK, nnz - b0), k1 = (int)(b0 + count);
    const long long k0 = b0 + lane * IPT;
    const int valid = std::max(0, std::min(IPT, count - lane * IPT));
    const bool full = ALIGNED && valid == IPT;
    int c[IPT];
    T v[IPT], xv[IPT];
    load_i32_run<IPT>(col + k0, full, valid, c, 0);
    load_val_run<V, IPT>(val + k0, full, valid, v);
    // row pointers of the first 32 rows that may end here, ahead of the gathers
    int e = r + lane < rend ? __ldg(rowptr + r + lane + 1) : INT_MAX;
    int first = r < rend ? __ldg(rowptr + r) : INT_MAX;
    if (lane < FLAT_CHUNK / 32) end[lane] = 0;
    __syncwarp();
#pragma unroll
    for (int q = 0; q < IPT; ++q) xv[q] = q < valid ? __ldg(x + c[q]) : (T)0;
    // the rows that end in the chunk, 32 at a time
    int nrows = 0;
    for (;;) {
      const int mine = r + lane;
      int s = __shfl_up_sync(FULL, e, 1);
      if (lane == 0) s = first;
      const bool ends = mine < rend && e <= k1, some = ends && s < e;
      const unsigned b = __ballot_sync(FULL, some);
      if (some) {
        const int at = (int)(e - 1 - b0);
        atomicOr(&end[at >> 5], 1u << (at & 31));
        rows[nrows + __popc(b & ((1u << lane) - 1u))] = mine;
      } else if (ends && write_empty) {
        y[mine] = ep((T)0, y, (long long)mine);
      }
      nrows += __popc(b);
      const int done = __popc(__ballot_sync(FULL, ends));
      r += done;
      if (done < 32) break;
      first = __shfl_sync(FULL, e, 31);
      // nothing but empty rows: skip the rest of them when they are not ours to write
      if (b == 0 && !write_empty) r = row_past(rowptr, r, rend, first);
      e = r + lane < rend ? __ldg(rowptr + r + lane + 1) : INT_MAX;
    }
    __syncwarp();
    const unsigned ends = (end[lane >> 2] >> ((lane & 3) * 8)) & 0xffu;  // of this lane's entries
    int before = __popc(ends);  // rows that end in earlier lanes
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int p = __shfl_up_sync(FULL, before, o);
      if (lane >= o) before += p;
    }
    before -= __popc(ends);
    T acc = lane == 0 ? run : (T)0;
    int at = before;
#pragma unroll
    for (int q = 0; q < IPT; ++q) {
      if (q < valid) acc = fused(acc, v[q], xv[q]);
      if ((ends >> q) & 1u) {
        sum[at++] = acc;
        acc = 0;
      }
    }
    const T in = warp_carries<T>(ends != 0, acc, &run);
    if (ends && lane > 0) sum[before] = in + sum[before];
    last_end = (int)((end[(count - 1) >> 5] >> ((count - 1) & 31)) & 1u);
    __syncwarp();
    for (int i = lane; i < nrows; i += 32) {
      const long long row = rows[i];
      y[row] = ep(sum[i], y, row);
    }
    __syncwarp();  // sum, rows and end are free again
  }
  if (lane == 0) {
    carry_row[tile] = last_end ? -1 : r;
    carry_val[tile] = last_end ? (T)0 : run;
  }
}

struct FlatArgs {
  const int32_t *rowptr, *col;
  const void *val;
  long long m, nnz, tiles;
  int log2_chunks;  // chunks per tile
  int32_t *tile_row, *carry_row;
  void *carry_val;
  bool rows_pass;   // tile_row is not known yet: the pass that finds it also writes the empty rows
  bool empty_pass;  // the empty rows are written by a pass of their own
};

template <typename V, int MODE>
cudaError_t flat_mode(const FlatArgs &a, typename Compute<V>::T alpha, const void *x_p, typename Compute<V>::T beta,
                      void *y_p, cudaStream_t s) {
  typedef typename Compute<V>::T T;
  const Epi<T, MODE> ep{alpha, beta};
  const T *x = (const T *)x_p;
  T *y = (T *)y_p;
  cudaError_t e = cudaSuccess;
  const dim3 by_row(grid_for(a.m, 256, 152 * 16)), nt(256);
  if (a.rows_pass)
    e = launch_pdl(flat_rows_kernel<T, MODE, true>, by_row, nt, 0, s, a.rowptr, a.m, FLAT_SHIFT + a.log2_chunks,
                   a.tiles, a.tile_row, ep, y);
  else if (a.empty_pass)
    e = launch_pdl(flat_empty_kernel<T, MODE>, by_row, nt, 0, s, a.rowptr, a.m, ep, y);
  if (e != cudaSuccess || a.tiles == 0) return e;
  const bool aligned = ((uintptr_t)a.col % 32) == 0 && ((uintptr_t)a.val % (sizeof(V) == 2 ? 16 : 32)) == 0;
  e = launch_pdl(aligned ? csr_flat_kernel<V, T, MODE, true> : csr_flat_kernel<V, T, MODE, false>,
                 dim3((unsigned)((a.tiles + FLAT_WARPS - 1) / FLAT_WARPS)), dim3(FLAT_NT), 0, s, a.rowptr, a.col,
                 (const V *)a.val, x, ep, y, a.nnz, (const int32_t *)a.tile_row, a.tiles, 1 << a.log2_chunks,
                 !a.rows_pass && !a.empty_pass, a.carry_row, (T *)a.carry_val);
  if (e != cudaSuccess || a.tiles == 1) return e;
  return launch_pdl(carry_kernel<T, MODE>, dim3(grid_for(a.tiles, 256, 152 * 8)), nt, 0, s, (const int32_t *)nullptr,
                    (const int32_t *)a.carry_row, (const T *)a.carry_val, a.tiles, ep, y);
}

template <typename V>
cudaError_t flat_typed(const FlatArgs &a, const void *alpha_p, const void *x, const void *beta_p, void *y,
                       cudaStream_t s) {
  typedef typename Compute<V>::T T;
  const T alpha = *(const T *)alpha_p, beta = *(const T *)beta_p;
  switch (epi_mode((double)alpha, (double)beta)) {
    case EPI_COPY: return flat_mode<V, EPI_COPY>(a, alpha, x, beta, y, s);
    case EPI_SCALE: return flat_mode<V, EPI_SCALE>(a, alpha, x, beta, y, s);
    default: return flat_mode<V, EPI_AXPBY>(a, alpha, x, beta, y, s);
  }
}

cudaError_t flat_product(const FlatArgs &a, smat_dtype_t dtype, const void *alpha, const void *x, const void *beta,
                         void *y, cudaStream_t s) {
  switch (dtype) {
    case SMAT_F64: return flat_typed<double>(a, alpha, x, beta, y, s);
    case SMAT_F32: return flat_typed<float>(a, alpha, x, beta, y, s);
    default: return flat_typed<__nv_bfloat16>(a, alpha, x, beta, y, s);
  }
}

}  // namespace

long long flat_tiles(long long nnz) { return (nnz + FLAT_CHUNK - 1) / FLAT_CHUNK; }

cudaError_t launch_flat_rows(const smat_s *h, int32_t *tile_row, int *gaps, cudaStream_t s) {
  const long long tiles = flat_tiles(h->nnz);
  flat_rows_kernel<float, EPI_COPY, false><<<grid_for(h->m, 256, 152 * 16), 256, 0, s>>>(
      h->rowptr, h->m, FLAT_SHIFT, tiles, tile_row, Epi<float, EPI_COPY>{1.0f, 0.0f}, nullptr);
  flat_gaps_kernel<<<grid_for(tiles, 256, 152 * 8), 256, 0, s>>>(tile_row, tiles, gaps);
  return cudaGetLastError();
}

cudaError_t launch_csr_flat(const smat_s *h, const Scratch &sc, const void *alpha, const void *x, const void *beta,
                            void *y, cudaStream_t s) {
  FlatArgs a{};
  a.rowptr = h->rowptr; a.col = h->colidx; a.val = h->val;
  a.m = h->m; a.nnz = h->nnz; a.tiles = flat_tiles(h->nnz);
  a.tile_row = h->flat_row;
  a.carry_row = (int32_t *)sc.carry;
  a.carry_val = (char *)sc.carry + (a.tiles * 4 + 15) / 16 * 16;
  a.empty_pass = h->flat_gaps || h->nnz == 0;
  return flat_product(a, h->dtype, alpha, x, beta, y, s);
}

// ---------------------------------------------------------------------------
// The product that allocates nothing.
//
// Some callers cannot call cudaMalloc: a solver that runs under a memory
// manager owning every device byte, code that must not synchronise the device
// (cudaMalloc/cudaFree may), or a host whose allocation calls are forbidden
// once its time-critical loop has started.  For them this entry point keeps
// the only scratch the kernels need -- one carry (row, partial sum) and one
// first row per tile -- in a fixed array in the library's own device memory.
// Every GPU that loads the library holds that array (1 MiB) until the process
// exits.  The array's address is looked up once per device, on the
// first call made with that device current; make that first call before any
// stream capture.  All calls share the array, so calls whose kernels overlap on
// the GPU race: order them on one stream, or synchronise between them.  Nothing
// in the array has to start at zero: each call writes every carry and first row
// that it later reads.
// ---------------------------------------------------------------------------
namespace {

// The array holds three regions, for at most 65,536 tiles:
constexpr long long NOALLOC_MAX_TILES = 65536;
// [0, 256 KiB): each tile's carry row, int32
constexpr size_t NOALLOC_ROW_BYTES = NOALLOC_MAX_TILES * 4;
// [256 KiB, 768 KiB): each tile's carry value, 8 bytes (FP64) or 4 (FP32)
constexpr size_t NOALLOC_VAL_BYTES = NOALLOC_MAX_TILES * 8;
// [768 KiB, 1 MiB + 4 B): the row of each tile's first entry, int32, and m
constexpr size_t NOALLOC_FIRST_OFFSET = NOALLOC_ROW_BYTES + NOALLOC_VAL_BYTES;
constexpr size_t NOALLOC_BYTES = NOALLOC_FIRST_OFFSET + (NOALLOC_MAX_TILES + 1) * 4;
// Rows and entries together of the largest matrix taken.
constexpr long long NOALLOC_MAX_ITEMS = NOALLOC_MAX_TILES * 2048;
static __device__ __align__(256) unsigned char g_noalloc_scratch[NOALLOC_BYTES];

constexpr int NOALLOC_MAX_DEVICES = 64;
std::mutex g_noalloc_mu;
void *g_noalloc_ptr[NOALLOC_MAX_DEVICES] = {};

// Device address of the scratch array for the current device, looked up on
// the first call with that device current and kept for the process's life:
// after cudaDeviceReset the kept address is stale, so this entry point must
// not be called again in a process that has reset a device it used.
cudaError_t noalloc_scratch(void **out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= NOALLOC_MAX_DEVICES) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_noalloc_mu);
  if (!g_noalloc_ptr[dev]) {
    void *p = nullptr;
    e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) return e;
    g_noalloc_ptr[dev] = p;
  }
  *out = g_noalloc_ptr[dev];
  return cudaSuccess;
}

}  // namespace
}  // namespace smat

extern "C" smat_status_t smat_spmv_csr_merge_noalloc(int64_t m, int64_t n, int64_t nnz, const int32_t *rowptr,
                                                     const int32_t *colidx, const void *vals, smat_dtype_t dtype,
                                                     const void *alpha, const void *x, const void *beta, void *y,
                                                     void *stream) {
  using namespace smat;
  if (m < 0 || n < 0 || nnz < 0 || !alpha || !beta) return SMAT_ERR_INVALID_ARG;
  if (dtype != SMAT_F64 && dtype != SMAT_F32 && dtype != SMAT_BF16) return SMAT_ERR_INVALID_ARG;
  if (m == 0) return SMAT_OK;
  if (!rowptr || !y || (nnz > 0 && (!colidx || !vals || !x))) return SMAT_ERR_INVALID_ARG;
  if (m > INT32_MAX - 1 || n > INT32_MAX || nnz > INT32_MAX) return SMAT_ERR_UNSUPPORTED;
  if (m + nnz > NOALLOC_MAX_ITEMS) return SMAT_ERR_UNSUPPORTED;
  void *scratch = nullptr;
  if (noalloc_scratch(&scratch) != cudaSuccess) return SMAT_ERR_CUDA;
  cudaStream_t s = (cudaStream_t)stream;
  // alpha == 0: y = beta*y (0 when beta == 0), reading neither A nor x, as in
  // smat_spmv, so that non-finite values in x cannot reach y
  if (dtype == SMAT_F64 ? *(const double *)alpha == 0.0 : *(const float *)alpha == 0.0f)
    return launch_beta_only(dtype, m, beta, y, s) == cudaSuccess ? SMAT_OK : SMAT_ERR_CUDA;
  FlatArgs a{};
  a.rowptr = rowptr; a.col = colidx; a.val = vals;
  a.m = m; a.nnz = nnz;
  // one chunk per tile, more when the carries of that many tiles would not fit
  while ((a.tiles = (flat_tiles(nnz) + (1 << a.log2_chunks) - 1) >> a.log2_chunks) > NOALLOC_MAX_TILES) ++a.log2_chunks;
  a.carry_row = (int32_t *)scratch;
  a.carry_val = (char *)scratch + NOALLOC_ROW_BYTES;
  a.tile_row = (int32_t *)((char *)scratch + NOALLOC_FIRST_OFFSET);
  a.rows_pass = true;
  return flat_product(a, dtype, alpha, x, beta, y, s) == cudaSuccess ? SMAT_OK : SMAT_ERR_CUDA;
}
