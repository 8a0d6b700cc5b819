// CSR -> COO / ELL / DIA conversions (arXiv 1210.2536, Sec. 2.1: the four
// basic storage formats; Table "Performance features of the four formats")
// and the value casts used for reduced-precision storage.
//
// Layouts (the paper's figure of the data structures is not available; these
// are the standard definitions):
//   ELL  col/val[s * P + i] = s-th stored entry of row i, s < K = max_RD;
//        padding (and rows M..P-1) hold column -1 and value +0.
//   DIA  val[t * P + i] = a(i, i + off[t]) or +0 where not stored; offsets
//        ascending.
//   COO  row[k] for every stored entry, in CSR order (col and val are CSR's).
//        The products read the row ends as bits (RowEnds); row[k] itself is
//        written only for an export.
// Every output element is written exactly once, with coalesced stores, and
// values are moved as raw bits.
#include "smat_internal.h"

namespace smat {
namespace {

constexpr unsigned FULL = 0xffffffffu;

template <int B> struct Bits;
template <> struct Bits<8> { typedef unsigned long long T; };
template <> struct Bits<4> { typedef unsigned int T; };
template <> struct Bits<2> { typedef unsigned short T; };

// Row ends of a list: a thread per row marks its last entry, and writes its
// ordinal for the tiles of 256 entries that start in it (a warp together where
// they are many) and its row for the ordinal.
template <bool CSR>
__global__ void __launch_bounds__(256) row_ends_kernel(const int32_t *__restrict__ rowptr,
                                                       const long long *__restrict__ scan, long long m, RowEnds re) {
  const int lane = threadIdx.x & 31;
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long r0 = (long long)blockIdx.x * blockDim.x + threadIdx.x - lane; r0 < m; r0 += stride) {
    const long long r = r0 + lane;
    long long t0 = 0, t1 = 0;  // the tiles that start in row r
    int ord = 0;
    if (r < m) {
      const long long s = CSR ? rowptr[r] : (long long)(unsigned)scan[r];
      const long long e = CSR ? rowptr[r + 1] : (long long)(unsigned)scan[r + 1];
      if (s < e) {
        ord = scan ? (int)(scan[r] >> 32) : (int)r;
        atomicOr(&re.ends[(e - 1) >> 5], 1u << ((e - 1) & 31));
        if (re.row) re.row[ord] = (int32_t)r;
        t0 = (s + 255) >> 8;
        t1 = ((e - 1) >> 8) + 1;
      }
    }
    const bool many = t1 - t0 > 8;
    if (!many)
      for (long long t = t0; t < t1; ++t) re.ord[t] = ord;
    for (unsigned left = __ballot_sync(FULL, many); left; left &= left - 1) {
      const int src = __ffs(left) - 1;
      const long long a = __shfl_sync(FULL, t0, src), b = __shfl_sync(FULL, t1, src);
      const int o = __shfl_sync(FULL, ord, src);
      for (long long t = a + lane; t < b; t += 32) re.ord[t] = o;
    }
  }
}

// The row of every entry, from the row ends: a warp per tile.
__global__ void __launch_bounds__(256) expand_rows_kernel(RowEnds re, long long n, int32_t *__restrict__ row) {
  const int lane = threadIdx.x & 31;
  const long long tile = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (tile * 256 >= n) return;
  int ord = re.ord[tile];
  for (int w = 0; w < 8; ++w) {
    const long long k = tile * 256 + w * 32 + lane;
    const unsigned ends = re.ends[tile * 8 + w];
    const int o = ord + __popc(ends & ((1u << lane) - 1u));
    if (k < n) row[k] = re.row ? re.row[o] : o;
    ord += __popc(ends);
  }
}

__global__ void empty_rows_kernel(const int32_t *__restrict__ rowptr, long long m, int32_t *list, int *count) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < m;
       i += (long long)gridDim.x * blockDim.x)
    if (rowptr[i + 1] == rowptr[i]) list[atomicAdd(count, 1)] = (int32_t)i;
}

__global__ void nonempty_rows_kernel(const int32_t *__restrict__ rowptr, long long m, long long *__restrict__ flag) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < m;
       i += (long long)gridDim.x * blockDim.x)
    flag[i] = (long long)(rowptr[i + 1] > rowptr[i]) << 32;
}

// ELL: thread per row (and per pad row up to P).
template <typename B>
__global__ void to_ell_kernel(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ col,
                              const B *__restrict__ val, long long m, long long P, long long K,
                              int32_t *__restrict__ ecol, B *__restrict__ eval) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < P;
       i += (long long)gridDim.x * blockDim.x) {
    long long s = 0, rd = 0;
    if (i < m) { s = rowptr[i]; rd = rowptr[i + 1] - s; }
#pragma unroll 8
    for (long long q = 0; q < K; ++q) {
      const long long pos = q * P + i;
      const int c = q < rd ? col[s + q] : -1;
      const B v = q < rd ? val[s + q] : (B)0;
      ecol[pos] = c;
      eval[pos] = v;
    }
  }
}

// DIA: thread per row; the row's sorted columns are merged against the
// ascending offsets, so each output element is produced in one pass.
template <typename B>
__global__ void to_dia_kernel(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ col,
                              const B *__restrict__ val, long long m, long long P,
                              const int32_t *__restrict__ off, long long nd, B *__restrict__ dval) {
  extern __shared__ int32_t s_off[];
  const bool in_smem = nd <= 4096;
  if (in_smem) {
    for (long long t = threadIdx.x; t < nd; t += blockDim.x) s_off[t] = off[t];
    __syncthreads();
  }
  const int32_t *o = in_smem ? s_off : off;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < P;
       i += (long long)gridDim.x * blockDim.x) {
    long long k = 0, e = 0;
    if (i < m) { k = rowptr[i]; e = rowptr[i + 1]; }
    for (long long t = 0; t < nd; ++t) {
      long long j = i + o[t];
      while (k < e && col[k] < j) ++k;
      B v = (B)0;
      if (k < e && col[k] == j) { v = val[k]; ++k; }
      dval[t * P + i] = v;
    }
  }
}

__global__ void cast_f32_kernel(const double *__restrict__ in, float *__restrict__ out, long long n) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    out[i] = __double2float_rn(in[i]);
}

__global__ void cast_bf16_kernel(const double *__restrict__ in, uint16_t *__restrict__ out, long long n) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    out[i] = __bfloat16_as_ushort(__double2bfloat16(in[i]));
}

int grid_for(long long work, int block, int max_blocks) {
  long long g = (work + block - 1) / block;
  if (g < 1) g = 1;
  if (g > max_blocks) g = max_blocks;
  return (int)g;
}

}  // namespace

size_t row_ends_words(int64_t n) { return (size_t)((n + 255) / 256 * 8); }

cudaError_t launch_row_ends(const RowEnds &re, int64_t m, const int32_t *rowptr, const long long *scan,
                            cudaStream_t s) {
  if (m <= 0) return cudaSuccess;
  const int g = grid_for(m, 256, 152 * 16);
  if (rowptr) row_ends_kernel<true><<<g, 256, 0, s>>>(rowptr, scan, m, re);
  else row_ends_kernel<false><<<g, 256, 0, s>>>(rowptr, scan, m, re);
  return cudaGetLastError();
}

cudaError_t launch_expand_rows(const RowEnds &re, int64_t n, int32_t *row, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  expand_rows_kernel<<<(unsigned)((n + 2047) / 2048), 256, 0, s>>>(re, n, row);
  return cudaGetLastError();
}

cudaError_t launch_empty_rows(const smat_s *h, int32_t *list, int *d_count, cudaStream_t s) {
  if (h->m <= 0) return cudaSuccess;
  empty_rows_kernel<<<grid_for(h->m, 256, 152 * 8), 256, 0, s>>>(h->rowptr, h->m, list, d_count);
  return cudaGetLastError();
}

cudaError_t launch_nonempty_rows(const smat_s *h, long long *flag, cudaStream_t s) {
  if (h->m <= 0) return cudaSuccess;
  nonempty_rows_kernel<<<grid_for(h->m, 256, 152 * 16), 256, 0, s>>>(h->rowptr, h->m, flag);
  return cudaGetLastError();
}

cudaError_t launch_to_ell(const smat_s *h, int64_t K, int32_t *col, void *val, cudaStream_t s) {
  if (h->P <= 0 || K <= 0) return cudaSuccess;
  int g = grid_for(h->P, 256, 152 * 16);
  switch (h->esz) {
    case 8: to_ell_kernel<<<g, 256, 0, s>>>(h->rowptr, h->colidx, (const Bits<8>::T *)h->val, h->m, h->P, K,
                                              col, (Bits<8>::T *)val); break;
    case 4: to_ell_kernel<<<g, 256, 0, s>>>(h->rowptr, h->colidx, (const Bits<4>::T *)h->val, h->m, h->P, K,
                                              col, (Bits<4>::T *)val); break;
    default: to_ell_kernel<<<g, 256, 0, s>>>(h->rowptr, h->colidx, (const Bits<2>::T *)h->val, h->m, h->P, K,
                                               col, (Bits<2>::T *)val); break;
  }
  return cudaGetLastError();
}

cudaError_t launch_to_dia(const smat_s *h, const int32_t *d_off, int64_t nd, void *val, cudaStream_t s) {
  if (h->P <= 0 || nd <= 0) return cudaSuccess;
  int g = grid_for(h->P, 256, 152 * 16);
  size_t sm = nd <= 4096 ? (size_t)nd * sizeof(int32_t) : 0;
  switch (h->esz) {
    case 8: to_dia_kernel<<<g, 256, sm, s>>>(h->rowptr, h->colidx, (const Bits<8>::T *)h->val, h->m, h->P,
                                               d_off, nd, (Bits<8>::T *)val); break;
    case 4: to_dia_kernel<<<g, 256, sm, s>>>(h->rowptr, h->colidx, (const Bits<4>::T *)h->val, h->m, h->P,
                                               d_off, nd, (Bits<4>::T *)val); break;
    default: to_dia_kernel<<<g, 256, sm, s>>>(h->rowptr, h->colidx, (const Bits<2>::T *)h->val, h->m, h->P,
                                                d_off, nd, (Bits<2>::T *)val); break;
  }
  return cudaGetLastError();
}

}  // namespace smat

extern "C" smat_status_t smat_cast_f64_to_f32(const double *in, float *out, int64_t n, void *stream) {
  if (n < 0 || (n > 0 && (!in || !out))) return SMAT_ERR_INVALID_ARG;
  if (n == 0) return SMAT_OK;
  smat::cast_f32_kernel<<<smat::grid_for(n, 256, 152 * 16), 256, 0, (cudaStream_t)stream>>>(in, out, n);
  return cudaGetLastError() == cudaSuccess ? SMAT_OK : SMAT_ERR_CUDA;
}

extern "C" smat_status_t smat_cast_f64_to_bf16(const double *in, uint16_t *out, int64_t n, void *stream) {
  if (n < 0 || (n > 0 && (!in || !out))) return SMAT_ERR_INVALID_ARG;
  if (n == 0) return SMAT_OK;
  smat::cast_bf16_kernel<<<smat::grid_for(n, 256, 152 * 16), 256, 0, (cudaStream_t)stream>>>(in, out, n);
  return cudaGetLastError() == cudaSuccess ? SMAT_OK : SMAT_ERR_CUDA;
}
