// Row-major to column-major copy of an m x n matrix (the layout torch hands
// over against the library's own).
//
// Bound by HBM: 16 bytes per entry.  A block moves a 64 x 32 tile through
// shared memory: it reads 256 consecutive bytes of each of 64 rows and writes
// 512 consecutive bytes of each of 32 columns (an odd row stride in shared
// memory keeps both sides free of bank conflicts), so every sector that
// crosses HBM is whole; a thread has its eight loads in flight together.
#include "cqr.h"
#include "cqr_common.cuh"

namespace cqr {

namespace {

constexpr int kTrRows = 64, kTrCols = 32, kTrThreads = 256;
constexpr int kTrPer = kTrRows * kTrCols / kTrThreads;

__global__ void __launch_bounds__(kTrThreads) transpose_kernel(i64 m, int n, const double* A, i64 lda, double* Q,
                                                               i64 ldq, int tiles_n) {
  __shared__ double tile[kTrRows * (kTrCols + 1)];
  stream_wait();
  const i64 r0 = (i64)(blockIdx.x / tiles_n) * kTrRows;
  const int c0 = (int)(blockIdx.x % tiles_n) * kTrCols, t = threadIdx.x;
  const int c = t % kTrCols, r = t / kTrCols;
  double v[kTrPer];
#pragma unroll
  for (int k = 0; k < kTrPer; ++k) {
    const i64 row = r0 + r + k * (kTrThreads / kTrCols);
    v[k] = row < m && c0 + c < n ? A[row * lda + c0 + c] : 0.0;
  }
#pragma unroll
  for (int k = 0; k < kTrPer; ++k) tile[(r + k * (kTrThreads / kTrCols)) * (kTrCols + 1) + c] = v[k];
  __syncthreads();
  const int rr = t % kTrRows;
#pragma unroll
  for (int k = 0; k < kTrPer; ++k) {
    const int cc = t / kTrRows + k * (kTrThreads / kTrRows);
    if (r0 + rr < m && c0 + cc < n) Q[(r0 + rr) + (i64)(c0 + cc) * ldq] = tile[rr * (kTrCols + 1) + cc];
  }
}

}  // namespace

cudaError_t colmajor_copy(i64 m, i64 n, const double* A, i64 lda, double* Q, i64 ldq, cudaStream_t st) {
  const i64 tiles_m = (m + kTrRows - 1) / kTrRows, tiles_n = (n + kTrCols - 1) / kTrCols;
  if (tiles_m * tiles_n > 0x7fffffffll) return cudaErrorInvalidValue;
  prof_begin(kMisc, st);
  launch(transpose_kernel, (unsigned)(tiles_m * tiles_n), kTrThreads, 0, st, m, (int)n, A, lda, Q, ldq, (int)tiles_n);
  prof_end(kMisc, 0.0, st);
  return cudaGetLastError();
}

}  // namespace cqr

extern "C" int cqr_colmajor(int64_t m, int64_t n, const double* A, int64_t lda, double* Q, int64_t ldq,
                            cqr_stream_t stream) {
  if (m < 1) return -1;
  if (n < 1 || n > 0x7fffffffll) return -2;
  if (!A) return -3;
  if (lda < n) return -4;
  if (!Q) return -5;
  if (ldq < m) return -6;
  {  // the extents of A (m rows of n, lda) and Q (n columns of m, ldq) must not overlap
    const char *a0 = (const char*)A, *a1 = (const char*)(A + (m - 1) * lda + n);
    const char *q0 = (const char*)Q, *q1 = (const char*)(Q + (n - 1) * ldq + m);
    if (a0 < q1 && q0 < a1) return -5;
  }
  cudaGetLastError();
  return cqr::colmajor_copy(m, n, A, lda, Q, ldq, (cudaStream_t)stream) == cudaSuccess ? 0 : CQR_ERR_CUDA;
}
