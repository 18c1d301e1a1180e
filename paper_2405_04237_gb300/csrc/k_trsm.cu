// Row-wise triangular solves.
//
// trsm_rows: Q = X U^{-1} (Alg. 1 step 3).  Every row x of X is solved by
// forward substitution, q_c = (x_c - sum_{i<c} q_i U_ic) * (1/U_cc), the
// sum taken in ascending i -- the same operation order as the plain
// definition, with the division replaced by a multiplication by the
// reciprocal that the Cholesky kernel computed once (a division costs about
// ten FP64 instructions; the substitution itself costs b(b-1)/2 FMAs per
// row).  No inverse of U is formed: substitution keeps each row backward
// stable, so the residual ||A - Q R|| stays at rounding level even when U
// is ill-conditioned.
//
// trsm_rows_transposed: Abar = B U^{-T} for the adjoint of A = QR, by back
// substitution a_c = (b_c - sum_{i>c} a_i U_ci) * (1/U_cc), descending c.
//
// One thread owns one row and keeps it in registers (b rounded up to a
// multiple of four is a template argument, so that every index is static; 64
// entries take 128 registers); 128 rows per block.  When a column is solved
// its multiples are subtracted from all later ones at once: every element
// sees its terms in ascending i, and the multiply-adds of a step are
// independent, so that one warp per scheduler keeps the FP64 pipe busy (a
// warp's FP64 instruction takes 64 clocks).  U lies in shared memory (every
// thread reads the same entry: a broadcast), the row loads are in flight
// while it arrives.  Against rows in shared memory: eight solves of 2^20 x 64
// 29.7 -> 28.3 ms (0.97 of the pipe), of 2000 x 4 79 -> 50 us.
#include <type_traits>

#include "cqr_common.cuh"

namespace cqr {

namespace {

constexpr int kRows = 128;
// Wide rows: three blocks per SM even if a few entries spill (2^20 x 64: 28.3
// against 29.3 ms for eight solves with two).
template <int B>
constexpr int kMinBlocks = B > 40 ? 3 : 1;

// The row's entries from and to memory.  The pointer of the store is made
// opaque: kept from the loads, the addresses of 64 columns take as many
// registers as the entries.
template <int B>
__device__ __forceinline__ void load_row(double (&x)[B], const double* p, i64 ld, bool live, int b) {
#pragma unroll
  for (int c = 0; c < B; ++c) {
    x[c] = live && c < b ? *p : 0.0;
    p += ld;
  }
}
template <int B>
__device__ __forceinline__ void store_row(const double (&x)[B], double* p, i64 ld, bool live, int b) {
  asm volatile("" : "+l"(p), "+l"(ld));
#pragma unroll
  for (int c = 0; c < B; ++c) {
    if (live && c < b) *p = x[c];
    p += ld;
  }
}

// U's upper triangle (zero elsewhere) into Us [B][B + 1] and its reciprocals,
// zero beyond b.
template <int B>
__device__ __forceinline__ void load_factor(int b, const double* U, i64 ldu, const double* rinv, double* Us,
                                            double* rv) {
  for (int e = threadIdx.x; e < B * B; e += kRows) {
    const int i = e % B, c = e / B;
    Us[i * (B + 1) + c] = i <= c && c < b ? U[i + (i64)c * ldu] : 0.0;
  }
  for (int e = threadIdx.x; e < B; e += kRows) rv[e] = e < b ? rinv[e] : 0.0;
}

template <int B>
__global__ void __launch_bounds__(kRows, kMinBlocks<B>)
    trsm_rows_kernel(i64 m, int b, double* X, i64 ldx, const double* U, i64 ldu, const double* rinv, const int* status,
                     const int* skip) {
  stream_wait();
  __shared__ double Us[B * (B + 1)], rv[B];
  if (status && *status) return;
  if (skip && *skip) return;  // U = I: the solve would leave X unchanged
  const i64 r = (i64)blockIdx.x * kRows + threadIdx.x;
  const bool live = r < m;
  double x[B];
  load_row<B>(x, X + (live ? r : 0), ldx, live, b);
  load_factor<B>(b, U, ldu, rinv, Us, rv);
  __syncthreads();
#pragma unroll
  for (int i = 0; i < B; ++i) {
    x[i] *= rv[i];
#pragma unroll
    for (int c = i + 1; c < B; ++c) x[c] = fma(-x[i], Us[i * (B + 1) + c], x[c]);
  }
  store_row<B>(x, X + r, ldx, live, b);
}

template <int B>
__global__ void __launch_bounds__(kRows, kMinBlocks<B>)
    trsm_rows_t_kernel(i64 m, int b, double* X, i64 ldx, const double* U, i64 ldu, const double* rinv) {
  stream_wait();
  __shared__ double Us[B * (B + 1)], rv[B];
  const i64 r = (i64)blockIdx.x * kRows + threadIdx.x;
  const bool live = r < m;
  double x[B];
  load_row<B>(x, X + (live ? r : 0), ldx, live, b);
  load_factor<B>(b, U, ldu, rinv, Us, rv);
  __syncthreads();
#pragma unroll
  for (int i = B - 1; i >= 0; --i) {
    x[i] *= rv[i];
#pragma unroll
    for (int c = 0; c < i; ++c) x[c] = fma(-x[i], Us[c * (B + 1) + i], x[c]);
  }
  store_row<B>(x, X + r, ldx, live, b);
}

// f(std::integral_constant<int, B>) for B = b rounded up to a multiple of 4
template <int B = 4, class F>
void with_width(int b, F&& f) {
  if constexpr (B <= kTrsmMaxB) {
    if (b <= B)
      f(std::integral_constant<int, B>());
    else
      with_width<B + 4>(b, f);
  }
}

}  // namespace

cudaError_t trsm_rows(i64 m, int b, double* X, i64 ldx, const double* U, i64 ldu, const double* rinv,
                      const int* status, cudaStream_t st, const int* skip, bool early) {
  if (m <= 0 || b <= 0) return cudaSuccess;
  if (b > kTrsmMaxB) return cudaErrorInvalidValue;
  const i64 blocks = (m + kRows - 1) / kRows;
  prof_begin(kTrsm, st);
  with_width(b, [&](auto B) {
    launch(early ? Work64{(double)m * b * b} : kNotEarly, trsm_rows_kernel<B>, (unsigned)blocks, kRows, 0, st, m, b, X,
           ldx, U, ldu, rinv, status, skip);
  });
  prof_end(kTrsm, (double)m * b * b, st);
  return cudaGetLastError();
}

cudaError_t trsm_rows_transposed(i64 m, int b, double* X, i64 ldx, const double* U, i64 ldu,
                                 const double* rinv, cudaStream_t st) {
  if (m <= 0 || b <= 0) return cudaSuccess;
  if (b > kTrsmMaxB) return cudaErrorInvalidValue;
  const i64 blocks = (m + kRows - 1) / kRows;
  prof_begin(kTrsm, st);
  with_width(b, [&](auto B) {
    launch(Work64{(double)m * b * b}, trsm_rows_t_kernel<B>, (unsigned)blocks, kRows, 0, st, m, b, X, ldx, U, ldu,
           rinv);
  });
  prof_end(kTrsm, (double)m * b * b, st);
  return cudaGetLastError();
}

}  // namespace cqr
