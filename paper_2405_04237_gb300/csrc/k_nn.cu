// C = beta*C + alpha*A*B: the Gram-Schmidt update A_{j:k} -= Q_{j-1} Y
// (Alg. 6 step 7, Alg. 9 step 4), the re-orthogonalisation update
// P -= Q_{1:j-1} Z (Alg. 9 step 7), the blocked part of wide triangular
// solves, the adjoint's Q copyltu(M) product, and the small triangular
// products R = R2 R1 (Alg. 3 step 3, Alg. 7 step 3), R_jj = S2 S1 and
// R_{1:j-1,j} += Z S1 of Alg. 9 (these two in one launch).
//
// Each block computes a TM x TN output tile (256 threads, one MT x MT register
// micro-tile per thread, TM * TN = 256 MT^2); K is staged through shared
// memory in chunks.  MT is 2 from one block per SM on, else 1, so that the
// multiply-adds (64 clocks each for a warp) are spread over the SMs: a 64 x 64
// x 64 product took 81 us in one block of 4 x 4 micro-tiles.  The FP64 pipe is
// so slow that 2 x 2 already hides the shared-memory loads, and its smaller
// blocks even out the last wave and the partial tiles: against 4 x 4, CQR2GS
// 30011 x 90 takes 1717 instead of 1814 us, 60000 x 256 14.94 instead of 15.40
// ms, 2^18 x 256 58.47 instead of 58.59 ms.  Every element sees the same
// operations in the same order whatever the tile.  With beta = 1 the
// accumulator starts from C and every term is one fused multiply-add (negated
// operand when alpha = -1), so the update issues exactly one FP64 instruction
// per multiply-add.  Threads whose columns all lie beyond N skip the
// arithmetic (warp-uniform when N is a multiple of 8), so narrow outputs do
// not pay for padding.
#include "cqr_common.cuh"

namespace cqr {

namespace {

constexpr int kNnThreads = 256;

struct NnArgs {
  const double* A;
  i64 lda;
  const double* B;
  i64 ldb;
  double* C;
  i64 ldc;
  i64 M;
  int N, K;
  int beta, a_upper, b_upper, transb;
  int tiles_n;
  const int* status;
  // a second product with the same B, N and K in the blocks from `first` on (kPair)
  const double* A2;
  i64 lda2;
  double* C2;
  i64 ldc2, M2;
  int beta2, a_upper2;
  i64 first;
};

template <int TM, int TN, int MT>
struct NnShape {
  static constexpr int NTM = TM / MT;
  static constexpr int KC = 16;
  static constexpr int SA = TM + 2, SB = TN + 2;
  static_assert(TM % MT == 0 && TN % MT == 0, "MT x MT micro-tiles");
  static_assert(NTM * (TN / MT) == kNnThreads, "one micro-tile per thread covers the TM x TN tile");
  static_assert(KC * (SA + SB) * (int)sizeof(double) <= 48 * 1024, "static shared memory limit");
};

// MT consecutive doubles of a shared-memory row
template <int MT>
__device__ __forceinline__ void lds_micro(const double* p, double (&v)[MT]) {
  if constexpr (MT == 2) {
    const double2 x = *reinterpret_cast<const double2*>(p);
    v[0] = x.x;
    v[1] = x.y;
  } else {
    v[0] = p[0];
  }
}

template <int TM, int TN, int MT, bool NEG, bool kPair = false>
__global__ void __launch_bounds__(kNnThreads) nn_kernel(NnArgs a) {
  stream_wait();
  using Sh = NnShape<TM, TN, MT>;
  __shared__ __align__(16) double As[Sh::KC * Sh::SA];
  __shared__ __align__(16) double Bs[Sh::KC * Sh::SB];
  if (a.status && *a.status) return;
  i64 bid = blockIdx.x;
  if (kPair && bid >= a.first) {
    bid -= a.first;
    a.A = a.A2;
    a.lda = a.lda2;
    a.C = a.C2;
    a.ldc = a.ldc2;
    a.M = a.M2;
    a.beta = a.beta2;
    a.a_upper = a.a_upper2;
  }
  const int tn_i = (int)(bid % a.tiles_n);
  const i64 m0 = (bid / a.tiles_n) * TM;
  const int n0 = tn_i * TN;
  const int t = threadIdx.x;
  const int mi = t % Sh::NTM, nj = t / Sh::NTM;
  const bool cols_live = n0 + MT * nj < a.N;
  const bool rows_live = m0 + MT * mi < a.M;
  const bool live = cols_live && rows_live;

  int klo = 0, khi = a.K;
  if (a.a_upper) klo = (int)(m0 < (i64)a.K ? m0 : (i64)a.K);
  if (a.b_upper) khi = min(a.K, n0 + TN);

  double acc[MT][MT];
#pragma unroll
  for (int i = 0; i < MT; ++i)
#pragma unroll
    for (int j = 0; j < MT; ++j) {
      double v = 0.0;
      if (a.beta) {
        const i64 r = m0 + MT * mi + i;
        const int c = n0 + MT * nj + j;
        if (r < a.M && c < a.N) v = a.C[r + (i64)c * a.ldc];
      }
      acc[i][j] = v;
    }

  for (int k0 = klo; k0 < khi; k0 += Sh::KC) {
    for (int e = t; e < Sh::KC * TM; e += kNnThreads) {
      const int mm = e % TM, kk = e / TM;
      const i64 r = m0 + mm;
      const int k = k0 + kk;
      double v = 0.0;
      if (r < a.M && k < khi) v = a.A[r + (i64)k * a.lda];
      As[kk * Sh::SA + mm] = v;
    }
    if (a.transb) {
      for (int e = t; e < Sh::KC * TN; e += kNnThreads) {
        const int nn = e % TN, kk = e / TN;
        const int c = n0 + nn, k = k0 + kk;
        double v = 0.0;
        if (c < a.N && k < khi) v = a.B[c + (i64)k * a.ldb];
        Bs[kk * Sh::SB + nn] = v;
      }
    } else {
      for (int e = t; e < Sh::KC * TN; e += kNnThreads) {
        const int kk = e % Sh::KC, nn = e / Sh::KC;
        const int c = n0 + nn, k = k0 + kk;
        double v = 0.0;
        if (c < a.N && k < khi) v = a.B[k + (i64)c * a.ldb];
        Bs[kk * Sh::SB + nn] = v;
      }
    }
    __syncthreads();
    if (live) {
#pragma unroll 4
      for (int kk = 0; kk < Sh::KC; ++kk) {
        double av[MT], bv[MT];
        lds_micro<MT>(&As[kk * Sh::SA + MT * mi], av);
        lds_micro<MT>(&Bs[kk * Sh::SB + MT * nj], bv);
#pragma unroll
        for (int i = 0; i < MT; ++i)
#pragma unroll
          for (int j = 0; j < MT; ++j) acc[i][j] = NEG ? fma(-av[i], bv[j], acc[i][j]) : fma(av[i], bv[j], acc[i][j]);
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < MT; ++i)
#pragma unroll
    for (int j = 0; j < MT; ++j) {
      const i64 r = m0 + MT * mi + i;
      const int c = n0 + MT * nj + j;
      if (r < a.M && c < a.N) a.C[r + (i64)c * a.ldc] = acc[i][j];
    }
}

template <int TM, int TN, int MT>
void launch_nn(const NnArgs& a, bool neg, bool pair, cudaStream_t st) {
  const i64 blocks = ((a.M + TM - 1) / TM) * a.tiles_n;
  const Work64 w{2.0 * (double)(a.M + a.M2) * a.N * a.K};
  if (pair) {
    NnArgs b = a;
    b.first = blocks;
    launch(w, nn_kernel<TM, TN, MT, false, true>, (unsigned)(blocks + ((a.M2 + TM - 1) / TM) * a.tiles_n), kNnThreads,
           0, st, b);
  } else if (neg) {
    launch(w, nn_kernel<TM, TN, MT, true>, (unsigned)blocks, kNnThreads, 0, st, a);
  } else {
    launch(w, nn_kernel<TM, TN, MT, false>, (unsigned)blocks, kNnThreads, 0, st, a);
  }
}

// Column tile for N columns and micro-tiles of MT (the widest is 16 MT).
int nn_tile_n(int N, int MT) {
  int t = 8;
  while (t < N && t < 16 * MT) t *= 2;
  return t;
}
i64 nn_blocks(i64 M, int N, int MT) {
  const int TN = nn_tile_n(N, MT), TM = 256 * MT * MT / TN;
  return (M + TM - 1) / TM * ((N + TN - 1) / TN);
}

// Tile by size, then the launch (the FP64 operations of a pair count together).
void run_nn(NnArgs& a, bool neg, bool pair, cudaStream_t st) {
  const int MT = nn_blocks(a.M + a.M2, a.N, 2) >= kSMs ? 2 : 1;
  const int TN = nn_tile_n(a.N, MT);
  a.tiles_n = (a.N + TN - 1) / TN;
  prof_begin(kUpdate, st);
  if (MT == 2) {
    switch (TN) {
      case 8: launch_nn<128, 8, 2>(a, neg, pair, st); break;
      case 16: launch_nn<64, 16, 2>(a, neg, pair, st); break;
      default: launch_nn<32, 32, 2>(a, neg, pair, st); break;
    }
  } else {
    if (TN == 8)
      launch_nn<32, 8, 1>(a, neg, pair, st);
    else
      launch_nn<16, 16, 1>(a, neg, pair, st);
  }
  prof_end(kUpdate, 2.0 * (double)(a.M + a.M2) * a.N * a.K, st);
}

}  // namespace

cudaError_t nn_product(i64 M, int N, int K, const double* A, i64 lda, const double* B, i64 ldb, double* C,
                       i64 ldc, double alpha, int beta, int a_upper, int b_upper, const int* status,
                       cudaStream_t st) {
  return nn_product_t(M, N, K, A, lda, B, ldb, 0, C, ldc, alpha, beta, a_upper, b_upper, status, st);
}

cudaError_t nn_product_t(i64 M, int N, int K, const double* A, i64 lda, const double* B, i64 ldb, int transb,
                         double* C, i64 ldc, double alpha, int beta, int a_upper, int b_upper, const int* status,
                         cudaStream_t st) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  NnArgs a{};
  a.A = A;
  a.lda = lda;
  a.B = B;
  a.ldb = ldb;
  a.C = C;
  a.ldc = ldc;
  a.M = M;
  a.N = N;
  a.K = K;
  a.beta = beta;
  a.a_upper = a_upper;
  a.b_upper = b_upper;
  a.transb = transb;
  a.status = status;
  const bool neg = alpha < 0.0;
  run_nn(a, neg, false, st);
  return cudaGetLastError();
}

cudaError_t r_products(i64 jb, int b, const double* S2, const double* S1, const double* Z, double* R, i64 ldr,
                       const int* status, cudaStream_t st) {
  if (b <= 0) return cudaSuccess;
  NnArgs a{};
  a.A = S2;
  a.lda = b;
  a.B = S1;
  a.ldb = b;
  a.C = R + jb + jb * ldr;
  a.ldc = ldr;
  a.M = b;
  a.N = b;
  a.K = b;
  a.a_upper = 1;
  a.b_upper = 1;
  a.status = status;
  a.A2 = Z;
  a.lda2 = jb;
  a.C2 = R + jb * ldr;
  a.ldc2 = ldr;
  a.M2 = jb;
  a.beta2 = 1;
  run_nn(a, false, jb > 0, st);
  return cudaGetLastError();
}

}  // namespace cqr
