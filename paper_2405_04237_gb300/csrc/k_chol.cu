// Cholesky factorisation W = U^T U of a b x b Gram matrix (Alg. 1 step 2;
// Alg. 2 step 5), right-looking:
//   for j = 0..b-1:  d = W_jj;  breakdown unless d > 0 and finite;
//                    U_jj = sqrt(d);  U_jc = W_jc / U_jj  (c > j);
//                    W_ac -= U_ja U_jc  (j < a <= c).
// Each W_jc receives its updates in ascending j, i.e. the same order as the
// row-by-row definition U_jc = (W_jc - sum_{i<j} U_ij U_ic) / U_jj.
//
// The b x b problem is a serial island between two streaming passes over
// the m rows, bound by the chain of dependent FP64 operations per column
// (64 clocks each) and, for wide panels, by one SM's two FP64 multiply-adds
// per clock.  b <= 64 runs in one block (fused with the sum of the Gram
// partials), wider panels in a cluster of eight.
//
// A breakdown (the Gram matrix is not numerically positive definite,
// Sec. 3) sets the status word to col0 + j + 1 with an atomic
// compare-and-swap, so the first breakdown of a factorisation is kept; the
// unfinished rows of U and their reciprocals become NaN.  Nothing traps.
#include "cqr.h"
#include "chol_device.cuh"
#include "cqr_common.cuh"

namespace cqr {

namespace {

constexpr double kIdentityTol = 8.0 * 0x1p-53;

constexpr int kSmallT = 256;
constexpr int kSmallChol = 64;           // widest Gram matrix of the one-block kernels
constexpr int kTrapMax = 96;             // most columns kb + nx
constexpr int kTrapTab = 2560;           // most elements (64 x 64: 2080; 32 x (32 + 61): 2480)

struct TrapWork {
  double rows[8 * kTrapMax];
  double dg[kSmallChol];
  unsigned short tab[kTrapTab];
  int broken;
};

// ---------------------------------------------------------------------------
// b <= kSmallChol: one block.
constexpr int kSmallLd = kSmallChol + 1;

struct CholArgs {
  int b;
  double* W;     // reduced Gram matrix (upper triangle read; scratch), ldw
  i64 ldw;
  double* U;
  i64 ldu;
  double* rinv;
  int col0;
  int* status;
  int shift;
  i64 m;
  int* skip;
  int* reject;
};

struct SmallChol {
  double Ws[kSmallChol * kSmallLd];
  TrapWork w;
  int far_from_identity;
};

// (max U_jj / min U_jj)^2 > 1 / (64 u): the panel test of the adaptive width
__device__ __forceinline__ int panel_rejected(double dmax, double dmin) {
  return dmax * dmax * 64.0 * 0x1p-53 > dmin * dmin;
}

__device__ void chol_small(const CholArgs& a, SmallChol& s) {
  const int b = a.b, t = threadIdx.x;
  if (t == 0) s.far_from_identity = 0;
  for (int e = t; e < b * b; e += kSmallT) {
    const int r = e % b, c = e / b;
    if (r <= c) s.Ws[r * kSmallLd + c] = __ldcg(a.W + r + (i64)c * a.ldw);
  }
  if (a.shift) {
    __syncthreads();
    // Alg. 4 steps 2-3: s = sqrt(m) u ||A||_F^2 with ||A||_F^2 = trace(W)
    if (t == 0) {
      double fro2 = 0.0;
      for (int j = 0; j < b; ++j) fro2 += s.Ws[j * kSmallLd + j];
      const double sh = sqrt((double)a.m) * 0x1p-53 * fro2;
      for (int j = 0; j < b; ++j) s.Ws[j * kSmallLd + j] += sh;
    }
  }
  const int jb = chol_trapezoid<kSmallT>(s.Ws, kSmallLd, b, 0, s.w.rows, kTrapMax, s.w.dg, s.w.tab, &s.w.broken);
  // A breakdown of a panel wider than one column under the panel test is a
  // rejection, not a failure of the factorisation.
  if (t == 0 && jb >= 0 && a.status && !(a.reject && b > 1)) atomicCAS(a.status, 0, a.col0 + jb + 1);
  if (a.reject && t == 0) {
    int rej = 0;
    if (b > 1) {
      if (jb >= 0) {
        rej = 1;
      } else {
        double dmax = s.w.dg[0], dmin = s.w.dg[0];
        for (int j = 1; j < b; ++j) {
          const double d = s.w.dg[j];
          if (d > dmax) dmax = d;
          if (d < dmin) dmin = d;
        }
        rej = panel_rejected(dmax, dmin);
      }
    }
    *a.reject = rej;
  }
  // Runtime choice of the second CholeskyQR pass (Sec. 7): when every entry
  // of U - I is within 8u the panel is already orthonormal to working
  // precision; U becomes I exactly and the triangular solve is skipped
  // (with U = I it would leave the panel unchanged).
  bool identity = false;
  if (a.skip) {
    if (jb < 0) {
      for (int e = t; e < b * b; e += kSmallT) {
        const int i = e % b, c = e / b;
        if (i <= c && !(fabs(i == c ? s.w.dg[i] - 1.0 : s.Ws[i * kSmallLd + c]) <= kIdentityTol))
          s.far_from_identity = 1;
      }
    }
    __syncthreads();
    identity = (jb < 0) && !s.far_from_identity;
    if (t == 0) *a.skip = identity ? 1 : 0;
  }
  const double nan = __longlong_as_double(0x7ff8000000000000LL);
  for (int e = t; e < b * b; e += kSmallT) {
    const int i = e % b, c = e / b;
    double v = 0.0;
    if (identity)
      v = (i == c) ? 1.0 : 0.0;
    else if (i <= c)
      v = (jb >= 0 && i >= jb) ? nan : (i == c ? s.w.dg[i] : s.Ws[i * kSmallLd + c]);
    a.U[i + (i64)c * a.ldu] = v;
  }
  if (t < b) a.rinv[t] = identity ? 1.0 : ((jb >= 0 && t >= jb) ? nan : 1.0 / s.w.dg[t]);
}

__global__ void __launch_bounds__(kSmallT) chol_small_kernel(CholArgs a) {
  stream_wait();
  __shared__ SmallChol s;
  if (a.status && *a.status) return;
  chol_small(a, s);
}

// The Gram partials' sum (16 entries of the upper triangle per block, 16
// contiguous parts each, see split_sum16) and, in the block that finishes
// last, the Cholesky factorisation: one launch instead of two for every
// CholeskyQR.  `counter` is zero at entry and left zero.
__global__ void __launch_bounds__(kSmallT) gram_chol_kernel(const double* part, i64 P, CholArgs a,
                                                            unsigned int* counter) {
  stream_wait();
  __shared__ SmallChol s;
  __shared__ double red[16 * 17];
  __shared__ unsigned int order;
  if (a.status && *a.status) return;
  const int b = a.b;
  const int u = blockIdx.x * 16 + (threadIdx.x & 15);
  const bool live = u < b * (b + 1) / 2;
  int r = 0, c = 0;
  if (live) decode_upper(u, r, c);
  const double* p = part + r + c * b;
  const i64 bb = (i64)b * b;
  const double v = split_sum16(P, live, red, [p, bb](i64 k) { return p[k * bb]; });
  if (threadIdx.x < 16 && live) a.W[r + (i64)c * a.ldw] = v;
  if (gridDim.x > 1) {
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) order = atomicAdd(counter, 1u);
    __syncthreads();
    if (order != gridDim.x - 1) return;
    __threadfence();
    if (threadIdx.x == 0) *counter = 0;
  } else {
    __threadfence_block();
    __syncthreads();
  }
  chol_small(a, s);
}

// ---------------------------------------------------------------------------
// 64 < b <= 512: one cluster of eight blocks, W in global memory (L2), row
// tiles of 32.  Per tile: every block factors the 32 x 32 diagonal block for
// itself, with its own share of the row panel's columns as the trapezoid's
// further columns (so the factor needs no broadcast); after a cluster
// barrier the trailing triangle is updated element by element over all eight
// blocks (32 fused multiply-adds each, ascending rows, the order of the
// right-looking definition), and a second barrier ends the step.  One SM
// delivers two FP64 multiply-adds per clock, so the b^3/6 of them alone took
// 85 us (b = 128) or 680 us (b = 256) in one block.
constexpr int kClu = 8;
constexpr int kCluTile = 32;
constexpr int kCluLd = kTrapMax + 1;

inline size_t chol_cluster_smem(int b) { return sizeof(double) * (size_t)kCluTile * (size_t)(b - kCluTile); }
static_assert((CQR_MAX_PANEL - kCluTile + kClu - 1) / kClu + kCluTile <= kTrapMax, "a block's columns of a tile");

__device__ __forceinline__ void cluster_barrier() {
  __threadfence();
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__global__ void __cluster_dims__(kClu, 1, 1) __launch_bounds__(kSmallT) chol_cluster_kernel(CholArgs a) {
  stream_wait();
  extern __shared__ __align__(16) double pan[];  // [kCluTile][rem]: the tile's row panel
  __shared__ double Ws[kCluTile * kCluLd];
  __shared__ TrapWork s;
  __shared__ double sh_shift, sh_dmax, sh_dmin;
  __shared__ int sh_far;
  if (a.status && *a.status) return;  // uniform over the cluster: set by earlier launches only
  const int t = threadIdx.x, rank = blockIdx.x, b = a.b, gt = rank * kSmallT + t;
  if (t < 32 && a.shift) {
    // Alg. 4 steps 2-3: s = sqrt(m) u ||A||_F^2 with ||A||_F^2 = trace(W)
    double fro2 = 0.0;
    for (int j = t; j < b; j += 32) fro2 += __ldcg(a.W + j + (i64)j * a.ldw);
    for (int o = 16; o > 0; o >>= 1) fro2 += __shfl_xor_sync(0xffffffffu, fro2, o);
    if (t == 0) sh_shift = sqrt((double)a.m) * 0x1p-53 * fro2;
  }
  if (t == 0) {
    sh_far = 0;
    if (rank == 0 && a.skip) *a.skip = 1;
  }
  for (int e = gt; e < b * b; e += kClu * kSmallT) {
    const int i = e % b, c = e / b;
    if (i > c) a.U[i + (i64)c * a.ldu] = 0.0;
  }
  cluster_barrier();  // the trace has been read everywhere; *skip = 1 is set
  int jb = -1;
  for (int k0 = 0; k0 < b; k0 += kCluTile) {
    const int kb = min(kCluTile, b - k0), k1 = k0 + kb, rem = b - k1;
    const int per = (rem + kClu - 1) / kClu;                      // columns of the row panel per block
    const int c0 = min(rank * per, rem), nx = min(per, rem - c0);  // this block's: k1 + c0 .. + nx
    for (int e = t; e < kb * (kb + nx); e += kSmallT) {
      const int i = e % kb, c = e / kb, gc = c < kb ? k0 + c : k1 + c0 + c - kb;
      if (c >= i) {
        const double w = __ldcg(a.W + (k0 + i) + (i64)gc * a.ldw);
        Ws[i * kCluLd + c] = (a.shift && c == i) ? w + sh_shift : w;
      }
    }
    jb = chol_trapezoid<kSmallT>(Ws, kCluLd, kb, nx, s.rows, kTrapMax, s.dg, s.tab, &s.broken);
    const int rows = jb >= 0 ? jb : kb;  // finished rows
    bool far = false;
    for (int e = t; e < rows * (kb + nx); e += kSmallT) {
      const int i = e % rows, c = e / rows;
      if (c < i || (c < kb && rank != 0)) continue;  // block 0 writes the diagonal block
      const double v = c == i ? s.dg[i] : Ws[i * kCluLd + c];
      a.U[(k0 + i) + (i64)(c < kb ? k0 + c : k1 + c0 + c - kb) * a.ldu] = v;
      far |= !(fabs(c == i ? v - 1.0 : v) <= kIdentityTol);
    }
    if (far) sh_far = 1;
    if (rank == 0 && t < rows) a.rinv[k0 + t] = 1.0 / s.dg[t];
    if (t == 0)
      for (int j = 0; j < rows; ++j) {
        const double d = s.dg[j];
        if (k0 + j == 0 || d > sh_dmax) sh_dmax = d;
        if (k0 + j == 0 || d < sh_dmin) sh_dmin = d;
      }
    cluster_barrier();  // the row panel is in U
    if (jb >= 0) {
      jb += k0;
      break;
    }
    if (rem > 0) {
      for (int e = t; e < kb * rem; e += kSmallT) {
        const int i = e % kb, c = e / kb;
        pan[i * rem + c] = __ldcg(a.U + (k0 + i) + (i64)(k1 + c) * a.ldu);
      }
      __syncthreads();
      const int cnt = rem * (rem + 1) / 2;
      for (int e = gt; e < cnt; e += kClu * kSmallT) {
        int i, c;
        decode_upper(e, i, c);
        double* w = a.W + (k1 + i) + (i64)(k1 + c) * a.ldw;
        double acc = __ldcg(w);
        const double *pi = pan + i, *pc = pan + c;
#pragma unroll 8
        for (int k = 0; k < kb; ++k) acc = fma(-pi[k * rem], pc[k * rem], acc);
        *w = acc;
      }
      cluster_barrier();
    }
  }
  if (gt == 0) {
    if (jb >= 0 && a.status && !a.reject) atomicCAS(a.status, 0, a.col0 + jb + 1);
    if (a.reject) *a.reject = jb >= 0 ? 1 : panel_rejected(sh_dmax, sh_dmin);
  }
  if (jb >= 0) {  // breakdown: the unfinished rows are NaN
    const double nan = __longlong_as_double(0x7ff8000000000000LL);
    for (int e = gt; e < b * b; e += kClu * kSmallT) {
      const int i = e % b, c = e / b;
      if (i <= c && i >= jb) a.U[i + (i64)c * a.ldu] = nan;
    }
    if (rank == 0)
      for (int e = jb + t; e < b; e += kSmallT) a.rinv[e] = nan;
  }
  if (a.skip) {
    // the runtime choice of the second pass (see chol_small): U := I when every entry of U - I is within 8u
    __syncthreads();
    if (t == 0 && (jb >= 0 || sh_far)) *a.skip = 0;
    cluster_barrier();
    if (__ldcg(a.skip) && jb < 0) {
      for (int e = gt; e < b * b; e += kClu * kSmallT) {
        const int i = e % b, c = e / b;
        if (i <= c) a.U[i + (i64)c * a.ldu] = i == c ? 1.0 : 0.0;
      }
      if (rank == 0)
        for (int e = t; e < b; e += kSmallT) a.rinv[e] = 1.0;
    }
  }
}

// M := copyltu(T - G): M_ac = T_ac - G_ac for a >= c, mirrored above.
__global__ void backward_middle_kernel(int n, const double* T, const double* G, double* M) {
  stream_wait();
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n * n) return;
  const int a = e % n, c = e / n;
  const int lo = a >= c ? a : c, hi = a >= c ? c : a;  // (lo, hi) in the lower triangle
  M[e] = T[lo + (i64)hi * n] - G[lo + (i64)hi * n];
}

__global__ void diag_reciprocal_kernel(int n, const double* R, i64 ldr, double* rinv) {
  stream_wait();
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < n) rinv[j] = 1.0 / R[j + (i64)j * ldr];
}

}  // namespace

cudaError_t chol_factor(int b, double* W, i64 ldw, double* U, i64 ldu, double* rinv, int col0, int* status,
                        int shift_fro, i64 m, cudaStream_t st, int* skip, int* reject) {
  if (b <= 0) return cudaSuccess;
  prof_begin(kCholesky, st);
  const CholArgs a{b, W, ldw, U, ldu, rinv, col0, status, shift_fro, m, skip, reject};
  if (b <= kSmallChol) {
    launch(chol_small_kernel, 1, kSmallT, 0, st, a);
  } else {
    static PerDevice<bool> attr;
    if (bool& set = attr.here(); !set) {
      cudaFuncSetAttribute(chol_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)chol_cluster_smem(CQR_MAX_PANEL));
      set = true;
    }
    launch(chol_cluster_kernel, kClu, kSmallT, chol_cluster_smem(b), st, a);
  }
  prof_end(kCholesky, (double)b * b * b / 3.0, st);
  return cudaGetLastError();
}

cudaError_t gram_chol(i64 m, int b, const double* X, i64 ldx, double* part, double* W, i64 ldw, double* U, i64 ldu,
                      double* rinv, int col0, int* status, int shift_fro, unsigned int* counter, cudaStream_t st,
                      int* skip, int* reject) {
  if (b <= 0) return cudaSuccess;
  if (b > kSmallChol || m <= 0) {
    const cudaError_t e = tn_product(m, b, b, X, ldx, X, ldx, 1, part, W, ldw, status, st);
    if (e != cudaSuccess) return e;
    return chol_factor(b, W, ldw, U, ldu, rinv, col0, status, shift_fro, m, st, skip, reject);
  }
  const i64 P = gram_partials(m, b, X, ldx, part, status, st);
  const CholArgs a{b, W, ldw, U, ldu, rinv, col0, status, shift_fro, m, skip, reject};
  prof_begin(kCholesky, st);
  // early only behind a Gram kernel that leaves SMs free (its blocks take 44 KB of shared memory each)
  launch(P <= kSMs ? Work64{0.0} : kNotEarly, gram_chol_kernel, (b * (b + 1) / 2 + 15) / 16, kSmallT, 0, st, part, P, a,
         counter);
  prof_end(kCholesky, (double)b * b * b / 3.0, st);
  return cudaGetLastError();
}

cudaError_t backward_middle(int n, const double* T, const double* G, double* M, cudaStream_t st) {
  const int thr = 256;
  prof_begin(kMisc, st);
  launch(backward_middle_kernel, (n * n + thr - 1) / thr, thr, 0, st, n, T, G, M);
  prof_end(kMisc, (double)n * n, st);
  return cudaGetLastError();
}

cudaError_t diag_reciprocal(int n, const double* R, i64 ldr, double* rinv, cudaStream_t st) {
  prof_begin(kMisc, st);
  launch(diag_reciprocal_kernel, (n + 255) / 256, 256, 0, st, n, R, ldr, rinv);
  prof_end(kMisc, (double)n, st);
  return cudaGetLastError();
}

}  // namespace cqr
