// Sums of register accumulators inside a block, shared by the split-m
// products (k_tn.cu) and the persistent batched kernel (k_batched.cu).
#pragma once
#include <cuda_runtime.h>

namespace cqr {

// ---------------------------------------------------------------------------
// Fixed-order sums of per-thread 4 x 4 accumulators inside a block.  The
// accumulators lie in shared memory entry-major (red[e * T + thread], entry
// e = u * 4 + v).  Output o = e * ntile + tile is the sum over k < nv of
// red[e * T + tile * st + k * sk].  A dependent FP64 add takes 64 clocks and
// a warp's add costs the same with one live lane as with 32, so the outputs
// are spread over all T threads: where there are fewer than T / 2 of them
// every output is cut into S parts, summed by S threads and then over the
// parts.  (One thread per tile adding all its values in a row took 200-330
// us per Gram matrix for b <= 16, most of the time of a small
// factorisation; spread it takes 1-2 us.)  `scratch` holds T doubles and
// may be `red` itself.
template <int T, class Store>
__device__ __forceinline__ void block_sums(const double* red, double* scratch, int ntile, int nv, int st, int sk,
                                           Store store) {
  const int t = threadIdx.x;
  const int O = 16 * ntile;
  const int S = 2 * O <= T ? T / O : 1;
  if (S == 1) {
    for (int o = t; o < O; o += T) {
      const int e = o / ntile, tile = o - e * ntile;
      const double* p = red + e * T + tile * st;
      double x = 0.0;
      for (int k = 0; k < nv; ++k) x += p[k * sk];
      store(tile, e, x);
    }
  } else {
    const int s = t / O, o = t - s * O;
    const int e = o / ntile, tile = o - e * ntile;
    double part = 0.0;
    if (s < S) {
      const double* p = red + e * T + tile * st;
      const int k1 = (s + 1) * nv / S;
      for (int k = s * nv / S; k < k1; ++k) part += p[k * sk];
    }
    if (scratch == red) __syncthreads();
    if (s < S) scratch[s * O + o] = part;
    __syncthreads();
    if (t < O) {
      double x = scratch[t];
      for (int q = 1; q < S; ++q) x += scratch[q * O + t];
      store(tile, e, x);  // s == 0 here: (tile, e) is output t
    }
  }
}

__device__ __forceinline__ void spill_acc(double* red, int T, const double (&acc)[4][4]) {
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v) red[(u * 4 + v) * T + threadIdx.x] = acc[u][v];
}

}  // namespace cqr
