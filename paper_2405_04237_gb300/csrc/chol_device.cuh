// Cholesky factorisation of a small Gram matrix inside one block: shared by
// the single-matrix kernels (k_chol.cu) and the persistent batched kernel.
#pragma once
#include <cuda_runtime.h>

namespace cqr {

// A normal float as a double, in integer operations (a conversion takes 64
// clocks like every FP64 instruction).
__device__ __forceinline__ double widen(float f) {
  const unsigned b = __float_as_uint(f);
  return __hiloint2double((int)((b >> 3) + (896u << 20)), (int)(b << 29));  // f > 0
}

// sqrt(d) and 1/sqrt(d) of a positive normal d by Newton's iteration.  The
// FP64 pipe of an SM takes 64 clocks for every warp instruction, also for a
// single live lane, so the chain of FP64 operations per column is what the
// factorisation of a small matrix costs (sqrt() and 1/x take 600 and 354
// clocks).  Here the reciprocal square root starts from the FP32 one of the
// scaled mantissa m = d 2^(-2k) in [1, 4), and its Newton step is evaluated
// in pairs of FP32 numbers (residual 1 - m r0^2 to 2^-46), which leaves r a
// relative error of about 2^-44 for one FP64 addition; one correction step
// u = u0 + (m - u0^2) r / 2 with an exact (fused) residual then gives the
// root itself (Markstein, IBM J. Res. Dev. 34 (1990): a correction with the
// fused residual rounds correctly but for near-ties; an exact root comes out
// exact).
__device__ __forceinline__ void sqrt_rsqrt(double d, double& u, double& r) {
  const int hi = __double2hiint(d), lo = __double2loint(d);
  const int ex = (hi >> 20) - 1023;
  if (ex == -1023) {  // subnormal
    u = sqrt(d);
    r = 1.0 / u;
    return;
  }
  const int k = ex >> 1, odd = ex & 1;
  const int mh = hi - (k << 21);  // m = d 2^(-2k)
  const double md = __hiloint2double(mh, lo);
  const float f = __uint_as_float((unsigned)((127 + odd) << 23) | ((unsigned)(hi & 0xFFFFF) << 3) |
                                  ((unsigned)lo >> 29));
  const float fl = __uint2float_rn((unsigned)lo & 0x1FFFFFFFu) * (odd ? 0x1p-51f : 0x1p-52f);  // m = f + fl
  const float r0 = rsqrtf(f);
  const float ph = __fmul_rn(r0, r0), pl = __fmaf_rn(r0, r0, -ph);
  float t = __fmaf_rn(-f, ph, 1.0f);
  t = __fmaf_rn(-f, pl, t);
  t = __fmaf_rn(-fl, ph, t);                                      // 1 - m r0^2
  const float c = r0 * t * __fmaf_rn(0.375f, t, 0.5f);            // r0 ((1 - t)^(-1/2) - 1)
  const double rm = widen(r0) + (double)c;
  const double hr = __hiloint2double(__double2hiint(rm) - (1 << 20), __double2loint(rm));  // rm / 2
  const double u0 = md * rm;
  const double um = fma(fma(-u0, u0, md), hr, u0);
  u = __hiloint2double(__double2hiint(um) + (k << 20), __double2loint(um));
  r = __hiloint2double(__double2hiint(rm) - (k << 20), __double2loint(rm));
}

// w / d for a positive d as w times the reciprocal: the FP32 reciprocal r0 of
// the mantissa m (24 bits), then r0 (1 + e + e^2) with the residual e = 1 - m
// r0 (third order Newton: relative error e^3 < 2^-66 before rounding).  Where d
// or 1/d is subnormal (1/d of a subnormal d overflows, 1/d below 2^-1022 loses
// bits) both are scaled first; w^2 <= d W_cc keeps w 2^54 finite.
__device__ __forceinline__ double over_pivot(double w, double d) {
  int hi = __double2hiint(d), ex = (hi >> 20) - 1023;
  if (ex == -1023 || ex > 1020) {
    const double s = ex < 0 ? 0x1p54 : 0x1p-54;
    w *= s;
    d *= s;
    hi = __double2hiint(d);
    ex = (hi >> 20) - 1023;
  }
  const int lo = __double2loint(d);
  const double m = __hiloint2double(hi - (ex << 20), lo);
  const float f = __uint_as_float((127u << 23) | ((unsigned)(hi & 0xFFFFF) << 3) | ((unsigned)lo >> 29));
  const double r0 = widen(__frcp_rn(f));
  const double e = fma(-m, r0, 1.0);
  const double r = fma(r0, fma(e, e, e), r0);
  return w * __hiloint2double(__double2hiint(r) - (ex << 20), __double2loint(r));
}

// ---------------------------------------------------------------------------
// The rows of a trapezoid in shared memory: Ws (row-major, ld) holds the
// upper triangle of a kb x kb diagonal block and nx further columns of the
// same rows; on return row j of both is row j of the factor (the diagonal in
// dg).  T threads, one barrier per two rows.  The rows are eliminated in the
// square-root-free form (pivots d_j, rows w_jc, multipliers l_jc = w_jc / d_j,
// W_ac -= l_ja w_jc) and scaled by 1 / sqrt(d_j) at the end, all at once.  In
// step j (even) the pivot warps apply the updates of rows j - 2 and j - 1 to
// rows j and j + 1 and eliminate the two; lanes 0 and 1 of each hold columns
// j and j + 1 (the pivots travel by shuffles), the others 30 further columns.
// Meanwhile the other warps apply the updates of rows j - 2 and j - 1 to the
// rows below.  A column's chain is six dependent FP64 operations (64 clocks
// each), and two columns share a barrier and a round trip through shared
// memory.  Every pivot warp reads rows j and j + 1 in columns j and j + 1, so
// none of these four is written in step j: a warp's own entries are those
// beyond column j + 1, the pivots go to dg, and the updated entry (j, j + 1)
// waits for the end in the unused place (j + 1, j) below the diagonal (two
// warps never touch one entry between two barriers, unless to read).
// At the end U_jc = w / u is w r corrected with the fused residual,
// so exact quotients stay exact.  The elements of the rows below are
// enumerated from the last row up (tab), so the live ones are always a prefix
// and no lane idles.  While they are few, the warps that share a scheduler
// (warp mod 4) with a pivot warp leave the update to the others: their FP64
// instructions would come between those of the pivot's chain.  Returns the row
// that broke down, or -1.  Scratch in shared memory: rows (8 x us, us >= kb
// + nx), tab (an entry per element), broken.  kb + nx <= 30 (T / 32 - 1).

// Elements per scheduler up to which the update fits behind the pivots' chain
// (about 1100 clocks: 8 elements a lane, two instructions of 64 each).
constexpr int kQuietLen = 256;

__device__ __forceinline__ bool good_pivot(double d) {
  // d > 0 and finite, in integers (an FP64 comparison takes 64 clocks of the chain)
  const int hi = __double2hiint(d);
  return hi < 0x7FF00000 && (hi > 0 || (hi == 0 && __double2loint(d) != 0));
}

template <int T>
__device__ int chol_trapezoid(double* Ws, int ld, int kb, int nx, double* rows, int us, double* dg,
                              unsigned short* tab, int* broken) {
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  if (t == 0) *broken = -1;
  const int total = kb * (kb + 1) / 2 + kb * nx;
  for (int e = t; e < total; e += T) {  // row kb-1-k starts at k (k + 1) / 2 + k nx
    const float h = (float)nx + 0.5f;
    int k = (int)(sqrtf(h * h + 2.0f * (float)e) - h);
    while ((k + 1) * (k + 2) / 2 + (k + 1) * nx <= e) ++k;
    while (k * (k + 1) / 2 + k * nx > e) --k;
    const int row = kb - 1 - k;
    tab[e] = (unsigned short)((row << 8) | (row + e - k * (k + 1) / 2 - k * nx));
  }
  __syncthreads();
  for (int j = 0; j < kb; j += 2) {
    int bad = 0;
    // rows j - 2, j - 1 (w, l each) and this step's
    const double* pw = rows + ((j >> 1) + 1 & 1) * 4 * us;
    double* cw = rows + (j >> 1 & 1) * 4 * us;
    const double *pl = pw + us, *pw2 = pw + 2 * us, *pl2 = pw + 3 * us;
    const int rest = kb + nx - j - 2;  // columns beyond the two pivots'
    const int np = rest > 30 ? (rest + 29) / 30 : 1;
    if (warp < np) {
      const bool two = j + 1 < kb;
      const int c = lane < 2 ? j + lane : j + 30 * warp + lane;
      const bool live = c < kb + nx && (lane != 1 || two || warp == 0);
      double *r1 = Ws + j * ld, *r2 = r1 + ld;
      double w1 = live ? r1[c] : 0.0, w2 = live && two && c > j ? r2[c] : 0.0;
      if (j > 0 && live) {
        const double x1 = pw[c], x2 = pw2[c];
        w1 = fma(-pl[j], x1, w1);
        w1 = fma(-pl2[j], x2, w1);
        if (two) {
          w2 = fma(-pl[j + 1], x1, w2);
          w2 = fma(-pl2[j + 1], x2, w2);
        }
      }
      const double d1 = __shfl_sync(0xffffffffu, w1, 0);
      if (good_pivot(d1)) {
        const double l1 = over_pivot(w1, d1);
        const bool own = live && (lane >= 2 || warp == 0);
        if (own && c > j) {
          cw[c] = w1;
          cw[us + c] = l1;
          *(c > j + 1 || !two ? r1 + c : r2 + j) = w1;
        }
        if (t == 0) dg[j] = d1;
        if (two) {
          w2 = fma(-__shfl_sync(0xffffffffu, l1, 1), w1, w2);
          const double d2 = __shfl_sync(0xffffffffu, w2, 1);
          if (good_pivot(d2)) {
            const double l2 = over_pivot(w2, d2);
            if (own && c > j + 1) {
              cw[2 * us + c] = w2;
              cw[3 * us + c] = l2;
              r2[c] = w2;
            }
            if (t == 0) dg[j + 1] = d2;
          } else {
            bad = 1;
            if (t == 0) *broken = j + 1;
          }
        }
      } else {
        bad = 1;
        if (t == 0) *broken = j;
      }
    } else if (j > 0) {
      const int k = kb - 2 - j, len = k > 0 ? k * (k + 1) / 2 + k * nx : 0;  // rows j+2 .. kb-1
      int w = warp - np, nw = T / 32 - np;
      if (np < 4 && len <= kQuietLen * (4 - np)) {
        const int q = warp & 3;
        w = q < np ? -1 : (warp >> 2) * (4 - np) + q - np;
        nw = (T / 128) * (4 - np);
      }
      if (w >= 0)
        for (int e = 32 * w + lane; e < len; e += 32 * nw) {
          const int i = tab[e] >> 8, c = tab[e] & 255;
          const double v = fma(-pl[i], pw[c], Ws[i * ld + c]);
          Ws[i * ld + c] = fma(-pl2[i], pw2[c], v);
        }
    }
    if (__syncthreads_or(bad)) break;
  }
  const int jb = *broken, done = jb >= 0 ? jb : kb;
  double* rs = rows;  // 1 / sqrt(d_j)
  for (int j = t; j < done; j += T) {
    double u, r;
    sqrt_rsqrt(dg[j], u, r);
    dg[j] = u;
    rs[j] = r;
  }
  __syncthreads();
  for (int e = t; e < total; e += T) {
    const int j = tab[e] >> 8, c = tab[e] & 255;
    if (c > j && j < done) {
      double* from = Ws + j * ld + c;
      if (c == j + 1 && c < kb && !(j & 1)) from = Ws + c * ld + j;  // entry (j, j + 1) of a pair of rows
      const double w = *from, r = rs[j], q = w * r;
      *from = 0.0;
      Ws[j * ld + c] = fma(fma(-q, dg[j], w), r, q);
    }
  }
  __syncthreads();
  return jb;
}

}  // namespace cqr
