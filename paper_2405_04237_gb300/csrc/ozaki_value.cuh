// The value of an emulated product's level sums (k_ozaki.cu).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace cqr {

constexpr int kLevelLo = 9;  // lowest weight level i + j kept

// sum_L S_L 32^L = 32^9 (g0 + 2^30 g1), times 2^(ex + ey - 108), rounded to
// the nearest double (halves to even) in integer operations (|g0| < 2^51, |g1|
// < 2^46): the FP64 pipe takes 64 clocks an instruction, and the epilogue of an
// update tile is bound by its issue slots and that pipe together.  The 77-bit
// sum is cut to its sign and a 64-bit window; where low bits are cut off, at
// least 57 significant ones are left, and the window's last bit, which is
// below the rounding position, tells whether any of them was set.  Outside the
// normal range the library's ldexp.
__device__ __forceinline__ double group_value(long long g0, long long g1, int exy) {
  const long long h = g1 + (g0 >> 30);
  const uint32_t l = (uint32_t)g0 & 0x3FFFFFFFu;  // sum = h 2^30 + l
  const bool neg = h < 0;
  const uint32_t lo = neg ? (0u - l) & 0x3FFFFFFFu : l;
  const unsigned long long hi = (unsigned long long)(neg ? -h - (l != 0u) : h);  // |sum| = hi 2^30 + lo, hi < 2^47
  const uint32_t top = (uint32_t)(hi >> 32);
  const int k = top >= 256u ? 17 : (top >= 4u ? 24 : 30);  // hi < 2^47, 2^40, 2^34
  const unsigned long long w = (hi << k) | (lo >> (30 - k)) | ((lo & ((1u << (30 - k)) - 1u)) != 0u);
  if (w == 0ull) return 0.0;
  const int z = __clzll((long long)w);
  const int E = exy - 108 + 5 * kLevelLo + (30 - k) + 63 - z + 1023;  // biased exponent
  if (E <= 0 || E >= 2046) {
    const double v = ldexp((double)w, exy - 108 + 5 * kLevelLo + 30 - k);
    return neg ? -v : v;
  }
  const unsigned long long n = w << z;
  // 2^52 .. 2^53: up when the eleven bits below are more than half, or half and the last one kept is odd
  const uint32_t low = (uint32_t)n;
  const unsigned long long m = (n >> 11) + ((low & 0x7FFu) + ((low >> 11) & 1u) > 0x400u);
  return __longlong_as_double((long long)(m + ((unsigned long long)(E - 1) << 52) + ((unsigned long long)neg << 63)));
}

}  // namespace cqr
