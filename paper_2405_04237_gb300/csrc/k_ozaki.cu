// FP64-accurate split-m products on the 5th-generation (tcgen05) FP8 tensor
// cores, with the Ozaki error-free splitting (Ozaki, Ogita, Oishi, Numer.
// Algorithms 59 (2012)), for the emulated variant of Alg. 9 (opt-in,
// CQR_EMULATED): the projections C = X^T Y of steps 3 and 7 and the updates
// C -= X Y of steps 4 and 7.
//
// Splitting.  For C = X^T Y, rows are cut into sub-chunks of kSub = 4096.
// Within a sub-chunk every column c of X (and of Y) gets a power-of-two
// scale 2^e_c with |x| < 2^e_c, and each entry becomes the fixed-point
// integer X = x * 2^(54 - e_c) (rounded, |X| <= 2^54), written in base 32
// with eleven balanced digits: X = sum_i d_i 32^i, -16 <= d_i <= 15 (16 for
// the top digit).  An integer of magnitude up to 16 is exact in e4m3: the
// code is the sign and |d|, read as |d| 2^-9 (e4m3's subnormals and the two
// binades above them are evenly spaced), so no table is needed and every
// product carries a factor 2^-18.  Balanced digits need 11 planes and 76
// plane pairs where sign-magnitude nibbles needed 14 and 105, and the pairs
// left out have no common sign: the error against exact sums (rms, in units
// of 2^-53 |x| |y|) is 0.02 to 0.1 at K = 4096 to 64 where the nibbles' was
// 0.1 to 0.8, and 0.13 for the diagonal of X^T X where it was 16 (their
// neglected products were all positive).  With 66 pairs (levels from 10) it
// is 0.1 to 0.5, and a factorisation of 60013 x 360 was 12 % further from
// the exact Q than with the nibbles.  For
// C -= X Y the contraction runs over the columns of X: each row of X gets its
// own scale over (at most kSub of) its entries and takes a column's place;
// Y (K x N) is split by columns.
//
// Plane layout.  One "stage" is 32 contraction indices.  Columns are grouped
// in tiles of T (128 on the X side, 32 on the Y side), and the planes are
// stored tile-major: for each tile, each stage, each plane i, the T x 32
// digits in the tensor cores' canonical K-major layout without swizzling
// (8-column groups of 256 bytes, each two 8 x 16-byte core matrices holding
// indices 0..15, then 16..31).  The 11 planes of one stage of one tile are
// thus one contiguous run (44 KiB for X, 11 KiB for Y), and a stage arrives
// in shared memory with two bulk asynchronous copies (for a Gram matrix
// X^T X, whose Y tiles are 32-column slices of the X planes, one copy for X
// and one per plane for Y).
//
// Products.  x_a y_b = 2^(e_a + e_b - 108) sum_{i,j} d^x_i d^y_j 32^(i+j).
// The 76 plane pairs with i + j >= 9 (the 12 most significant weight
// levels) are multiplied with tcgen05.mma kind::f8f6f4 (e4m3 x e4m3 -> f32)
// into one TMEM accumulator per level: TMEM region r (32 columns, r = 0..11)
// holds level r + 9.  The Y planes of one stage lie in shared memory one
// after the other, so planes j0 .. j0+n-1 form one operand of N = 32 n rows,
// and one instruction A_i x [Y_j0; ...; Y_j0+n-1] (128 x 32n x 32) adds pair
// (i, j0 + v) into region i + j0 + v - 9 for v < n.  16 such instructions
// (N = 32 .. 256) cover the 76 pairs.  Per level the sum over at most 4096
// contraction indices is below 11 * 256 * 4096 < 2^24 in magnitude, so the
// FP32 accumulation is exact (an integer times 2^-18).  The dropped levels
// weigh at most about 2^-56.6 of the scales' product per index.
//
// Schedule.  A block of 16 warps computes a 128 x 32 tile of C over its
// contraction range (a sub-chunk of a projection, all of K for an update).
// Four shared-memory stages of 55 KiB rotate: one thread issues the bulk
// copies of a stage (completion counted in bytes on the stage's "full"
// mbarrier), one thread issues its 16 MMAs and commits them to the stage's
// "empty" mbarrier, which frees the stage for the copy four stages later.
// At the end every thread reads the 12 level sums of its row from TMEM,
// combines levels 9..14 and 15..20 exactly in 64-bit integers (below 2^51)
// and rounds the two to a double in integer operations (group_value), so the
// FP64 pipe does nothing for a projection and one subtraction per entry of an
// update.  Every wait is bounded in time
// (kWaitNs of the global nanosecond timer, 2 s: a stage arrives within
// microseconds); on expiry the block records CQR_STATUS_TIMEOUT, waits
// (bounded) for its copies in flight, frees its TMEM and returns.  A
// one-shot host-side test hook (cqr_test_arm_wait_expiry) makes the next
// launch of one of the two kernels withhold the copies of one stage, with a
// short bound, so that the expiry path runs and can be checked.
#include <mutex>

#include "cqr_common.cuh"
#include "cqr.h"
#include "ozaki_value.cuh"

namespace cqr {

namespace {

constexpr int kSub = 4096;          // rows per sub-chunk (exact FP32 level sums)
constexpr int kPlanes = 11;         // balanced base-32 digits of a 54-bit magnitude and its sign
constexpr int kLevels = 2 * kPlanes - 1 - kLevelLo;
constexpr int kLowLevels = 6;       // levels of the low 64-bit group; the others form the high one
constexpr int kStage = 32;          // contraction indices per stage (one MMA K step for 8-bit types)
constexpr int kStagesPerSub = kSub / kStage;
constexpr int kExpZero = -100000;   // scale of an all-zero column
constexpr int kExpBad = 100000;     // a column holding Inf or NaN

constexpr int kTcM = 128;           // rows of the tile (X side, TMEM lanes)
constexpr int kTcN = 32;            // columns of the tile (Y side)
constexpr int kTcThreads = 512;     // warp 0 copies, warp 1 issues, all 16 run the epilogue
constexpr int kTcRing = 4;
constexpr int kTcABytes = kPlanes * kTcM * kStage;    // 45056
constexpr int kTcBBytes = kPlanes * kTcN * kStage;    // 11264
constexpr int kTcStageBytes = kTcABytes + kTcBBytes;  // 56320
constexpr int kTcSmem = kTcRing * kTcStageBytes + 1024;  // + alignment slack
constexpr uint32_t kTcCols = 512;   // TMEM columns: the levels' regions (384), rounded up to a power of 2
constexpr int kMaxDynSmem = 227 * 1024 - 1024;  // opt-in dynamic shared memory per block, less static use
static_assert(kTcSmem <= kMaxDynSmem, "projection ring fits in shared memory");
static_assert(kTcCols >= 32 && kTcCols <= 512 && (kTcCols & (kTcCols - 1)) == 0,
              "TMEM allocation: power of 2, 32..512");
constexpr int kRegionLo = kLevelLo;  // level of TMEM region 0
static_assert(kLevels * kTcN <= (int)kTcCols, "level regions fit in the TMEM allocation");
static_assert(kLevelLo == 9 && kLevels == 2 * kLowLevels, "the MMA schedule and the groups of six levels");
static_assert((long long)kPlanes * 256 * kSub < (1 << 24), "exact FP32 level sums");
// Instruction descriptor of tcgen05.mma kind::f8f6f4 without N: D f32 (bits
// 4-5 = 1), A and B e4m3 (bits 7-9, 10-12 = 0), both K-major (bits 15, 16 =
// 0), M >> 4 at bits 24-28; N >> 3 goes to bits 17-22.
constexpr uint32_t kTcIdescM = (1u << 4) | ((uint32_t)(kTcM >> 4) << 24);
constexpr unsigned long long kWaitNs = 2000000000ull;  // bound of every mbarrier wait (ns of %globaltimer)

inline int round_up(int x, int t) { return (x + t - 1) / t * t; }

// x * 2^(54 - e) rounded to an integer, plus 16 in every base-32 digit, of one
// FP64 value (raw bits b) against scale e: the fields of 5 bits (the top one
// 6) are the balanced digits plus 16.  Zeros, subnormals and the entries of a
// bad column (e far above any exponent) count as 0.
constexpr unsigned long long kDigitBias = 16ull * (((1ull << 50) - 1) / 31) + (16ull << 50);

__device__ __forceinline__ unsigned long long biased_digits(unsigned long long b, int e) {
  const uint32_t hi = (uint32_t)(b >> 32), lo = (uint32_t)b;
  const int E = (int)((hi >> 20) & 0x7FFu);
  // the mantissa with its leading one at bit 62; |x| 2^(54-e) = M 2^(E - 1031 - e), E <= e + 1022
  const unsigned long long M =
      ((unsigned long long)((__funnelshift_l(lo, hi, 10) & 0x3FFFFFFFu) | 0x40000000u) << 32) | (lo << 10);
  const int s = E ? min(e + 1030 - E, 63) : 63;
  const unsigned long long mag = ((M >> s) + 1) >> 1;
  const unsigned long long neg = (unsigned long long)((long long)b >> 63);
  return (mag ^ neg) + (kDigitBias - neg);
}

// e4m3 codes, sign and magnitude, of four digits given as bytes u = d + 16
// (0 .. 31; kTop: 0 .. 32).
template <bool kTop>
__device__ __forceinline__ uint32_t e4m3_of_digits(uint32_t u) {
  const uint32_t six = kTop ? (u >> 1) & 0x10101010u : 0u;    // d = 16
  const uint32_t n = (~(u | six) >> 4) & 0x01010101u;         // d < 0
  return ((u & 0x0F0F0F0Fu) ^ (n * 15u)) + (n * 129u + six);  // 16 - u's low bits, sign bit
}

// out[i] = byte i of w[0..3] (i < N)
template <int N>
__device__ __forceinline__ void transpose4(const uint32_t (&w)[4], uint32_t* out) {
  const uint32_t a = __byte_perm(w[0], w[1], 0x5140), c = __byte_perm(w[2], w[3], 0x5140);
  out[0] = __byte_perm(a, c, 0x5410);
  out[1] = __byte_perm(a, c, 0x7632);
  const uint32_t b = __byte_perm(w[0], w[1], 0x7362), d = __byte_perm(w[2], w[3], 0x7362);
  out[2] = __byte_perm(b, d, 0x5410);
  if (N == 4) out[3] = __byte_perm(b, d, 0x7632);
}

// The 5-bit field at bit 5 I of four values given bytewise (w[q] = byte q of
// each): one byte, or the upper bits of one and the lower of the next.
template <int I>
__device__ __forceinline__ uint32_t field(const uint32_t* w) {
  constexpr int q = 5 * I / 8, r = 5 * I % 8;
  constexpr uint32_t all = I == kPlanes - 1 ? 0x3F3F3F3Fu : 0x1F1F1F1Fu;
  if (r <= 3) return (w[q] >> r) & all;
  constexpr uint32_t low = 0x01010101u * ((1u << ((8 - r) & 7)) - 1u);
  return ((w[q] >> r) & low) | ((w[q + 1] << ((8 - r) & 7)) & (all & ~low));
}

// Digits of four FP64 values (raw bits b[0..3]) against scale e: byte k of
// word i is the e4m3 code of digit i of value k.  The fixed-point values are
// transposed bytewise first, so that every later step works on four digits at
// once: about 45 instructions a value in all (the splitting kernels are bound
// by the integer pipes; extracting the fields of each value by itself took 70).
__device__ __forceinline__ void digits4(const unsigned long long (&b)[4], int e, uint32_t (&w)[kPlanes]) {
  uint32_t lo[4], hi[4], v[8];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const unsigned long long x = biased_digits(b[k], e);
    lo[k] = (uint32_t)x;
    hi[k] = (uint32_t)(x >> 32);
  }
  transpose4<4>(lo, v);
  transpose4<3>(hi, v + 4);
  v[7] = 0u;
  w[0] = e4m3_of_digits<false>(field<0>(v));
  w[1] = e4m3_of_digits<false>(field<1>(v));
  w[2] = e4m3_of_digits<false>(field<2>(v));
  w[3] = e4m3_of_digits<false>(field<3>(v));
  w[4] = e4m3_of_digits<false>(field<4>(v));
  w[5] = e4m3_of_digits<false>(field<5>(v));
  w[6] = e4m3_of_digits<false>(field<6>(v));
  w[7] = e4m3_of_digits<false>(field<7>(v));
  w[8] = e4m3_of_digits<false>(field<8>(v));
  w[9] = e4m3_of_digits<false>(field<9>(v));
  w[10] = e4m3_of_digits<true>(field<10>(v));
}
static_assert(kPlanes == 11 && 5 * (kPlanes - 1) + 6 <= 56, "eleven fields in the first seven bytes");

// Byte offset, within one (stage, plane) block, of the 16 indices
// 16*half .. 16*half+15 of column col (canonical K-major layout).
__device__ __forceinline__ i64 plane_off(i64 col, int half) {
  return (col >> 3) * 256 + half * 128 + (col & 7) * 16;
}

// ---------------------------------------------------------------------------
// Column splitting: X (rows r0 .. r0 + nsub*kSub of an m x c matrix) ->
// planes.  Grid (ceil(c / 4), nsub), 512 threads: block (g, s) takes columns
// 4g .. 4g+3 over sub-chunk s.  Warp w takes stages 16 it + w, it = 0..7 (only
// those below nst, for the short Y of an update); lane l handles rows 4 (l mod
// 8) .. + 3 of the stage in column 4g + l / 8.  A warp load thus reads whole
// lines and a warp store writes two runs of 64 bytes of a plane (4 columns x
// 16 indices each).  Two passes over the sub-chunk: the column maxima
// (scales), then the digits; the second pass re-reads from L2 what two blocks
// an SM leave there (128 KiB each, 40 MB over the chip).
// Tiles of T columns (T a multiple of 8); plane block
// (s, tile, st, i) starts at byte
// (((s * ntile + tile) * kStagesPerSub + st) * kPlanes + i) * T * 32 with
// ntile = ceil(c / T); exps: [s * c + col].  Columns past c of the last
// group are written as zero digits (the tile padding; never read).
constexpr int kSplitCols = 4;
constexpr int kSplitWarps = 16;

// 4 consecutive entries xc[row .. row+3] (zero past m or for a column past
// c); 16-byte loads when `vec` (an odd leading dimension puts every other
// column off the 16-byte grid).
__device__ __forceinline__ void load4(const double* xc, i64 row, i64 m, bool colok, bool vec,
                                      unsigned long long (&bits)[4]) {
  if (vec && colok && row + 3 < m) {
    const double2* p = reinterpret_cast<const double2*>(xc + row);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const double2 v = __ldg(p + k);
      bits[2 * k] = (unsigned long long)__double_as_longlong(v.x);
      bits[2 * k + 1] = (unsigned long long)__double_as_longlong(v.y);
    }
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k)
      bits[k] = (unsigned long long)__double_as_longlong((colok && row + k < m) ? xc[row + k] : 0.0);
  }
}

__global__ void __launch_bounds__(32 * kSplitWarps, 2) ozaki_split_kernel(const double* X, i64 ldx, i64 m, i64 r0,
                                                                          int c, int T, int nst, uint8_t* planes,
                                                                          int* exps, const int* status) {
  stream_wait();
  if (status && *status) return;
  const int g = blockIdx.x, s = blockIdx.y, t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int cl = lane >> 3, quad = lane & 7;
  const int col = kSplitCols * g + cl;
  const bool colok = col < c;
  const i64 base = r0 + (i64)s * kSub + 4 * quad;
  const double* xc = X + (i64)(colok ? col : 0) * ldx;
  const bool vec = (ldx & 1) == 0 && (reinterpret_cast<uintptr_t>(X + r0) & 15) == 0;  // rows are multiples of 4
  // pass 1: the column's largest exponent (zeros and subnormals do not set the scale) and Inf/NaN
  int emax = 0;
#pragma unroll 4
  for (int st = warp; st < nst; st += kSplitWarps) {
    unsigned long long b[4];
    load4(xc, base + st * kStage, m, colok, vec, b);
#pragma unroll
    for (int k = 0; k < 4; ++k) emax = max(emax, (int)(b[k] >> 52) & 0x7FF);
  }
  // the eight lanes of a column
#pragma unroll
  for (int o = 1; o < 8; o *= 2) emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, o));
  __shared__ int red_max[kSplitWarps][kSplitCols];
  __shared__ int e_col[kSplitCols];
  if (quad == 0) red_max[warp][cl] = emax;
  __syncthreads();
  if (t < kSplitCols) {
    int E = 0;
    for (int w = 0; w < kSplitWarps; ++w) E = max(E, red_max[w][t]);
    // |x| < 2^(E - 1022) for biased exponent E; scale e with |x| < 2^e: e = E - 1022
    const int e = E == 0x7FF ? kExpBad : (E == 0 ? kExpZero : E - 1022);
    e_col[t] = e;
    if (kSplitCols * g + t < c) exps[(i64)s * c + kSplitCols * g + t] = e;
  }
  __syncthreads();
  const int e = e_col[cl];
  // pass 2: digits, 4 bytes per plane; the stage after the next is fetched while this one's digits are formed
  const int ntile = (c + T - 1) / T;
  uint8_t* dst = planes +
                 (((i64)s * ntile + col / T) * kStagesPerSub + warp) * kPlanes * T * kStage +
                 plane_off(col % T, quad >> 2) + 4 * (quad & 3);
  unsigned long long b[2][4];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int st = warp + h * kSplitWarps;
    load4(xc, base + st * kStage, m, colok && st < nst, vec, b[h]);
  }
#pragma unroll 1
  for (int st0 = warp; st0 < nst; st0 += 2 * kSplitWarps) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int st = st0 + h * kSplitWarps, next = st + 2 * kSplitWarps;
      uint32_t w[kPlanes];
      digits4(b[h], e, w);
      load4(xc, base + next * kStage, m, colok && next < nst, vec, b[h]);
      if (st < nst) {
#pragma unroll
        for (int i = 0; i < kPlanes; ++i) *reinterpret_cast<uint32_t*>(dst + (i64)i * T * kStage) = w[i];
      }
      dst += (i64)kSplitWarps * kPlanes * T * kStage;
    }
  }
}

// Row splitting for C -= X Y: rows r0 .. r0 + rows of X (m x K, ldx) over the
// contraction columns k0 .. k0 + kc (kc <= kSub).  Thread = row; every row
// gets its own scale over its kc entries (first pass), then its digits for
// 16 columns at a time (second pass) go to plane block (tile, st, i) at
// byte ((tile * nst + st) * kPlanes + i) * 128 * 32 with tile = row / 128,
// rows in the role of columns.  rows is a multiple of 128; rows at or past m
// split as zeros.
__global__ void __launch_bounds__(128) ozaki_rowsplit_kernel(const double* X, i64 ldx, i64 m, i64 r0, int rows,
                                                             i64 k0, int kc, uint8_t* planes, int* exps,
                                                             const int* status) {
  stream_wait();
  if (status && *status) return;
  const int row = blockIdx.x * 128 + threadIdx.x;
  if (row >= rows) return;
  const i64 r = r0 + row;
  const bool live = r < m;
  const double* xr = X + (live ? r : 0) + k0 * ldx;
  int emax = -2000;
  bool bad = false;
  if (live) {
#pragma unroll 8
    for (int k = 0; k < kc; ++k) {
      const unsigned long long b = (unsigned long long)__double_as_longlong(xr[(i64)k * ldx]);
      const int E = (int)((b >> 52) & 0x7FF);
      bad |= E == 0x7FF;
      if (E != 0 && E > emax) emax = E;
    }
  }
  const int e = bad ? kExpBad : (emax < 0 ? kExpZero : emax - 1022);
  exps[row] = e;
  const int nst = (kc + kStage - 1) / kStage;
  for (int st = 0; st < nst; ++st) {
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
      const int kb = st * kStage + 16 * h;
      uint32_t words[kPlanes][4];
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        unsigned long long b4[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int kk = kb + 4 * g + k;
          b4[k] = (unsigned long long)__double_as_longlong((live && kk < kc) ? xr[(i64)kk * ldx] : 0.0);
        }
        uint32_t w[kPlanes];
        digits4(b4, e, w);
#pragma unroll
        for (int i = 0; i < kPlanes; ++i) words[i][g] = w[i];
      }
      uint8_t* dst = planes + ((i64)(row / kTcM) * nst + st) * kTcABytes + plane_off(row % kTcM, h);
#pragma unroll
      for (int i = 0; i < kPlanes; ++i) {
        uint4 v = make_uint4(words[i][0], words[i][1], words[i][2], words[i][3]);
        *reinterpret_cast<uint4*>(dst + (i64)i * kTcM * kStage) = v;
      }
    }
  }
}

// The same for contractions of up to four stages (kc <= 128), in one pass: a
// block of nst warps takes 32 rows, warp w the 32 columns of stage w, which
// each lane keeps in registers between the maximum and the digits.  (Two
// passes re-read the rows from DRAM: the blocks in flight hold more than L2.)
constexpr int kRowStages = 4;

__global__ void __launch_bounds__(32 * kRowStages) ozaki_rowsplit_short_kernel(const double* X, i64 ldx, i64 m, i64 r0,
                                                                               i64 k0, int kc, uint8_t* planes,
                                                                               int* exps, const int* status) {
  stream_wait();
  if (status && *status) return;
  __shared__ int red[kRowStages][32];
  const int lane = threadIdx.x & 31, st = threadIdx.x >> 5, nst = blockDim.x >> 5;
  const int row = blockIdx.x * 32 + lane;
  const i64 r = r0 + row;
  const bool live = r < m;
  const double* xr = X + (live ? r : 0) + (k0 + st * kStage) * ldx;
  const int w = min(kStage, kc - st * kStage);  // live columns of the stage
  unsigned long long b[kStage];
  int emax = 0;
#pragma unroll
  for (int k = 0; k < kStage; ++k)
    b[k] = (unsigned long long)__double_as_longlong(live && k < w ? xr[(i64)k * ldx] : 0.0);
#pragma unroll
  for (int k = 0; k < kStage; ++k) emax = max(emax, (int)(b[k] >> 52) & 0x7FF);
  red[st][lane] = emax;
  __syncthreads();
  for (int q = 0; q < nst; ++q) emax = max(emax, red[q][lane]);
  const int e = emax == 0x7FF ? kExpBad : (emax == 0 ? kExpZero : emax - 1022);
  if (st == 0) exps[row] = e;
  uint8_t* dst0 = planes + ((i64)(row / kTcM) * nst + st) * kTcABytes + plane_off(row % kTcM, 0);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    uint32_t words[kPlanes][4];
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const int o = 16 * h + 4 * g;
      const unsigned long long b4[4] = {b[o], b[o + 1], b[o + 2], b[o + 3]};
      uint32_t d[kPlanes];
      digits4(b4, e, d);
#pragma unroll
      for (int i = 0; i < kPlanes; ++i) words[i][g] = d[i];
    }
#pragma unroll
    for (int i = 0; i < kPlanes; ++i)
      *reinterpret_cast<uint4*>(dst0 + 128 * h + (i64)i * kTcM * kStage) =
          make_uint4(words[i][0], words[i][1], words[i][2], words[i][3]);
  }
}

// ---------------------------------------------------------------------------
// tcgen05, TMEM, bulk copies and mbarriers (inline PTX).
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor: canonical K-major layout without
// swizzling; leading (K-direction) core-matrix offset 128 bytes, stride
// between 8-row groups 256 bytes; version 1 (bit 46).
__device__ __forceinline__ uint64_t tc_desc(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFF) >> 4) | ((uint64_t)(128 >> 4) << 16) | ((uint64_t)(256 >> 4) << 32) |
         ((uint64_t)1 << 46);
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(done)
      : "r"(bar), "r"(parity)
      : "memory");
  return done != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Wait bounded in time; false when the bound (ns) expired first.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, unsigned long long limit_ns) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = global_ns();
  for (;;) {
    if (mbar_try_wait(bar, parity)) return true;
    if (global_ns() - t0 > limit_ns) return false;
  }
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
// D (TMEM) = A x B^T (acc = 0) or D += A x B^T (acc = 1), N = 32 * nb
__device__ __forceinline__ void tc_mma(uint32_t d, uint64_t ad, uint64_t bd, int nb, uint32_t acc) {
  const uint32_t idesc = kTcIdescM | ((uint32_t)(kTcN * nb >> 3) << 17);
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
      "l"(ad), "l"(bd), "r"(idesc), "r"(acc));
}

// The MMA schedule of one stage: (plane i of X, first plane j0 of Y, count n).
// The first three write every region (levels 9..20) without overlap, so in the
// first stage of a tile they run with acc = 0 and initialise the accumulators.
// An instruction reads 4 KiB of X and n KiB of Y from shared memory (128 B per
// clock) for 16 n clocks of arithmetic, so the splits are even: 5 + 4 rather
// than 8 + 1.
struct TcMma {
  int i, j0, n;
};
constexpr int kTcMmas = 16, kTcInit = 3;
#define CQR_TC_SCHEDULE                                                                \
  {10, 0, 6}, {10, 6, 5}, {9, 0, 1},                              /* every level once */ \
      {9, 1, 5}, {9, 6, 5}, {8, 1, 5}, {8, 6, 5}, {7, 2, 5}, {7, 7, 4}, /* j >= 9 - i */  \
      {6, 3, 8}, {5, 4, 7}, {4, 5, 6}, {3, 6, 5}, {2, 7, 4}, {1, 8, 3}, {0, 9, 2}
__device__ constexpr TcMma kTcSchedule[kTcMmas] = {CQR_TC_SCHEDULE};

// Compile-time check of the same entries: every digit pair (i, j) of a kept
// level exactly once and no other, every instruction within the planes,
// N = 32 n <= 256, every region in TMEM, and the first kTcInit instructions
// writing each region exactly once (they run with the accumulate flag off).
constexpr TcMma kTcScheduleCheck[kTcMmas] = {CQR_TC_SCHEDULE};
constexpr bool tc_schedule_ok() {
  int count[kPlanes][kPlanes] = {};
  int first[kLevels] = {};
  for (int u = 0; u < kTcMmas; ++u) {
    const TcMma e = kTcScheduleCheck[u];
    if (e.i < 0 || e.i >= kPlanes || e.j0 < 0 || e.n < 1 || e.j0 + e.n > kPlanes || kTcN * e.n > 256) return false;
    for (int v = 0; v < e.n; ++v) {
      const int j = e.j0 + v, region = e.i + j - kRegionLo;
      if (region < 0 || region >= kLevels) return false;
      ++count[e.i][j];
      if (u < kTcInit) ++first[region];
    }
  }
  for (int i = 0; i < kPlanes; ++i)
    for (int j = 0; j < kPlanes; ++j)
      if (count[i][j] != (i + j >= kLevelLo ? 1 : 0)) return false;
  for (int r = 0; r < kLevels; ++r)
    if (first[r] != 1) return false;
  return true;
}
static_assert(tc_schedule_ok(),
              "MMA schedule: kept pairs once, regions in range, the first ones initialise the regions");
#undef CQR_TC_SCHEDULE
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// 4 consecutive 32-bit TMEM columns of this thread's lane
__device__ __forceinline__ void tc_ld4(uint32_t taddr, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
}
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Contraction length up to which every level sum is below 2^22 units (11
// pairs x 256 x K < 2^22): then the FP32 value f (a multiple of 2^-18) is read
// exactly as bits(f + 48) - bits(48), one full-rate FP32 add and integer
// arithmetic, instead of a quarter-rate conversion.
constexpr int kMagicMaxK = 1312;
static_assert(kPlanes * 256 * kMagicMaxK < (1 << 22), "level sums below 2^22");
constexpr float kMagicF = 48.0f;        // 1.5 * 2^5: steps of 2^-18
constexpr int kMagicBits = 0x42400000;  // its encoding

// Columns of the epilogue's register step; warps that read one TMEM lane
// quarter (each takes kEpiCols columns of the tile), of 16 epilogue warps.
constexpr int kEpiStep = 4, kEpiCols = 8;
constexpr int kEpiWarps = 4 * (kTcN / kEpiCols);

// The level sums of columns c0 .. c0+3 of this thread's TMEM lane.
__device__ __forceinline__ void load_levels(uint32_t lane_base, int c0, uint32_t (&v)[kLevels][kEpiStep]) {
#pragma unroll
  for (int l = 0; l < kLevels; ++l) tc_ld4(lane_base + (uint32_t)((kLevelLo - kRegionLo + l) * kTcN + c0), v[l]);
  tc_wait_ld();
}

// g0 = sum_{l < 6} s_l 32^l and g1 = sum_{l >= 6} s_l 32^(l - 6) of column j's
// level sums s_l (integers).  kMagic (|s_l| < 2^22): neighbouring levels first
// combine in unsigned 32-bit arithmetic (the offsets cancel modulo 2^32 and
// |s_l + 32 s_l+1| < 2^28, so the two's-complement reading is the value).
template <bool kMagic>
__device__ __forceinline__ void group_sums(const uint32_t (&v)[kLevels][kEpiStep], int j, long long& g0,
                                           long long& g1) {
  if (kMagic) {
    uint32_t b[kLevels];
#pragma unroll
    for (int l = 0; l < kLevels; ++l) b[l] = __float_as_uint(__fadd_rn(__uint_as_float(v[l][j]), kMagicF));
    const uint32_t off = 33u * (uint32_t)kMagicBits;  // modulo 2^32
    auto two = [&](int l) { return (long long)(int)(b[l] + 32u * b[l + 1] - off); };
    g0 = two(4) * 1048576 + (two(2) * 1024 + two(0));
    g1 = two(10) * 1048576 + (two(8) * 1024 + two(6));
  } else {
    auto lev = [&](int l) { return (long long)__float2int_rz(__uint_as_float(v[l][j]) * 262144.0f); };
    g0 = g1 = 0;
#pragma unroll
    for (int l = kLowLevels - 1; l >= 0; --l) g0 = g0 * 32 + lev(l);
#pragma unroll
    for (int l = kLevels - 1; l >= kLowLevels; --l) g1 = g1 * 32 + lev(l);
  }
}

struct OzArgs {
  const uint8_t* px;  // planes of X (the tile's rows: projection columns p / update rows)
  const uint8_t* py;  // planes of Y (the tile's columns q)
  const int* ex;
  const int* ey;
  int p, q;           // extents (projection: p x q; update: rows of the chunk x N)
  int tiles_p;        // tiles of X in the plane layout (projection: per sub-chunk)
  int y_in_x;         // projection X^T X: the Y tiles are read from the X planes (32-column slices)
  int nst;            // stages per tile (projection: kStagesPerSub)
  int tiles_q;
  int s_off;          // projection: sub-chunk index offset of this launch in the partial buffer
  double* part;       // projection: [s][p * q] column-major p x q
  double* C;          // update: C (ldc) of the chunk's first row
  i64 ldc;
  int* status;
  unsigned long long wait_ns;  // bound of every mbarrier wait (kWaitNs unless the test hook is armed)
  int withhold;                // test hook: the producer issues no copies from this stage on (-1: none)
};

// Projections: one 128 x 32 tile of one sub-chunk per block, grid
// (tiles_q, tiles_p, nsub) with the q tile fastest (the blocks running
// together share the X planes of a sub-chunk in L2); the tile goes to the
// sub-chunk's partial.
__global__ void __launch_bounds__(kTcThreads, 1) ozaki_tc_kernel(OzArgs a) {
  stream_wait();
  extern __shared__ uint8_t tc_raw[];
  __shared__ __align__(8) uint64_t full_bar[kTcRing], empty_bar[kTcRing], done_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ int give_up;
  if (a.status && *a.status) return;  // uniform across the block, before any allocation
  const int q0 = blockIdx.x * kTcN, p0 = blockIdx.y * kTcM, s = blockIdx.z;
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  uint8_t* ring = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(tc_raw) + 1023) & ~(uintptr_t)1023);
  // scales of the epilogue, fetched first so that their latency hides behind the contraction
  __shared__ int ey_s[kTcN];
  const int r = 32 * (warp & 3) + lane;  // tile row = TMEM lane
  const int pr = p0 + r;
  const bool live = pr < a.p;
  const int exr = live ? a.ex[(i64)s * a.p + pr] : kExpZero;
  if (t < kTcN) ey_s[t] = q0 + t < a.q ? a.ey[(i64)s * a.q + q0 + t] : kExpZero;
  if (t == 0) {
    for (int i = 0; i < kTcRing; ++i) {
      mbar_init(smem_u32(&full_bar[i]), 1);
      mbar_init(smem_u32(&empty_bar[i]), 1);
    }
    mbar_init(smem_u32(&done_bar), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    give_up = 0;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(kTcCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  const int nst = a.nst;
  // this tile's stages: tile-major plane layout, kStagesPerSub stages per (sub-chunk, tile)
  const uint8_t* gx = a.px + ((i64)s * a.tiles_p + p0 / kTcM) * kStagesPerSub * kTcABytes;
  // Y tile: its own planes, or (X^T X) the 32-column slice q0 of the X tile holding it
  const uint8_t* gy = a.y_in_x ? a.px + ((i64)s * a.tiles_p + q0 / kTcM) * kStagesPerSub * kTcABytes +
                                     (i64)(q0 % kTcM) * kStage
                               : a.py + ((i64)s * a.tiles_q + q0 / kTcN) * kStagesPerSub * kTcBBytes;

  if (warp == 0 && lane == 0) {
    // producer: bulk copies of stage st into ring slot st % kTcRing
    int issued = 0;
    for (int st = 0; st < nst; ++st) {
      const int slot = st % kTcRing;
      if (st >= kTcRing && !mbar_wait(smem_u32(&empty_bar[slot]), (uint32_t)((st / kTcRing - 1) & 1), a.wait_ns)) {
        atomicExch(&give_up, 1);
        break;
      }
      if (*(volatile int*)&give_up || st == a.withhold) break;
      const uint32_t fb = smem_u32(&full_bar[slot]);
      const uint32_t sa = smem_u32(ring + slot * kTcStageBytes), sb = sa + kTcABytes;
      mbar_expect_tx(fb, kTcStageBytes);
      bulk_g2s(sa, gx + (i64)st * kTcABytes, kTcABytes, fb);
      if (a.y_in_x) {
#pragma unroll 1
        for (int i = 0; i < kPlanes; ++i)
          bulk_g2s(sb + i * (kTcN * kStage), gy + (i64)st * kTcABytes + i * (kTcM * kStage), kTcN * kStage, fb);
      } else {
        bulk_g2s(sb, gy + (i64)st * kTcBBytes, kTcBBytes, fb);
      }
      issued = st + 1;
    }
    // before leaving, every issued copy must have landed (bounded)
    for (int st = issued - kTcRing < 0 ? 0 : issued - kTcRing; st < issued; ++st)
      mbar_wait(smem_u32(&full_bar[st % kTcRing]), (uint32_t)((st / kTcRing) & 1), a.wait_ns);
  } else if (warp == 1 && lane == 0) {
    // MMA issuer: the 16 instructions of each stage (the 76 pairs, level L = i + j into region L - 9)
    for (int st = 0; st < nst; ++st) {
      const int slot = st % kTcRing;
      if (!mbar_wait(smem_u32(&full_bar[slot]), (uint32_t)((st / kTcRing) & 1), a.wait_ns)) {
        atomicExch(&give_up, 1);
        break;
      }
      if (*(volatile int*)&give_up) break;
      tc_fence_after();
      const uint32_t sa = smem_u32(ring + slot * kTcStageBytes), sb = sa + kTcABytes;
      const uint64_t ad0 = tc_desc(sa), bd0 = tc_desc(sb);
#pragma unroll
      for (int u = 0; u < kTcMmas; ++u) {
        const TcMma e = kTcSchedule[u];
        const uint64_t ad = ad0 + (uint64_t)((e.i * kTcM * kStage) >> 4);
        const uint64_t bd = bd0 + (uint64_t)((e.j0 * kTcN * kStage) >> 4);
        tc_mma(tmem + (uint32_t)((e.i + e.j0 - kRegionLo) * kTcN), ad, bd, e.n, (st > 0 || u >= kTcInit) ? 1u : 0u);
      }
      tc_commit(smem_u32(&empty_bar[slot]));
    }
    tc_commit(smem_u32(&done_bar));  // arrives when every MMA issued above has completed
  }
  __syncwarp();
  const bool done = mbar_wait(smem_u32(&done_bar), 0, a.wait_ns);
  // one decision for the whole block, and converged warps for tcgen05.ld
  const int failed = __syncthreads_or(!done || *(volatile int*)&give_up);
  tc_fence_after();
  if (failed) {
    if (t == 0 && a.status) atomicCAS(a.status, 0, CQR_STATUS_TIMEOUT);
  } else {
    // epilogue: row r of the tile (TMEM lane r), this warp's columns
    const uint32_t lane_base = tmem + ((uint32_t)(32 * (warp & 3)) << 16);
    const int cw = kEpiCols * (warp >> 2);
#pragma unroll
    for (int c0 = cw; c0 < cw + kEpiCols; c0 += kEpiStep) {
      uint32_t v[kLevels][kEpiStep];
      load_levels(lane_base, c0, v);
#pragma unroll
      for (int j = 0; j < kEpiStep; ++j) {
        const int qc = q0 + c0 + j;
        if (!live || qc >= a.q) continue;
        const int eyc = ey_s[c0 + j];
        double x;
        if (exr == kExpBad || eyc == kExpBad) {
          x = __longlong_as_double(0x7ff8000000000000LL);
        } else if (exr == kExpZero || eyc == kExpZero) {
          x = 0.0;
        } else {
          long long g0, g1;
          group_sums<false>(v, j, g0, g1);
          x = group_value(g0, g1, exr + eyc);
        }
        a.part[(i64)(a.s_off + s) * a.p * a.q + pr + (i64)qc * a.p] = x;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTcCols));
}

// ---------------------------------------------------------------------------
// Updates C -= X Y as a persistent, warp-specialised kernel.  Warp 0 streams
// the stages of the block's tiles into two rings of four slots, one for X (44
// KiB each) and one for Y (11 KiB each), warp
// 1 issues the MMAs of a tile into the one set of TMEM level regions, and
// warps 2-17 (TMEM lane quarter warp mod 4, eight columns each) run the
// epilogue in two phases:
// first the level sums become the exact 64-bit group sums, kept in registers
// (two per column of the thread's row), and the regions are handed back to
// warp 1 at once; then, while the next tile's MMAs run, the group sums are
// scaled, added and subtracted from C, whose entries were fetched before the
// wait for the MMAs.  The epilogue is about 120 instructions per entry, long
// chains of integer operations: with one warp per lane quarter (one per
// scheduler) it took 27000 clocks a tile, five times the MMAs.  A tile of K =
// 128 now takes 5.9 us, the MMAs (3.3) and the first phase one after the other.
// Two sets of regions with 16-column tiles do not overlap them either (8.2 us
// for 32 columns, the MMAs re-read X twice as often), nor does holding the
// second phases back until all first ones are done.
//
// Tile T is row tile T / tiles_q, column tile T % tiles_q.  X is four
// fifths of a stage's bytes.  Contractions of up to four stages (K <= 128:
// every product with one panel) therefore keep the row tile's X stages in their four slots while the
// block, which takes a contiguous run of tiles, goes through its column
// tiles.  Longer contractions stream X with Y, and block c takes tiles c,
// c + G, c + 2G, ... (G = grid size), so that the blocks running together
// share row tiles in L2.
constexpr int kUpRing = 4;
constexpr int kUpThreads = 64 + 32 * kEpiWarps;
constexpr int kUpSmem = 1024 + kUpRing * kTcStageBytes;  // X slots, then Y slots
static_assert(kUpSmem <= kMaxDynSmem, "update ring fits in shared memory");

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

template <bool kMagic>
__global__ void __launch_bounds__(kUpThreads, 1) ozaki_tc_update_kernel(OzArgs a, int ntiles) {
  stream_wait();
  extern __shared__ uint8_t up_raw[];
  __shared__ __align__(8) uint64_t full_a[kUpRing], empty_a[kUpRing], full_b[kUpRing], empty_b[kUpRing];
  __shared__ __align__(8) uint64_t acc_full, acc_empty, mma_done;
  __shared__ uint32_t tmem_slot;
  __shared__ int give_up;
  if (a.status && *a.status) return;  // uniform across the block, before any allocation
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  uint8_t* ring = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(up_raw) + 1023) & ~(uintptr_t)1023);
  if (t == 0) {
    for (int i = 0; i < kUpRing; ++i) {
      mbar_init(smem_u32(&full_a[i]), 1);
      mbar_init(smem_u32(&empty_a[i]), 1);
      mbar_init(smem_u32(&full_b[i]), 1);
      mbar_init(smem_u32(&empty_b[i]), 1);
    }
    mbar_init(smem_u32(&acc_full), 1);
    mbar_init(smem_u32(&acc_empty), kEpiWarps);  // one arrival per epilogue warp
    mbar_init(smem_u32(&mma_done), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    give_up = 0;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(kTcCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  const int nst = a.nst;
  const bool keep_x = nst <= kUpRing;
  // this block's tiles: t_first, t_first + t_step, .. below t_last
  const int t_step = keep_x ? 1 : (int)gridDim.x;
  const int t_first = keep_x ? (int)((i64)blockIdx.x * ntiles / gridDim.x) : (int)blockIdx.x;
  const int t_last = keep_x ? (int)((i64)(blockIdx.x + 1) * ntiles / gridDim.x) : ntiles;
  const uint32_t xs = smem_u32(ring), ys = xs + kUpRing * kTcABytes;

  if (warp == 0) {
    if (lane == 0) {  // producer
      int ga = 0, gb = 0;  // X and Y stages issued; X stage h goes to slot h % nst (kept) or h % kUpRing
      const int xr = keep_x ? nst : kUpRing;
      bool stop = false;
      for (int T = t_first; T < t_last && !stop; T += t_step) {
        // tile-major planes: nst stages per X tile, kStagesPerSub per Y tile
        const uint8_t* gx = a.px + (i64)(T / a.tiles_q) * nst * kTcABytes;
        const uint8_t* gy = a.py + (i64)(T % a.tiles_q) * kStagesPerSub * kTcBBytes;
        const bool load_x = !keep_x || T == t_first || T % a.tiles_q == 0;
        for (int st = 0; st < nst; ++st) {
          const int sa = ga % xr, sb = gb % kUpRing;
          if ((load_x && ga >= xr && !mbar_wait(smem_u32(&empty_a[sa]), (uint32_t)((ga / xr - 1) & 1), a.wait_ns)) ||
              (gb >= kUpRing && !mbar_wait(smem_u32(&empty_b[sb]), (uint32_t)((gb / kUpRing - 1) & 1), a.wait_ns))) {
            atomicExch(&give_up, 1);
            stop = true;
            break;
          }
          if (*(volatile int*)&give_up || gb == a.withhold) {
            stop = true;
            break;
          }
          if (load_x) {
            const uint32_t fa = smem_u32(&full_a[sa]);
            mbar_expect_tx(fa, kTcABytes);
            bulk_g2s(xs + sa * kTcABytes, gx + (i64)st * kTcABytes, kTcABytes, fa);
            ++ga;
          }
          const uint32_t fb = smem_u32(&full_b[sb]);
          mbar_expect_tx(fb, kTcBBytes);
          bulk_g2s(ys + sb * kTcBBytes, gy + (i64)st * kTcBBytes, kTcBBytes, fb);
          ++gb;
        }
      }
      // every issued copy must have landed before the block leaves (bounded)
      for (int h = ga - xr < 0 ? 0 : ga - xr; h < ga; ++h)
        mbar_wait(smem_u32(&full_a[h % xr]), (uint32_t)((h / xr) & 1), a.wait_ns);
      for (int h = gb - kUpRing < 0 ? 0 : gb - kUpRing; h < gb; ++h)
        mbar_wait(smem_u32(&full_b[h % kUpRing]), (uint32_t)((h / kUpRing) & 1), a.wait_ns);
    }
  } else if (warp == 1) {
    if (lane == 0) {  // MMA issuer
      int ga = 0, gb = 0, k = 0;  // X stage of the tile's first one (kept) or of this one; Y stage; tile
      const int xr = keep_x ? nst : kUpRing;
      bool stop = false;
      for (int T = t_first; T < t_last && !stop; T += t_step, ++k) {
        if (k >= 1 && !mbar_wait(smem_u32(&acc_empty), (uint32_t)((k - 1) & 1), a.wait_ns)) {
          atomicExch(&give_up, 1);
          break;
        }
        tc_fence_after();
        const bool free_x = !keep_x || T + 1 == t_last || (T + 1) % a.tiles_q == 0;
        for (int st = 0; st < nst; ++st) {
          const int ha = keep_x ? ga + st : ga;
          const int sa = ha % xr, sb = gb % kUpRing;
          if (!mbar_wait(smem_u32(&full_a[sa]), (uint32_t)((ha / xr) & 1), a.wait_ns) ||
              !mbar_wait(smem_u32(&full_b[sb]), (uint32_t)((gb / kUpRing) & 1), a.wait_ns) ||
              *(volatile int*)&give_up) {
            atomicExch(&give_up, 1);
            stop = true;
            break;
          }
          tc_fence_after();
          const uint64_t ad0 = tc_desc(xs + sa * kTcABytes), bd0 = tc_desc(ys + sb * kTcBBytes);
#pragma unroll
          for (int u = 0; u < kTcMmas; ++u) {
            const TcMma e = kTcSchedule[u];
            const uint64_t ad = ad0 + (uint64_t)((e.i * kTcM * kStage) >> 4);
            const uint64_t bd = bd0 + (uint64_t)((e.j0 * kTcN * kStage) >> 4);
            tc_mma(tmem + (uint32_t)((e.i + e.j0 - kRegionLo) * kTcN), ad, bd, e.n, (st > 0 || u >= kTcInit) ? 1u : 0u);
          }
          if (free_x) tc_commit(smem_u32(&empty_a[sa]));
          tc_commit(smem_u32(&empty_b[sb]));
          if (!keep_x) ++ga;
          ++gb;
        }
        if (keep_x && free_x) ga += nst;
        tc_commit(smem_u32(&acc_full));
      }
      tc_commit(smem_u32(&mma_done));  // every MMA issued above has completed when this arrives
      mbar_wait(smem_u32(&mma_done), 0, a.wait_ns);
    }
  } else {
    // epilogue: TMEM lane quarter qw, tile row r, columns cw .. cw + 7
    const int qw = warp & 3, r = 32 * qw + lane, cw = kEpiCols * ((warp - 2) >> 2);
    const uint32_t lane_base = tmem + ((uint32_t)(32 * qw) << 16);
    int k = 0;
    for (int T = t_first; T < t_last; T += t_step, ++k) {
      const int pr = (T / a.tiles_q) * kTcM + r, q0 = (T % a.tiles_q) * kTcN + cw;
      const bool live = pr < a.p;
      double* C = a.C + pr + (i64)q0 * a.ldc;
      const int exr = live ? a.ex[pr] : kExpZero;
      int eyc[kEpiCols];
      double cv[kEpiCols];
#pragma unroll
      for (int j = 0; j < kEpiCols; ++j) {
        const bool ok = live && q0 + j < a.q;
        eyc[j] = ok ? a.ey[q0 + j] : kExpZero;
        cv[j] = ok ? C[(i64)j * a.ldc] : 0.0;
      }
      const bool ok = mbar_wait(smem_u32(&acc_full), (uint32_t)(k & 1), a.wait_ns);
      if (!__all_sync(0xffffffffu, ok) || __any_sync(0xffffffffu, *(volatile int*)&give_up)) {
        atomicExch(&give_up, 1);
        break;
      }
      tc_fence_after();
      // phase 1: level sums -> exact group sums g0 (levels 9..14), g1 (15..20), kept in registers
      long long g0[kEpiCols], g1[kEpiCols];
#pragma unroll
      for (int c0 = 0; c0 < kEpiCols; c0 += kEpiStep) {
        uint32_t v[kLevels][kEpiStep];
        load_levels(lane_base, cw + c0, v);
#pragma unroll
        for (int j = 0; j < kEpiStep; ++j) group_sums<kMagic>(v, j, g0[c0 + j], g1[c0 + j]);
      }
      // hand the regions back to the MMA warp (the next tile's first stage overwrites them)
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&acc_empty));
      // phase 2 (overlaps the next tile's MMAs): scale, add the two groups, subtract from C
#pragma unroll
      for (int j = 0; j < kEpiCols; ++j) {
        if (!live || q0 + j >= a.q) continue;
        double v;
        if (exr == kExpBad || eyc[j] == kExpBad) {
          v = __longlong_as_double(0x7ff8000000000000LL);
        } else if (exr == kExpZero || eyc[j] == kExpZero) {
          v = 0.0;
        } else {
          v = group_value(g0[j], g1[j], exr + eyc[j]);
        }
        C[(i64)j * a.ldc] = cv[j] - v;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (t == 0 && give_up && a.status) atomicCAS(a.status, 0, CQR_STATUS_TIMEOUT);
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTcCols));
}

// C = sum of the sub-chunks' partials, 16 entries per block (split_sum16).
__global__ void __launch_bounds__(256) ozaki_reduce_kernel(const double* part, i64 nsub, int p, int q, double* C,
                                                           i64 ldc, const int* status) {
  stream_wait();
  __shared__ double red[16 * 17];
  if (status && *status) return;
  const i64 pq = (i64)p * q, e = (i64)blockIdx.x * 16 + (threadIdx.x & 15);
  const bool live = e < pq;
  const double s = split_sum16(nsub, live, red, [=](i64 k) { return part[k * pq + e]; });
  if (threadIdx.x < 16 && live) C[e % p + (e / p) * ldc] = s;
}

void up_attr() {
  static PerDevice<bool> done;
  if (bool& set = done.here(); !set) {
    cudaFuncSetAttribute(ozaki_tc_update_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kUpSmem);
    cudaFuncSetAttribute(ozaki_tc_update_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kUpSmem);
    set = true;
  }
}

void tc_attr() {
  static PerDevice<bool> done;
  if (bool& set = done.here(); !set) {
    cudaFuncSetAttribute(ozaki_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kTcSmem);
    set = true;
  }
}

// One-shot test hook of the bounded waits (cqr_test_arm_wait_expiry): the
// next launch of kernel `g_fault_kernel` (0 = ozaki_tc_kernel, 1 =
// ozaki_tc_update_kernel) gets the armed stage to withhold and wait bound,
// then the hook disarms itself.
std::mutex g_fault_mu;
int g_fault_kernel = -1, g_fault_stage = -1;
unsigned long long g_fault_ns = 0;

void take_fault(int kernel, OzArgs& a) {
  a.wait_ns = kWaitNs;
  a.withhold = -1;
  std::lock_guard<std::mutex> lk(g_fault_mu);
  if (g_fault_kernel == kernel) {
    a.wait_ns = g_fault_ns;
    a.withhold = g_fault_stage;
    g_fault_kernel = -1;
  }
}

// Rows per update chunk: the X planes of one chunk take about 1 GiB.
inline i64 oz_nn_rows(int nst) {
  i64 rows = ((i64)1 << 30) / ((i64)kPlanes * kStage * nst);
  rows = rows / kTcM * kTcM;
  return rows < kTcM ? kTcM : rows;
}

}  // namespace

// Rows per splitting chunk of a projection: planes of one chunk take 1 to
// 2 GiB.  A launch has (column tiles) x (sub-chunks) blocks of equal length,
// one per SM, so a partly filled last wave costs a whole one; of the
// sub-chunk counts between the 1 GiB budget and twice it, the one with the
// fewest waves per sub-chunk is taken (the smallest among equals).
i64 oz_chunk_rows(int p, int q) {
  const i64 cpx = round_up(p, kTcM), cpy = round_up(q, kTcN);
  i64 base = ((i64)1 << 30) / ((i64)kPlanes * (cpx + cpy) * kSub);
  if (base < 1) base = 1;
  const i64 tiles = (cpx / kTcM) * (cpy / kTcN);
  i64 best = base;
  for (i64 n = base + 1; n <= 2 * base; ++n) {
    // waves(n) / n < waves(best) / best, in integers
    const i64 wn = (tiles * n + kSMs - 1) / kSMs, wb = (tiles * best + kSMs - 1) / kSMs;
    if (wn * best < wb * n) best = n;
  }
  return best * kSub;
}

size_t ozaki_workspace_bytes(i64 m, int p, int q) {
  if (m <= 0 || p <= 0 || q <= 0) return 0;
  const int cpx = round_up(p, kTcM), cpy = round_up(q, kTcN);
  const i64 nsub_total = (m + kSub - 1) / kSub;
  i64 ch = oz_chunk_rows(p, q);
  const i64 mr = nsub_total * kSub;
  if (ch > mr) ch = mr;
  const i64 nsub_ch = ch / kSub;
  size_t b = 0;
  b += (size_t)nsub_ch * kPlanes * (cpx + cpy) * kSub;        // planes of one chunk
  b = (b + 255) & ~(size_t)255;
  b += sizeof(int) * (size_t)nsub_ch * (p + q);               // scales
  b = (b + 255) & ~(size_t)255;
  b += sizeof(double) * (size_t)nsub_total * p * q;           // partials
  return (b + 255) & ~(size_t)255;
}

cudaError_t tn_product_emulated(i64 m, int p, int q, const double* X, i64 ldx, const double* Y, i64 ldy,
                                void* ws, double* C, i64 ldc, const int* status, cudaStream_t st) {
  if (p <= 0 || q <= 0) return cudaSuccess;
  const int cpx = round_up(p, kTcM), cpy = round_up(q, kTcN);
  const i64 nsub_total = (m + kSub - 1) / kSub;
  i64 ch = oz_chunk_rows(p, q);
  const i64 mr = nsub_total * kSub;
  if (ch > mr) ch = mr;
  const i64 nsub_ch = ch / kSub;
  uint8_t* planes = (uint8_t*)ws;
  size_t off = (size_t)nsub_ch * kPlanes * (cpx + cpy) * kSub;
  off = (off + 255) & ~(size_t)255;
  int* exps = (int*)((char*)ws + off);
  off += sizeof(int) * (size_t)nsub_ch * (p + q);
  off = (off + 255) & ~(size_t)255;
  double* part = (double*)((char*)ws + off);
  tc_attr();
  uint8_t* px = planes;
  uint8_t* py = planes + (size_t)nsub_ch * kPlanes * cpx * kSub;
  int* ex = exps;
  int* ey = exps + nsub_ch * p;
  const int tiles_p = cpx / kTcM, tiles_q = cpy / kTcN;
  const bool same = X == Y && ldx == ldy && p == q;  // X^T X: split once
  for (i64 r0 = 0; r0 < m; r0 += ch) {
    const i64 nsub = ((m - r0 < ch ? m - r0 : ch) + kSub - 1) / kSub;
    prof_begin(kMisc, st);
    launch(ozaki_split_kernel, dim3((unsigned)((p + kSplitCols - 1) / kSplitCols), (unsigned)nsub), 32 * kSplitWarps,
           0, st, X, ldx, m, r0, p, kTcM, kStagesPerSub, px, ex, status);
    prof_end(kMisc, 0.0, st);
    if (!same) {
      prof_begin(kMisc, st);
      launch(ozaki_split_kernel, dim3((unsigned)((q + kSplitCols - 1) / kSplitCols), (unsigned)nsub),
             32 * kSplitWarps, 0, st, Y, ldy, m, r0, q, kTcN, kStagesPerSub, py, ey, status);
      prof_end(kMisc, 0.0, st);
    }
    OzArgs a{};
    a.px = px;
    a.py = same ? px : py;
    a.ex = ex;
    a.ey = same ? ex : ey;
    a.p = p;
    a.q = q;
    a.tiles_p = tiles_p;
    a.y_in_x = same ? 1 : 0;
    a.nst = kStagesPerSub;
    a.tiles_q = tiles_q;
    a.s_off = (int)(r0 / kSub);
    a.part = part;
    a.status = const_cast<int*>(status);
    take_fault(0, a);
    prof_begin(kProjection, st);
    launch(ozaki_tc_kernel, dim3((unsigned)tiles_q, (unsigned)tiles_p, (unsigned)nsub), kTcThreads, kTcSmem, st, a);
    prof_end(kProjection, 2.0 * (double)(nsub * kSub < m - r0 ? nsub * kSub : m - r0) * p * q, st);
  }
  const i64 pq = (i64)p * q;
  prof_begin(kReduce, st);
  launch(ozaki_reduce_kernel, (unsigned)((pq + 15) / 16), 256, 0, st, part, nsub_total, p, q, C, ldc, status);
  prof_end(kReduce, (double)nsub_total * pq, st);
  return cudaGetLastError();
}

size_t ozaki_nn_workspace_bytes(i64 M, int N, int K) {
  if (M <= 0 || N <= 0 || K <= 0) return 0;
  const int kc = K < kSub ? K : kSub;
  const int nst = (kc + kStage - 1) / kStage;
  const int cpy = round_up(N, kTcN);
  i64 rows = oz_nn_rows(nst);
  const i64 mr = (M + kTcM - 1) / kTcM * kTcM;
  if (rows > mr) rows = mr;
  size_t b = (size_t)rows * nst * kStage * kPlanes;  // X planes of one chunk
  b = (b + 255) & ~(size_t)255;
  b += (size_t)kSub * kPlanes * cpy;                 // Y planes (one sub-chunk)
  b = (b + 255) & ~(size_t)255;
  b += sizeof(int) * ((size_t)rows + N);             // scales
  return (b + 255) & ~(size_t)255;
}

cudaError_t nn_update_emulated(i64 M, int N, int K, const double* X, i64 ldx, const double* Y, i64 ldy, double* C,
                               i64 ldc, void* ws, const int* status, cudaStream_t st) {
  if (M <= 0 || N <= 0 || K <= 0) return cudaSuccess;
  const int kcmax = K < kSub ? K : kSub;
  const int nstmax = (kcmax + kStage - 1) / kStage;
  const int cpy = round_up(N, kTcN);
  i64 rows = oz_nn_rows(nstmax);
  const i64 mr = (M + kTcM - 1) / kTcM * kTcM;
  if (rows > mr) rows = mr;
  uint8_t* px = (uint8_t*)ws;
  size_t off = ((size_t)rows * nstmax * kStage * kPlanes + 255) & ~(size_t)255;
  uint8_t* py = (uint8_t*)ws + off;
  off = (off + (size_t)kSub * kPlanes * cpy + 255) & ~(size_t)255;
  int* ex = (int*)((char*)ws + off);
  int* ey = ex + rows;
  up_attr();
  const int tiles_q = cpy / kTcN;
  for (i64 k0 = 0; k0 < K; k0 += kSub) {
    const int kc = (int)(K - k0 < kSub ? K - k0 : kSub);
    const int nst = (kc + kStage - 1) / kStage;
    prof_begin(kMisc, st);
    launch(ozaki_split_kernel, dim3((unsigned)((N + kSplitCols - 1) / kSplitCols), 1u), 32 * kSplitWarps, 0, st, Y, ldy,
           k0 + kc, k0, N, kTcN, nst, py, ey, status);
    prof_end(kMisc, 0.0, st);
    for (i64 r0 = 0; r0 < M; r0 += rows) {
      const i64 live = M - r0 < rows ? M - r0 : rows;
      const int rws = (int)((live + kTcM - 1) / kTcM * kTcM);
      prof_begin(kMisc, st);
      if (nst <= kRowStages)
        launch(ozaki_rowsplit_short_kernel, (unsigned)(rws / 32), 32 * nst, 0, st, X, ldx, M, r0, k0, kc, px, ex,
               status);
      else
        launch(ozaki_rowsplit_kernel, (unsigned)(rws / 128), 128, 0, st, X, ldx, M, r0, rws, k0, kc, px, ex, status);
      prof_end(kMisc, 0.0, st);
      OzArgs a{};
      a.px = px;
      a.py = py;
      a.ex = ex;
      a.ey = ey;
      a.p = (int)live;
      a.q = N;
      a.tiles_p = rws / kTcM;
      a.nst = nst;
      a.tiles_q = tiles_q;
      a.C = C + r0;
      a.ldc = ldc;
      a.status = const_cast<int*>(status);
      take_fault(1, a);
      const int ntiles = (rws / kTcM) * tiles_q;
      prof_begin(kUpdate, st);
      const unsigned grid = (unsigned)(ntiles < kSMs ? ntiles : kSMs);
      if (nst * kStage <= kMagicMaxK)
        launch(ozaki_tc_update_kernel<true>, grid, kUpThreads, kUpSmem, st, a, ntiles);
      else
        launch(ozaki_tc_update_kernel<false>, grid, kUpThreads, kUpSmem, st, a, ntiles);
      prof_end(kUpdate, 2.0 * (double)live * N * kc, st);
    }
  }
  return cudaGetLastError();
}

}  // namespace cqr

extern "C" int cqr_test_arm_wait_expiry(int kernel, int stage, long long wait_ns) {
  if (kernel < -1 || kernel > 1) return -1;
  if (kernel == -1) {  // disarm
    std::lock_guard<std::mutex> lk(cqr::g_fault_mu);
    cqr::g_fault_kernel = -1;
    return 0;
  }
  if (stage < 0) return -2;
  if (wait_ns < 1 || wait_ns > (long long)cqr::kWaitNs) return -3;
  std::lock_guard<std::mutex> lk(cqr::g_fault_mu);
  cqr::g_fault_kernel = kernel;
  cqr::g_fault_stage = stage;
  cqr::g_fault_ns = (unsigned long long)wait_ns;
  return 0;
}
