// Split-m transposed products: the Gram matrix W = X^T X (Alg. 1 step 1,
// syrk semantics as in the caption of Table 1) and the projections
// Y = Q^T A (Alg. 6 step 6, Alg. 9 steps 3 and 7).
//
// The m-row sum is the "Gram reduce" of Alg. 2 step 4 / Alg. 8 steps 3 and 8,
// done inside one GPU: persistent thread blocks each own a contiguous range
// of (output tile, row block) work items, write one partial tile per
// (block, tile) segment, and a second kernel adds the partials in ascending
// row order.  The item ranges are static, so the summation order -- and the
// result -- is the same on every run.
//
// Each thread owns a 4 x 4 micro-tile of the output and, per row, issues 16
// FP64 FMAs on operands staged in shared memory (row-major, padded).  For
// small outputs several thread groups split the rows of a block and are
// summed in group order at the end.
#include "block_sums.cuh"
#include "cqr_common.cuh"

namespace cqr {

namespace {

constexpr int kTnThreads = 256;
constexpr int kSyrkThreads = 512;  // 16 warps
// Persistent blocks per SM for the split-m grids (at most what the
// registers allow).  Each block stalls in the load burst at the start of a
// row block; with three resident blocks the others keep the FP64 pipe busy
// meanwhile (projection: 1.195 -> 1.213 TFLOP/s on GB300 against two).
constexpr int kMaxResident = 3;
constexpr int kFullRows = 32;  // staged rows of a 64 x 64 tile

// [begin, end) of the items of persistent block c when T items are split
// over P blocks.
__host__ __device__ inline void item_range(i64 c, i64 T, i64 P, i64& begin, i64& end) {
  begin = (c * T) / P;
  end = ((c + 1) * T) / P;
}
// The persistent block whose range contains item i.
__host__ __device__ inline i64 owner_of(i64 i, i64 T, i64 P) { return ((i + 1) * P - 1) / T; }

__device__ inline double2 lds2(const double* p) { return *reinterpret_cast<const double2*>(p); }

__device__ __forceinline__ void cp_async8_zfill(double* dst, const double* src, bool ok) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(d), "l"(src), "r"(ok ? 8 : 0) : "memory");
}

// ---------------------------------------------------------------------------
// Gram (syrk) kernel for b <= 128, T threads.  The upper triangle is cut into
// cnt = n4(n4+1)/2 tiles of 4 x 4 (n4 = ceil(b/4)).  M of them are "main"
// tiles: thread t < M * RG owns main tile t % M on the rows r = t / M (mod
// RG) of each staged row block.  The E = cnt - M other tiles are "extra":
// each is owned by T / E threads that split the rows round-robin.  Where
// cnt * (T / cnt) threads fill the block to 93 %, every tile is a main tile
// (no second accumulator to sum at the end); otherwise M is the largest
// power of two <= cnt and every thread carries one main and at most one
// extra accumulator, so no lane idles.
struct SyrkArgs {
  const double* X;
  i64 ldx, m;
  int b, bp;       // width, padded width (multiple of 4)
  int M, RG;       // main tiles, row groups
  int E, tpt;      // extra tiles, threads per extra tile
  int rb;          // rows per staged block
  i64 P;           // persistent blocks; block c owns rows [c m / P, (c + 1) m / P)
  double* part;    // [P][b*b]
  const int* status;
};

__device__ __forceinline__ void syrk_tile_row(const double* row, int i, int j, double (&acc)[4][4]) {
  const double2 p0 = lds2(row + 4 * i), p1 = lds2(row + 4 * i + 2);
  const double2 q0 = lds2(row + 4 * j), q1 = lds2(row + 4 * j + 2);
  const double xv[4] = {p0.x, p0.y, p1.x, p1.y};
  const double yv[4] = {q0.x, q0.y, q1.x, q1.y};
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v) acc[u][v] = fma(xv[u], yv[v], acc[u][v]);
}

template <int T>
__global__ void __launch_bounds__(T) syrk_partial_kernel(SyrkArgs a) {
  stream_wait();
  extern __shared__ __align__(16) double sm[];
  if (a.status && *a.status) return;
  const int t = threadIdx.x;
  const int sp = a.bp + 2;  // padded row stride (even: keeps 16-byte alignment)
  int mi, mj;
  decode_upper(t % a.M, mi, mj);
  const int g = t / a.M;
  const bool extra = a.E > 0 && t < a.E * a.tpt;
  int ei = 0, ej = 0;
  const int ek = extra ? t % a.tpt : 0;
  if (extra) decode_upper(a.M + t / a.tpt, ei, ej);
  double am[4][4], ae[4][4];
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v) am[u][v] = ae[u][v] = 0.0;

  i64 rbeg, rend;
  item_range(blockIdx.x, a.m, a.P, rbeg, rend);
  const int rb = a.rb;
  for (i64 r0 = rbeg; r0 < rend; r0 += rb) {
    const int nrow = (int)imin64(rb, rend - r0);
    // stage X[r0:r0+nrow, 0:bp] row-major; zero beyond b.  Asynchronous
    // copies: every load of the block is in flight before the one wait,
    // instead of one memory latency per loop iteration.
    for (int e = t; e < rb * a.bp; e += T) {
      const int r = e % rb, c = e / rb;
      const bool ok = r < nrow && c < a.b;
      cp_async8_zfill(sm + r * sp + c, ok ? a.X + (r0 + r) + (i64)c * a.ldx : a.X, ok);
    }
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    if (g < a.RG) {
#pragma unroll 2
      for (int r = g; r < nrow; r += a.RG) syrk_tile_row(sm + r * sp, mi, mj, am);
    }
    if (extra)
      for (int r = ek; r < nrow; r += a.tpt) syrk_tile_row(sm + r * sp, ei, ej, ae);
    __syncthreads();
  }
  // fixed-order sums: main tiles over the row groups, extra tiles over their threads
  double* P = a.part + (i64)blockIdx.x * a.b * a.b;
  const int b = a.b, M = a.M;
  auto store = [P, b](int id, int e, double x) {
    int i, j;
    decode_upper(id, i, j);
    const int r = 4 * i + (e >> 2), c = 4 * j + (e & 3);
    if (r <= c && c < b) P[r + c * b] = x;
  };
  double* scratch = sm + 16 * T;
  spill_acc(sm, T, am);
  __syncthreads();
  block_sums<T>(sm, scratch, M, a.RG, 1, M, store);
  if (a.E > 0) {
    __syncthreads();
    spill_acc(sm, T, ae);
    __syncthreads();
    block_sums<T>(sm, scratch, a.E, a.tpt, a.tpt, 1, [store, M](int id, int e, double x) { store(M + id, e, x); });
  }
}

// W[r + c*ldw] = sum_{s<P} part[s][r + c*b] for r <= c, mirrored.  16 entries
// of the upper triangle (column by column) per block of 256 threads.
__global__ void __launch_bounds__(256) syrk_reduce_kernel(const double* part, int b, i64 P, double* W, i64 ldw,
                                                          const int* status) {
  stream_wait();
  __shared__ double red[16 * 17];
  if (status && *status) return;
  const int u = blockIdx.x * 16 + (threadIdx.x & 15);
  const bool live = u < b * (b + 1) / 2;
  int r = 0, c = 0;
  if (live) decode_upper(u, r, c);
  const double* p = part + r + c * b;
  const i64 bb = (i64)b * b;
  const double s = split_sum16(P, live, red, [p, bb](i64 k) { return p[k * bb]; });
  if (threadIdx.x < 16 && live) {
    W[r + (i64)c * ldw] = s;
    if (r != c) W[c + (i64)r * ldw] = s;
  }
}

// ---------------------------------------------------------------------------
// General C = X^T Y (no symmetry).  Tile tp x tq (multiples of 4, at most
// 64), 256 threads: ntg = tp tq / 16 micro-tiles of 4 x 4, G = 256 / ntg row
// groups; thread t < ntg * G owns micro-tile t % ntg on the rows r = t / ntg
// (mod G).  The 64 x 64 tile (every product of two multiples of 64) has its
// sizes at compile time: the address arithmetic of the run-time form costs
// it 0.8 % (projections at 2^18 x 1024, b = 128: 395.0 -> 392.0 ms).
struct TnArgs {
  const double* X;
  i64 ldx;
  const double* Y;
  i64 ldy;
  i64 m;
  int p, q;
  int tp, tq, rb;
  int tiles_p;
  i64 nb, T, P;  // row blocks per tile, total items, persistent blocks
  double* part;  // [P + ntiles][tp * tq]
  const int* status;
};

template <bool kFull>
__global__ void __launch_bounds__(kTnThreads) tn_partial_kernel(TnArgs a) {
  stream_wait();
  extern __shared__ __align__(16) double sm[];
  if (a.status && *a.status) return;
  const int t = threadIdx.x;
  const int atp = kFull ? 64 : a.tp, atq = kFull ? 64 : a.tq;
  const int NP = atp >> 2, ntg = NP * (atq >> 2), G = kTnThreads / ntg;
  const int g = t / ntg, u = t - g * ntg;
  const int mj = u / NP, mi = u - mj * NP;
  const int SP = atp + 2, SQ = atq + 2;
  const int rb = kFull ? kFullRows : a.rb;
  double* Xs = sm;
  double* Ys = sm + rb * SP;

  i64 ib, ie;
  item_range(blockIdx.x, a.T, a.P, ib, ie);
  i64 item = ib;
  while (item < ie) {
    const i64 tile = item / a.nb;
    const i64 tile_end = imin64(ie, (tile + 1) * a.nb);
    const int p0 = (int)(tile % a.tiles_p) * atp, q0 = (int)(tile / a.tiles_p) * atq;
    double acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = 0.0;
    for (; item < tile_end; ++item) {
      const i64 r0 = (item - tile * a.nb) * rb;
      const int nrow = (int)imin64(rb, a.m - r0);
      // asynchronous staging (zero-filled beyond p, q): all loads in flight before one wait
      for (int e = t; e < rb * atp; e += kTnThreads) {
        const int r = e % rb, c = e / rb;
        const bool ok = r < nrow && p0 + c < a.p;
        cp_async8_zfill(Xs + r * SP + c, ok ? a.X + (r0 + r) + (i64)(p0 + c) * a.ldx : a.X, ok);
      }
      for (int e = t; e < rb * atq; e += kTnThreads) {
        const int r = e % rb, c = e / rb;
        const bool ok = r < nrow && q0 + c < a.q;
        cp_async8_zfill(Ys + r * SQ + c, ok ? a.Y + (r0 + r) + (i64)(q0 + c) * a.ldy : a.Y, ok);
      }
      asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
      __syncthreads();
      if (g < G) {
        const double* xi = Xs + 4 * mi;
        const double* yj = Ys + 4 * mj;
#pragma unroll 2
        for (int r = g; r < nrow; r += G) {
          const double2 p0v = lds2(xi + r * SP), p1v = lds2(xi + r * SP + 2);
          const double2 q0v = lds2(yj + r * SQ), q1v = lds2(yj + r * SQ + 2);
          const double xv[4] = {p0v.x, p0v.y, p1v.x, p1v.y};
          const double yv[4] = {q0v.x, q0v.y, q1v.x, q1v.y};
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = fma(xv[i], yv[j], acc[i][j]);
        }
      }
      __syncthreads();
    }
    // segment id = persistent block + tile (unique, increasing in rows)
    double* Pp = a.part + ((i64)blockIdx.x + tile) * (atp * atq);
    if (G > 1) {
      spill_acc(sm, kTnThreads, acc);
      __syncthreads();
      block_sums<kTnThreads>(sm, sm + 16 * kTnThreads, ntg, G, 1, ntg, [Pp, atp, NP](int id, int e, double x) {
        const int j = id / NP, i = id - j * NP;
        Pp[(4 * i + (e >> 2)) + (4 * j + (e & 3)) * atp] = x;
      });
      __syncthreads();
    } else if (g == 0) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) Pp[(4 * mi + i) + (4 * mj + j) * atp] = acc[i][j];
    }
  }
}

// C[r + c*ldc] = sum over the segments of tile(r, c), ascending rows.
__global__ void __launch_bounds__(256) tn_reduce_kernel(const double* part, int p, int q, int TP, int TQ, int tiles_p,
                                                        i64 nb, i64 T, i64 P, double* C, i64 ldc, const int* status) {
  stream_wait();
  __shared__ double red[16 * 17];
  if (status && *status) return;
  const i64 e = (i64)blockIdx.x * 16 + (threadIdx.x & 15);
  const bool live = e < (i64)p * q;
  const int r = (int)(e % p), c = (int)(e / p);
  i64 nseg = 0;  // T == 0, no rows: the empty sum
  const double* src = part;
  const i64 tt = (i64)TP * TQ;
  if (live && T > 0) {
    const i64 tile = (i64)(r / TP) + (i64)(c / TQ) * tiles_p;
    const i64 c_lo = owner_of(tile * nb, T, P);
    const i64 c_hi = owner_of((tile + 1) * nb - 1, T, P);
    nseg = c_hi - c_lo + 1;
    src = part + (c_lo + tile) * tt + (r % TP) + (c % TQ) * TP;
  }
  const double s = split_sum16(nseg, live, red, [src, tt](i64 k) { return src[k * tt]; });
  if (threadIdx.x < 16 && live) C[r + (i64)c * ldc] = s;
}

// ---------------------------------------------------------------------------
struct SyrkPlan {
  int T, bp, M, RG, E, tpt, rb, P;
  size_t smem;
};

// Row count x tile count (the work) below which the 128-thread kernel is used,
// for up to 256 tiles: its smaller blocks spread a short matrix over more SMs.
// Times of a panel, two Gram matrices each, with 128 / 512 threads, us: work
// 1e5: b = 8 66 / 67, 16 81 / 83, 24 99 / 102, 32 125 / 125, 48 213 / 215, 64
// 320 / 321, 80 439 / 424; work 1.2e6: 209 / 206, 224 / 211, 220 / 213, 240 /
// 226, 317 / 273, 402 / 365, 515 / 472.  So it gains up to 3 % below 3e5 and
// costs 2 to 16 % from 6e5 up to the line, which lies too far up: at 3e5 it
// would cost nothing.
constexpr i64 kSyrkSmall = 1200000;

// Doubles of partial triangles up to which the 128-thread kernel takes more
// than one block per SM: 5.8 MB of a small call's workspace.  It binds for 41
// to 69 columns.  A panel of 48 columns, work 1.2e6: 318 us, 372 with one block
// per SM, 285 without a limit; 64 columns: 403, 393 and 383.
constexpr i64 kPartCap = 730000;

struct SyrkOcc {
  int o[2][129];
};
PerDevice<SyrkOcc> g_occ_syrk;

SyrkPlan syrk_plan(i64 m, int b) {
  SyrkPlan s;
  const int n4 = (b + 3) / 4;
  s.bp = 4 * n4;
  const int cnt = n4 * (n4 + 1) / 2;
  const bool small = cnt <= 256 && m * cnt < kSyrkSmall;
  s.T = small ? 128 : kSyrkThreads;
  if (cnt <= s.T && (s.T / cnt) * cnt * 100 >= s.T * 93) {
    s.M = cnt;
  } else {
    s.M = 1;
    while (s.M * 2 <= cnt && s.M * 2 <= s.T) s.M *= 2;
  }
  s.RG = s.T / s.M;
  s.E = cnt - s.M;
  s.tpt = s.E > 0 ? s.T / s.E : 0;
  // staged doubles per row block: half the reduction area of the large
  // kernel, twice that of the small one
  const int per = (small ? 4096 : 8192) / (s.bp + 2);
  s.rb = per >= s.RG ? per / s.RG * s.RG : s.RG;
  // Blocks: at least 32 rows each, at most kMaxResident per SM, and above one
  // per SM at most kPartCap doubles of partial triangles.
  const i64 min_rows = 32;
  i64 want = (m + min_rows - 1) / min_rows;
  if (want < 1) want = 1;
  if (small) {
    const i64 cap = kPartCap / ((i64)b * b);
    const i64 most = cap > kSMs ? cap : (i64)kSMs;
    if (want > most) want = most;
  }
  const size_t tile = (size_t)s.rb * (s.bp + 2), red = (size_t)17 * s.T;
  s.smem = (tile > red ? tile : red) * sizeof(double);
  int& occ = g_occ_syrk.here().o[small ? 0 : 1][b];
  if (occ == 0) {
    int o = 0;
    if (small) {
      cudaFuncSetAttribute(syrk_partial_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, syrk_partial_kernel<128>, 128, s.smem);
    } else {
      cudaFuncSetAttribute(syrk_partial_kernel<kSyrkThreads>, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, syrk_partial_kernel<kSyrkThreads>, kSyrkThreads, s.smem);
    }
    occ = o > 0 ? o : 1;
  }
  const i64 slots = (i64)kSMs * min(occ, kMaxResident);
  s.P = (int)(want < slots ? want : slots);
  return s;
}

// Tile of the general product: of the cuts of p and q into equal tiles of at
// most 64, the one that wastes the fewest lanes (tile padding and threads
// beyond ntg * G); among equals the largest tile.
void tn_tile(int p, int q, int& tp, int& tq) {
  const int kp = (p + 63) / 64, kq = (q + 63) / 64;
  double best = -1.0;
  tp = tq = 64;
  for (int ip = kp; ip <= kp + 2; ++ip)
    for (int iq = kq; iq <= kq + 2; ++iq) {
      const int a = ((p + ip - 1) / ip + 3) / 4 * 4, b = ((q + iq - 1) / iq + 3) / 4 * 4;
      const int np = (p + a - 1) / a, nq = (q + b - 1) / b;
      const int ntg = (a / 4) * (b / 4);
      const double util = (double)p * q / ((double)np * a * nq * b) * ((double)(kTnThreads / ntg * ntg) / kTnThreads);
      if (util > best * 1.001) {
        best = util;
        tp = a;
        tq = b;
      }
    }
}

size_t tn_smem(int tp, int tq, int rb) {
  const size_t tile = (size_t)rb * (tp + tq + 4), red = (size_t)17 * kTnThreads;
  return (tile > red ? tile : red) * sizeof(double);
}

PerDevice<int> g_occ_tn;  // run-time form, at the largest shared-memory size

int tn_occupancy() {
  int& occ = g_occ_tn.here();
  if (occ == 0) {
    cudaFuncSetAttribute(tn_partial_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 48 * 1024);
    int o = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, tn_partial_kernel<false>, kTnThreads, 48 * 1024);
    occ = o > 0 ? o : 1;
  }
  return occ;
}

}  // namespace

TnPlan tn_plan(i64 m, int p, int q, int sym) {
  TnPlan P{};
  if (sym && p <= 128) {
    const SyrkPlan s = syrk_plan(m, p);
    P.tp = P.tq = s.bp;
    P.tiles_p = P.tiles_q = 1;
    P.ntiles = 1;
    P.rb = s.rb;
    P.S = s.P;
    return P;
  }
  tn_tile(p, q, P.tp, P.tq);
  P.tiles_p = (p + P.tp - 1) / P.tp;
  P.tiles_q = (q + P.tq - 1) / P.tq;
  P.ntiles = P.tiles_p * P.tiles_q;
  // Rows per item: about 4096 staged doubles, but where m is too short for
  // every block to get that many, an even share (rounded up to the row
  // groups, so that no block gets a second item), at least 32.
  const i64 slots = (i64)kSMs * min(tn_occupancy(), kMaxResident);
  const int G = kTnThreads / ((P.tp / 4) * (P.tq / 4));
  i64 rb = 4096 / (P.tp + P.tq);
  if (rb > G) rb = rb / G * G;
  i64 even = (m * P.ntiles + slots - 1) / slots;
  if (even < 32) even = 32;
  if (even > G) even = (even + G - 1) / G * G;
  if (rb > even) rb = even;
  P.rb = (int)rb;
  const i64 T = (m + P.rb - 1) / P.rb * P.ntiles;
  P.S = (int)(T < slots ? (T > 0 ? T : 1) : slots);
  return P;
}

size_t tn_partial_doubles(i64 m, int p, int q, int sym) {
  if (p <= 0 || q <= 0) return 0;
  if (sym && p > 128) {
    // blocked into 128-wide pieces: the largest piece dominates
    size_t mx = 0;
    for (int i = 0; i < p; i += 128)
      for (int j = i; j < p; j += 128) {
        int pi = p - i < 128 ? p - i : 128, pj = p - j < 128 ? p - j : 128;
        size_t d = tn_partial_doubles(m, pi, pj, i == j);
        if (d > mx) mx = d;
      }
    return mx;
  }
  TnPlan P = tn_plan(m, p, q, sym);
  if (sym) return (size_t)P.S * p * p;
  return (size_t)(P.S + P.ntiles) * P.tp * P.tq;
}

size_t tn_nominal_doubles(i64 m, int p, int q, int sym) {
  if (p <= 0 || q <= 0) return 0;
  if (sym && p > 128) {
    size_t mx = 0;
    for (int i = 0; i < p; i += 128)
      for (int j = i; j < p; j += 128) {
        const int pi = p - i < 128 ? p - i : 128, pj = p - j < 128 ? p - j : 128;
        const size_t d = tn_nominal_doubles(m, pi, pj, i == j);
        if (d > mx) mx = d;
      }
    return mx;
  }
  if (sym) {  // 512 threads, about 8192 staged doubles a block, one block per SM
    const int n4 = (p + 3) / 4, cnt = n4 * (n4 + 1) / 2;
    int M = 1;
    while (M * 2 <= cnt && M * 2 <= kSyrkThreads) M *= 2;
    const int RG = kSyrkThreads / M, per = 8192 / (4 * n4 + 2);
    const i64 rb = per >= RG ? per / RG * RG : RG;
    const i64 nb = (m + rb - 1) / rb;
    return (size_t)(nb < kSMs ? nb : kSMs) * p * p;
  }
  auto tile = [](int d) { return d <= 8 ? 8 : d <= 16 ? 16 : d <= 32 ? 32 : 64; };
  const int tp = tile(p), tq = tile(q);
  const int G = kTnThreads / ((tp / 4) * (tq / 4)), unit = G > 8 ? G : 8;
  const i64 rb = (4096 / (tp + tq)) / unit * unit;
  const i64 nt = (i64)((p + tp - 1) / tp) * ((q + tq - 1) / tq), T = (m + rb - 1) / rb * nt;
  return (size_t)((T < kSMs * kMaxResident ? T : kSMs * kMaxResident) + nt) * tp * tq;
}

i64 gram_partials(i64 m, int b, const double* X, i64 ldx, double* part, const int* status, cudaStream_t st) {
  if (m <= 0) return 0;
  const SyrkPlan s = syrk_plan(m, b);
  SyrkArgs a;
  a.X = X;
  a.ldx = ldx;
  a.m = m;
  a.b = b;
  a.bp = s.bp;
  a.M = s.M;
  a.RG = s.RG;
  a.E = s.E;
  a.tpt = s.tpt;
  a.rb = s.rb;
  a.P = s.P;
  a.part = part;
  a.status = status;
  prof_begin(kGram, st);
  if (s.T == 128)
    launch(Work64{(double)m * b * (b + 1)}, syrk_partial_kernel<128>, s.P, 128, s.smem, st, a);
  else
    launch(syrk_partial_kernel<kSyrkThreads>, s.P, kSyrkThreads, s.smem, st, a);
  prof_end(kGram, (double)m * b * (b + 1), st);
  return s.P;
}

cudaError_t tn_product(i64 m, int p, int q, const double* X, i64 ldx, const double* Y, i64 ldy, int sym,
                       double* part, double* C, i64 ldc, const int* status, cudaStream_t st) {
  if (p <= 0 || q <= 0) return cudaSuccess;
  if (sym && p > 128) {
    // W = [X1 X2 ...]^T [X1 X2 ...] by 128-wide blocks; upper blocks, mirrored.
    for (int j = 0; j < p; j += 128) {
      for (int i = 0; i <= j; i += 128) {
        const int pi = p - i < 128 ? p - i : 128, pj = p - j < 128 ? p - j : 128;
        cudaError_t e;
        if (i == j) {
          e = tn_product(m, pi, pi, X + (i64)i * ldx, ldx, X + (i64)i * ldx, ldx, 1, part, C + i + (i64)i * ldc,
                         ldc, status, st);
        } else {
          e = tn_product(m, pi, pj, X + (i64)i * ldx, ldx, X + (i64)j * ldx, ldx, 0, part, C + i + (i64)j * ldc,
                         ldc, status, st);
        }
        if (e != cudaSuccess) return e;
      }
    }
    return cudaSuccess;
  }
  if (sym) {
    const i64 nsum = gram_partials(m, p, X, ldx, part, status, st);  // m == 0: none, the empty sum W = 0
    prof_begin(kReduce, st);
    launch(Work64{(double)nsum * p * (p + 1) / 2}, syrk_reduce_kernel, (p * (p + 1) / 2 + 15) / 16, 256, 0, st, part, p,
           nsum, C, ldc, status);
    prof_end(kReduce, (double)nsum * p * (p + 1) / 2, st);
    return cudaGetLastError();
  }
  const TnPlan P = tn_plan(m, p, q, sym);
  TnArgs a;
  a.X = X;
  a.ldx = ldx;
  a.Y = Y;
  a.ldy = ldy;
  a.m = m;
  a.p = p;
  a.q = q;
  a.tp = P.tp;
  a.tq = P.tq;
  a.rb = P.rb;
  a.tiles_p = P.tiles_p;
  a.nb = (m + P.rb - 1) / P.rb;
  a.T = a.nb * P.ntiles;
  a.P = P.S;
  a.part = part;
  a.status = status;
  if (m > 0) {
    prof_begin(kProjection, st);
    const size_t smem = tn_smem(P.tp, P.tq, P.rb);
    if (P.tp == 64 && P.tq == 64 && P.rb == kFullRows)
      launch(tn_partial_kernel<true>, (unsigned)P.S, kTnThreads, smem, st, a);
    else
      launch(Work64{2.0 * (double)m * p * q}, tn_partial_kernel<false>, (unsigned)P.S, kTnThreads, smem, st, a);
    prof_end(kProjection, 2.0 * (double)m * p * q, st);
  }
  const i64 pq = (i64)p * q;
  prof_begin(kReduce, st);
  launch(Work64{(double)(P.S + P.ntiles) / P.ntiles * pq}, tn_reduce_kernel, (unsigned)((pq + 15) / 16), 256, 0, st,
         part, p, q, P.tp, P.tq, P.tiles_p, a.nb, m > 0 ? a.T : 0, m > 0 ? a.P : 1, C, ldc, status);
  prof_end(kReduce, m > 0 ? (double)(P.S + P.ntiles) / P.ntiles * pq : 0.0, st);
  return cudaGetLastError();
}

}  // namespace cqr
