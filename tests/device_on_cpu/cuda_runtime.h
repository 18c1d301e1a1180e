// Device code on the CPU: the part of CUDA's language that the small
// single-block headers of the library use, for tests that have to choose the
// order in which warps run.  A block is run by run_block(): one fiber per
// thread, a barrier or a warp shuffle suspends it.  Between two barriers the
// warps run one after the other in the order given (the lanes of a warp
// advance together from shuffle to shuffle), so a value that one warp reads
// and another writes without a barrier between them comes out differently for
// different orders.
#pragma once
#include <math.h>
#include <stdint.h>
#include <string.h>
#include <ucontext.h>

#include <algorithm>
#include <functional>
#include <vector>

#define __host__
#define __device__
#define __forceinline__ inline
#define __noinline__
#define __restrict__

struct Dim1 {
  int x;
};
inline Dim1 threadIdx;

inline long long __double_as_longlong(double d) {
  long long v;
  memcpy(&v, &d, 8);
  return v;
}
inline double __longlong_as_double(long long v) {
  double d;
  memcpy(&d, &v, 8);
  return d;
}
inline int __double2hiint(double d) { return (int)(__double_as_longlong(d) >> 32); }
inline int __double2loint(double d) { return (int)__double_as_longlong(d); }
inline double __hiloint2double(int hi, int lo) {
  return __longlong_as_double((long long)(((uint64_t)(uint32_t)hi << 32) | (uint32_t)lo));
}
inline unsigned __float_as_uint(float f) {
  unsigned v;
  memcpy(&v, &f, 4);
  return v;
}
inline float __uint_as_float(unsigned v) {
  float f;
  memcpy(&f, &v, 4);
  return f;
}
inline float __fmul_rn(float a, float b) { return a * b; }
inline float __fmaf_rn(float a, float b, float c) { return fmaf(a, b, c); }
inline float __uint2float_rn(unsigned v) { return (float)v; }
inline float __frcp_rn(float a) { return 1.0f / a; }
inline float rsqrtf(float a) { return 1.0f / sqrtf(a); }
inline int __clzll(long long v) { return v ? __builtin_clzll((unsigned long long)v) : 64; }

namespace device_on_cpu {

struct Thread {
  ucontext_t ctx;
  std::vector<char> stack;
  int state;     // 0 ready, 1 at a barrier, 2 at a shuffle, 3 done
  double out;    // value offered to a shuffle
  int src, vote;
};

inline std::vector<Thread> threads;
inline ucontext_t scheduler;
inline int current, any_vote;
inline std::function<void()> body;

inline void suspend(int state) {
  Thread& t = threads[current];
  t.state = state;
  swapcontext(&t.ctx, &scheduler);
}

inline void entry() {
  body();
  threads[current].state = 3;
  swapcontext(&threads[current].ctx, &scheduler);
}

// Runs f in n threads; order[k] is the warp that runs k-th after each barrier.
// Returns false if some threads of the block wait at a barrier that others left out.
inline bool run_block(int n, const std::vector<int>& order, std::function<void()> f) {
  body = f;
  threads.assign(n, Thread());
  for (int i = 0; i < n; ++i) {
    Thread& t = threads[i];
    t.stack.resize(64 * 1024);
    t.state = 0;
    getcontext(&t.ctx);
    t.ctx.uc_stack.ss_sp = t.stack.data();
    t.ctx.uc_stack.ss_size = t.stack.size();
    t.ctx.uc_link = nullptr;
    makecontext(&t.ctx, entry, 0);
  }
  for (;;) {
    for (int w : order)
      for (bool again = true; again;) {
        again = false;
        for (int i = 32 * w; i < 32 * w + 32; ++i)
          if (threads[i].state == 0) {
            current = threadIdx.x = i;
            swapcontext(&scheduler, &threads[i].ctx);
          }
        for (int i = 32 * w; i < 32 * w + 32; ++i)
          if (threads[i].state == 2) {  // the whole warp shuffles together
            threads[i].state = 0;
            again = true;
          }
      }
    int done = 0;
    any_vote = 0;
    for (Thread& t : threads) {
      done += t.state == 3;
      any_vote |= t.state == 1 && t.vote;
    }
    if (done == n) return true;
    if (done) return false;
    for (Thread& t : threads) t.state = 0;
  }
}

}  // namespace device_on_cpu

inline int __syncthreads_or(int v) {
  device_on_cpu::threads[device_on_cpu::current].vote = v;
  device_on_cpu::suspend(1);
  return device_on_cpu::any_vote;
}
inline void __syncthreads() { __syncthreads_or(0); }
inline double __shfl_sync(unsigned, double v, int src) {
  using namespace device_on_cpu;
  threads[current].out = v;
  suspend(2);
  const double got = threads[(current & ~31) + src].out;
  suspend(2);  // nobody offers its next value before all have read
  return got;
}
