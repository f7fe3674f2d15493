// A CTA on the host, for tests of device code without a GPU: every thread is a coroutine that runs
// alone up to its next barrier, in ascending or descending order of the threads, so that code whose
// threads exchange data without a barrier between them gives a wrong result in one of the orders.
// Warp collectives (shuffles, votes, reductions) count as barriers of the warp.
#pragma once

#include <ucontext.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <memory>
#include <type_traits>
#include <vector>

#include <vector_functions.h>
#include <vector_types.h>

#undef __device__
#undef __host__
#undef __global__
#undef __shared__
#undef __forceinline__
#undef __noinline__
#undef __launch_bounds__
#define __device__
#define __host__
#define __global__
#define __shared__ static
#define __forceinline__ inline
#define __noinline__
#define __launch_bounds__(...)

namespace simt {

struct Index { unsigned x = 0, y = 0, z = 0; };
enum State { READY, AT_WARP, AT_BLOCK, DONE };

struct Thread {
  ucontext_t ctx;
  std::unique_ptr<char[]> stack;
  State state = READY;
};

struct Block {
  std::vector<Thread> t;
  std::vector<uint64_t> box;         // a value per thread for the warp collectives
  std::function<void()> body;
  ucontext_t main;
  int cur = 0;
};
inline Block* B = nullptr;

inline void wait_at(State s) {
  const int me = B->cur;
  B->t[me].state = s;
  swapcontext(&B->t[me].ctx, &B->main);
}
inline void entry() {
  B->body();
  B->t[B->cur].state = DONE;
  swapcontext(&B->t[B->cur].ctx, &B->main);
}

}  // namespace simt

inline simt::Index threadIdx, blockIdx, blockDim, gridDim;

namespace simt {

// `body` by nthreads threads; false when some of them wait for ever
inline bool run_block(int nthreads, bool descending, std::function<void()> body) {
  Block b;
  B = &b;
  b.t.resize(nthreads);
  b.box.assign(nthreads, 0);
  b.body = std::move(body);
  blockDim.x = nthreads;
  constexpr size_t kStack = 1 << 16;
  for (auto& t : b.t) {
    t.stack.reset(new char[kStack]);
    getcontext(&t.ctx);
    t.ctx.uc_stack.ss_sp = t.stack.get();
    t.ctx.uc_stack.ss_size = kStack;
    t.ctx.uc_link = &b.main;
    makecontext(&t.ctx, (void (*)())entry, 0);
  }
  for (;;) {
    bool ran = false;
    for (int k = 0; k < nthreads; ++k) {
      const int i = descending ? nthreads - 1 - k : k;
      if (b.t[i].state != READY) continue;
      ran = true;
      b.cur = i;
      threadIdx.x = i;
      swapcontext(&b.main, &b.t[i].ctx);
    }
    // barriers that everybody who still runs has reached
    bool all_block = true, any = false;
    for (int w = 0; w < nthreads; w += 32) {
      bool all_warp = true, waits = false;
      for (int i = w; i < std::min(nthreads, w + 32); ++i) {
        any |= b.t[i].state != DONE;
        all_warp &= b.t[i].state == AT_WARP || b.t[i].state == DONE;
        waits |= b.t[i].state == AT_WARP;
        all_block &= b.t[i].state == AT_BLOCK || b.t[i].state == DONE;
      }
      if (all_warp && waits) {
        for (int i = w; i < std::min(nthreads, w + 32); ++i)
          if (b.t[i].state == AT_WARP) b.t[i].state = READY;
        ran = true;
      }
    }
    if (!any) return true;
    if (all_block) {
      for (auto& t : b.t)
        if (t.state == AT_BLOCK) t.state = READY;
      ran = true;
    }
    if (!ran) return false;
  }
}

template <typename T>
inline T exchange(T v, int src) {
  uint64_t u = 0;
  std::memcpy(&u, &v, sizeof(T));
  const int me = B->cur, w = me & ~31;
  B->box[me] = u;
  wait_at(AT_WARP);
  u = B->box[w + (src & 31)];
  T r;
  std::memcpy(&r, &u, sizeof(T));
  wait_at(AT_WARP);
  return r;
}
template <typename T, typename F>
inline T warp_fold(T v, F f) {
  T r = exchange(v, 0);
  for (int i = 1; i < 32; ++i) r = f(r, exchange(v, i));
  return r;
}

}  // namespace simt

inline void __syncwarp(unsigned = 0xffffffffu) { simt::wait_at(simt::AT_WARP); }
inline void __syncthreads() { simt::wait_at(simt::AT_BLOCK); }
inline int __syncthreads_or(int v) {
  static int any;
  any = 0;
  __syncthreads();
  any |= v;
  __syncthreads();
  return any != 0;
}
template <typename T> inline T __shfl_xor_sync(unsigned, T v, int m) { return simt::exchange(v, (threadIdx.x & 31) ^ m); }
template <typename T> inline T __shfl_sync(unsigned, T v, int src) { return simt::exchange(v, src); }
inline int __reduce_add_sync(unsigned, int v) { return simt::warp_fold(v, [](int a, int b) { return a + b; }); }
inline unsigned __reduce_max_sync(unsigned, unsigned v) {
  return simt::warp_fold(v, [](unsigned a, unsigned b) { return a > b ? a : b; });
}
inline unsigned __reduce_min_sync(unsigned, unsigned v) {
  return simt::warp_fold(v, [](unsigned a, unsigned b) { return a < b ? a : b; });
}
inline long long __double_as_longlong(double v) { long long u; std::memcpy(&u, &v, 8); return u; }
inline double __longlong_as_double(long long u) { double v; std::memcpy(&v, &u, 8); return v; }
inline int __double2hiint(double v) { return (int)(__double_as_longlong(v) >> 32); }
inline int __double2loint(double v) { return (int)__double_as_longlong(v); }
inline float __uint_as_float(unsigned u) { float v; std::memcpy(&v, &u, 4); return v; }
inline unsigned __float_as_uint(float v) { unsigned u; std::memcpy(&u, &v, 4); return u; }
inline int __clzll(long long v) { return v ? __builtin_clzll((unsigned long long)v) : 64; }
inline int atomicExch(int* p, int v) { const int o = *p; *p = v; return o; }
inline int atomicAdd(int* p, int v) { const int o = *p; *p += v; return o; }
inline int __reduce_max_sync(unsigned, int v) {
  return simt::warp_fold(v, [](int a, int b) { return a > b ? a : b; });
}
inline double rsqrt(double v) { return 1.0 / std::sqrt(v); }
using std::max;
using std::min;
using std::isfinite;
