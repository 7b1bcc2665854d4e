// A thread block on the host: every thread is a fibre, a warp advances in step from one warp operation
// (__shfl_sync, __syncwarp) to the next, and between two block barriers the warps run one after another
// in a given order. Code whose result depends on how far another warp has come between two barriers
// gives different results for different orders.
#pragma once
#include <ucontext.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <functional>
#include <vector>

#define __device__
#define __forceinline__ inline
#define __shared__ static
using std::fma;
using std::max;
using std::min;

namespace simt {
enum State { kRun, kWarpOp, kBarrier, kDone };
struct Thread {
  ucontext_t ctx;
  std::vector<char> stack;
  State state;
  unsigned ops;  // warp operations so far
};
struct Block {
  std::vector<Thread> threads;
  std::vector<double> slots;  // two sets of 32 published values per warp
  ucontext_t main;
  std::function<void()> body;
  int current = 0;
};
inline Block* g = nullptr;

inline void yield(State s) {
  Thread& t = g->threads[g->current];
  t.state = s;
  swapcontext(&t.ctx, &g->main);
}
inline void entry() {
  g->body();
  g->threads[g->current].state = kDone;
}
inline void resume(int id);

// runs one thread block of n threads; order: a permutation of its warps
inline void run(int n, const std::vector<int>& order, std::function<void()> body);
}  // namespace simt

struct ThreadIndex { int x; };
inline ThreadIndex threadIdx;

inline void simt::resume(int id) {
  g->current = id;
  threadIdx.x = id;
  g->threads[id].state = kRun;
  swapcontext(&g->main, &g->threads[id].ctx);
}

inline void simt::run(int n, const std::vector<int>& order, std::function<void()> body) {
  Block block;
  g = &block;
  block.body = std::move(body);
  block.threads.resize(n);
  block.slots.resize(2 * n);
  for (Thread& t : block.threads) {
    t.stack.resize(64 * 1024);
    getcontext(&t.ctx);
    t.ctx.uc_stack.ss_sp = t.stack.data();
    t.ctx.uc_stack.ss_size = t.stack.size();
    t.ctx.uc_link = &block.main;
    makecontext(&t.ctx, entry, 0);
    t.state = kRun;
    t.ops = 0;
  }
  for (bool alive = true; alive;) {
    alive = false;
    for (int w : order) {
      if (block.threads[32 * w].state == kDone) continue;
      for (;;) {  // this warp, up to the next block barrier or its end
        for (int l = 0; l < 32; ++l) resume(32 * w + l);
        const State s = block.threads[32 * w].state;
        for (int l = 0; l < 32; ++l)
          if (block.threads[32 * w + l].state != s) {
            std::fprintf(stderr, "warp %d: lanes apart at a warp operation or a barrier\n", w);
            std::exit(2);
          }
        if (s != kWarpOp) {
          alive |= s == kBarrier;
          break;
        }
      }
    }
  }
  g = nullptr;
}

inline void __syncthreads() { simt::yield(simt::kBarrier); }
inline void __syncwarp() { simt::yield(simt::kWarpOp); }
inline double __shfl_sync(unsigned, double v, int src) {
  const int id = simt::g->current;
  const unsigned op = simt::g->threads[id].ops++;
  double* slots = simt::g->slots.data() + 64 * (id / 32) + 32 * (op & 1);  // (a lane is one operation ahead at most)
  slots[id % 32] = v;
  simt::yield(simt::kWarpOp);
  return slots[src];
}
inline double rsqrt(double x) { return 1.0 / std::sqrt(x); }
inline int atomicCAS(int* p, int expect, int v) {
  const int old = *p;
  if (old == expect) *p = v;
  return old;
}
