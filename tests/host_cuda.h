// Runs a CUDA kernel's source on the CPU under chosen schedules: every thread is a coroutine, and at each
// synchronisation (flag, barrier, warp exchange) the scheduler picks the next one at random and now and then holds a
// warp back until nothing else can go on.  Orders that a GPU takes once in a blue moon then happen in every run: a
// read that no wait covers returns the poison that the buffers start with, a barrier that not all threads reach is
// reported as a deadlock.  Memory is sequentially consistent here, so only missing waits show, not missing fences.
#pragma once

#include <math.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>
#include <sys/mman.h>
#include <ucontext.h>

#include <algorithm>
#include <functional>
#include <memory>
#include <vector>

#define __device__
#define __global__
#define __forceinline__ inline
#define __noinline__
#define __launch_bounds__(...)
#define __align__(n)

struct double2 { double x, y; };
inline double2 make_double2(double x, double y) { return {x, y}; }
struct Index3 { int x, y, z; };

namespace emu {

struct Cta;
struct Thread {
  ucontext_t ctx;
  Index3 tid{0, 0, 0};
  Cta* cta = nullptr;
  int warp = 0, lane = 0;
  bool done = false, ready = false;
  const int* polled = nullptr;  // the flag it last read, and what it saw
  int saw = 0;
  void* stack = nullptr;
};
struct Barrier {
  int count = 0, generation = 0, any[2] = {0, 0}, all[2] = {1, 1};
  std::vector<Thread*> waiting;
};
struct Warp {
  Barrier sync;
  uint64_t box[2][32];
  bool held = false;
  std::vector<Thread*> parked;  // its threads that could run
};
struct Cta {
  Index3 bid{0, 0, 0};
  int live = 0;
  std::vector<std::unique_ptr<Thread>> threads;
  std::vector<Warp> warps;
  Barrier bars[16];
  std::vector<unsigned char> smem;
  int ints[8] = {0};
};

struct Scheduler {
  uint64_t seed = 1;
  double hold_release = 0.0, hold_barrier = 0.0;  // chance that a warp is held back after a release, after a barrier
  int64_t steps = 0, work = 0;
  Thread* cur = nullptr;
  ucontext_t main;
  std::vector<Thread*> ready, polling;
  std::vector<Warp*> held;
  std::function<void()> body;
  Index3 grid{1, 1, 1}, block{1, 1, 1};

  uint64_t rnd() {
    seed ^= seed << 13;
    seed ^= seed >> 7;
    seed ^= seed << 17;
    return seed;
  }
  double uniform() { return (double)(rnd() >> 11) * 0x1p-53; }
  void wake(Thread* t) {
    Warp& w = t->cta->warps[t->warp];
    if (t->ready) return;
    t->ready = true;
    (w.held ? w.parked : ready).push_back(t);
  }
  void wake_polling() {
    std::vector<Thread*> v;
    v.swap(polling);
    for (Thread* t : v) wake(t);
  }
  void to_main() { swapcontext(&cur->ctx, &main); }
  void yield(double hold = 0.0) {
    Warp& w = cur->cta->warps[cur->warp];
    if (cur->lane == 0 && !w.held && hold > 0 && uniform() < hold) {
      w.held = true;
      held.push_back(&w);
    }
    ++work;
    wake(cur);
    to_main();
  }
  // A look at something that another thread changes: looks again when something has happened.
  void poll() {
    polling.push_back(cur);
    to_main();
  }
  // Everything that can run has run: the pollers look again (several times, as they do while a warp is delayed), then
  // a warp held back goes on, then time passes.
  bool idle() {
    if (!polling.empty() && (work > 0 || (!held.empty() && rnd() % 64))) {
      work = 0;
      wake_polling();
    } else if (!held.empty()) {
      const size_t i = rnd() % held.size();
      Warp* w = held[i];
      held.erase(held.begin() + i);
      w->held = false;
      ready.insert(ready.end(), w->parked.begin(), w->parked.end());
      w->parked.clear();
      work = 1;
    } else if (!polling.empty()) {
      steps += 100000;
      wake_polling();
    } else {
      return false;
    }
    return true;
  }
  static constexpr size_t kStack = 48 << 10;
  static void entry() {
    extern Scheduler sched;
    sched.body();
    sched.cur->done = true;
    sched.to_main();
  }
  std::unique_ptr<Cta> start(int b, size_t smem) {
    auto c = std::make_unique<Cta>();
    c->bid.x = b;
    c->smem.assign(smem + 64, 0xff);
    c->warps.resize((block.x + 31) / 32);
    c->live = block.x;
    for (int t = 0; t < block.x; ++t) {
      auto th = std::make_unique<Thread>();
      th->tid.x = t;
      th->warp = t / 32;
      th->lane = t % 32;
      th->cta = c.get();
      th->stack = mmap(nullptr, kStack, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS, -1, 0);
      getcontext(&th->ctx);
      th->ctx.uc_stack.ss_sp = th->stack;
      th->ctx.uc_stack.ss_size = kStack;
      th->ctx.uc_link = nullptr;
      makecontext(&th->ctx, entry, 0);
      wake(th.get());
      c->threads.push_back(std::move(th));
    }
    return c;
  }
  // Runs the grid with at most `resident` CTAs at a time, started in order; false on a deadlock.
  bool launch(int ctas, int threads, size_t smem, int resident, std::function<void()> kernel) {
    body = std::move(kernel);
    grid = {ctas, 1, 1};
    block = {threads, 1, 1};
    ready.clear();
    polling.clear();
    held.clear();
    steps = 0;
    std::vector<std::unique_ptr<Cta>> live;
    int next = 0;
    while (next < ctas && (int)live.size() < resident) live.push_back(start(next++, smem));
    while (!live.empty()) {
      if (ready.empty()) {
        if (!idle()) return false;
        continue;
      }
      ++steps;
      const size_t i = rnd() % ready.size();
      Thread* t = ready[i];
      ready[i] = ready.back();
      ready.pop_back();
      t->ready = false;
      cur = t;
      swapcontext(&main, &t->ctx);
      if (t->done) {
        munmap(t->stack, kStack);
        if (--t->cta->live == 0) {
          for (size_t k = 0; k < live.size(); ++k)
            if (live[k].get() == t->cta) {
              live.erase(live.begin() + k);
              break;
            }
          if (next < ctas) live.push_back(start(next++, smem));
        }
      }
    }
    return true;
  }
};
extern Scheduler sched;

// Arrives at a barrier of n threads; waits for the others when block is set.  Returns its generation.
inline int arrive(Barrier& b, int n, bool block, bool pred = false) {
  const int g = b.generation;
  b.any[g & 1] |= pred;
  b.all[g & 1] &= pred;
  if (++b.count == n) {
    b.count = 0;
    ++b.generation;
    b.any[b.generation & 1] = 0;
    b.all[b.generation & 1] = 1;
    for (Thread* t : b.waiting) sched.wake(t);
    b.waiting.clear();
  } else if (block) {
    b.waiting.push_back(sched.cur);
    while (b.generation == g) sched.to_main();
  }
  return g;
}
inline void warp_sync() { arrive(sched.cur->cta->warps[sched.cur->warp].sync, 32, true); }
template <typename T>
T shuffle(T v, int src) {
  Warp& w = sched.cur->cta->warps[sched.cur->warp];
  const int g = w.sync.generation & 1;
  memcpy(&w.box[g][sched.cur->lane], &v, sizeof(T));
  warp_sync();
  T r;
  memcpy(&r, &w.box[g][src], sizeof(T));
  return r;
}
inline int& shared_int(int i) { return sched.cur->cta->ints[i]; }
inline unsigned char* shared_memory() {
  return (unsigned char*)(((uintptr_t)sched.cur->cta->smem.data() + 15) & ~(uintptr_t)15);
}

}  // namespace emu

#define threadIdx (emu::sched.cur->tid)
#define blockIdx (emu::sched.cur->cta->bid)
#define gridDim (emu::sched.grid)
#define blockDim (emu::sched.block)

using std::max;
using std::min;
inline double __fma_rn(double a, double b, double c) { return __builtin_fma(a, b, c); }
inline double __dmul_rn(double a, double b) { return a * b; }
inline double __dsub_rn(double a, double b) { return a - b; }
inline float rsqrtf(float x) { return 1.0f / sqrtf(x); }
inline long long __double_as_longlong(double x) { long long r; memcpy(&r, &x, 8); return r; }
inline double __longlong_as_double(long long x) { double r; memcpy(&r, &x, 8); return r; }
inline int __double2hiint(double x) { return (int)(__double_as_longlong(x) >> 32); }
template <typename T> T __shfl_sync(unsigned, T v, int src) { return emu::shuffle(v, src); }
inline void __syncwarp() { emu::warp_sync(); }
inline void __threadfence() {}
inline void __threadfence_block() {}
inline void __nanosleep(unsigned) {}
inline void bar_sync(int id, int n) { emu::arrive(emu::sched.cur->cta->bars[id], n, true); emu::sched.yield(emu::sched.hold_barrier); }
inline void bar_arrive(int id, int n) { emu::arrive(emu::sched.cur->cta->bars[id], n, false); emu::sched.yield(); }
inline bool bar_or(int id, int n, bool pred) {
  emu::Barrier& b = emu::sched.cur->cta->bars[id];
  const int g = emu::arrive(b, n, true, pred);
  const bool r = b.any[g & 1] != 0;  // the next use of this slot needs every thread of this one back first
  emu::sched.yield(emu::sched.hold_barrier);
  return r;
}
inline void __syncthreads() { bar_sync(0, emu::sched.block.x); }
inline bool __syncthreads_and(bool pred) {
  emu::Barrier& b = emu::sched.cur->cta->bars[0];
  const int g = emu::arrive(b, emu::sched.block.x, true, pred);
  const bool r = b.all[g & 1] != 0;
  emu::sched.yield();
  return r;
}
inline int atomicAdd(int* p, int v) { emu::sched.yield(); const int o = *p; *p += v; return o; }
inline int ld_acquire(const int* p) {
  emu::Thread* t = emu::sched.cur;
  const int now = *(volatile const int*)p;
  if (t->polled == p && t->saw == now)
    emu::sched.poll();
  else
    emu::sched.yield();
  t->polled = p;
  return t->saw = *(volatile const int*)p;
}
// Whoever is held back here has told the others to go on.
inline void red_release(int* p, int v) { *p += v; emu::sched.yield(emu::sched.hold_release); }
inline void or_release(int* p, int v) { *p |= v; emu::sched.yield(emu::sched.hold_release); }
inline double2 ld2(const double2* p) { return *p; }
inline uint64_t globaltimer() { emu::sched.poll(); return (uint64_t)emu::sched.steps * 10; }
