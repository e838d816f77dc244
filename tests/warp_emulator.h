// A CPU stand-in for one warp at a time of a generated kernel: every lane is a fiber, the lanes run one after another,
// each up to its next warp-wide operation, which completes when every lane of its mask has come to it.  Lanes that come
// to different operations of the same mask, or that wait for lanes that have finished, end the run with exit code 3: on
// a GPU, where nothing orders lanes between such operations, the warp could hang.  The order in which the lanes run
// between two operations is a parameter, so code that is right only while a warp happens to stay converged shows.
#pragma once
#include <ucontext.h>

#include <algorithm>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#define __device__
#define __global__
#define __forceinline__ inline
#define __noinline__ __attribute__((noinline))
#define __launch_bounds__(...)
#define __grid_constant__
#define __shared__ static
#define __align__(n) __attribute__((aligned(n)))

struct uint2 {
  unsigned x, y;
};
struct uint4 {
  unsigned x, y, z, w;
};
static inline uint2 make_uint2(unsigned x, unsigned y) { return {x, y}; }
static inline uint4 make_uint4(unsigned x, unsigned y, unsigned z, unsigned w) { return {x, y, z, w}; }
struct Dim {
  unsigned x;
};
static Dim threadIdx, blockIdx;

template <class T>
static inline T min(T a, T b) { return b < a ? b : a; }
template <class T>
static inline T __ldg(const T* p) { return *p; }
static inline int __ffs(unsigned x) { return __builtin_ffs((int)x); }
static inline int __popc(unsigned x) { return __builtin_popcount(x); }
static inline unsigned __funnelshift_r(unsigned lo, unsigned hi, unsigned s) {
  return (unsigned)(((uint64_t)hi << 32 | lo) >> (s & 31));
}
static inline unsigned __byte_perm(unsigned a, unsigned b, unsigned s) {
  const uint64_t v = (uint64_t)b << 32 | a;
  unsigned r = 0;
  for (int i = 0; i < 4; ++i) r |= (unsigned)((v >> (8 * (s >> (4 * i) & 7))) & 255) << (8 * i);
  return r;
}
static inline unsigned lop3(unsigned a, unsigned b, unsigned c, unsigned lut) {
  unsigned r = 0;
  for (int i = 0; i < 8; ++i)
    if (lut >> i & 1) r |= (i & 4 ? a : ~a) & (i & 2 ? b : ~b) & (i & 1 ? c : ~c);
  return r;
}
static inline unsigned atomicAdd(unsigned* p, unsigned v) { const unsigned o = *p; *p += v; return o; }
static inline unsigned atomicOr(unsigned* p, unsigned v) { const unsigned o = *p; *p |= v; return o; }

namespace warp {
enum Op { kRunning, kSync, kAny, kMatch, kShfl, kDone };
struct Lane {
  ucontext_t ctx;
  std::vector<char> stack;
  Op op = kRunning;
  unsigned mask = 0;
  uint64_t in = 0, out = 0;
  int src = 0;
  bool arrived = false;
};
static Lane lanes[32];
static ucontext_t scheduler;
static int current = 0;

static inline uint64_t meet(Op op, unsigned mask, uint64_t in, int src = 0) {
  const int me = current;
  Lane& l = lanes[me];
  l.op = op, l.mask = mask, l.in = in, l.src = src, l.arrived = true;
  swapcontext(&l.ctx, &scheduler);
  return lanes[me].out;
}

// runs one warp of `kernel` (threads 32 w .. 32 w + 31 of block b); order: 0 ascending lanes, 1 descending, else a
// different order each time
template <class F>
void run(unsigned b, unsigned w, int order, F&& kernel) {
  static F* f;
  f = &kernel;
  blockIdx.x = b;
  for (int i = 0; i < 32; ++i) {
    Lane& l = lanes[i];
    if (l.stack.empty()) l.stack.resize(256 << 10);
    getcontext(&l.ctx);
    l.ctx.uc_stack.ss_sp = l.stack.data();
    l.ctx.uc_stack.ss_size = l.stack.size();
    l.ctx.uc_link = nullptr;
    l.arrived = false;
    l.op = kRunning;
    makecontext(&l.ctx, +[] {
      (*f)();
      lanes[current].op = kDone;
      swapcontext(&lanes[current].ctx, &scheduler);
    }, 0);
  }
  uint64_t random = 88172645463325252ull + b * 64 + w + (uint64_t)order * 7919;
  for (;;) {
    int at[32];
    for (int i = 0; i < 32; ++i) at[i] = order == 1 ? 31 - i : i;
    if (order > 1)
      for (int i = 31; i > 0; --i) {
        random ^= random << 13, random ^= random >> 7, random ^= random << 17;
        std::swap(at[i], at[random % (i + 1)]);
      }
    bool ran = false;
    for (int i : at) {
      if (lanes[i].op == kDone || lanes[i].arrived) continue;
      ran = true;
      current = i;
      threadIdx.x = 32 * w + i;
      swapcontext(&scheduler, &lanes[i].ctx);
    }
    // operations whose lanes are all there
    bool done = true, resolved = false;
    for (int i = 0; i < 32; ++i) {
      if (lanes[i].op == kDone) continue;
      done = false;
      if (!lanes[i].arrived) continue;
      const unsigned mask = lanes[i].mask;
      if (!(mask >> i & 1)) {
        fprintf(stderr, "lane %d is not in its mask %08x\n", i, mask);
        exit(3);
      }
      bool all = true;
      for (int k = 0; k < 32; ++k)
        if (mask >> k & 1) all = all && lanes[k].arrived && lanes[k].op == lanes[i].op && lanes[k].mask == mask;
      if (!all) continue;
      uint64_t any = 0;
      for (int k = 0; k < 32; ++k)
        if (mask >> k & 1) any |= lanes[k].in;
      for (int k = 0; k < 32; ++k) {
        if (!(mask >> k & 1)) continue;
        Lane& l = lanes[k];
        if (l.op == kAny) l.out = any != 0;
        if (l.op == kShfl) l.out = lanes[l.src].in;
        if (l.op == kMatch) {
          l.out = 0;
          for (int j = 0; j < 32; ++j)
            if ((mask >> j & 1) && lanes[j].in == l.in) l.out |= 1ull << j;
        }
      }
      for (int k = 0; k < 32; ++k)
        if (mask >> k & 1) lanes[k].arrived = false;
      resolved = true;
    }
    if (done) return;
    if (!ran && !resolved) {
      fprintf(stderr, "block %u warp %u: lanes wait for each other at different operations\n", b, w);
      exit(3);
    }
  }
}
}  // namespace warp

static inline void __syncwarp(unsigned mask = ~0u) { warp::meet(warp::kSync, mask, 0); }
static inline bool __any_sync(unsigned mask, bool v) { return warp::meet(warp::kAny, mask, v) != 0; }
static inline unsigned __match_any_sync(unsigned mask, unsigned long long v) {
  return (unsigned)warp::meet(warp::kMatch, mask, v);
}
static inline unsigned __shfl_sync(unsigned mask, unsigned v, int src) {
  return (unsigned)warp::meet(warp::kShfl, mask, v, src);
}
