// A warp on the CPU: 32 fibers in lockstep, so that device code that uses warp intrinsics alone can be compiled
// and run by a plain C++ compiler.  Every collective hands the warp's 32 values round; a lane that has ended
// counts as arrived.
#pragma once
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <ucontext.h>

#include <functional>
#include <vector>

#define __device__
#define __host__
#define __forceinline__ inline

namespace warp {
constexpr int kLanes = 32;
inline int lane;
inline uint32_t slot[2][kLanes];
inline int turn[kLanes];
inline bool done[kLanes];
inline ucontext_t ctx[kLanes], host;
inline std::function<void()> body;

inline void fiber() {
  body();
  done[lane] = true;
  for (;;) swapcontext(&ctx[lane], &host);
}

// Every lane's value (the slots alternate: a lane may be one collective ahead of the others, never two).
inline const uint32_t *exchange(uint32_t x) {
  const int t = turn[lane]++ & 1;
  slot[t][lane] = x;
  swapcontext(&ctx[lane], &host);
  return slot[t];
}

// Runs f in all lanes, one collective after another.
inline void run(std::function<void()> f) {
  static std::vector<char> stacks((size_t)kLanes << 16);
  body = std::move(f);
  for (int i = 0; i < kLanes; i++) {
    getcontext(&ctx[i]);
    ctx[i].uc_stack.ss_sp = stacks.data() + ((size_t)i << 16);
    ctx[i].uc_stack.ss_size = (size_t)1 << 16;
    ctx[i].uc_link = &host;
    makecontext(&ctx[i], fiber, 0);
    done[i] = false;
    turn[i] = 0;
  }
  for (bool any = true; any;) {
    any = false;
    for (lane = 0; lane < kLanes; lane++)
      if (!done[lane]) {
        swapcontext(&host, &ctx[lane]);
        any = any || !done[lane];
      }
  }
}
}  // namespace warp

inline unsigned lane_id() { return (unsigned)warp::lane; }
inline unsigned lanemask_lt() { return (1u << warp::lane) - 1u; }
inline int __popc(unsigned x) { return __builtin_popcount(x); }
inline int __ffs(unsigned x) { return __builtin_ffs((int)x); }
inline int __shfl_sync(unsigned, int x, int from) { return (int)warp::exchange((uint32_t)x)[from & 31]; }
inline int __shfl_up_sync(unsigned, int x, int d) {
  const uint32_t *v = warp::exchange((uint32_t)x);
  return warp::lane >= d ? (int)v[warp::lane - d] : x;
}
inline unsigned __ballot_sync(unsigned, bool p) {
  const uint32_t *v = warp::exchange(p);
  unsigned m = 0;
  for (int i = 0; i < warp::kLanes; i++) m |= v[i] << i;
  return m;
}
inline bool __all_sync(unsigned m, bool p) { return __ballot_sync(m, p) == 0xFFFFFFFFu; }
inline unsigned __reduce_or_sync(unsigned, unsigned x) {
  const uint32_t *v = warp::exchange(x);
  unsigned m = 0;
  for (int i = 0; i < warp::kLanes; i++) m |= v[i];
  return m;
}
