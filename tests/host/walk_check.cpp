// EntryWalk on the CPU: every entry is handed out once, in order, with its row; on offsets that decrease
// somewhere the walk ends and stays within the offsets' range; and the work is even over the warps, also
// where entries or rows lie unevenly.
#include "warp.h"

#include "walk.cuh"

static unsigned rng_state = 12345;
static unsigned rnd(unsigned m) {
  rng_state = rng_state * 1664525u + 1013904223u;
  return (unsigned)(((uint64_t)(rng_state >> 4) * m) >> 28);
}

static int walk(const std::vector<int32_t> &xadj, int nw, bool monotone) {
  const int n = (int)xadj.size() - 1;
  const int64_t lo = xadj[0], hi = xadj[n];
  int64_t expect = lo;
  int bad = 0;
  for (int w = 0; w < nw; w++)
    warp::run([&] {
      int64_t steps = 0;
      for (gp::EntryWalk wk(xadj.data(), n, w, nw); wk.next();) {
        if (++steps > hi - lo) { bad |= 1; break; }
        if (lane_id() == 0) {
          if (wk.e0 < lo || wk.e1 > hi || wk.e1 <= wk.e0) bad |= 2;
          if (monotone && wk.e0 != expect) bad |= 4;
          expect = wk.e1;
        }
        for (int f = wk.e0; f < wk.e1; f += 32) {
          const int q = wk.owner(f), e = f + (int)lane_id();
          const int64_t r = wk.u0 + q;
          if (e < wk.e1 && monotone && !(r < n && xadj[r] <= e && e < xadj[r + 1])) bad |= 8;
        }
      }
    });
  if (monotone && expect != hi) bad |= 16;
  return bad;
}

// Most collectives a warp of a walk takes to go over its share.
static int most(const std::vector<int32_t> &xadj, int nw) {
  const int n = (int)xadj.size() - 1;
  int m = 0;
  for (int w = 0; w < nw; w++) {
    warp::run([&] {
      for (gp::EntryWalk wk(xadj.data(), n, w, nw); wk.next();)
        for (int f = wk.e0; f < wk.e1; f += 32) wk.owner(f);
    });
    m = warp::turn[0] > m ? warp::turn[0] : m;
  }
  return m;
}

static int even() {
  int bad = 0;
  const int n = 1 << 17, sms = 8;
  for (int kind = 0; kind < 6; kind++) {
    std::vector<int32_t> x(n + 1);
    for (int i = 0; i < n; i++) {  // few entries anywhere | at one end | one hub | even | none | a dense end
      const int deg = kind == 0 ? i % 9973 == 17 : kind == 1 ? i < 16 : kind == 2 ? (i == 70000 ? 100000 : i % 64 == 0)
                    : kind == 3 ? 2 : kind == 4 ? 0 : i < 4096 ? 64 : i % 1024 == 3;
      x[i + 1] = x[i] + deg;
    }
    const int blocks = gp::walk_grid(n, x[n], sms, 8), nw = blocks * 8;
    // a warp takes the search, a window's five collectives per 32 units and an owner's seven per 32 entries
    const int64_t units = (int64_t)n + x[n], per = units / nw + 1;
    const int got = most(x, nw), allowed = 40 + (int)(per * (5.0 / 32 + 7.0 / 32));
    if (got > allowed) {
      printf("kind=%d blocks=%d: %d collectives, %d allowed\n", kind, blocks, got, allowed);
      bad = 32;
    }
    if (blocks < (units < 8 * 576 * 4 * sms ? 1 : 4 * sms)) bad |= 64;
  }
  // millions of nodes fill the device whatever the entries
  if (gp::walk_grid(8 << 20, 0, 152, 8) < 152 * 8 || gp::walk_grid(1, 0, 152, 8) != 1) bad |= 64;
  return bad;
}

int main(int argc, char **argv) {
  if (argc > 1 && argv[1][0] == 'e') return even();
  const bool monotone = argc > 1 && argv[1][0] == 'm';
  int bad = 0;
  if (monotone) {
    for (int n : {0, 1, 2, 31, 32, 33, 64, 65, 500})
      for (int kind = 0; kind < 6; kind++)
        for (int nw : {1, 2, 7, 40}) {
          std::vector<int32_t> x(n + 1);
          x[0] = kind == 5 ? 17 : 0;
          for (int i = 0; i < n; i++) {
            const int deg = kind == 0 ? 1 : kind == 1 ? (int)rnd(9) : kind == 2 ? (i % 70 == 69 ? 5 : 0)
                          : kind == 3 ? (i == n / 2 ? 3000 : (int)rnd(2)) : kind == 4 ? 0 : 1 + (int)rnd(40);
            x[i + 1] = x[i] + deg;
          }
          const int b = walk(x, nw, true);
          if (b) printf("n=%d kind=%d nw=%d: %d\n", n, kind, nw, b);
          bad |= b;
        }
  } else {
    // row 19 is found for entry 10, and its window of 32 rows ends at entry 5
    std::vector<int32_t> x(65, 200);
    for (int i = 0; i < 20; i++) x[i] = i == 0 ? 0 : 5;
    x[51] = 5;
    x[64] = 100;
    for (int nw : {1, 2, 3, 10}) bad |= walk(x, nw, false);
    for (int rep = 0; rep < 2000; rep++) {
      const int n = 1 + (int)rnd(150);
      std::vector<int32_t> y(n + 1);
      for (int i = 0; i <= n; i++) y[i] = (int)rnd(300);
      if (rep & 1)
        for (int i = 1; i <= n; i++) y[i] = rnd(8) ? y[i - 1] + (int)rnd(4) : y[i];
      bad |= walk(y, 1 + (int)rnd(6), false);
    }
  }
  printf("bad=%d\n", bad);
  return bad != 0;
}
