// walk.cuh -- how kernels that go over all CSR entries split them: the walk of a warp over its share, and the
// grids of such kernels.  Uses lane_id and lanemask_lt (gp_internal.cuh) and the warp intrinsics, nothing else.
#pragma once
#include <stdint.h>

namespace gp {

inline int grid_for(int64_t items, int per_block, int cap) {
  int64_t g = (items + per_block - 1) / per_block;
  if (g < 1) g = 1;
  if (g > cap) g = cap;
  return (int)g;
}

// A walk of one warp over its share of a graph's CSR entries, 32 consecutive rows (a window) at a
// time.  Rows and entries are split together: a row counts one unit and each of its entries another, and
// every warp gets an even share of the units, in whole rows but for rows of more than kWalkWhole entries.
// With 32 rows per warp step one warp walked a hub's whole row (4e5 entries of the scale-24 R-MAT graph)
// while the rest of the device waited; with even shares of the entries alone one warp walked all the empty
// rows between two of them (8.4M nodes with 840 edges: modularity 1.3 ms, against .18 with 32 rows per warp step and
// .14 now; sparsification .79, .13 and .14).
//
//   for (EntryWalk w(xadj, n, wid, nw); w.next(); )
//     entries [w.e0, w.e1) lie in rows [w.u0, w.u0 + 32); lane i's row is [w.xs, w.xe) (past n: empty);
//     lane 0's may begin before e0, the others begin at or after it
//
// Every step of next() goes 32 rows on and e0, e1 stay between the first and the last offset and never go
// back, also when offsets in between decrease (not every caller checks them).
//
// On graphs of short rows the kernels are bound by instructions (75 % of the issue slots), of which a window
// costs a fixed number, and by the blocks an SM holds: the state is 32 bits a word (rows + entries stay below
// 2^32; with 64 the kernels took 40 to 48 registers instead of 32), and a few entries left in a window take a
// short form of the body (walk_entries).
constexpr int kWalkWhole = 128;

struct EntryWalk {
  const int32_t *xadj;
  unsigned n;
  int hi;            // the last offset
  unsigned until;    // the share ends at this unit
  int pos;           // entries still to walk
  unsigned row;      // the next window's first row
  int start;         // where it begins
  unsigned u0;       // this window's first row
  int e0, e1;
  int xs, xe;        // this lane's row
  int split;         // the lane whose row goes on in the next share (-1: none)
  bool no_empty;     // no row of the window is empty
  int ended;         // rows of the window that end at or before the entry that owner is asked for next
  __device__ __forceinline__ EntryWalk(const int32_t *x, int nn, int wid, int nw) : xadj(x), n((unsigned)nn) {
    // the search's first 32 places, at doubling distances around where even degrees would put the share: read
    // together with the first and the last offset
    const int lane = (int)lane_id();
    const int64_t g = (int64_t)((float)wid / (float)nw * (float)nn);
    const int64_t at = lane < 16 ? g - (1 << (15 - lane)) : g + (1 << (lane - 16)) - 1;
    const unsigned p = at < 0 || nn == 0 ? 0u : at < (int64_t)n ? (unsigned)at : n - 1;
    const int v = nn > 0 ? x[p] : 0, lo = nn > 0 ? x[0] : 0;
    hi = nn > 0 ? x[nn] : 0;
    // row r's units: r + xadj[r] for itself, then r + 1 + e for each of its entries e
    const int64_t all = (int64_t)nn + hi, per = (all - lo + nw - 1) / nw;
    int64_t from = lo + per * wid, to = from + per;
    if (to > all) to = all;
    until = (unsigned)to;
    row = n;
    pos = hi;
    start = 0;
    if (from < to) {
      int next;
      row = first((unsigned)from, p, v, start, next);
      pos = cut(row, start, next, (unsigned)from);
      if (pos < lo) pos = lo;
    }
    u0 = 0; e0 = e1 = xs = xe = 0; split = -1; no_empty = false; ended = 0;
  }
  __device__ __forceinline__ bool next() {
    while (row < n) {
      u0 = row;
      const unsigned end = u0 + lane_id() + 1, u = end < n ? end : n;
      xe = xadj[u];
      xs = __shfl_up_sync(0xFFFFFFFFu, xe, 1);
      if (lane_id() == 0) xs = start;
      start = __shfl_sync(0xFFFFFFFFu, xe, 31);
      int stop = start;
      // the share ends in the first row whose units reach past it; the last one's rows end with row n
      const unsigned past = __ballot_sync(0xFFFFFFFFu, u + (unsigned)xe > until);
      row = u0 + 32;
      if (past) {
        const int j = __ffs(past) - 1;
        const int b = __shfl_sync(0xFFFFFFFFu, xs, j), e = __shfl_sync(0xFFFFFFFFu, xe, j);
        stop = cut(u0 + j, b, e, until);
        split = stop > b ? j : -1;
        row = n;
      }
      if (stop > hi) stop = hi;
      if (stop <= pos) continue;  // no entries here
      e0 = pos;
      e1 = pos = stop;
      no_empty = __all_sync(0xFFFFFFFFu, xs < xe);
      ended = 0;
      return true;
    }
    return false;
  }
  // The entry at which a share begins, or ends, whose unit t lies in row r with entries [b, e).
  __device__ __forceinline__ static int cut(unsigned r, int b, int e, unsigned t) {
    const int c = (int)(t - r - 1);
    return e - b <= kWalkWhole || c < b ? b : c;
  }
  // Row of unit t and its offsets, from 32 ascending places p with their offsets v, then by 32 parts a step: one
  // or two dependent reads where the degrees are near even; they are what a small graph's kernel waits for.
  __device__ __forceinline__ unsigned first(unsigned t, unsigned p, int v, int &begin, int &end) const {
    const int lane = (int)lane_id();
    int k = __popc(__ballot_sync(0xFFFFFFFFu, p + (unsigned)v <= t));  // the reached places come first
    unsigned a = (unsigned)__shfl_sync(0xFFFFFFFFu, (int)p, k > 0 ? k - 1 : 0);
    unsigned b = (unsigned)__shfl_sync(0xFFFFFFFFu, (int)p, k < 32 ? k : 31);
    if (k == 0) a = 0;            // row a is reached (its first unit is at or before t), row b is not
    if (k == 32) b = n;
    if (b <= a) b = a + 1;        // offsets that decrease
    while (b - a > 1) {           // the last step's parts are rows, row a among them for its offset
      const unsigned step = (b - a + 31) / 32;
      p = a + lane * step < b ? a + lane * step : b;
      v = xadj[p];
      k = __popc(__ballot_sync(0xFFFFFFFFu, p < b && p + (unsigned)v <= t));
      a += step * (k > 0 ? k - 1 : 0);
      b = a + step < b ? a + step : b;
    }
    const unsigned lower = __ballot_sync(0xFFFFFFFFu, p == a), upper = __ballot_sync(0xFFFFFFFFu, p == b);
    begin = __shfl_sync(0xFFFFFFFFu, v, lower ? __ffs(lower) - 1 : 0);
    end = __shfl_sync(0xFFFFFFFFu, v, upper ? __ffs(upper) - 1 : 0);
    if (!lower) begin = xadj[a];
    if (!upper) end = xadj[b];
    return a;
  }
  // Lane index of the row that holds entry f + lane (f the same in the whole warp, 32 on from the call before in
  // this window): the lanes whose row ends at or before it.  Without empty rows in the window every row end is
  // another position, so the ends among the 32 entries form a bit mask, and a count of its lower bits replaces
  // the search (one reduction instead of five dependent shuffles).
  __device__ __forceinline__ int owner(int f) {
    if (no_empty) {
      const unsigned d = (unsigned)(xe - f - 1);
      const unsigned ends = __reduce_or_sync(0xFFFFFFFFu, d < 32 ? 1u << d : 0u);
      const int q = ended + __popc(ends & lanemask_lt());
      ended += __popc(ends);
      return q;
    }
    const int e = f + (int)lane_id();
    int q = 0;
#pragma unroll
    for (int step = 16; step > 0; step >>= 1) {
      const int val = __shfl_sync(0xFFFFFFFFu, xe, q + step - 1);
      if (val <= e) q += step;
    }
    return q;
  }
};

// Entries [e0, e1) in steps of 32 R, 64 or 32: body(c, f) takes the entries f + 32 r + lane, r < c.value, that lie
// before e1.
template <int V> struct Steps { static constexpr int value = V; };
template <int R, typename F>
__device__ __forceinline__ void walk_entries(int e0, int e1, F body) {
  for (int f = e0; f < e1;) {
    const int left = e1 - f;
    if (left > 64) {
      body(Steps<R>{}, f);
      f = left > 32 * R ? f + 32 * R : e1;
    } else if (left > 32) {
      body(Steps<2>{}, f);
      f = e1;
    } else {
      body(Steps<1>{}, f);
      f = e1;
    }
  }
}

// Blocks of 256 threads for an EntryWalk: 28 rows a warp, which fit one window, or 576 units where the rows are long;
// on small graphs 112 units until every SM holds four blocks.  No more blocks than the device holds at once
// (per_sm of the kernel an SM) while that leaves a warp at most 4096 units: every block begins with a search, which takes as
// long as a window or two.  Beyond that up to 16 an SM, which evens out what the shares do not.
inline int walk_grid(int64_t n, int64_t m2, int num_sms, int per_sm) {
  const int64_t units = n + m2, few = units / (8 * 112), rows = n / (8 * 28), most = units / (8 * 576);
  int64_t b = few < 4 * (int64_t)num_sms ? few : 4 * (int64_t)num_sms;
  if (b < rows) b = rows;
  if (b < most) b = most;
  return grid_for(b, 1, units / (8 * 4096) <= (int64_t)per_sm * num_sms ? per_sm * num_sms : num_sms * 16);
}

}  // namespace gp
