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
// time.  The entries are split evenly over the warps, not the rows: with 32 rows per warp step one warp
// walked a hub's whole row (4e5 entries of the scale-24 R-MAT graph) while the rest of the device
// waited.  One search per warp (32 probes a step) finds the first row; a window without entries (a long
// run of empty rows) is left by another search.
//
//   for (EntryWalk w(xadj, n, wid, nw); w.next(); )
//     entries [w.e0, w.e1) lie in rows [w.u0, w.u0 + 32); lane i's row ends at w.xe (INT_MAX past n)
struct EntryWalk {
  const int32_t *xadj;
  int n;
  int64_t pos, end;  // entries still to walk
  int64_t u0, row;   // this window's first row, the next one's
  int e0, e1, xe;
  bool no_empty;     // no row of the window is empty
  __device__ __forceinline__ EntryWalk(const int32_t *x, int nn, int wid, int nw) : xadj(x), n(nn) {
    const int64_t lo = nn > 0 ? x[0] : 0, hi = nn > 0 ? x[nn] : 0;
    const int64_t per = (((hi - lo + nw - 1) / nw) + 31) & ~(int64_t)31;
    pos = lo + per * wid;
    end = pos + per < hi ? pos + per : hi;
    row = pos < end ? first(lo, hi) : 0;
    u0 = 0; e0 = e1 = xe = 0; no_empty = false;
  }
  __device__ __forceinline__ bool next() {
    while (pos < end) {
      u0 = row;
      const int64_t u = u0 + lane_id();
      xe = u < n ? xadj[u + 1] : 0x7FFFFFFF;
      const int last = (int)((n - u0) < 32 ? (n - u0) : 32) - 1;
      const int64_t wend = __shfl_sync(0xFFFFFFFFu, xe, last);
      if (wend <= pos) {  // nothing here: jump
        row = find(pos);
        if (row == u0) pos = end;  // this window was that row's: the offsets decrease somewhere (not checked by
        continue;                  // every caller); the walk ends instead of asking again for ever
      }
      e0 = (int)pos;
      e1 = (int)(wend < end ? wend : end);
      const int before = __shfl_up_sync(0xFFFFFFFFu, xe, 1);
      no_empty = __all_sync(0xFFFFFFFFu, lane_id() == 0 || u >= n || before < xe);
      pos = e1;
      row = u0 + 32;
      return true;
    }
    return false;
  }
  // Row of entry pos: where even degrees would put it, else by the search.
  __device__ __forceinline__ int64_t first(int64_t lo, int64_t hi) const {
    int64_t g = (int64_t)((float)(pos - lo) / (float)(hi - lo) * (float)n) - 16;
    g = g < 0 ? 0 : g > n ? n : g;
    const int64_t p = g + lane_id();
    const unsigned m = __ballot_sync(0xFFFFFFFFu, p < n && (int64_t)xadj[p] <= pos);
    return (m & 1) && m != 0xFFFFFFFFu ? g + __popc(m) - 1 : find(pos);
  }
  // Row of entry e (xadj[0] <= e < xadj[n]); the whole warp asks for the same e.
  __device__ __forceinline__ int64_t find(int64_t e) const {
    int64_t a = 0, b = n;  // xadj[a] <= e < xadj[b]
    while (b - a > 1) {
      const int64_t step = (b - a + 32) / 33, p = a + (int64_t)(lane_id() + 1) * step;
      const unsigned m = __ballot_sync(0xFFFFFFFFu, p < b && (int64_t)xadj[p] <= e);
      a += step * __popc(m);
      b = a + step < b ? a + step : b;
    }
    return a;
  }
  // Lane index of the row that holds entry f + lane (f the same in the whole warp): the lanes whose row
  // ends at or before it.  Without empty rows in the window every row end is another position, so the
  // ends among the 32 entries form a bit mask, and a count of its lower bits replaces the search (one
  // reduction instead of five dependent shuffles).
  __device__ __forceinline__ int owner(int f) const {
    if (no_empty) {
      const int d = xe - f;
      const unsigned ends = __reduce_or_sync(0xFFFFFFFFu, d > 0 && d < 32 ? 1u << d : 0u);
      return __popc(__ballot_sync(0xFFFFFFFFu, d <= 0)) + __popc(ends & (lanemask_lt() | (1u << lane_id())));
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

// Blocks of 256 threads for an EntryWalk over m2 entries: 96 entries a warp (the 32 rows of a mesh hold 128) until
// every SM holds four blocks, then more entries a warp up to 512, then more blocks up to 16 an SM.  With
// 2048 entries a warp throughout, small graphs kept a few SMs busy with chains of a dozen steps (a small
// graph's scoring took 334 us against 201 with a warp per 32 rows; ER partition of 65,536 nodes 7.69 -> 7.5 ms); with 128 to 512 entries a warp small meshes'
// kernels took a second window's chain, some 3 us each.
inline int walk_grid(int64_t m2, int num_sms) {
  const int64_t b = m2 / (8 * 96) < 4 * (int64_t)num_sms ? m2 / (8 * 96) : 4 * (int64_t)num_sms;
  return grid_for(b * 256 > m2 / 16 ? b * 256 : m2 / 16, 256, num_sms * 16);
}

}  // namespace gp
