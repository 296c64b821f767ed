// contract.cu -- cluster contraction (Sec. 2): coarse node A weighs the sum
// of its members' weights; coarse edge {A, B}, A != B, weighs the total
// weight of the fine edges between the clusters.
//
// Three passes over the fine graph, each with coalesced streams:
//  reserve: every fine node reserves room for its row inside its coarse
//           node's segment (an atomic add on the segment length returns the
//           node's offset) and adds its weight to the coarse node;
//  map    : rows and entries are split evenly over the warps (EntryWalk),
//           which write (coarse id of the neighbour, weight) into the owner's
//           segment; entries inside the cluster are marked;
//  merge  : each segment is summed by coarse neighbour in a hash table (a
//           warp with a shared-memory table up to 128 entries, a block with
//           a 4096-slot shared table up to 2048, many blocks with a table in
//           global memory above, or a block each where those tables together
//           would pass the memory bound) and written back in place, compacted;
// and the merged rows are finally packed into the coarse CSR.  Row order
// inside a coarse row is unspecified.
#include "gp_internal.cuh"

namespace gp {

namespace {

constexpr unsigned FULL = 0xFFFFFFFFu;
constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kWarpSlots = 256;
constexpr int kWarpMaxUb = 128;
constexpr int kBlockSmemSlots = 4096;
constexpr int kMapUnroll = 8;
constexpr int kHugeSeg = 2048;       // segments above this many entries are merged by many blocks
constexpr int kSegChunk = 2048;      // their entries per block and step
constexpr int kSegTabChunk = 4096;   // and table slots
constexpr unsigned long long kEmptySlot = 0xFFFFFFFFull;  // the slot (-1, 0): neighbour in the low half

__device__ __forceinline__ unsigned slot_hash(int B, int bits) {
  return ((unsigned)B * 2654435761u) >> (32 - bits);
}

__device__ __forceinline__ void table_add(int *tk, int *tv, unsigned mask, int bits, int B, int w) {
  unsigned s = slot_hash(B, bits);
  for (unsigned probe = 0; probe <= mask; probe++) {  // bounded: more slots than keys
    const int prev = atomicCAS(&tk[s], -1, B);
    if (prev == -1 || prev == B) { atomicAdd(&tv[s], w); return; }
    s = (s + 1) & mask;
  }
}

// Distinct neighbours that a segment of len entries can have: no more than there are coarse nodes.
__host__ __device__ __forceinline__ int seg_keys(int len, int nc) { return len < nc ? len : nc; }

// Segment length (the member rows' total length) and weight of every coarse
// node; moff[v] = offset of v's row inside its coarse node's segment.
__global__ void k_reserve(const int32_t *xadj, const int32_t *vwgt, const int32_t *cmap, int n, int32_t *seg,
                          int32_t *cw, int32_t *moff) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x) {
    const int A = cmap[v];
    moff[v] = atomicAdd(&seg[A], xadj[v + 1] - xadj[v]);
    atomicAdd(&cw[A], vwgt[v]);
  }
}

// (coarse neighbour, weight) of every fine entry into its owner's segment;
// entries inside the owner's cluster get neighbour -1.
__global__ void __launch_bounds__(kThreads) k_map(const int32_t *xadj, const int32_t *adjncy,
                                                  const int32_t *adjwgt, const int32_t *cmap,
                                                  const int32_t *moff, const int32_t *tstart, int n,
                                                  int2 *temp, unsigned long long *units) {
  const int lane = (int)lane_id();
  const int wid = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int nw = (int)((gridDim.x * blockDim.x) >> 5);
  unsigned long long ue = 0;
  for (EntryWalk wk(xadj, n, wid, nw); wk.next();) {
    const int64_t u = wk.u0 + lane;
    int A = -2, base = 0;
    if (u < n) {
      A = cmap[u];
      base = tstart[A] + moff[u] - wk.xs;
    }
    const int e1 = wk.e1;
    if (lane == 0) ue += (unsigned long long)(e1 - wk.e0);
    // kMapUnroll entries per lane in flight: ids, then coarse ids, then the writes
    walk_entries<kMapUnroll>(wk.e0, e1, [&](auto steps, int f0) {
      constexpr int R = decltype(steps)::value;
      int e[R], bj[R], Aj[R], nb[R];
#pragma unroll
      for (int r = 0; r < R; r++) {
        e[r] = f0 + r * 32 + lane;
        const int j = wk.owner(f0 + r * 32);
        bj[r] = __shfl_sync(FULL, base, j);
        Aj[r] = __shfl_sync(FULL, A, j);
      }
#pragma unroll
      for (int r = 0; r < R; r++) nb[r] = e[r] < e1 ? __ldcs(adjncy + e[r]) : 0;  // read once: evict first
#pragma unroll
      for (int r = 0; r < R; r++) nb[r] = e[r] < e1 ? cmap[nb[r]] : 0;
#pragma unroll
      for (int r = 0; r < R; r++)
        if (e[r] < e1) temp[bj[r] + e[r]] = nb[r] == Aj[r] ? make_int2(-1, 0) : make_int2(nb[r], adjwgt ? __ldcs(adjwgt + e[r]) : 1);
    });
  }
  ue = warp_sum(ue);
  if (units && lane == 0) {
    atomicAdd(units + 0, ue);
    if (!adjwgt) atomicAdd(units + 5, ue);
  }
}

struct MergeArgs {
  const int32_t *tstart;
  int nc;
  int2 *temp;
  int32_t *rowcnt;
  int32_t *large, *nlarge;  // segments for a block each, from the front; huge ones (nlarge[1]) from the back
  int split_huge;           // 1: segments above kHugeSeg go to the huge list
  int32_t *gkeys, *gvals;
  int64_t gstride;
  unsigned long long *units;
};

// One warp per coarse node whose segment holds at most kWarpMaxUb entries.
__global__ void __launch_bounds__(kThreads) k_merge_warp(MergeArgs a) {
  __shared__ int s_k[kWarps][kWarpSlots];
  __shared__ int s_v[kWarps][kWarpSlots];
  const int lane = (int)lane_id(), wib = threadIdx.x >> 5;
  int *tk = s_k[wib], *tv = s_v[wib];
  for (int t = lane; t < kWarpSlots; t += 32) { tk[t] = -1; tv[t] = 0; }
  __syncwarp();
  const int wid = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int nw = (int)((gridDim.x * blockDim.x) >> 5);
  unsigned long long uout = 0;
  for (int A = wid; A < a.nc; A += nw) {
    const int s0 = a.tstart[A], s1 = a.tstart[A + 1];
    const int len = s1 - s0;
    if (len > kWarpMaxUb) {
      if (lane == 0) {
        if (a.split_huge && len > kHugeSeg) a.large[a.nc - atomicAdd(a.nlarge + 1, 1)] = A;
        else a.large[atomicAdd(a.nlarge, 1)] = A;
      }
      continue;
    }
    const int bits = table_bits(len, 5), tsize = 1 << bits;
    for (int i0 = s0; i0 < s1; i0 += 64) {  // two entries per lane in flight
      const int i1 = i0 + lane, i2 = i0 + 32 + lane;
      const int2 x1 = i1 < s1 ? __ldcs(a.temp + i1) : make_int2(-1, 0);
      const int2 x2 = i2 < s1 ? __ldcs(a.temp + i2) : make_int2(-1, 0);
      if (x1.x >= 0) table_add(tk, tv, tsize - 1, bits, x1.x, x1.y);
      if (x2.x >= 0) table_add(tk, tv, tsize - 1, bits, x2.x, x2.y);
    }
    __syncwarp();
    // extract in slot order and leave the table clean for the next node
    int cnt = 0;
    for (int t0 = 0; t0 < tsize; t0 += 32) {
      const int key = tk[t0 + lane];
      const bool occ = key >= 0;
      const unsigned m = __ballot_sync(FULL, occ);
      if (occ) {
        a.temp[s0 + cnt + __popc(m & lanemask_lt())] = make_int2(key, tv[t0 + lane]);
        tk[t0 + lane] = -1;
        tv[t0 + lane] = 0;
      }
      cnt += __popc(m);
    }
    if (lane == 0) a.rowcnt[A] = cnt;
    uout += cnt;
    __syncwarp();
  }
  if (a.units && lane == 0) atomicAdd(a.units + 3, uout);
}

// One block per coarse node of the large list.
__global__ void __launch_bounds__(kThreads) k_merge_block(MergeArgs a) {
  __shared__ int s_k[kBlockSmemSlots];
  __shared__ int s_v[kBlockSmemSlots];
  __shared__ int s_cnt;
  const int nl = *a.nlarge;
  int *gk = a.gkeys ? a.gkeys + (int64_t)blockIdx.x * a.gstride : nullptr;
  int *gv = a.gvals ? a.gvals + (int64_t)blockIdx.x * a.gstride : nullptr;
  unsigned long long uout = 0;
  for (int li = blockIdx.x; li < nl; li += gridDim.x) {
    const int A = a.large[li];
    const int s0 = a.tstart[A], s1 = a.tstart[A + 1];
    const int bits = table_bits(seg_keys(s1 - s0, a.nc), 5);
    const unsigned tsize = 1u << bits;
    const bool in_smem = tsize <= kBlockSmemSlots;
    int *tk = in_smem ? s_k : gk;
    int *tv = in_smem ? s_v : gv;
    for (unsigned t = threadIdx.x; t < tsize; t += blockDim.x) { tk[t] = -1; tv[t] = 0; }
    if (threadIdx.x == 0) s_cnt = 0;
    __syncthreads();
    for (int i = s0 + threadIdx.x; i < s1; i += blockDim.x) {
      const int2 x = a.temp[i];
      if (x.x >= 0) table_add(tk, tv, tsize - 1, bits, x.x, x.y);
    }
    __syncthreads();
    for (unsigned t = threadIdx.x; t < tsize; t += blockDim.x) {
      const int key = tk[t];
      if (key >= 0) a.temp[s0 + atomicAdd(&s_cnt, 1)] = make_int2(key, tv[t]);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      a.rowcnt[A] = s_cnt;
      uout += s_cnt;
    }
    __syncthreads();
  }
  if (a.units && threadIdx.x == 0) atomicAdd(a.units + 3, uout);
}

// Longest segment, number of huge ones and the keys their tables have to hold.
struct SegStats {
  int longest, huge;
  unsigned long long keys;
};

__global__ void k_seg_stats(const int32_t *x, int n, SegStats *out) {
  int m = 0, nh = 0;
  unsigned long long ns = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int l = x[i];
    m = l > m ? l : m;
    if (l > kHugeSeg) { nh++; ns += (unsigned long long)seg_keys(l, n); }
  }
  m = warp_max(m);
  if (lane_id() == 0 && m) atomicMax(&out->longest, m);
  if (__any_sync(FULL, nh)) {
    nh = warp_sum(nh);
    ns = warp_sum(ns);
    if (lane_id() == 0) { atomicAdd(&out->huge, nh); atomicAdd(&out->keys, ns); }
  }
}

// ------------------------------------- huge segments: many blocks a segment
//
// A coarse node that holds a hub has a segment of up to several 1e5 entries; one block with a table in
// global memory took milliseconds for it while the rest of the device waited (12 levels of the scale-24
// R-MAT graph: 131 ms of contraction).  k_seg_plan lists the huge segments with the prefix sums of their
// chunks, k_seg_insert sums 2048 entries at a time in a shared table and adds the sums to the segment's
// table in global memory (two slots a key where the memory bound allows, a key being an entry or, if there are
// fewer of them, a coarse node; one 64-bit exchange claims a
// slot), and k_seg_extract writes the occupied slots back to the
// segment.  Consecutive steps work on the same few tables, which stay in L2 meanwhile.

struct Seg {
  int A, s0, len, tsize;
  long long toff;
};

struct SegArgs {
  Seg *segs;
  int *chunk0, *tchunk0;  // prefix sums of entry chunks and table chunks; [count] = totals
  int2 *tab;              // (coarse neighbour, weight) slots
  int q4;                 // slots a key, in quarters
};

__global__ void __launch_bounds__(1024) k_seg_plan(MergeArgs a, SegArgs h) {
  __shared__ long long s_w[3][32];
  const int cnt = a.nlarge[1];
  const int lane = (int)lane_id(), wp = threadIdx.x >> 5;
  long long run[3] = {0, 0, 0};  // entry chunks, table chunks, table slots
  for (int b = 0; b < cnt; b += 1024) {
    const int i = b + (int)threadIdx.x;
    Seg x{};
    if (i < cnt) {
      x.A = a.large[a.nc - i];
      x.s0 = a.tstart[x.A];
      x.len = a.tstart[x.A + 1] - x.s0;
      x.tsize = tab_slots(seg_keys(x.len, a.nc), h.q4);
    }
    const long long val[3] = {chunks_of(x.len, kSegChunk), chunks_of(x.tsize, kSegTabChunk), x.tsize};
    long long ex[3];
#pragma unroll
    for (int q = 0; q < 3; q++) {
      long long y = val[q];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const long long z = __shfl_up_sync(FULL, y, o);
        if (lane >= o) y += z;
      }
      if (lane == 31) s_w[q][wp] = y;
      ex[q] = y - val[q];
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 3; q++) {
      long long before = run[q], total = run[q];
      for (int w = 0; w < 32; w++) {
        if (w < wp) before += s_w[q][w];
        total += s_w[q][w];
      }
      ex[q] += before;
      run[q] = total;
    }
    if (i < cnt) {
      x.toff = ex[2];
      h.segs[i] = x;
      h.chunk0[i] = (int)ex[0];
      h.tchunk0[i] = (int)ex[1];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    h.chunk0[cnt] = (int)run[0];
    h.tchunk0[cnt] = (int)run[1];
  }
}

__device__ __forceinline__ int seg_of(const int *first, int cnt, int it) {
  int lo = 0, hi = cnt;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (first[mid] <= it) lo = mid; else hi = mid;
  }
  return lo;
}

__global__ void k_seg_clear(int2 *tab, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    tab[i] = make_int2(-1, 0);
}

__global__ void __launch_bounds__(kThreads) k_seg_insert(MergeArgs a, SegArgs h) {
  __shared__ int s_k[2 * kSegChunk];
  __shared__ int s_v[2 * kSegChunk];
  constexpr int BITS = 12;
  static_assert((1 << BITS) == 2 * kSegChunk, "table size");
  const int cnt = a.nlarge[1], items = h.chunk0[cnt];
  for (int t = threadIdx.x; t < 2 * kSegChunk; t += blockDim.x) { s_k[t] = -1; s_v[t] = 0; }
  for (int it = blockIdx.x; it < items; it += gridDim.x) {
    const int si = seg_of(h.chunk0, cnt, it);
    const Seg x = h.segs[si];
    int2 *tab = h.tab + x.toff;
    const int c0 = (it - h.chunk0[si]) * kSegChunk, left = min(x.len - c0, kSegChunk);
    const int2 *in = a.temp + x.s0 + c0;
    constexpr int R = kSegChunk / kThreads;
    int2 e[R];
#pragma unroll
    for (int r = 0; r < R; r++) {
      const int j = r * kThreads + (int)threadIdx.x;
      e[r] = j < left ? __ldcs(in + j) : make_int2(-1, 0);
    }
    __syncthreads();  // the shared table is empty
#pragma unroll
    for (int r = 0; r < R; r++)
      if (e[r].x >= 0) table_add(s_k, s_v, 2 * kSegChunk - 1, BITS, e[r].x, e[r].y);
    __syncthreads();
    for (int t = threadIdx.x; t < 2 * kSegChunk; t += blockDim.x) {
      const int B = s_k[t];
      if (B < 0) continue;
      const int w = s_v[t];
      s_k[t] = -1;
      s_v[t] = 0;
      int s = (int)__umulhi((unsigned)B * 2654435761u, (unsigned)x.tsize);
      for (int probe = 0; probe < x.tsize; probe++) {  // bounded: more slots than keys
        const unsigned long long prev = atomicCAS((unsigned long long *)&tab[s], kEmptySlot,
                                                  ((unsigned long long)(unsigned)w << 32) | (unsigned)B);
        if (prev == kEmptySlot) break;
        if ((int)(unsigned)prev == B) { atomicAdd(&tab[s].y, w); break; }
        s = s + 1 == x.tsize ? 0 : s + 1;
      }
    }
  }
}

__global__ void __launch_bounds__(kThreads) k_seg_extract(MergeArgs a, SegArgs h) {
  const int cnt = a.nlarge[1], items = h.tchunk0[cnt];
  unsigned long long uout = 0;
  for (int it = blockIdx.x; it < items; it += gridDim.x) {
    const int si = seg_of(h.tchunk0, cnt, it);
    const Seg x = h.segs[si];
    const int2 *tab = h.tab + x.toff;
    const int t0 = (it - h.tchunk0[si]) * kSegTabChunk, t1 = min(x.tsize, t0 + kSegTabChunk);
    constexpr int R = 8;
    for (int b = t0 + (int)(threadIdx.x & ~31u); b < t1; b += kThreads * R) {  // a warp's R x 32 slots a step
      int2 e[R];
      unsigned m[R];
      int n = 0;
#pragma unroll
      for (int r = 0; r < R; r++) {
        const int t = b + r * kThreads + (int)lane_id();
        e[r] = t < t1 ? __ldcs(tab + t) : make_int2(-1, 0);
      }
#pragma unroll
      for (int r = 0; r < R; r++) {
        m[r] = __ballot_sync(FULL, e[r].x >= 0);
        n += __popc(m[r]);
      }
      int pos = 0;
      if (lane_id() == 0 && n) pos = atomicAdd(&a.rowcnt[x.A], n);
      pos = x.s0 + __shfl_sync(FULL, pos, 0);
#pragma unroll
      for (int r = 0; r < R; r++) {
        if (e[r].x >= 0) a.temp[pos + __popc(m[r] & lanemask_lt())] = e[r];
        pos += __popc(m[r]);
      }
      uout += (unsigned)n;
    }
  }
  if (a.units && lane_id() == 0 && uout) atomicAdd(a.units + 3, uout);
}

// Packs the merged rows from the segment layout into the final CSR.
__global__ void __launch_bounds__(kThreads) k_pack_rows(const int32_t *tstart, const int32_t *rowcnt,
                                                        const int32_t *xadj_out, int nc, const int2 *temp,
                                                        int32_t *adj, int32_t *w) {
  const int lane = (int)lane_id();
  const int wid = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int nw = (int)((gridDim.x * blockDim.x) >> 5);
  for (int A = wid; A < nc; A += nw) {
    const int src = tstart[A], dst = xadj_out[A], c = rowcnt[A];
    for (int j = lane; j < c; j += 32) {
      const int2 x = temp[src + j];
      adj[dst + j] = x.x;
      w[dst + j] = x.y;
    }
  }
}

}  // namespace

void contract_graph(gp_ctx *ctx, const DevGraph &g, const int32_t *cmap, int32_t nc, DevGraph &out) {
  TraceTimer trace(ctx);
  const int n = g.n;
  const int grid = grid_for(n, 256, ctx->num_sms * 8);
  DBuf<int32_t> seg(ctx, (size_t)nc + 1), cw(ctx, (size_t)nc + 1), tstart(ctx, (size_t)nc + 1);
  DBuf<int32_t> moff(ctx, (size_t)(n > 0 ? n : 1));
  {
    ProfScope ps(ctx, PROF_CONTRACT_AUX);
    seg.zero(); cw.zero();
    k_reserve<<<grid, 256, 0, ctx->stream>>>(g.xadj, g.vwgt, cmap, n, seg.get(), cw.get(), moff.get());
    GP_LAUNCH_CHECK();
    scan_exclusive_i32(ctx, seg.get(), tstart.get(), nc + 1, nullptr);
  }
  DBuf<int2> temp(ctx, (size_t)(g.m2 > 0 ? g.m2 : 1));
  DBuf<int32_t> rowcnt(ctx, (size_t)nc + 1), large(ctx, (size_t)nc + 1), nlarge(ctx, 2);
  rowcnt.zero();
  nlarge.zero();
  MergeArgs a{};
  a.tstart = tstart.get(); a.nc = nc; a.temp = temp.get(); a.rowcnt = rowcnt.get();
  a.large = large.get(); a.nlarge = nlarge.get();
  unsigned long long *units = ctx->d_units ? ctx->d_units + PROF_CONTRACT * PROF_UNITS : nullptr;
  a.units = units;
  // segments beyond the shared tables: tables of their own, or, when those together would take more memory
  // than the bound of table_blocks, per-block global tables
  DBuf<SegStats> sstats(ctx, 1);
  sstats.zero();
  k_seg_stats<<<grid_for(nc, 256, ctx->num_sms * 8), 256, 0, ctx->stream>>>(seg.get(), nc, sstats.get());
  GP_LAUNCH_CHECK();
  SegStats hs;
  read_back(ctx, sstats.get(), sizeof(hs), &hs);
  int lblocks = ctx->num_sms * 4;
  DBuf<int32_t> gk, gv;
  SegArgs sg{};
  DBuf<Seg> segs;
  DBuf<int> chunk0, tchunk0;
  DBuf<int2> tab;
  int64_t slots = 0;
  const int64_t table_bytes = ctx->limits.table_bytes(g.m2);
  for (sg.q4 = 8; sg.q4 > 4; sg.q4--) {  // two slots a key down to one and a quarter
    slots = (int64_t)hs.keys * sg.q4 / 4 + hs.huge;
    if (slots * (int64_t)sizeof(int2) <= table_bytes) break;
  }
  a.split_huge = hs.huge > 0 && sg.q4 > 4 ? 1 : 0;
  if (a.split_huge) {
    segs.reset(ctx, (size_t)hs.huge);
    chunk0.reset(ctx, (size_t)hs.huge + 1);
    tchunk0.reset(ctx, (size_t)hs.huge + 1);
    tab.reset(ctx, (size_t)slots);
    sg = SegArgs{segs.get(), chunk0.get(), tchunk0.get(), tab.get(), sg.q4};
  } else if (const int bits = table_bits(seg_keys(hs.longest, nc), 5); ((int64_t)1 << bits) > kBlockSmemSlots) {
    a.gstride = (int64_t)1 << bits;
    lblocks = table_blocks(table_bytes, a.gstride, lblocks);
    gk.reset(ctx, (size_t)(a.gstride * lblocks));
    gv.reset(ctx, (size_t)(a.gstride * lblocks));
    a.gkeys = gk.get();
    a.gvals = gv.get();
  }
  {
    ProfScope ps(ctx, PROF_CONTRACT);
    if (g.m2 > 0) {
      k_map<<<walk_grid(n, g.m2, ctx->num_sms, 5), kThreads, 0, ctx->stream>>>(
          g.xadj, g.adjncy, g.unit_w ? nullptr : g.adjwgt, cmap, moff.get(), tstart.get(), n, temp.get(), units);
      GP_LAUNCH_CHECK();
    }
    k_merge_warp<<<grid_for((int64_t)nc * 32, kThreads, ctx->num_sms * 8), kThreads, 0, ctx->stream>>>(a);
    GP_LAUNCH_CHECK();
    if (hs.longest > kWarpMaxUb) {
      k_merge_block<<<lblocks, kThreads, 0, ctx->stream>>>(a);
      GP_LAUNCH_CHECK();
    }
    if (a.split_huge) {
      k_seg_plan<<<1, 1024, 0, ctx->stream>>>(a, sg);
      GP_LAUNCH_CHECK();
      k_seg_clear<<<grid_for(slots, kThreads, ctx->num_sms * 8), kThreads, 0, ctx->stream>>>(tab.get(), slots);
      GP_LAUNCH_CHECK();
      k_seg_insert<<<ctx->num_sms * 6, kThreads, 0, ctx->stream>>>(a, sg);
      GP_LAUNCH_CHECK();
      k_seg_extract<<<ctx->num_sms * 8, kThreads, 0, ctx->stream>>>(a, sg);
      GP_LAUNCH_CHECK();
    }
  }
  DBuf<int32_t> total(ctx, 1);
  out.n = nc;
  out.bx.reset(ctx, (size_t)nc + 1);
  out.xadj = out.bx.get();
  scan_exclusive_i32(ctx, rowcnt.get(), out.xadj, nc + 1, total.get());
  const int32_t m2 = read_scalar(ctx, total.get());
  out.m2 = m2;
  out.ba.reset(ctx, (size_t)m2);
  out.bw.reset(ctx, (size_t)m2);
  out.adjncy = out.ba.get();
  out.adjwgt = out.bw.get();
  {
    ProfScope ps(ctx, PROF_CONTRACT_AUX);
    k_pack_rows<<<grid_for((int64_t)nc * 32, kThreads, ctx->num_sms * 8), kThreads, 0, ctx->stream>>>(
        tstart.get(), rowcnt.get(), out.xadj, nc, temp.get(), out.adjncy, out.adjwgt);
    GP_LAUNCH_CHECK();
  }
  out.bv.reset(ctx, (size_t)nc);
  out.vwgt = out.bv.get();
  if (trace.on())
    fprintf(stderr, "[gp contract] n=%d m2=%lld -> n=%d m2=%lld ms=%.2f\n", n, (long long)g.m2, nc,
            (long long)out.m2, trace.ms());
  if (nc > 0)
    GP_CUDA(cudaMemcpyAsync(out.vwgt, cw.get(), sizeof(int32_t) * nc, cudaMemcpyDeviceToDevice,
                            ctx->stream));
}

}  // namespace gp
