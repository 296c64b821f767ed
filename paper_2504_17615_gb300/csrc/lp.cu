// lp.cu -- size-constrained label propagation (Sec. 3 of the paper; the
// clustering of Sec. 4.1 and the refinement of Sec. 4.3) as synchronous
// sub-rounds with hash priorities:
//
//  per round r: nodes with neighbours are bucketed by (sub-round, degree
//  class); per sub-round s:
//   rate   : every active node sums the edge weight to each neighbouring
//            label on the snapshot and picks the admissible label of largest
//            rating (ties: smallest h32(TIE), then smallest label); it
//            proposes when that beats its own label's rating
//   decide : a target whose snapshot weight plus all incoming weight fits
//            the bound accepts everybody; the proposers of overflowing
//            targets are sorted by (target, h32(PRIO), node) and accepted
//            while the running weight fits (longest prefix)
//   apply  : labels and weights are updated; the non-empty clusters (the
//            labels of positive weight) are counted; the stop flag is raised
//            when that count reaches n_min or a round moved nothing.
#include "lp.cuh"
#include "lp_rate.cuh"

#include <chrono>

namespace gp {

namespace {

constexpr unsigned FULL = 0xFFFFFFFFu;
constexpr int kThreads = 256;
constexpr int kWarpsPerBlock = kThreads / 32;
constexpr int kMaxKeys = 64 * kNumBuckets;

struct RateArgs {
  const int32_t *xadj, *adjncy, *adjwgt, *vwgt, *label, *weight;
  const uint8_t *label8;  // optional narrow copy of label (fewer than 256 labels) for gathers
  const int4 *list;     // bucket list: (node, row offset, degree, node weight)
  const int32_t *offs;
  int key;
  int nkeys;            // k_rate_warp, k_rate_block: buckets of the launch, from key on
  int64_t bound;
  uint64_t ktie;
  int2 *prop;           // RATE_LP: per list position (proposed label or -1, own label)
  int32_t *incoming;    // RATE_LP: per label incoming weight
  uint64_t *fav_keys;   // RATE_FAV: per list position (fav << 32 | v)
  const int *stop;
  int32_t *gkeys, *gvals;  // large kernel global tables
  int64_t gstride;
  unsigned long long *units;
  int64_t m2;           // CSR entries
  int wlabels;          // labels whose weights a launch may copy to shared memory (<= 256)
  uint8_t *dirty;       // optional: per node, 0 = cannot move until a neighbour moves (rating skipped)
  const int32_t *ccount;  // optional: the list holds ccount[key] records from offs[key] (compacted)
};

__device__ __forceinline__ int list_end(const RateArgs &a, int key) {
  return a.ccount ? a.offs[key] + a.ccount[key] : a.offs[key + 1];
}
__device__ __forceinline__ int list_end(const RateArgs &a) { return list_end(a, a.key); }

// The first of a bucket's records [begin, end) for worker `id` of nw, which go through the buckets of a launch as if
// they were one list; done: records of the buckets before, modulo nw.
__device__ __forceinline__ int bucket_first(int begin, int end, int id, int nw, int &done) {
  const int at = id >= done ? id - done : id - done + nw;
  done = (int)(((unsigned)done + (unsigned)(end - begin)) % (unsigned)nw);
  return begin + at;
}

__device__ __forceinline__ void add_units(unsigned long long *units, unsigned long long e,
                                          unsigned long long v, unsigned long long c,
                                          unsigned long long p, bool narrow, bool implied) {
  if (!units) return;
  e = warp_sum(e); v = warp_sum(v); c = warp_sum(c); p = warp_sum(p);
  if (lane_id() == 0) {
    if (e) atomicAdd(units + 0, e);
    if (e && narrow) atomicAdd(units + 4, e);
    if (e && implied) atomicAdd(units + 5, e);
    if (v) atomicAdd(units + 1, v);
    if (c) atomicAdd(units + 2, c);
    if (p) atomicAdd(units + 3, p);
  }
}

__device__ __forceinline__ int label_of(const RateArgs &a, int u) {
  return a.label8 ? (int)a.label8[u] : a.label[u];
}

__device__ __forceinline__ unsigned slot_hash(int L, int bits) {
  return ((unsigned)L * 2654435761u) >> (32 - bits);
}

template <int MODE>
__device__ __forceinline__ void emit(const RateArgs &a, int i, int v, int best, int cv, int own) {
  if (MODE == RATE_LP) {
    a.prop[i] = make_int2(best, own);
    atomicAdd(&a.incoming[best], cv);
  } else {
    a.fav_keys[i] = ((uint64_t)(uint32_t)best << 32) | (uint32_t)v;
  }
}

// ------------------------------------- degree <= 32: a thread per node
//
// A thread loads its node's whole row (16 bytes a load where the arrays are aligned), gathers the labels,
// and adds up equal labels by comparing all pairs in registers.  It is the gather of the labels that
// should bound this step (about 300e9 random reads/s while the label array fits L2, 76e9/s from a 268 MB
// array); with 8 or 16 lanes per node and tables in shared memory a node of 20 neighbours took 225-300
// warp instructions, so that issue and latency bound it instead.  The pairs cost D (D - 1) / 2 x 3
// instructions per 32 nodes, a tenth of that, and every label of the row is in flight at once.
// A level of 16.8M nodes and 336M entries (clustering, contraction, sparsification, clustering of the result) went from
// 25.6 to 21.7 ms; where the label array passes L2 (2^26 nodes) clustering's rating stays at the rate of its misses
// (44 ms).  Refinement of that graph, unit weights, 128 one-byte labels: 59.6 ms with lane groups, 54.7 with this,
// 60.2 with byte counters per thread in shared memory instead of the pairs (a fifth of the instructions, but 39 % of
// the warps active and 28 % of the issue slots used).
//
// The choice is lazy in the label weights: candidates are ranked by (rating, tie hash, label) without the
// bound, and only the best one's weight is read; if it does not fit, the weights of all that are rated
// above the own label are read and those that do not fit dropped.  With one-byte labels (refinement: at
// most 255 labels) the label weights are copied to shared memory once per block and every candidate is
// checked up front.

// Label kinds: LK_WIDE int32 labels, LK_NARROW uint8 labels (fewer than 256).
enum LabelKind { LK_WIDE = 0, LK_NARROW = 1 };

template <int D>
struct ThreadShape {
  static constexpr int NT = D <= 16 ? 256 : 128;
  static constexpr int PER_SM = D <= 8 ? 5 : D <= 16 ? 3 : D <= 24 ? 5 : 4;  // blocks an SM holds
};

template <int MODE, int D, int LK>
__global__ void __launch_bounds__(ThreadShape<D>::NT, ThreadShape<D>::PER_SM) k_rate_thread(RateArgs a) {
  constexpr int NT = ThreadShape<D>::NT;
  constexpr bool kSmemW = MODE == RATE_LP && LK != LK_WIDE;
  __shared__ int s_w[kSmemW ? 256 : 1];
  if (a.stop && *a.stop) return;
  if (kSmemW) {
    for (int t = threadIdx.x; t < a.wlabels; t += NT) s_w[t] = a.weight[t];
    __syncthreads();
  }
  const bool vec = (((uintptr_t)a.adjncy | (uintptr_t)a.adjwgt) & 15) == 0;
  const int begin = a.offs[a.key], end = list_end(a);
  unsigned long long ue = 0, uv = 0, uc = 0, up = 0;
  for (int i0 = begin + (int)(blockIdx.x * NT); i0 < end; i0 += (int)(gridDim.x * NT)) {
    const int i = i0 + (int)threadIdx.x;
    int4 rec = i < end ? a.list[i] : make_int4(-1, 0, 0, 0);
    const int v = rec.x, cv = rec.w;
    // a clean node cannot move: neither its neighbours' labels nor its own changed since it last found no
    // label rated above its own
    const bool live = v >= 0 && !(a.dirty && !a.dirty[v]);
    const int st = live ? rec.y : 0, deg = live ? rec.z : 0;
    const int own = live ? (LK == LK_WIDE ? a.label[v] : (int)a.label8[v]) : -2;
    int L[D], w[D];
    load_row<D>(a.adjncy, st, deg, a.m2, vec, L);
#pragma unroll
    for (int q = 0; q < D; q++) L[q] = q < deg ? (LK == LK_WIDE ? a.label[L[q]] : (int)a.label8[L[q]]) : -1;
    if (a.adjwgt) {
      load_row<D>(a.adjwgt, st, deg, a.m2, vec, w);
    } else {
#pragma unroll
      for (int q = 0; q < D; q++) w[q] = 1;
    }
    bool stay;
    int nc;
    const int best = choose_row<D, MODE == RATE_FAV>(L, w, deg, live, v, own, cv, a.bound, a.ktie,
                                                     kSmemW ? s_w : nullptr, a.weight, stay, nc);
    uc += nc;
    if (a.dirty && live && stay) a.dirty[v] = 0;
    if (live) {
      ue += deg;
      uv += 1;
    }
    if (best >= 0) {
      emit<MODE>(a, i, v, best, cv, own);
      up += 1;
    } else if (MODE == RATE_LP && v >= 0) {
      a.prop[i] = make_int2(-1, 0);
    }
  }
  add_units(a.units, ue, uv, uc, up, a.label8 != nullptr, a.adjwgt == nullptr);
}

// ------------------------- degree <= 128, <= 512: warp/node, shared table
//
// The table has two slots per neighbour (a slot is the high half of hash x size, so any size will do) and
// kWarpUnroll neighbours per lane are in flight.  What costs here is the probing: a warp goes on until its
// unluckiest lane has found a slot, some ten probes with 4/3 slots per neighbour and about four with two.
// On the scale-24 R-MAT graph two slots (and more for blocks and hubs) took the partition from 468 to 425 ms.

constexpr int kWarpUnroll = 4;

constexpr int kTabQ4 = 8;     // shared tables: two slots per neighbour ...
constexpr int kTabQ4Last = 6; // ... one and a half in the largest class (an SM's whole shared memory)

template <int MODE>
__global__ void __launch_bounds__(kThreads) k_rate_warp(RateArgs a, int slots) {
  extern __shared__ int s_tab[];  // per warp: slots labels, slots ratings
  const int lane = (int)lane_id(), wib = threadIdx.x >> 5;
  int *tk = s_tab + wib * 2 * slots, *tv = tk + slots;
  for (int t = lane; t < slots; t += 32) { tk[t] = -1; tv[t] = 0; }
  __syncwarp();
  if (a.stop && *a.stop) return;
  const int wid = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int nw = (int)((gridDim.x * blockDim.x) >> 5);
  unsigned long long ue = 0, uv = 0, uc = 0, up = 0;
  for (int b = 0, done = 0; b < a.nkeys; b++) {
    const int begin = a.offs[a.key + b], end = list_end(a, a.key + b);
    for (int i = bucket_first(begin, end, wid, nw, done); i < end; i += nw) {
      const int4 rec = a.list[i];
      const int v = rec.x, start = rec.y, deg = rec.z, cv = rec.w;
      if (a.dirty && !a.dirty[v]) {  // clean: cannot move
        if (MODE == RATE_LP && lane == 0) a.prop[i] = make_int2(-1, 0);
        continue;
      }
      const int own = label_of(a, v);
      const int tsize = tab_slots(deg, kTabQ4);
      for (int j0 = lane; j0 < deg; j0 += 32 * kWarpUnroll) {
        int L[kWarpUnroll], w[kWarpUnroll];
#pragma unroll
        for (int r = 0; r < kWarpUnroll; r++) {
          const int j = j0 + r * 32;
          L[r] = j < deg ? __ldcs(a.adjncy + start + j) : -1;
          w[r] = j < deg && a.adjwgt ? __ldcs(a.adjwgt + start + j) : 1;
        }
#pragma unroll
        for (int r = 0; r < kWarpUnroll; r++) L[r] = L[r] >= 0 ? label_of(a, L[r]) : -1;
#pragma unroll
        for (int r = 0; r < kWarpUnroll; r++) {
          if (L[r] < 0) continue;
          int s = (int)__umulhi((unsigned)L[r] * 2654435761u, (unsigned)tsize);
          for (int probe = 0; probe < tsize; probe++) {  // bounded: more slots than neighbours
            const int prev = atomicCAS(&tk[s], -1, L[r]);
            if (prev == -1 || prev == L[r]) { atomicAdd(&tv[s], w[r]); break; }
            s = s + 1 == tsize ? 0 : s + 1;
          }
        }
      }
      __syncwarp();
      int own_loc = 0, rloc = -1, nc = 0, rall = 0;
      for (int t = lane; t < tsize; t += 32) {
        const int L = tk[t];
        if (L < 0) continue;
        const int r = tv[t];
        if (L == own) { own_loc = r; continue; }
        nc++;
        rall = r > rall ? r : rall;
        if (r > rloc && (MODE != RATE_LP || (int64_t)a.weight[L] + cv <= a.bound)) rloc = r;  // only a better one matters
      }
      const int own_r = __reduce_max_sync(FULL, own_loc);
      const int rmax = __reduce_max_sync(FULL, rloc);
      if (a.dirty && __reduce_max_sync(FULL, rall) <= own_r && lane == 0) a.dirty[v] = 0;
      ue += deg; uv += 1; uc += nc;
      const bool want = !(rmax < 0 || (MODE == RATE_LP && rmax <= own_r));
      uint64_t packed = ~0ull;
      for (int t = lane; t < tsize; t += 32) {
        const int L = tk[t];
        if (L < 0) continue;
        if (want && L != own && tv[t] == rmax && (MODE != RATE_LP || (int64_t)a.weight[L] + cv <= a.bound)) {
          const uint64_t p = ((uint64_t)h32(a.ktie, (uint32_t)v, (uint32_t)L) << 32) | (uint32_t)L;
          packed = p < packed ? p : packed;
        }
        tk[t] = -1;
        tv[t] = 0;
      }
      if (want) {
        packed = warp_min(packed);
        if (lane == 0) { emit<MODE>(a, i, v, (int)(uint32_t)packed, cv, own); up += 1; }
      } else if (MODE == RATE_LP && lane == 0) {
        a.prop[i] = make_int2(-1, 0);
      }
      __syncwarp();
    }
  }
  add_units(a.units, ue * (lane == 0), uv * (lane == 0), uc, up, a.label8 != nullptr, a.adjwgt == nullptr);
}

// ---- a block per node: favourites of degree > 128, and hubs when their tables would pass the memory bound

__device__ __forceinline__ int block_max_i32(int v, int *s_red) {
  v = warp_max(v);
  const int w = threadIdx.x >> 5;
  __syncthreads();
  if (lane_id() == 0) s_red[w] = v;
  __syncthreads();
  int r = s_red[0];
  for (int i = 1; i < kWarpsPerBlock; i++) r = s_red[i] > r ? s_red[i] : r;
  return r;
}

__device__ __forceinline__ uint64_t block_min_u64(uint64_t v, uint64_t *s_red) {
  v = warp_min(v);
  const int w = threadIdx.x >> 5;
  __syncthreads();
  if (lane_id() == 0) s_red[w] = v;
  __syncthreads();
  uint64_t r = s_red[0];
  for (int i = 1; i < kWarpsPerBlock; i++) r = s_red[i] < r ? s_red[i] : r;
  return r;
}

template <int MODE>
__global__ void __launch_bounds__(kThreads) k_rate_large(RateArgs a) {
  __shared__ int s_k[kLargeSmemSlots];
  __shared__ int s_v[kLargeSmemSlots];
  __shared__ int s_ri[kWarpsPerBlock];
  __shared__ uint64_t s_ru[kWarpsPerBlock];
  if (a.stop && *a.stop) return;
  for (int t = threadIdx.x; t < kLargeSmemSlots; t += blockDim.x) { s_k[t] = -1; s_v[t] = 0; }
  __syncthreads();
  const int begin = a.offs[a.key], end = list_end(a);
  int *gk = a.gkeys ? a.gkeys + (int64_t)blockIdx.x * a.gstride : nullptr;
  int *gv = a.gvals ? a.gvals + (int64_t)blockIdx.x * a.gstride : nullptr;
  unsigned long long ue = 0, uv = 0, uc = 0, up = 0;
  for (int i = begin + (int)blockIdx.x; i < end; i += (int)gridDim.x) {
    const int4 rec = a.list[i];
    const int v = rec.x, start = rec.y, deg = rec.z, cv = rec.w;
    if (a.dirty && !a.dirty[v]) {  // clean: cannot move (uniform in the block)
      if (MODE == RATE_LP && threadIdx.x == 0) a.prop[i] = make_int2(-1, 0);
      continue;
    }
    const int own = label_of(a, v);
    const int bits = table_bits(deg, 1);
    const unsigned tsize = 1u << bits;
    const bool in_smem = tsize <= kLargeSmemSlots;
    int *tk = in_smem ? s_k : gk;
    int *tv = in_smem ? s_v : gv;
    for (int j = threadIdx.x; j < deg; j += blockDim.x) {
      const int L = label_of(a, __ldcs(a.adjncy + start + j));
      const int w = a.adjwgt ? __ldcs(a.adjwgt + start + j) : 1;
      unsigned s = slot_hash(L, bits);
      for (unsigned probe = 0; probe < tsize; probe++) {  // bounded: the table never fills
        const int prev = atomicCAS(&tk[s], -1, L);
        if (prev == -1 || prev == L) { atomicAdd(&tv[s], w); break; }
        s = (s + 1) & (tsize - 1);
      }
    }
    __syncthreads();
    int own_loc = 0, rloc = -1, nc = 0, rall = 0;
    for (unsigned t = threadIdx.x; t < tsize; t += blockDim.x) {
      const int L = tk[t];
      if (L < 0) continue;
      const int r = tv[t];
      if (L == own) { own_loc = r; continue; }
      nc++;
      rall = r > rall ? r : rall;
      if (MODE == RATE_LP && (int64_t)a.weight[L] + cv > a.bound) continue;
      rloc = r > rloc ? r : rloc;
    }
    const int own_r = block_max_i32(own_loc, s_ri);
    const int rmax = block_max_i32(rloc, s_ri);
    if (a.dirty) {
      const int ra = block_max_i32(rall, s_ri);
      if (ra <= own_r && threadIdx.x == 0) a.dirty[v] = 0;
    }
    uc += nc;
    if (threadIdx.x == 0) { ue += deg; uv += 1; }
    if (!(rmax < 0 || (MODE == RATE_LP && rmax <= own_r))) {
      uint64_t packed = ~0ull;
      for (unsigned t = threadIdx.x; t < tsize; t += blockDim.x) {
        const int L = tk[t];
        if (L < 0 || L == own || tv[t] != rmax) continue;
        if (MODE == RATE_LP && (int64_t)a.weight[L] + cv > a.bound) continue;
        const uint64_t p = ((uint64_t)h32(a.ktie, (uint32_t)v, (uint32_t)L) << 32) | (uint32_t)L;
        packed = p < packed ? p : packed;
      }
      packed = block_min_u64(packed, s_ru);
      if (threadIdx.x == 0) { emit<MODE>(a, i, v, (int)(uint32_t)packed, cv, own); up += 1; }
    } else if (MODE == RATE_LP && threadIdx.x == 0) {
      a.prop[i] = make_int2(-1, 0);
    }
    __syncthreads();
    for (unsigned t = threadIdx.x; t < tsize; t += blockDim.x) { tk[t] = -1; tv[t] = 0; }
    __syncthreads();
  }
  add_units(a.units, ue, uv, uc, up, a.label8 != nullptr, a.adjwgt == nullptr);
}

// ------------------- 512 < degree <= 18432: block/node, shared table
//
// As k_rate_warp with a block's threads.  Nodes of 2049 .. 18432 neighbours held 172M of the 521M entries of
// the scale-24 R-MAT graph; their tables in shared memory take no global atomics, which limited them to
// 7e9 entries/s: clustering of that level 183 -> 115 ms.  With two slots instead of 4/3 a sub-round takes
// .35 instead of .47 ms in the 512-thread class, .40 instead of .45 in the 1024-thread one (one and a half).

constexpr int kBlockUnroll = 4;

template <int NT>
__device__ __forceinline__ int block_max_n(int v, int *s_red) {
  v = __reduce_max_sync(FULL, v);
  __syncthreads();
  if (lane_id() == 0) s_red[threadIdx.x >> 5] = v;
  __syncthreads();
  int r = s_red[0];
#pragma unroll
  for (int i = 1; i < NT / 32; i++) r = s_red[i] > r ? s_red[i] : r;
  return r;
}

template <int NT>
__device__ __forceinline__ uint64_t block_min_n(uint64_t v, uint64_t *s_red) {
  v = warp_min(v);
  __syncthreads();
  if (lane_id() == 0) s_red[threadIdx.x >> 5] = v;
  __syncthreads();
  uint64_t r = s_red[0];
#pragma unroll
  for (int i = 1; i < NT / 32; i++) r = s_red[i] < r ? s_red[i] : r;
  return r;
}

template <int NT>
__global__ void __launch_bounds__(NT) k_rate_block(RateArgs a, int slots, int q4) {
  extern __shared__ int s_tab[];  // slots labels, slots ratings
  __shared__ int s_ri[NT / 32], s_own;
  __shared__ uint64_t s_ru[NT / 32];
  if (a.stop && *a.stop) return;
  int *tk = s_tab, *tv = s_tab + slots;
  for (int t = threadIdx.x; t < slots; t += NT) { tk[t] = -1; tv[t] = 0; }
  unsigned long long ue = 0, uv = 0, uc = 0, up = 0;
  for (int b = 0, done = 0; b < a.nkeys; b++) {
    const int begin = a.offs[a.key + b], end = list_end(a, a.key + b);
    for (int i = bucket_first(begin, end, (int)blockIdx.x, (int)gridDim.x, done); i < end; i += (int)gridDim.x) {
      const int4 rec = a.list[i];
      const int v = rec.x, start = rec.y, deg = rec.z, cv = rec.w;
      if (a.dirty && !a.dirty[v]) {  // clean: cannot move (uniform in the block)
        if (threadIdx.x == 0) a.prop[i] = make_int2(-1, 0);
        continue;
      }
      const int own = label_of(a, v);
      const int tsize = tab_slots(deg, q4);
      if (threadIdx.x == 0) s_own = 0;
      __syncthreads();  // the table is empty, and the flag of the clean nodes was read before it may change
      for (int j0 = threadIdx.x; j0 < deg; j0 += NT * kBlockUnroll) {
        int L[kBlockUnroll], w[kBlockUnroll];
#pragma unroll
        for (int r = 0; r < kBlockUnroll; r++) {
          const int j = j0 + r * NT;
          L[r] = j < deg ? __ldcs(a.adjncy + start + j) : -1;
          w[r] = j < deg && a.adjwgt ? __ldcs(a.adjwgt + start + j) : 1;
        }
#pragma unroll
        for (int r = 0; r < kBlockUnroll; r++) L[r] = L[r] >= 0 ? label_of(a, L[r]) : -1;
#pragma unroll
        for (int r = 0; r < kBlockUnroll; r++) {
          if (L[r] < 0) continue;
          int s = (int)__umulhi((unsigned)L[r] * 2654435761u, (unsigned)tsize);
          for (int probe = 0; probe < tsize; probe++) {  // bounded: more slots than neighbours
            const int prev = atomicCAS(&tk[s], -1, L[r]);
            if (prev == -1 || prev == L[r]) { atomicAdd(&tv[s], w[r]); break; }
            s = s + 1 == tsize ? 0 : s + 1;
          }
        }
      }
      __syncthreads();
      int rloc = -1, rall = 0, nc = 0;
      for (int t = threadIdx.x; t < tsize; t += NT) {
        const int L = tk[t];
        if (L < 0) continue;
        const int r = tv[t];
        if (L == own) { s_own = r; continue; }
        nc++;
        rall = r > rall ? r : rall;
        if (r > rloc && (int64_t)a.weight[L] + cv <= a.bound) rloc = r;  // only what beats the thread's best matters
      }
      const int rmax = block_max_n<NT>(rloc, s_ri);  // its barriers also publish s_own
      const int own_r = s_own;
      if (a.dirty) {
        rall = block_max_n<NT>(rall, s_ri);
        if (rall <= own_r && threadIdx.x == 0) a.dirty[v] = 0;
      }
      uc += nc;
      const bool want = rmax >= 0 && rmax > own_r;
      uint64_t packed = ~0ull;
      for (int t = threadIdx.x; t < tsize; t += NT) {
        const int L = tk[t];
        if (L < 0) continue;
        if (want && L != own && tv[t] == rmax && (int64_t)a.weight[L] + cv <= a.bound) {
          const uint64_t p = ((uint64_t)h32(a.ktie, (uint32_t)v, (uint32_t)L) << 32) | (uint32_t)L;
          packed = p < packed ? p : packed;
        }
        tk[t] = -1;
        tv[t] = 0;
      }
      if (want) packed = block_min_n<NT>(packed, s_ru);
      if (threadIdx.x == 0) {
        ue += deg;
        uv += 1;
        if (want) { emit<RATE_LP>(a, i, v, (int)(uint32_t)packed, cv, own); up += 1; }
        else a.prop[i] = make_int2(-1, 0);
      }
      __syncthreads();
    }
  }
  add_units(a.units, ue, uv, uc, up, a.label8 != nullptr, a.adjwgt == nullptr);
}

// ------------------------------------------------- hubs: many blocks a node
//
// A node of more neighbours than that (with few labels: of more than 2048) is rated by as many blocks as
// its row has chunks.  With one block a node and a table in global memory, a sub-round waited for the
// block of the largest hub: 8 ms in every sub-round of the scale-24 R-MAT graph (4e5 neighbours), 330 ms
// for level 1.  k_hub_plan lists the sub-round's hubs with the prefix sums of their chunks; then
//  few labels (at most kHubDense: refinement): k_hub_dense counts a chunk per label in shared memory, adds
//    it to the hub's counters, and the block that finishes a hub's last chunk chooses;
//  many labels: k_hub_insert sums a chunk's labels in a shared table and adds the sums to the hub's table
//    in global memory (one 64-bit exchange claims a slot with its sum; three slots per neighbour where the
//    memory bound allows, since every probe is a round trip to L2), k_hub_table walks the tables (4096
//    slots a block) for the largest admissible rating, and then for the smallest (hash, label) of that
//    rating, and leaves them empty.
// The choice is the same as in the other kernels.

constexpr int kHubChunk = 2048;    // row entries per block and step
constexpr int kHubTabChunk = 4096; // table slots per block and step
constexpr int kHubDense = 1024;    // labels up to which a hub's ratings are counted per label
constexpr unsigned long long kEmptySlot = 0xFFFFFFFFull;  // the slot (-1, 0): label in the low half, rating in the high

struct Hub {
  int pos, v, st, deg, cv, own;  // list position, node, row offset, degree, weight, label
  int tsize, done;               // table slots; blocks that finished (dense, pick)
  long long toff;                // table offset
  int rmax, ownr, rall, pad;     // ratings: largest admissible, own label's, largest of any other label
  unsigned long long best;       // smallest (hash, label) of rating rmax
};

struct HubArgs {
  Hub *hubs;
  int *chunk0, *tchunk0;  // prefix sums of row chunks and of table chunks; [count] = totals
  int2 *tab;              // (label, rating) slots, empty (-1, 0) between sub-rounds
  int32_t *hist;          // dense: [hub][nlabels], zero between sub-rounds
  int nlabels;
  int q4;                 // slots per neighbour, in quarters
};

__global__ void __launch_bounds__(1024) k_hub_plan(RateArgs a, HubArgs h) {
  __shared__ long long s_w[3][32];
  if (a.stop && *a.stop) return;
  const int begin = a.offs[a.key], cnt = list_end(a) - begin;
  const int lane = (int)lane_id(), wp = threadIdx.x >> 5;
  long long run[3] = {0, 0, 0};  // row chunks, table chunks, table slots
  for (int b = 0; b < cnt; b += 1024) {
    const int i = b + (int)threadIdx.x;
    int deg = 0;
    Hub x{};
    if (i < cnt) {
      const int4 rec = a.list[begin + i];
      x.pos = begin + i; x.v = rec.x; x.st = rec.y; x.cv = rec.w;
      deg = a.dirty && !a.dirty[rec.x] ? 0 : rec.z;  // clean: cannot move
      if (deg == 0) a.prop[begin + i] = make_int2(-1, 0);
      x.deg = deg;
      x.own = label_of(a, rec.x);
      x.tsize = deg > 0 ? tab_slots(deg, h.q4) : 0;
      x.rmax = -1;
      x.best = ~0ull;
    }
    const long long val[3] = {chunks_of(deg, kHubChunk), chunks_of(x.tsize, kHubTabChunk), x.tsize};
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
      h.hubs[i] = x;
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

// The hub whose chunks hold item `it`: the last one with first[i] <= it.
__device__ __forceinline__ int hub_of(const int *first, int cnt, int it) {
  int lo = 0, hi = cnt;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (first[mid] <= it) lo = mid; else hi = mid;
  }
  return lo;
}

__device__ __forceinline__ void hub_emit(const RateArgs &a, const Hub &x, int rmax, int ownr, int rall,
                                         unsigned long long best) {
  if (a.dirty && rall <= ownr) a.dirty[x.v] = 0;
  if (rmax < 0 || rmax <= ownr) a.prop[x.pos] = make_int2(-1, 0);
  else emit<RATE_LP>(a, x.pos, x.v, (int)(uint32_t)best, x.cv, x.own);
}

__global__ void __launch_bounds__(kThreads) k_hub_dense(RateArgs a, HubArgs h) {
  extern __shared__ int s_hist[];  // nlabels
  __shared__ int s_ri[kWarpsPerBlock];
  __shared__ uint64_t s_ru[kWarpsPerBlock];
  __shared__ bool s_last;
  if (a.stop && *a.stop) return;
  const int cnt = list_end(a) - a.offs[a.key], items = h.chunk0[cnt];
  for (int t = threadIdx.x; t < h.nlabels; t += blockDim.x) s_hist[t] = 0;
  unsigned long long ue = 0, uv = 0;
  for (int it = blockIdx.x; it < items; it += gridDim.x) {
    const int hi = hub_of(h.chunk0, cnt, it);
    const Hub x = h.hubs[hi];
    const int c0 = (it - h.chunk0[hi]) * kHubChunk, c1 = min(x.deg, c0 + kHubChunk);
    constexpr int R = kHubChunk / kThreads;
    int u[R], w[R];
#pragma unroll
    for (int r = 0; r < R; r++) {
      const int j = c0 + r * kThreads + (int)threadIdx.x;
      u[r] = j < c1 ? __ldcs(a.adjncy + x.st + j) : -1;
      w[r] = j < c1 && a.adjwgt ? __ldcs(a.adjwgt + x.st + j) : 1;
    }
    __syncthreads();  // the counters are empty
#pragma unroll
    for (int r = 0; r < R; r++)
      if (u[r] >= 0) atomicAdd(&s_hist[label_of(a, u[r])], w[r]);
    __syncthreads();
    int32_t *hist = h.hist + (int64_t)hi * h.nlabels;
    for (int t = threadIdx.x; t < h.nlabels; t += blockDim.x) {
      const int c = s_hist[t];
      if (c) { atomicAdd(&hist[t], c); s_hist[t] = 0; }
    }
    __threadfence();
    __syncthreads();
    const int chunks = chunks_of(x.deg, kHubChunk);
    if (threadIdx.x == 0) {
      s_last = atomicAdd(&h.hubs[hi].done, 1) == chunks - 1;
      ue += c1 - c0;
    }
    __syncthreads();
    if (!s_last) continue;
    __threadfence();
    int rloc = -1, rall = 0;
    const int ownr = *(volatile int32_t *)&hist[x.own];
    for (int t = threadIdx.x; t < h.nlabels; t += blockDim.x) {
      const int r = *(volatile int32_t *)&hist[t];
      if (r == 0 || t == x.own) continue;
      rall = r > rall ? r : rall;
      if (r > rloc && (int64_t)a.weight[t] + x.cv <= a.bound) rloc = r;
    }
    const int rmax = block_max_i32(rloc, s_ri);
    rall = block_max_i32(rall, s_ri);
    uint64_t packed = ~0ull;
    for (int t = threadIdx.x; t < h.nlabels; t += blockDim.x) {
      const int r = *(volatile int32_t *)&hist[t];
      if (r != 0 && r == rmax && t != x.own && (int64_t)a.weight[t] + x.cv <= a.bound) {
        const uint64_t p = ((uint64_t)h32(a.ktie, (uint32_t)x.v, (uint32_t)t) << 32) | (uint32_t)t;
        packed = p < packed ? p : packed;
      }
    }
    packed = block_min_u64(packed, s_ru);
    __syncthreads();  // every thread has read the own label's count
    for (int t = threadIdx.x; t < h.nlabels; t += blockDim.x) hist[t] = 0;
    if (threadIdx.x == 0) {
      uv += 1;
      hub_emit(a, x, rmax, ownr, rall, packed);
    }
  }
  add_units(a.units, ue, uv, 0, 0, a.label8 != nullptr, a.adjwgt == nullptr);
}

__global__ void __launch_bounds__(kThreads) k_hub_insert(RateArgs a, HubArgs h) {
  __shared__ int s_k[2 * kHubChunk];
  __shared__ int s_v[2 * kHubChunk];
  if (a.stop && *a.stop) return;
  constexpr int BITS = 12;
  static_assert((1 << BITS) == 2 * kHubChunk, "table size");
  const int cnt = list_end(a) - a.offs[a.key], items = h.chunk0[cnt];
  for (int t = threadIdx.x; t < 2 * kHubChunk; t += blockDim.x) { s_k[t] = -1; s_v[t] = 0; }
  unsigned long long ue = 0;
  for (int it = blockIdx.x; it < items; it += gridDim.x) {
    const int hi = hub_of(h.chunk0, cnt, it);
    const Hub &x = h.hubs[hi];
    const int st = x.st, tsize = x.tsize;
    int2 *tab = h.tab + x.toff;
    const int c0 = (it - h.chunk0[hi]) * kHubChunk, c1 = min(x.deg, c0 + kHubChunk);
    constexpr int R = kHubChunk / kThreads;
    int L[R], w[R];
#pragma unroll
    for (int r = 0; r < R; r++) {
      const int j = c0 + r * kThreads + (int)threadIdx.x;
      L[r] = j < c1 ? __ldcs(a.adjncy + st + j) : -1;
      w[r] = j < c1 && a.adjwgt ? __ldcs(a.adjwgt + st + j) : 1;
    }
#pragma unroll
    for (int r = 0; r < R; r++) L[r] = L[r] >= 0 ? label_of(a, L[r]) : -1;
    __syncthreads();  // the shared table is empty
#pragma unroll
    for (int r = 0; r < R; r++) {
      if (L[r] < 0) continue;
      unsigned s = part_slot(L[r], BITS);
      for (int probe = 0; probe < 2 * kHubChunk; probe++) {  // bounded: at most half full
        const int prev = atomicCAS(&s_k[s], -1, L[r]);
        if (prev == -1 || prev == L[r]) { atomicAdd(&s_v[s], w[r]); break; }
        s = (s + 1) & (2 * kHubChunk - 1);
      }
    }
    __syncthreads();
    for (int t = threadIdx.x; t < 2 * kHubChunk; t += blockDim.x) {
      const int K = s_k[t];
      if (K < 0) continue;
      const int sum = s_v[t];
      s_k[t] = -1;
      s_v[t] = 0;
      int s = (int)__umulhi((unsigned)K * 2654435761u, (unsigned)tsize);
      for (int probe = 0; probe < tsize; probe++) {  // bounded: more slots than neighbours
        const unsigned long long prev = atomicCAS((unsigned long long *)&tab[s], kEmptySlot,
                                                  ((unsigned long long)(unsigned)sum << 32) | (unsigned)K);
        if (prev == kEmptySlot) break;
        if ((int)(unsigned)prev == K) { atomicAdd(&tab[s].y, sum); break; }
        s = s + 1 == tsize ? 0 : s + 1;
      }
    }
    if (threadIdx.x == 0) ue += c1 - c0;
  }
  add_units(a.units, ue, 0, 0, 0, a.label8 != nullptr, a.adjwgt == nullptr);
}

template <bool PICK>
__global__ void __launch_bounds__(kThreads) k_hub_table(RateArgs a, HubArgs h) {
  __shared__ int s_ri[kWarpsPerBlock];
  __shared__ uint64_t s_ru[kWarpsPerBlock];
  if (a.stop && *a.stop) return;
  const int cnt = list_end(a) - a.offs[a.key], items = h.tchunk0[cnt];
  unsigned long long uv = 0, uc = 0;
  for (int it = blockIdx.x; it < items; it += gridDim.x) {
    const int hi = hub_of(h.tchunk0, cnt, it);
    Hub *hp = &h.hubs[hi];
    const int own = hp->own, cv = hp->cv, v = hp->v;
    int2 *tab = h.tab + hp->toff;
    const int t0 = (it - h.tchunk0[hi]) * kHubTabChunk, t1 = min(hp->tsize, t0 + kHubTabChunk);
    constexpr int R = 8;
    if (!PICK) {
      int best = *(volatile int *)&hp->rmax, rall = 0;  // only ratings above what some block has found matter
      const int floor0 = best;
      for (int b = t0 + (int)threadIdx.x; b < t1; b += kThreads * R) {
        int2 e[R];
#pragma unroll
        for (int r = 0; r < R; r++) e[r] = b + r * kThreads < t1 ? tab[b + r * kThreads] : make_int2(-1, 0);
#pragma unroll
        for (int r = 0; r < R; r++) {
          if (e[r].x < 0) continue;
          if (e[r].x == own) { hp->ownr = e[r].y; continue; }  // one slot holds the own label
          uc++;
          rall = e[r].y > rall ? e[r].y : rall;
          if (e[r].y > best && (int64_t)a.weight[e[r].x] + cv <= a.bound) best = e[r].y;
        }
      }
      best = block_max_i32(best, s_ri);
      rall = block_max_i32(rall, s_ri);
      if (threadIdx.x == 0) {
        if (best > floor0) atomicMax(&hp->rmax, best);
        if (rall > 0) atomicMax(&hp->rall, rall);
      }
    } else {
      const int rmax = hp->rmax, ownr = hp->ownr;
      const bool want = rmax >= 0 && rmax > ownr;
      uint64_t packed = ~0ull;
      for (int b = t0 + (int)threadIdx.x; b < t1; b += kThreads * R) {
        int2 e[R];
#pragma unroll
        for (int r = 0; r < R; r++) e[r] = b + r * kThreads < t1 ? tab[b + r * kThreads] : make_int2(-1, 0);
#pragma unroll
        for (int r = 0; r < R; r++)
          if (e[r].x >= 0) tab[b + r * kThreads] = make_int2(-1, 0);
        if (!want) continue;
#pragma unroll
        for (int r = 0; r < R; r++) {
          if (e[r].x < 0 || e[r].x == own || e[r].y != rmax || (int64_t)a.weight[e[r].x] + cv > a.bound) continue;
          const uint64_t p = ((uint64_t)h32(a.ktie, (uint32_t)v, (uint32_t)e[r].x) << 32) | (uint32_t)e[r].x;
          packed = p < packed ? p : packed;
        }
      }
      packed = block_min_u64(packed, s_ru);
      if (threadIdx.x == 0) {
        if (packed != ~0ull) atomicMin(&hp->best, packed);
        __threadfence();
        const int chunks = chunks_of(hp->tsize, kHubTabChunk);
        if (atomicAdd(&hp->done, 1) == chunks - 1) {
          __threadfence();
          uv += 1;
          hub_emit(a, *hp, rmax, ownr, hp->rall, *(volatile unsigned long long *)&hp->best);
        }
      }
    }
    __syncthreads();
  }
  add_units(a.units, 0, uv, uc, 0, false, false);
}

// ------------------------------------------------------------- full nodes
//
// A cluster that a node rates holds the neighbour it was read from, so it weighs at least as much as the node's
// lightest neighbour: a node without room for that one can move to no cluster, in any sub-round, and is left
// out of the lists.  Only nodes above half the bound are looked at (a node up to that is full only among
// heavier ones).  On the coarse levels of a graph with hubs these nodes hold a third to nearly all of the
// entries (scale-24 R-MAT, levels 3 / 4 / 5: 23 of 77M, 24 of 45M, 27 of 28M; partition 365 -> 346 ms).
constexpr int kFullUnroll = 8;

__global__ void __launch_bounds__(kThreads) k_mark_full(const int32_t *xadj, const int32_t *adjncy,
                                                        const int32_t *vwgt, int n, int64_t bound,
                                                        uint8_t *full) {  // full: zero on entry
  const int lane = (int)lane_id();
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t step = ((int64_t)n + 31) / 32;  // a warp's nodes lie this far apart: hubs have neighbouring ids
  for (int64_t v0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; v0 < step; v0 += nw) {
    const int64_t v = v0 + lane * step;
    const int64_t c = v < n ? vwgt[v] : 0;
    int st = 0, en = 0;
    const bool heavy = 2 * c > bound;
    if (heavy) { st = xadj[v]; en = xadj[v + 1]; }
    bool mark = false;
    for (unsigned m = __ballot_sync(FULL, heavy && en > st); m; m &= m - 1) {
      const int l = __ffs(m) - 1;
      const int s = __shfl_sync(FULL, st, l), e = __shfl_sync(FULL, en, l);
      const int64_t room = bound - __shfl_sync(FULL, c, l);  // a neighbour up to this weight may let the node in
      bool fits = false;
      for (int f = s; f < e; f += 32 * kFullUnroll) {
        int u[kFullUnroll];
#pragma unroll
        for (int r = 0; r < kFullUnroll; r++) u[r] = f + r * 32 + lane < e ? adjncy[f + r * 32 + lane] : -1;
#pragma unroll
        for (int r = 0; r < kFullUnroll; r++) u[r] = u[r] >= 0 ? vwgt[u[r]] : INT32_MAX;
#pragma unroll
        for (int r = 0; r < kFullUnroll; r++) fits = fits || u[r] <= room;
        if (__any_sync(FULL, fits)) { fits = true; break; }
      }
      if (lane == l) mark = !fits;
    }
    if (mark) full[v] = 1;
  }
}

// ----------------------------------------------------- per-round buckets

struct BucketArgs {
  const int32_t *xadj, *label, *size, *vwgt;
  int n;
  uint64_t kact;
  int S;           // sub-rounds (1 for the favourite lists)
  int fav_mode;    // 0: all nodes with neighbours; 1: light singletons
  int64_t U;       // fav_mode: light means 2 c <= U
  const int *stop;
  const uint8_t *full;  // nodes that no cluster can have room for (k_mark_full); may be null
};

__device__ __forceinline__ int bucket_key(const BucketArgs &b, int v) {
  const int deg = b.xadj[v + 1] - b.xadj[v];
  if (deg == 0 || (b.full && b.full[v])) return -1;
  if (b.fav_mode) {
    if (b.size[b.label[v]] != 1 || 2 * (int64_t)b.vwgt[v] > b.U) return -1;
    return degree_bucket(deg);
  }
  const int s = (int)(h32(b.kact, (uint32_t)v, 0) % (uint32_t)b.S);
  return s * kNumBuckets + degree_bucket(deg);
}

constexpr int kChunk = kThreads * 16;

__global__ void __launch_bounds__(kThreads) k_bucket_count(BucketArgs b, int nkeys, int *cnt) {
  __shared__ int s_c[kMaxKeys];
  if (b.stop && *b.stop) return;
  for (int t = threadIdx.x; t < nkeys; t += blockDim.x) s_c[t] = 0;
  __syncthreads();
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < b.n;
       v += (int64_t)gridDim.x * blockDim.x) {
    const int k = bucket_key(b, (int)v);
    if (k >= 0) atomicAdd(&s_c[k], 1);
  }
  __syncthreads();
  for (int t = threadIdx.x; t < nkeys; t += blockDim.x)
    if (s_c[t]) atomicAdd(&cnt[t], s_c[t]);
}

// One block of kMaxKeys threads: a scan over the keys (one thread's loop over them took a dependent read
// from memory each).
__global__ void __launch_bounds__(kMaxKeys) k_bucket_offsets(const int *cnt, int nkeys, int *offs, int *cursor,
                                                             const int *stop) {
  __shared__ int s_w[kMaxKeys / 32];
  if (stop && *stop) return;
  const int t = threadIdx.x, lane = (int)lane_id();
  const int x = t < nkeys ? cnt[t] : 0;
  int y = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int z = __shfl_up_sync(FULL, y, o);
    if (lane >= o) y += z;
  }
  if (lane == 31) s_w[t >> 5] = y;
  __syncthreads();
  for (int w = 0; w < (t >> 5); w++) y += s_w[w];
  if (t < nkeys) {
    offs[t] = y - x;
    cursor[t] = y - x;
    if (t == nkeys - 1) offs[nkeys] = y;
  }
}

__global__ void __launch_bounds__(kThreads) k_bucket_scatter(BucketArgs b, int nkeys, int *cursor,
                                                             int4 *list) {
  __shared__ int s_c[kMaxKeys];
  __shared__ int s_base[kMaxKeys];
  if (b.stop && *b.stop) return;
  for (int64_t c0 = (int64_t)blockIdx.x * kChunk; c0 < b.n; c0 += (int64_t)gridDim.x * kChunk) {
    for (int t = threadIdx.x; t < nkeys; t += blockDim.x) s_c[t] = 0;
    __syncthreads();
    int keys[16];
#pragma unroll
    for (int j = 0; j < 16; j++) {
      const int64_t v = c0 + j * kThreads + threadIdx.x;
      keys[j] = v < b.n ? bucket_key(b, (int)v) : -1;
      if (keys[j] >= 0) atomicAdd(&s_c[keys[j]], 1);
    }
    __syncthreads();
    for (int t = threadIdx.x; t < nkeys; t += blockDim.x) {
      s_base[t] = s_c[t] ? atomicAdd(&cursor[t], s_c[t]) : 0;
      s_c[t] = 0;
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < 16; j++) {
      if (keys[j] < 0) continue;
      const int64_t v = c0 + j * kThreads + threadIdx.x;
      const int pos = s_base[keys[j]] + atomicAdd(&s_c[keys[j]], 1);
      const int st = b.xadj[v];
      list[pos] = make_int4((int)v, st, b.xadj[v + 1] - st, b.vwgt[v]);
    }
    __syncthreads();
  }
}

// ------------------------------------------------------ clean nodes
//
// Refinement keeps a flag per node: a node whose rating found no label rated
// above its own (admissible or not) cannot propose until one of its
// neighbours moves, so it is left out of the rating lists until then.

// The dirty records of the sub-round's buckets k0 .. k1-1, packed from the
// start of each bucket's range; ccount[key] receives the bucket's count.
__global__ void __launch_bounds__(kThreads) k_compact_dirty(const int4 *list, const int32_t *offs, int k0, int k1,
                                                            const uint8_t *dirty, int4 *clist, int32_t *ccount,
                                                            const int *stop) {
  if (stop && *stop) return;
  __shared__ int s_cnt[kNumBuckets], s_base[kNumBuckets];
  const int begin = offs[k0], end = offs[k1];
  const int lane = (int)lane_id();
  for (int base = begin + (int)(blockIdx.x * blockDim.x); base < end; base += gridDim.x * blockDim.x) {
    if (threadIdx.x < kNumBuckets) s_cnt[threadIdx.x] = 0;
    __syncthreads();
    const int i = base + (int)threadIdx.x;
    int bk = k1;  // bucket of the position (k1 past the end)
    int b = -1;   // bucket if the record is kept
    int4 rec = make_int4(0, 0, 0, 0);
    if (i < end) {
      bk = k0;
      while (bk + 1 < k1 && offs[bk + 1] <= i) bk++;
      rec = list[i];
      if (dirty[rec.x]) b = bk;
    }
    // consecutive lanes hold consecutive list positions, so a bucket's lanes form one run:
    // its kept lanes are the peers (no match over arbitrary keys needed)
    const int prev = __shfl_up_sync(FULL, bk, 1);
    const unsigned starts = __ballot_sync(FULL, lane == 0 || prev != bk);
    const unsigned kept = __ballot_sync(FULL, b >= 0);
    const unsigned le = lanemask_lt() | (1u << lane);
    const unsigned after = starts & ~le;  // run starts after this lane
    const unsigned run_lo = 31 - __clz(starts & le);
    const unsigned run_hi = after ? (unsigned)__ffs(after) - 1 : 32u;  // one past the run
    const unsigned run = (run_hi == 32 ? FULL : ((1u << run_hi) - 1u)) & ~((1u << run_lo) - 1u);
    const unsigned peers = kept & run;
    int pos = 0;
    if (b >= 0) {
      // the block's kept records of each bucket are counted in shared memory, and the bucket's
      // global cursor advances once per block and bucket
      const int leader = __ffs(peers) - 1;
      if (lane == leader) pos = atomicAdd(&s_cnt[b - k0], __popc(peers));
      pos = __shfl_sync(peers, pos, leader) + __popc(peers & lanemask_lt());
    }
    __syncthreads();
    if (threadIdx.x < kNumBuckets && s_cnt[threadIdx.x] > 0)
      s_base[threadIdx.x] = atomicAdd(&ccount[k0 + threadIdx.x], s_cnt[threadIdx.x]);
    __syncthreads();
    if (b >= 0) clist[offs[b] + s_base[b - k0] + pos] = rec;
  }
}
__global__ void __launch_bounds__(kThreads) k_mark_dirty(const int4 *mov, int nmov, const uint64_t *ov_key,
                                                         const uint32_t *ov_val, const uint8_t *ov_acc, int nov,
                                                         const uint64_t *cutoff, uint64_t kprio,
                                                         const int32_t *xadj, const int32_t *adjncy,
                                                         uint8_t *dirty) {
  const int lane = (int)lane_id();
  const int wid = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int nw = (int)((gridDim.x * blockDim.x) >> 5);
  const int total = nmov + nov;
  for (int t0 = 2 * wid; t0 < total; t0 += 2 * nw) {
    int v[2], e0[2], e1[2];
#pragma unroll
    for (int q = 0; q < 2; q++) {
      const int t = t0 + q;
      v[q] = -1;
      if (t < nmov) v[q] = mov[t].x;
      else if (t < total && ov_acc[t - nmov]) v[q] = (int)ov_val[t - nmov];
      if (v[q] >= 0 && cutoff &&
          ((((uint64_t)h32(kprio, (uint32_t)v[q], 0)) << 32) | (uint32_t)v[q]) >= *cutoff)
        v[q] = -1;
      e0[q] = v[q] >= 0 ? xadj[v[q]] : 0;
      e1[q] = v[q] >= 0 ? xadj[v[q] + 1] : 0;
    }
#pragma unroll
    for (int q = 0; q < 2; q++)
      if (lane == 0 && v[q] >= 0) dirty[v[q]] = 1;
    const int len = max(e1[0] - e0[0], e1[1] - e0[1]);
    for (int o = lane; o < len; o += 32) {
      const int a0 = e0[0] + o, a1 = e0[1] + o;
      const int u0 = a0 < e1[0] ? adjncy[a0] : -1, u1 = a1 < e1[1] ? adjncy[a1] : -1;
      if (u0 >= 0) dirty[u0] = 1;
      if (u1 >= 0) dirty[u1] = 1;
    }
  }
}

// ------------------------------------------------------------- acceptance

struct Counters {
  int stop;
  int nov;   // proposers of overflowing targets this sub-round
  int nmov;  // proposers accepted outright this sub-round
  int pad0;
  long long moved_sub;
  long long moved_round;
  long long moved_total;
  long long nonempty;   // clustering: change of the number of labels of positive weight in the sub-round
  long long nclusters;
};

// Every active node's proposal (written by the rating kernels at its list
// position) goes to the list of outright acceptances (the target's snapshot
// weight plus all incoming weight fits), as a (node, target, own label,
// weight) record, or to the list of proposers of overflowing targets.  Slots
// in both lists are reserved once per block and iteration.
__global__ void __launch_bounds__(kThreads) k_decide(const int4 *list, const int32_t *offs,
                                                     int k0, int k1, const int2 *prop,
                                                     const int32_t *weight, const int32_t *incoming,
                                                     int64_t bound, int4 *mov,
                                                     uint64_t *ov_key, uint32_t *ov_val, Counters *cnt,
                                                     uint64_t kprio, const int32_t *ccount) {
  __shared__ int s_a[kWarpsPerBlock + 1], s_o[kWarpsPerBlock + 1];
  if (cnt->stop) return;
  const int begin = offs[k0], end = offs[k1];
  const int stride = gridDim.x * blockDim.x;
  const int lane = (int)lane_id(), w = threadIdx.x >> 5;
  for (int base = begin + (int)(blockIdx.x * blockDim.x); base < end; base += stride) {
    const int i = base + (int)threadIdx.x;
    bool acc = false, over = false;
    int v = 0, K = -1, own = 0, c = 0;
    bool live = i < end;
    if (live && ccount) {  // compacted lists: positions past a bucket's count hold nothing
      int b = k0;
      while (b + 1 < k1 && offs[b + 1] <= i) b++;
      live = i < offs[b] + ccount[b];
    }
    if (live) {
      const int2 pr = prop[i];
      K = pr.x;
      if (K >= 0) {
        const int4 rec = list[i];
        v = rec.x; c = rec.w; own = pr.y;
        if ((int64_t)weight[K] + incoming[K] <= bound) acc = true;
        else over = true;
      }
    }
    const unsigned ma = __ballot_sync(0xFFFFFFFFu, acc), mo = __ballot_sync(0xFFFFFFFFu, over);
    if (lane == 0) { s_a[w] = __popc(ma); s_o[w] = __popc(mo); }
    __syncthreads();
    if (threadIdx.x == 0) {
      int ra = 0, ro = 0;
      for (int j = 0; j < kWarpsPerBlock; j++) {
        const int ca = s_a[j], co = s_o[j];
        s_a[j] = ra; s_o[j] = ro;
        ra += ca; ro += co;
      }
      s_a[kWarpsPerBlock] = ra ? atomicAdd(&cnt->nmov, ra) : 0;
      s_o[kWarpsPerBlock] = ro ? atomicAdd(&cnt->nov, ro) : 0;
    }
    __syncthreads();
    if (acc) {
      const int pos = s_a[kWarpsPerBlock] + s_a[w] + __popc(ma & lanemask_lt());
      mov[pos] = make_int4(v, K, own, c);
    }
    if (over) {
      const int pos = s_o[kWarpsPerBlock] + s_o[w] + __popc(mo & lanemask_lt());
      ov_key[pos] = ((uint64_t)(uint32_t)K << 32) | h32(kprio, (uint32_t)v, 0);
      ov_val[pos] = (uint32_t)v;
    }
    __syncthreads();
  }
}

// Runs of equal keys are ordered by node id (the last tie-break of R7).
__global__ void k_fix_runs(const uint64_t *keys, uint32_t *vals, int n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    if (i > 0 && keys[i - 1] == keys[i]) continue;
    if (i + 1 >= n || keys[i + 1] != keys[i]) continue;
    int e = i + 1;
    while (e < n && keys[e] == keys[i]) e++;
    for (int a = i + 1; a < e; a++) {
      uint32_t x = vals[a];
      int b = a - 1;
      while (b >= i && vals[b] > x) { vals[b + 1] = vals[b]; b--; }
      vals[b + 1] = x;
    }
  }
}

__global__ void k_ov_weights(const uint32_t *vals, int n, const int32_t *vwgt, int64_t *cs) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    cs[i] = vwgt[vals[i]];
}

// Sorted by (target, prio, node): accept while the running weight within the
// target's segment fits (ps = exclusive prefix sum of the weights).
__global__ void k_ov_accept(const uint64_t *keys, const uint32_t *vals, int n, const int64_t *ps,
                            const int32_t *vwgt, const int32_t *weight, int64_t bound, uint8_t *ov_acc) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const uint64_t k = keys[i];
    const uint64_t seg = k & 0xFFFFFFFF00000000ull;
    int lo = 0, hi = i;  // first index with key >= seg
    while (lo < hi) {
      int mid = (lo + hi) >> 1;
      if (keys[mid] < seg) lo = mid + 1; else hi = mid;
    }
    const int K = (int)(k >> 32);
    const int64_t incl = ps[i] - ps[lo] + vwgt[vals[i]];
    ov_acc[i] = (int64_t)weight[K] + incl <= bound ? 1 : 0;
  }
}

// ------------------------------------------ small overflow sets
//
// Up to kOvSmall proposers of overflowing targets are ordered by (target,
// priority, node) with a bitonic sort in one block's shared memory; a block
// scan of their weights gives every proposer its running weight within its
// target, and it is accepted iff the target's weight plus that fits.

constexpr int kOvSmall = 2048;
constexpr int kOvSmallThreads = 1024;

__global__ void __launch_bounds__(kOvSmallThreads) k_ov_small(uint64_t *key, uint32_t *val, int nov,
                                                              const int32_t *vwgt, const int32_t *weight,
                                                              int64_t bound, uint8_t *acc) {
  __shared__ uint64_t s_k[kOvSmall];
  __shared__ uint32_t s_v[kOvSmall];
  __shared__ long long s_w[kOvSmallThreads / 32];
  int P = 1;
  while (P < nov) P <<= 1;
  const int t = threadIdx.x;
  for (int i = t; i < P; i += blockDim.x) {
    s_k[i] = i < nov ? key[i] : ~0ull;
    s_v[i] = i < nov ? val[i] : 0xFFFFFFFFu;
  }
  __syncthreads();
  for (int size = 2; size <= P; size <<= 1) {
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      for (int i = t; i < P / 2; i += blockDim.x) {
        const int lo = 2 * i - (i & (stride - 1));  // pairs (lo, lo + stride)
        const int hi = lo + stride;
        const bool up = (lo & size) == 0;
        const uint64_t ka = s_k[lo], kb = s_k[hi];
        const uint32_t va = s_v[lo], vb = s_v[hi];
        const bool gt = ka > kb || (ka == kb && va > vb);
        if (gt == up) { s_k[lo] = kb; s_k[hi] = ka; s_v[lo] = vb; s_v[hi] = va; }
      }
      __syncthreads();
    }
  }
  // sorted order written back; inclusive running weights (their total is at most
  // the graph's node weight, below 2^31) replace the node ids in shared memory
  long long carry = 0;
  const int lane = (int)lane_id(), wp = t >> 5, nwp = blockDim.x >> 5;
  for (int c0 = 0; c0 < nov; c0 += blockDim.x) {
    const int i = c0 + t;
    long long x = 0;
    if (i < nov) {
      const uint32_t v = s_v[i];
      key[i] = s_k[i];
      val[i] = v;
      x = vwgt[v];
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const long long y = __shfl_up_sync(FULL, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) s_w[wp] = x;
    __syncthreads();
    long long before = carry, chunk = 0;
    for (int q = 0; q < nwp; q++) {
      if (q < wp) before += s_w[q];
      chunk += s_w[q];
    }
    if (i < nov) s_v[i] = (uint32_t)(before + x);
    carry += chunk;
    __syncthreads();
  }
  for (int i = t; i < nov; i += blockDim.x) {
    // first proposer of i's target: lower bound of (target << 32) in the sorted keys
    const uint64_t seg = s_k[i] & 0xFFFFFFFF00000000ull;
    int a = 0, b = i;
    while (a < b) {
      const int mid = (a + b) >> 1;
      if (s_k[mid] < seg) a = mid + 1; else b = mid;
    }
    const long long incl = (long long)s_v[i] - (a > 0 ? (long long)s_v[a - 1] : 0);
    const int K = (int)(s_k[i] >> 32);
    acc[i] = (int64_t)weight[K] + incl <= bound ? 1 : 0;
  }
}

// ------------------------------------------ overflow with few labels
//
// The proposers of overflowing targets are not sorted.  Per target, a
// histogram of their weights over the top bits of the priority locates the
// bucket in which the running weight (in priority order) crosses the
// target's free room: proposers in earlier buckets fit (the accepted prefix
// contains them), proposers in later ones do not, and only the crossing
// bucket's proposers are ranked exactly by (priority, node), in one block per
// target.  The result equals the longest-prefix rule of the sorted order.

constexpr int kOvBuckets = 4096;   // priority buckets per label (top 12 bits)
constexpr int kOvMaxLabels = 256;  // labels handled this way
constexpr int kOvSmem = 2048;      // crossing-bucket proposers ranked in shared memory

__global__ void k_ovb_hist(const uint64_t *key, const uint32_t *val, int nov, const int32_t *vwgt,
                           unsigned long long *hw, int32_t *hc) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nov; i += gridDim.x * blockDim.x) {
    const uint64_t k = key[i];
    const int64_t slot = (int64_t)(k >> 32) * kOvBuckets + (int)((uint32_t)k >> 20);
    atomicAdd(&hw[slot], (unsigned long long)vwgt[val[i]]);
    atomicAdd(&hc[slot], 1);
  }
}

// One block per label: the crossing bucket, the weight before it and the
// number of proposers in it.
__global__ void __launch_bounds__(256) k_ovb_cut(const unsigned long long *hw, const int32_t *hc,
                                                 const int32_t *weight, int64_t bound, int32_t *cut,
                                                 long long *base, int32_t *mcnt) {
  constexpr int PER = kOvBuckets / 256;
  __shared__ long long s_w[8];
  __shared__ int s_cut;
  const int K = blockIdx.x;
  const unsigned long long *h = hw + (int64_t)K * kOvBuckets;
  const int t = threadIdx.x, lane = (int)lane_id(), wp = t >> 5;
  long long loc = 0;
#pragma unroll
  for (int q = 0; q < PER; q++) loc += (long long)h[t * PER + q];
  long long incl = loc;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long y = __shfl_up_sync(FULL, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) s_w[wp] = incl;
  if (t == 0) s_cut = kOvBuckets;
  __syncthreads();
  long long excl = incl - loc;
  for (int q = 0; q < wp; q++) excl += s_w[q];
  const long long room = bound - (long long)weight[K];
  long long run = excl;
  int mine = kOvBuckets;
  long long before = 0;
  for (int q = 0; q < PER; q++) {
    const long long x = (long long)h[t * PER + q];
    if (x > 0 && run + x > room) { mine = t * PER + q; before = run; break; }
    run += x;
  }
  if (mine < kOvBuckets) atomicMin(&s_cut, mine);
  __syncthreads();
  if (mine == s_cut && mine < kOvBuckets) {
    cut[K] = mine;
    base[K] = before;
    mcnt[K] = hc[(int64_t)K * kOvBuckets + mine];
  }
  if (t == 0 && s_cut == kOvBuckets) { cut[K] = kOvBuckets; base[K] = 0; mcnt[K] = 0; }
}

__global__ void __launch_bounds__(1024) k_ovb_offsets(const int32_t *mcnt, int nlabels, int32_t *roff,
                                                      int32_t *cursor) {
  if (threadIdx.x == 0) {
    int run = 0;
    for (int K = 0; K < nlabels; K++) { roff[K] = run; cursor[K] = run; run += mcnt[K]; }
    roff[nlabels] = run;
  }
}

// Earlier buckets accepted, later ones rejected, the crossing bucket's
// proposers listed per label.
__global__ void k_ovb_class(const uint64_t *key, const uint32_t *val, int nov, const int32_t *cut,
                            int32_t *cursor, uint8_t *acc, uint64_t *bkey, int32_t *bidx) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nov; i += gridDim.x * blockDim.x) {
    const uint64_t k = key[i];
    const int K = (int)(k >> 32), b = (int)((uint32_t)k >> 20), c = cut[K];
    acc[i] = b < c ? 1 : 0;
    if (b == c) {
      const int j = atomicAdd(&cursor[K], 1);
      bkey[j] = ((uint64_t)(uint32_t)k << 32) | val[i];  // (priority, node)
      bidx[j] = i;
    }
  }
}

// One block per label: ranks the crossing bucket's proposers by (priority,
// node) and accepts those whose running weight still fits.
__global__ void __launch_bounds__(256) k_ovb_resolve(const uint64_t *bkey, const int32_t *bidx,
                                                     const int32_t *roff, const int32_t *vwgt,
                                                     const int32_t *weight, const long long *base,
                                                     int64_t bound, uint8_t *acc) {
  __shared__ uint64_t s_k[kOvSmem];
  __shared__ int s_c[kOvSmem];
  const int K = blockIdx.x;
  const int r0 = roff[K], m = roff[K + 1] - r0;
  if (m == 0) return;
  const bool in_smem = m <= kOvSmem;
  if (in_smem) {
    for (int j = threadIdx.x; j < m; j += blockDim.x) {
      s_k[j] = bkey[r0 + j];
      s_c[j] = vwgt[(uint32_t)bkey[r0 + j]];
    }
    __syncthreads();
  }
  const long long room = bound - (long long)weight[K] - base[K];
  for (int i = threadIdx.x; i < m; i += blockDim.x) {
    const uint64_t ki = in_smem ? s_k[i] : bkey[r0 + i];
    long long incl = 0;
    for (int j = 0; j < m; j++) {  // weight of the proposers up to and including i
      const uint64_t kj = in_smem ? s_k[j] : bkey[r0 + j];
      if (kj <= ki) incl += in_smem ? s_c[j] : vwgt[(uint32_t)kj];
    }
    acc[bidx[r0 + i]] = incl <= room ? 1 : 0;
  }
}

struct ApplyArgs {
  const int4 *mov;  // outright moves: (node, target, own label, node weight)
  const uint64_t *ov_key;
  const uint32_t *ov_val;
  const uint8_t *ov_acc;
  int nmov, nov;
  const int32_t *vwgt;
  int32_t *label, *weight, *incoming;
  uint8_t *label8;
  int nshared;       // > 0: few labels; weight changes summed per block in shared memory
  Counters *cnt;
  const uint64_t *cutoff;  // 2.5x cap: only moves with key (h32(PRIO), v) below *cutoff apply (null: all)
  uint64_t kprio;
  int track;  // clustering: count the labels whose weight reaches or leaves 0
};

__device__ __forceinline__ uint64_t move_key(uint64_t kprio, int v) {
  return ((uint64_t)h32(kprio, (uint32_t)v, 0) << 32) | (uint32_t)v;
}

__device__ __forceinline__ void proposal(const ApplyArgs &a, int t, int &v, int &K, int &own, int &c,
                                         bool &mv) {
  if (t < a.nmov) {
    const int4 r = a.mov[t];
    v = r.x; K = r.y; own = r.z; c = r.w; mv = true;
  } else {
    const int j = t - a.nmov;
    v = (int)a.ov_val[j]; K = (int)(a.ov_key[j] >> 32); mv = a.ov_acc[j] != 0;
    own = mv ? a.label[v] : 0;
    c = mv ? a.vwgt[v] : 0;
  }
}

// Moves every accepted proposer (outright or through the overflow order).
__global__ void __launch_bounds__(kThreads) k_apply(ApplyArgs a) {
  extern __shared__ int s_dw[];
  for (int t = threadIdx.x; t < a.nshared; t += blockDim.x) s_dw[t] = 0;
  if (a.nshared) __syncthreads();
  const int total = a.nmov + a.nov;
  long long moved = 0, dne = 0;  // dne: labels whose weight left 0 minus labels whose weight reached 0
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
    int v, K, own, c;
    bool mv;
    proposal(a, t, v, K, own, c, mv);
    if (mv && a.cutoff && move_key(a.kprio, v) >= *a.cutoff) mv = false;
    if (mv) {
      a.label[v] = K;
      if (a.label8) a.label8[v] = (uint8_t)K;

      if (a.nshared) {
        atomicAdd(&s_dw[K], c);
        atomicSub(&s_dw[own], c);
      } else {
        // every update's transition 0 <-> non-0 counted: their sum is the net change
        const int ok = atomicAdd(&a.weight[K], c);
        const int oo = atomicSub(&a.weight[own], c);
        if (a.track) dne += (ok == 0 ? 1 : 0) - (oo == c ? 1 : 0);
      }
      moved++;
    }
  }
  if (a.nshared) {
    __syncthreads();
    for (int t = threadIdx.x; t < a.nshared; t += blockDim.x)
      if (s_dw[t]) {
        const int o = atomicAdd(&a.weight[t], s_dw[t]);
        if (a.track) dne += ((o + s_dw[t] > 0) ? 1 : 0) - ((o > 0) ? 1 : 0);
      }
  }
  moved = warp_sum(moved);
  dne = warp_sum(dne);
  if (lane_id() == 0 && moved)
    atomicAdd((unsigned long long *)&a.cnt->moved_sub, (unsigned long long)moved);
  if (lane_id() == 0 && dne) atomicAdd((unsigned long long *)&a.cnt->nonempty, (unsigned long long)dne);
}

// ------------------------------------------------------- the 2.5x cap
//
// The node reduction of a clustering is at most 2.5x (Sec. 4.3): with c
// clusters at the start of a sub-round, its moves may empty at most D =
// c - n_min of them.  A cluster all of whose weight leaves is emptied at the
// largest move key (h32(PRIO), node) among its departures (arrivals are not
// counted); if more than D clusters are emptied, only the moves below the
// (D+1)-th smallest emptying key apply.  These kernels run before k_apply, on
// the snapshot labels and weights, and only in sub-rounds whose accepted moves
// could exceed D.

// Departure weight and latest departure key per source cluster.
__global__ void __launch_bounds__(kThreads) k_cap_depart(ApplyArgs a, int32_t *depw,
                                                         unsigned long long *dkey) {
  const int total = a.nmov + a.nov;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
    int v, K, own, c;
    bool mv;
    proposal(a, t, v, K, own, c, mv);
    if (!mv) continue;
    atomicAdd(&depw[own], c);
    atomicMax(&dkey[own], (unsigned long long)move_key(a.kprio, v));
  }
}

// The emptying key of every emptied cluster (listed once, by its latest mover);
// then clears the per-cluster state of the sources.
__global__ void __launch_bounds__(kThreads) k_cap_collect(ApplyArgs a, const int32_t *depw,
                                                          const unsigned long long *dkey,
                                                          uint64_t *ekeys, int *ecount) {
  const int total = a.nmov + a.nov;
  for (int base = blockIdx.x * blockDim.x; base < total; base += gridDim.x * blockDim.x) {
    const int t = base + (int)threadIdx.x;
    bool emit_key = false;
    uint64_t key = 0;
    if (t < total) {
      int v, K, own, c;
      bool mv;
      proposal(a, t, v, K, own, c, mv);
      if (mv) {
        key = move_key(a.kprio, v);
        emit_key = depw[own] == a.weight[own] && key == dkey[own];
      }
    }
    const int pos = warp_append(ecount, emit_key);
    if (emit_key) ekeys[pos] = key;
  }
}

__global__ void __launch_bounds__(kThreads) k_cap_clear(ApplyArgs a, int32_t *depw, unsigned long long *dkey) {
  const int total = a.nmov + a.nov;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
    int v, K, own, c;
    bool mv;
    proposal(a, t, v, K, own, c, mv);
    if (!mv) continue;
    depw[own] = 0;
    dkey[own] = 0;
  }
}

// Closes a sub-round in one launch: clears the incoming weights of its
// targets, counts the non-empty clusters (node weights are positive, so a
// label is in use iff its weight is), and the last block to finish updates
// the counters: cluster count, moves, the stop flag (cluster count at n_min;
// at the end of a round, a round without moves), and clears the proposal
// list sizes for the next sub-round.
__global__ void __launch_bounds__(kThreads) k_close(ApplyArgs a, int64_t count_labels, long long n_min,
                                                    int round_end, unsigned *done) {
  Counters *cnt = a.cnt;
  if (cnt->stop) return;
  const int total = a.nmov + a.nov;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
    const int K = t < a.nmov ? a.mov[t].y : (int)(a.ov_key[t - a.nmov] >> 32);
    a.incoming[K] = 0;
  }
  __syncthreads();
  __shared__ bool s_last;
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = atomicAdd(done, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last || threadIdx.x != 0) return;
  __threadfence();
  volatile Counters *vc = cnt;
  if (count_labels > 0) vc->nclusters = vc->nclusters + vc->nonempty;  // k_apply's net change
  vc->nonempty = 0;
  const long long moved = vc->moved_sub;
  vc->moved_round = vc->moved_round + moved;
  vc->moved_total = vc->moved_total + moved;
  vc->moved_sub = 0;
  vc->nov = 0;
  vc->nmov = 0;
  if (count_labels > 0 && vc->nclusters <= n_min) vc->stop = 1;
  if (round_end) {
    if (!vc->stop && vc->moved_round == 0) vc->stop = 1;
    vc->moved_round = 0;
  }
  *done = 0;
}

__global__ void k_counters_init(Counters *cnt, long long nclusters) {
  cnt->stop = 0; cnt->nov = 0; cnt->nmov = 0; cnt->pad0 = 0; cnt->moved_sub = 0; cnt->moved_round = 0;
  cnt->moved_total = 0; cnt->nonempty = 0; cnt->nclusters = nclusters;
}

// Largest degree, number of nodes above kBlockDeg0, number of hubs and their neighbours.
struct DegStats {
  int maxdeg, big, hubs, pad;
  unsigned long long hubdeg;
};

__global__ void k_max_degree(const int32_t *xadj, int n, DegStats *out) {
  int m = 0, nb = 0, nh = 0;
  unsigned long long ns = 0;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x) {
    const int d = xadj[v + 1] - xadj[v];
    m = d > m ? d : m;
    if (d > kBlockDeg0) nb++;
    if (d > kHubDeg) { nh++; ns += (unsigned long long)d; }
  }
  m = warp_max(m);
  if (lane_id() == 0 && m) atomicMax(&out->maxdeg, m);
  if (__any_sync(FULL, nb)) {
    nb = warp_sum(nb);
    nh = warp_sum(nh);
    ns = warp_sum(ns);
    if (lane_id() == 0) { atomicAdd(&out->big, nb); atomicAdd(&out->hubs, nh); atomicAdd(&out->hubdeg, ns); }
  }
}

__global__ void k_fill_slots(int2 *tab, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    tab[i] = make_int2(-1, 0);
}

struct RateTables {
  DBuf<int32_t> gkeys, gvals;
  int64_t stride = 0;
  int blocks = 0;
  // hubs (HubArgs), when the graph has some and their tables stay within the bound of table_blocks
  bool hubs = false;
  int q4 = 0;          // the hub tables' slots per neighbour, in quarters
  bool dense = false;  // few labels: nodes above kBlockDeg0 are counted per label
  DBuf<Hub> hub;
  DBuf<int> chunk0, tchunk0;
  DBuf<int2> tab;
  DBuf<int32_t> hist;
};

// What the kernels for nodes beyond the shared tables need: the hubs' plan and tables (nlabels > 0: label
// propagation), or per-block hash tables in global memory (favourites, and graphs whose hubs' tables
// together would take more memory than that).
void make_tables(gp_ctx *ctx, const DevGraph &g, int64_t nlabels, RateTables &t) {
  DBuf<DegStats> ds(ctx, 1);
  ds.zero();
  k_max_degree<<<grid_for(g.n, 256, ctx->num_sms * 8), 256, 0, ctx->stream>>>(g.xadj, g.n, ds.get());
  GP_LAUNCH_CHECK();
  DegStats h;
  read_back(ctx, ds.get(), sizeof(h), &h);
  const int maxdeg = h.maxdeg;
  t.blocks = ctx->num_sms * 4;
  if (nlabels > 0) {
    const int64_t cap = ctx->limits.table_bytes(g.m2) / (int64_t)sizeof(int2);
    t.dense = nlabels <= kHubDense && (int64_t)h.big * nlabels <= 2 * cap;
    const int64_t hubs = t.dense ? h.big : h.hubs;
    int64_t slots = 0;
    for (t.q4 = 12; t.q4 > 4; t.q4 -= 2) {  // three slots per neighbour down to one and a half
      slots = (int64_t)h.hubdeg * t.q4 / 4 + hubs;
      if (slots <= cap) break;
    }
    t.hubs = hubs > 0 && (t.dense || t.q4 > 4);
    if (t.hubs) {
      t.hub.reset(ctx, (size_t)hubs);
      t.chunk0.reset(ctx, (size_t)hubs + 1);
      t.tchunk0.reset(ctx, (size_t)hubs + 1);
      if (t.dense) {
        t.hist.reset(ctx, (size_t)(hubs * nlabels));
        t.hist.zero();
      } else {
        t.tab.reset(ctx, (size_t)slots);
        k_fill_slots<<<grid_for(slots, 256, ctx->num_sms * 8), 256, 0, ctx->stream>>>(t.tab.get(), slots);
        GP_LAUNCH_CHECK();
      }
    }
    if (t.hubs || maxdeg <= kHubDeg) return;
  }
  const int bits = table_bits(maxdeg, 1);
  if (((int64_t)1 << bits) > kLargeSmemSlots) {
    t.stride = (int64_t)1 << bits;
    t.blocks = table_blocks(ctx->limits.table_bytes(g.m2), t.stride, t.blocks);
    t.gkeys.reset(ctx, (size_t)(t.stride * t.blocks));
    t.gvals.reset(ctx, (size_t)(t.stride * t.blocks));
    t.gkeys.fill_bytes(0xFF);
    t.gvals.zero();
  }
}

// Grid for `count` listed nodes, `per_block` nodes per block and iteration
// (count < 0: unknown, the full grid).
inline int rate_grid(gp_ctx *ctx, int64_t count, int per_block, int cap) {
  if (count < 0) return cap;
  return grid_for(count, per_block, cap);
}

// One class of degree <= D; count < 0: unknown, the full grid.
template <int MODE, int D, int LK>
void launch_threads(gp_ctx *ctx, RateArgs a, int key, int count) {
  if (count == 0) return;
  a.key = key;
  constexpr int NT = ThreadShape<D>::NT;
  k_rate_thread<MODE, D, LK><<<rate_grid(ctx, count, NT, ctx->num_sms * ThreadShape<D>::PER_SM * 4), NT, 0,
                               ctx->stream>>>(a);
  GP_LAUNCH_CHECK();
}

// hcnt: the bucket sizes of this sub-round when the host knows them (empty buckets are then not
// launched), else nullptr
template <int MODE, int LK>
void launch_groups(gp_ctx *ctx, const RateArgs &a, int base, const int *hcnt) {
  launch_threads<MODE, 8, LK>(ctx, a, base + 0, hcnt ? hcnt[0] : -1);
  launch_threads<MODE, 16, LK>(ctx, a, base + 1, hcnt ? hcnt[1] : -1);
  launch_threads<MODE, 24, LK>(ctx, a, base + 2, hcnt ? hcnt[2] : -1);
  launch_threads<MODE, 32, LK>(ctx, a, base + 3, hcnt ? hcnt[3] : -1);
}

template <int NT>
void launch_block(gp_ctx *ctx, const RateArgs &a, int maxdeg, int q4, int grid) {
  const int slots = tab_slots(maxdeg, q4);
  const size_t smem = 2 * sizeof(int) * (size_t)slots;
  if (smem > 48 * 1024)
    GP_CUDA(cudaFuncSetAttribute(k_rate_block<NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  k_rate_block<NT><<<grid, NT, smem, ctx->stream>>>(a, slots, q4);
  GP_LAUNCH_CHECK();
}

template <int MODE>
void launch_warps(gp_ctx *ctx, const RateArgs &a, int maxdeg, int count) {
  const int slots = tab_slots(maxdeg, kTabQ4);
  const size_t smem = 2 * sizeof(int) * (size_t)slots * kWarpsPerBlock;
  if (smem > 48 * 1024)
    GP_CUDA(cudaFuncSetAttribute(k_rate_warp<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  k_rate_warp<MODE><<<rate_grid(ctx, count, kWarpsPerBlock, ctx->num_sms * 8), kThreads, smem, ctx->stream>>>(a, slots);
  GP_LAUNCH_CHECK();
}

// A sub-round of few nodes is a chain of launches of some 5 us each, one per class that is not empty.  The classes
// up to kWarpMaxDeg go through k_rate_warp together while they hold at most Limits::few_nodes nodes an SM for each launch
// that this saves (24 warps an SM take about 1.5 us for a node each), and up to one node an SM of the block
// classes through the largest of these.  A launch per class / together, on the per-phase path: refinement with k = 64 of
// scale-10, -14 and -18 R-MAT graphs 4.5 / 3.0, 5.9 / 4.1 and 7.6 / 5.9 ms, of an ER graph of 65,536 nodes 4.4 / 3.2; clustering
// of the scale-14 and -18 graphs 5.6 / 3.5 and 8.3 / 5.1 ms.  With one class (a mesh) nothing is saved and a warp per
// node takes longer.

// nlabels: number of labels
template <int MODE>
void launch_rate(gp_ctx *ctx, RateArgs a, int bucket_key_base, const RateTables &t, int64_t nlabels,
                 const int *hcnt) {
  a.nkeys = 1;
  int warps = 0, warp_classes = 0, blocks = 0, block_classes = 0;
  if (hcnt) {
    for (int b = 0; b < kMediumBucket + 2; b++) {
      warps += hcnt[b];
      warp_classes += hcnt[b] > 0;
    }
    for (int b = kMediumBucket + 2; b < kMediumBucket + 5; b++) {
      blocks += hcnt[b];
      block_classes += hcnt[b] > 0;
    }
  }
  const int few = ctx->limits.few_nodes * ctx->num_sms;
  if (MODE == RATE_LP && warp_classes > 1 && warps <= (int64_t)few * (warp_classes - 1)) {
    a.key = bucket_key_base;
    a.nkeys = kMediumBucket + 2;
    launch_warps<MODE>(ctx, a, kWarpMaxDeg, warps);
    a.nkeys = 1;
  } else {
    if (MODE == RATE_LP && a.label8) launch_groups<MODE, MODE == RATE_LP ? LK_NARROW : LK_WIDE>(ctx, a, bucket_key_base, hcnt);
    else launch_groups<MODE, LK_WIDE>(ctx, a, bucket_key_base, hcnt);
    for (int q = 0; q < 2; q++) {  // a warp per node; favourites of larger nodes: k_rate_large
      const int b = kMediumBucket + q;
      if ((hcnt && hcnt[b] == 0) || (q == 1 && MODE != RATE_LP)) continue;
      a.key = bucket_key_base + b;
      launch_warps<MODE>(ctx, a, q == 0 ? kMediumMaxDeg : kWarpMaxDeg, hcnt ? hcnt[b] : -1);
    }
  }
  const bool together =
      MODE == RATE_LP && few > 0 && !(t.hubs && t.dense) && block_classes > 1 && blocks <= ctx->num_sms;
  if (together) {
    a.key = bucket_key_base + kMediumBucket + 2;
    a.nkeys = 3;
    launch_block<1024>(ctx, a, kHubDeg, kTabQ4Last, blocks);
    a.nkeys = 1;
  }
  const int hgrid = ctx->num_sms * 6;
  for (int q = MODE == RATE_LP ? 0 : -1; q < 4; q++) {  // the three block classes, the hubs
    const int b = kMediumBucket + 2 + q;
    const int c = hcnt ? hcnt[b] : -1;
    if (c == 0 || (together && q < 3)) continue;
    a.key = bucket_key_base + b;
    if (MODE == RATE_LP && t.hubs && (q == 3 || (q > 0 && t.dense))) {
      HubArgs h{t.hub.get(), t.chunk0.get(), t.tchunk0.get(), t.tab.get(), t.hist.get(), (int)nlabels, t.q4};
      k_hub_plan<<<1, 1024, 0, ctx->stream>>>(a, h);
      GP_LAUNCH_CHECK();
      if (t.dense) {
        k_hub_dense<<<hgrid, kThreads, sizeof(int) * (size_t)nlabels, ctx->stream>>>(a, h);
        GP_LAUNCH_CHECK();
      } else {
        k_hub_insert<<<hgrid, kThreads, 0, ctx->stream>>>(a, h);
        GP_LAUNCH_CHECK();
        k_hub_table<false><<<hgrid, kThreads, 0, ctx->stream>>>(a, h);
        GP_LAUNCH_CHECK();
        k_hub_table<true><<<hgrid, kThreads, 0, ctx->stream>>>(a, h);
        GP_LAUNCH_CHECK();
      }
    } else if (MODE == RATE_LP && q < 3) {
      if (q == 0) launch_block<256>(ctx, a, kBlockDeg0, kTabQ4, rate_grid(ctx, c, 1, ctx->num_sms * 6));
      else if (q == 1) launch_block<512>(ctx, a, kBlockDeg1, kTabQ4, rate_grid(ctx, c, 1, ctx->num_sms * 2));
      else launch_block<1024>(ctx, a, kHubDeg, kTabQ4Last, rate_grid(ctx, c, 1, ctx->num_sms));
    } else {
      a.gkeys = t.gkeys.get();
      a.gvals = t.gvals.get();
      a.gstride = t.stride;
      k_rate_large<MODE><<<rate_grid(ctx, c, 1, t.blocks), kThreads, 0, ctx->stream>>>(a);
      GP_LAUNCH_CHECK();
    }
  }
}

}  // namespace

int bits_for(int64_t x) {
  int b = 0;
  while (((int64_t)1 << b) <= x) b++;
  return b < 1 ? 1 : b;
}

LpResult lp_run(gp_ctx *ctx, const DevGraph &g, int32_t *label, int32_t *weight, int64_t nlabels, uint64_t seed, const LpParams &p, int64_t *nclusters_dev,
                uint8_t *label8) {
  LpResult res;
  const int n = g.n;
  DBuf<uint8_t> full;
  if (p.count_clusters && n > 0) {
    ProfScope ps(ctx, PROF_ROUND_SETUP);
    full.reset(ctx, (size_t)n);
    full.zero();
    k_mark_full<<<grid_for(n, kThreads, ctx->num_sms * 8), kThreads, 0, ctx->stream>>>(g.xadj, g.adjncy, g.vwgt, n,
                                                                                       p.bound, full.get());
    GP_LAUNCH_CHECK();
  }
  if (lp_small_applicable(g, p) &&
      lp_run_small(ctx, g, label, weight, nlabels, seed, p, nclusters_dev, label8, full.get(), res))
    return res;
  const int S = p.subrounds;
  GP_REQUIRE(S >= 1 && S <= 64, GP_ERR_INVALID, "lp_subrounds must be in [1, 64]");
  const int nkeys = S * kNumBuckets;
  DBuf<int4> list(ctx, (size_t)n);
  DBuf<int2> prop(ctx, (size_t)n);
  DBuf<int32_t> incoming(ctx, (size_t)nlabels);
  DBuf<int32_t> cnt(ctx, (size_t)nkeys), offs(ctx, (size_t)nkeys + 1), cursor(ctx, (size_t)nkeys);
  DBuf<int4> mov(ctx, (size_t)n);
  DBuf<uint64_t> ov_key(ctx, (size_t)n);
  DBuf<uint32_t> ov_val(ctx, (size_t)n);
  DBuf<uint8_t> ov_acc(ctx, (size_t)n);
  // few labels (refinement): bucketed overflow resolution, no sort
  const bool few = nlabels <= kOvMaxLabels;
  DBuf<unsigned long long> ovb_hw;
  DBuf<int32_t> ovb_hc, ovb_cut, ovb_m, ovb_roff, ovb_cursor, ovb_idx;
  DBuf<long long> ovb_base;
  DBuf<uint64_t> ovb_key;
  if (few) {
    ovb_hw.reset(ctx, (size_t)nlabels * kOvBuckets);
    ovb_hc.reset(ctx, (size_t)nlabels * kOvBuckets);
    ovb_cut.reset(ctx, (size_t)nlabels);
    ovb_m.reset(ctx, (size_t)nlabels);
    ovb_roff.reset(ctx, (size_t)nlabels + 1);
    ovb_cursor.reset(ctx, (size_t)nlabels);
    ovb_base.reset(ctx, (size_t)nlabels);
    ovb_key.reset(ctx, (size_t)n);
    ovb_idx.reset(ctx, (size_t)n);
  }
  DBuf<Counters> counters(ctx, 1);
  Counters *C = counters.get();
  // refinement: nodes that must be rated (all at first; a node with no label rated above its
  // own is left out until a neighbour moves: it cannot propose, so results are unchanged)
  const bool use_dirty = !p.count_clusters;
  DBuf<uint8_t> dirty;
  DBuf<int4> clist;
  DBuf<int32_t> ccount;
  if (use_dirty) {
    dirty.reset(ctx, (size_t)n);
    dirty.fill_bytes(1);
    clist.reset(ctx, (size_t)n);
    ccount.reset(ctx, (size_t)nkeys);
  }
  // the 2.5x cap (clustering): departure weight and latest key per cluster, emptying keys
  DBuf<int32_t> cap_w;
  DBuf<unsigned long long> cap_k;
  DBuf<uint64_t> cap_e;
  DBuf<int> cap_n;
  DBuf<unsigned> done(ctx, 1);
  done.zero();
  incoming.zero();
  int64_t ncl0 = 0;
  if (p.count_clusters && nclusters_dev) read_back(ctx, nclusters_dev, sizeof(int64_t), &ncl0);
  k_counters_init<<<1, 1, 0, ctx->stream>>>(C, ncl0);
  GP_LAUNCH_CHECK();
  RateTables tables;
  make_tables(ctx, g, nlabels, tables);
  unsigned long long *units_rate = ctx->profile && ctx->d_units ? ctx->d_units + p.prof_rate * PROF_UNITS : nullptr;

  TraceTimer trace(ctx);
  const int grid = ctx->num_sms * 8;
  std::vector<int32_t> hoffs((size_t)nkeys + 1);
  double sync_s = 0;  // host time blocked in the per-sub-round read of the counters (tracing)
  const auto t_host0 = std::chrono::steady_clock::now();
  const bool agg = nlabels <= 4096;  // refinement: few labels, aggregate weight updates
  bool stop = n == 0 || (p.count_clusters && ncl0 <= p.n_min);
  int32_t subs = 0;
  for (int r = 0; r < p.rounds && !stop; r++) {
    const uint64_t kact = stream_key(seed, p.tag_act, (uint32_t)p.level, (uint32_t)r);
    const uint64_t ktie = stream_key(seed, p.tag_tie, (uint32_t)p.level, (uint32_t)r);
    const uint64_t kprio = stream_key(seed, p.tag_prio, (uint32_t)p.level, (uint32_t)r);
    {
      ProfScope ps(ctx, PROF_ROUND_SETUP);
      BucketArgs b{g.xadj, label, nullptr, g.vwgt, n, kact, S, 0, 0, &C->stop, full.get()};
      cnt.zero();
      k_bucket_count<<<grid_for(n, kThreads, grid), kThreads, 0, ctx->stream>>>(b, nkeys, cnt.get());
      GP_LAUNCH_CHECK();
      k_bucket_offsets<<<1, kMaxKeys, 0, ctx->stream>>>(cnt.get(), nkeys, offs.get(), cursor.get(), &C->stop);
      GP_LAUNCH_CHECK();
      k_bucket_scatter<<<grid_for(n, kChunk, grid), kThreads, 0, ctx->stream>>>(b, nkeys, cursor.get(),
                                                                               list.get());
      GP_LAUNCH_CHECK();
    }
    // bucket sizes of the round (launch shapes, empty buckets skipped) and the stop flag
    int stop_now = 0;
    read_back(ctx, &C->stop, sizeof(int), &stop_now);
    if (stop_now) { stop = true; break; }
    read_back(ctx, offs.get(), sizeof(int32_t) * (nkeys + 1), hoffs.data());
    for (int s = 0; s < S; s++) {
      if (p.dbg_max_subrounds >= 0 && subs >= p.dbg_max_subrounds) { stop = true; break; }
      RateArgs a{};
      a.xadj = g.xadj; a.adjncy = g.adjncy; a.adjwgt = g.unit_w ? nullptr : g.adjwgt; a.vwgt = g.vwgt;
      a.label = label; a.weight = weight; a.list = list.get(); a.offs = offs.get();
      a.bound = p.bound; a.ktie = ktie; a.prop = prop.get(); a.incoming = incoming.get();
      a.stop = &C->stop; a.units = units_rate; a.label8 = label8; a.m2 = g.m2;
      a.wlabels = label8 ? (int)nlabels : 0;
      a.dirty = dirty.get();
      if (use_dirty && r > 0) {  // in round 0 every node is still marked: the lists stay as they are
        const int k0c = s * kNumBuckets;
        GP_CUDA(cudaMemsetAsync(ccount.get() + k0c, 0, sizeof(int32_t) * kNumBuckets, ctx->stream));
        const int act = hoffs[k0c + kNumBuckets] - hoffs[k0c];
        if (act > 0) {
          k_compact_dirty<<<grid_for(act, kThreads, grid), kThreads, 0, ctx->stream>>>(
              list.get(), offs.get(), k0c, k0c + kNumBuckets, dirty.get(), clist.get(), ccount.get(), &C->stop);
          GP_LAUNCH_CHECK();
        }
        a.list = clist.get();
        a.ccount = ccount.get();
      }
      {
        ProfScope ps(ctx, p.prof_rate);
        int hcnt[kNumBuckets];
        for (int b = 0; b < kNumBuckets; b++) hcnt[b] = hoffs[s * kNumBuckets + b + 1] - hoffs[s * kNumBuckets + b];
        launch_rate<RATE_LP>(ctx, a, s * kNumBuckets, tables, nlabels, hcnt);
      }
      const int k0 = s * kNumBuckets, k1 = s * kNumBuckets + kNumBuckets;
      const int active = hoffs[k1] - hoffs[k0];
      {
        ProfScope ps(ctx, p.prof_accept);
        k_decide<<<grid_for(active, kThreads, grid), kThreads, 0, ctx->stream>>>(
            use_dirty && r > 0 ? clist.get() : list.get(), offs.get(), k0, k1, prop.get(), weight, incoming.get(),
            p.bound, mov.get(), ov_key.get(), ov_val.get(), C, kprio, use_dirty && r > 0 ? ccount.get() : nullptr);
        GP_LAUNCH_CHECK();
      }
      Counters hdr;
      const auto t_sync0 = std::chrono::steady_clock::now();
      read_back(ctx, C, sizeof(hdr), &hdr);
      sync_s += std::chrono::duration<double>(std::chrono::steady_clock::now() - t_sync0).count();
      if (hdr.stop) { stop = true; break; }
      const int nov = hdr.nov, nmov = hdr.nmov;
      subs++;
      res.overflow_total += nov;
      if (nov > res.overflow_max) res.overflow_max = nov;
      res.proposals += nov + nmov;
      if (nov > 0 && few) {
        ProfScope ps(ctx, p.prof_overflow);
        const int gsmall = grid_for(nov, 256, grid);
        GP_CUDA(cudaMemsetAsync(ovb_hw.get(), 0, sizeof(unsigned long long) * ovb_hw.count, ctx->stream));
        GP_CUDA(cudaMemsetAsync(ovb_hc.get(), 0, sizeof(int32_t) * ovb_hc.count, ctx->stream));
        k_ovb_hist<<<gsmall, 256, 0, ctx->stream>>>(ov_key.get(), ov_val.get(), nov, g.vwgt, ovb_hw.get(),
                                                    ovb_hc.get());
        GP_LAUNCH_CHECK();
        k_ovb_cut<<<(int)nlabels, 256, 0, ctx->stream>>>(ovb_hw.get(), ovb_hc.get(), weight, p.bound,
                                                        ovb_cut.get(), ovb_base.get(), ovb_m.get());
        GP_LAUNCH_CHECK();
        k_ovb_offsets<<<1, 32, 0, ctx->stream>>>(ovb_m.get(), (int)nlabels, ovb_roff.get(), ovb_cursor.get());
        GP_LAUNCH_CHECK();
        k_ovb_class<<<gsmall, 256, 0, ctx->stream>>>(ov_key.get(), ov_val.get(), nov, ovb_cut.get(),
                                                     ovb_cursor.get(), ov_acc.get(), ovb_key.get(),
                                                     ovb_idx.get());
        GP_LAUNCH_CHECK();
        k_ovb_resolve<<<(int)nlabels, 256, 0, ctx->stream>>>(ovb_key.get(), ovb_idx.get(), ovb_roff.get(),
                                                            g.vwgt, weight, ovb_base.get(), p.bound,
                                                            ov_acc.get());
        GP_LAUNCH_CHECK();
      } else if (nov > 0 && nov <= kOvSmall) {
        ProfScope ps(ctx, p.prof_overflow);
        k_ov_small<<<1, kOvSmallThreads, 0, ctx->stream>>>(ov_key.get(), ov_val.get(), nov, g.vwgt, weight,
                                                           p.bound, ov_acc.get());
        GP_LAUNCH_CHECK();
      } else if (nov > 0) {
        ProfScope ps(ctx, p.prof_overflow);
        const int kbits = bits_for(nlabels) + 32;
        radix_sort_pairs(ctx, ov_key.get(), ov_val.get(), nov, kbits);
        const int gsmall = grid_for(nov, 256, grid);
        k_fix_runs<<<gsmall, 256, 0, ctx->stream>>>(ov_key.get(), ov_val.get(), nov);
        GP_LAUNCH_CHECK();
        DBuf<int64_t> cs(ctx, (size_t)nov);
        k_ov_weights<<<gsmall, 256, 0, ctx->stream>>>(ov_val.get(), nov, g.vwgt, cs.get());
        GP_LAUNCH_CHECK();
        scan_exclusive_i64(ctx, cs.get(), cs.get(), nov, nullptr);
        k_ov_accept<<<gsmall, 256, 0, ctx->stream>>>(ov_key.get(), ov_val.get(), nov, cs.get(), g.vwgt,
                                                     weight, p.bound, ov_acc.get());
        GP_LAUNCH_CHECK();
      }
      {
        ProfScope ps(ctx, p.prof_apply);
        ApplyArgs aa{};
        aa.mov = mov.get(); aa.ov_key = ov_key.get(); aa.ov_val = ov_val.get();
        aa.ov_acc = ov_acc.get(); aa.nmov = nmov; aa.nov = nov; aa.vwgt = g.vwgt; aa.label = label;
        aa.weight = weight; aa.incoming = incoming.get(); aa.label8 = label8;
        aa.nshared = agg ? (int)nlabels : 0; aa.cnt = C;
        aa.kprio = kprio;
        aa.track = p.count_clusters ? 1 : 0;

        const int ga = grid_for((int64_t)nmov + nov, kThreads, grid);
        // the 2.5x cap: only when the accepted moves could empty more than D clusters
        const int64_t D = hdr.nclusters - p.n_min;
        if (p.count_clusters && (int64_t)nmov + nov > D) {
          if (!cap_w.get()) {
            cap_w.reset(ctx, (size_t)nlabels);
            cap_k.reset(ctx, (size_t)nlabels);
            cap_w.zero();
            cap_k.zero();
            cap_e.reset(ctx, (size_t)n);
            cap_n.reset(ctx, 1);
          }
          cap_n.zero();
          k_cap_depart<<<ga, kThreads, 0, ctx->stream>>>(aa, cap_w.get(), cap_k.get());
          GP_LAUNCH_CHECK();
          k_cap_collect<<<ga, kThreads, 0, ctx->stream>>>(aa, cap_w.get(), cap_k.get(), cap_e.get(), cap_n.get());
          GP_LAUNCH_CHECK();
          k_cap_clear<<<ga, kThreads, 0, ctx->stream>>>(aa, cap_w.get(), cap_k.get());
          GP_LAUNCH_CHECK();
          const int E = read_scalar(ctx, cap_n.get());
          if (E > D) {
            DBuf<uint32_t> dummy(ctx, (size_t)E);
            radix_sort_pairs(ctx, cap_e.get(), dummy.get(), E, 64);
            aa.cutoff = cap_e.get() + D;
            res.capped++;
          }
        }
        if (nmov + nov > 0) {
          k_apply<<<ga, kThreads, sizeof(int) * aa.nshared, ctx->stream>>>(aa);
          GP_LAUNCH_CHECK();
          if (use_dirty) {
            k_mark_dirty<<<grid_for((int64_t)(nmov + nov) * 16, kThreads, grid), kThreads, 0, ctx->stream>>>(
                mov.get(), nmov, ov_key.get(), ov_val.get(), ov_acc.get(), nov, aa.cutoff, kprio, g.xadj, g.adjncy,
                dirty.get());
            GP_LAUNCH_CHECK();
          }
        }
        const int64_t count_labels = p.count_clusters ? nlabels : 0;
        const int gc = grid_for((int64_t)nmov + nov, kThreads, grid);
        k_close<<<gc, kThreads, 0, ctx->stream>>>(aa, count_labels, (long long)p.n_min, s == S - 1 ? 1 : 0,
                                                  done.get());
        GP_LAUNCH_CHECK();
      }
    }
    if (stop) break;
  }
  Counters hc;
  read_back(ctx, C, sizeof(Counters), &hc);
  res.subrounds = subs;
  res.moves = hc.moved_total;
  res.nclusters = hc.nclusters;
  if (trace.on()) {
    const double host_s = std::chrono::duration<double>(std::chrono::steady_clock::now() - t_host0).count();
    fprintf(stderr,
            "[gp lp] %s level=%d n=%d m2=%lld labels=%lld subrounds=%d moves=%lld proposals=%lld "
            "overflow_total=%lld overflow_max=%lld capped=%d host_ms=%.2f sync_ms=%.2f ms=%.2f\n",
            p.count_clusters ? "cluster" : "refine", p.level, n, (long long)g.m2, (long long)nlabels, subs,
            (long long)res.moves, (long long)res.proposals, (long long)res.overflow_total,
            (long long)res.overflow_max, res.capped, 1000 * host_s, 1000 * sync_s, trace.ms());
  }
  if (p.count_clusters && nclusters_dev)
    GP_CUDA(cudaMemcpyAsync(nclusters_dev, &C->nclusters, sizeof(int64_t), cudaMemcpyDeviceToDevice,
                            ctx->stream));
  return res;
}

// ------------------------------------------------------- 2-hop favourites

namespace {
__global__ void k_fill_u64(uint64_t *a, int64_t n, uint64_t v) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    a[i] = v;
}
}  // namespace

void favourites_bucketed(gp_ctx *ctx, const DevGraph &g, const int32_t *label, const int32_t *size,
                         int64_t U, uint64_t kfav, DBuf<uint64_t> &keys, int32_t &count) {
  const int n = g.n;
  const int nkeys = kNumBuckets;
  const int grid = ctx->num_sms * 8;
  DBuf<int4> list(ctx, (size_t)n);
  DBuf<int32_t> cnt(ctx, (size_t)nkeys), offs(ctx, (size_t)nkeys + 1),
      cursor(ctx, (size_t)nkeys);
  BucketArgs b{g.xadj, label, size, g.vwgt, n, 0, 1, 1, U, nullptr, nullptr};
  cnt.zero();
  k_bucket_count<<<grid_for(n, kThreads, grid), kThreads, 0, ctx->stream>>>(b, nkeys, cnt.get());
  GP_LAUNCH_CHECK();
  k_bucket_offsets<<<1, kMaxKeys, 0, ctx->stream>>>(cnt.get(), nkeys, offs.get(), cursor.get(), nullptr);
  GP_LAUNCH_CHECK();
  k_bucket_scatter<<<grid_for(n, kChunk, grid), kThreads, 0, ctx->stream>>>(b, nkeys, cursor.get(),
                                                                           list.get());
  GP_LAUNCH_CHECK();
  int32_t total = 0;
  read_back(ctx, offs.get() + nkeys, sizeof(int32_t), &total);
  count = total;
  keys.reset(ctx, (size_t)(total > 0 ? total : 1));
  if (total == 0) return;
  k_fill_u64<<<grid_for(total, 256, grid), 256, 0, ctx->stream>>>(keys.get(), total, ~0ull);
  GP_LAUNCH_CHECK();
  RateTables tables;
  make_tables(ctx, g, 0, tables);
  RateArgs a{};
  a.xadj = g.xadj; a.adjncy = g.adjncy; a.adjwgt = g.unit_w ? nullptr : g.adjwgt; a.vwgt = g.vwgt;
  a.label = label; a.weight = nullptr; a.list = list.get(); a.offs = offs.get();
  a.bound = U; a.ktie = kfav; a.fav_keys = keys.get(); a.stop = nullptr; a.m2 = g.m2;
  launch_rate<RATE_FAV>(ctx, a, 0, tables, 0, nullptr);
}

}  // namespace gp
