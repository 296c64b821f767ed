// ip.cu -- initial partitioning of the coarsest graph by recursive
// bisection (Sec. 4.3), plus the greedy rebalancer.
//
// All subproblems of one depth of the bisection tree are split together;
// every (subproblem, trial) pair runs in its own block.  A trial grows side 1
// greedily: among nodes that still fit under L1, frontier nodes (connected
// to side 1) of largest gain 2 conn(v) - deg'(v), ties by the smallest id;
// when no frontier node fits, the node of smallest (h32(key(IP, 0, bid), v,
// t), v).  It stops once side 1 weighs >= T1.  The trial with the smallest
// cut (ties: lowest trial) wins.
//
// Each growing step takes up to B = 1 + n'/1024 frontier nodes in order of
// their gains at the start of the step, skipping those that no longer fit
// (one node per step below 1024 nodes).
//
// A trial is one chain of a few hundred dependent steps, so the kernel is
// bound by the latency of a step and built to shorten it:
//  * a node is ONE word: its state, gain and id packed so that a signed
//    maximum over words is the choice (gain first, then the smallest id).
//    32 bits hold it when the weighted degrees stay below 2^15 and the
//    subproblem below 2^15 nodes; a maximum over the warp is then one
//    instruction.  Otherwise words have 64 bits.
//  * every 64-node chunk keeps the largest word of its frontier nodes, raised
//    by an atomic maximum when a neighbour's connection grows and recomputed
//    for the chunk of a node just taken; each lane keeps the maximum over its
//    chunks in a register.
//  * rows are copied to shared memory where they fit (below the first depths
//    only a subproblem's internal edges are left); the row bounds of a taken
//    node are fetched while the next one is being chosen.
//  * steps of up to kSoloB nodes run in one warp without block barriers;
//  * steps of kBatchB nodes or more select them together: a histogram of the
//    chunk maxima's gains gives the gain of the B-th largest maximum, the nodes
//    of at least that gain in the (at most B) chunks that can hold the step's
//    nodes are ranked by counting, and one warp walks them in order.  One pick
//    after another is a chain of some 460 cycles each.
// A picked node that no longer fits is retired for good (side 1 only gets
// heavier), which leaves the choice among the nodes that fit unchanged.
// The fallback scans all nodes the first few times; after that, the nodes
// still free are put in the order of the top bits of their hash (a counting
// sort) and a cursor walks them, 32 at a time (a node that left the free state
// or stopped fitting never comes back).
//
// Measured (20,480 nodes, 204,800 edges, k = 128, 8 trials; the whole initial partition): 17.0 ms with 64-bit
// keys in separate arrays, block barriers in every step and a sort of the chunk maxima; 9.0 ms with the
// words, one pick after another everywhere; 7.8 ms with the steps of kBatchB nodes selected together.
#include "ip_words.cuh"

#include <algorithm>

namespace gp {

namespace {

constexpr int kUpdUnroll = 4;
constexpr int kSmemBatch = 64;  // the nodes of a growing step live in shared memory up to this many
constexpr int kIpWarps = 8;     // warps per (subproblem, trial)
constexpr int kSoloB = 4;       // steps of up to this many nodes run in one warp
constexpr int kBatchB = 8;      // steps of at least this many select them together
constexpr int kBins = 512;      // gains below the largest one that the selection tells apart
constexpr int kCands = 256;     // nodes ranked per selection; more: picked one by one
constexpr int kStaticSmem = 8192;      // room for the kernel's static shared variables
constexpr int kSmSmem = 228 * 1024;    // shared memory of an SM; every resident block reserves another 1 KiB
constexpr int kMaxSmemBytes = 227 * 1024 - kStaticSmem;

template <int V> struct IntC { static constexpr int value = V; };

struct Sub {
  int32_t start, count;  // node list range
  int32_t bid;           // heap id of the bisection
  int32_t pad;
  int64_t T1, L1;        // side-1 target and limit
};

__device__ __forceinline__ uint32_t lds_u32(uint32_t p) {
  uint32_t x;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(x) : "r"(p) : "memory");
  return x;
}
__device__ __forceinline__ int lds_u16(uint32_t p) {
  uint16_t x;
  asm volatile("ld.shared.u16 %0, [%1];" : "=h"(x) : "r"(p) : "memory");
  return (int)x;
}

struct IpArgs {
  const int32_t *lxadj;            // local CSR of every subproblem (by list position)
  const int2 *ladj;                // (local index, weight) of internal neighbours
  const int32_t *vtx, *cvl, *dpl;  // by list position: node id, weight, deg'
  const Sub *subs;
  int trials;
  int n;
  uint64_t seed;
  int smem_bytes;                  // dynamic shared memory of a block
  int cv16;                        // node weights fit 16 bits: kept in shared memory
  void *gx, *gbest, *gsup;         // [trial][n] words when a subproblem's do not fit in shared memory, ...
  int32_t *gbatch;                 // per block: the nodes taken in the current step
  int batch_cap;
  int64_t bstride, sstride;        // their chunk maxima and maxima over 32 chunks, per trial
  uint2 *ford;                     // [trial][n] fallback order (words in shared memory only): (hash, node)
  int32_t *fcur;                   // and its buckets' places, hstride per trial
  int64_t hstride;
  unsigned long long *trace;       // optional: [0] growing steps, [1] fallbacks, [2] retired nodes
  int64_t *trial_cut;              // per block
  uint8_t *flags;                  // [trial][n] side-1 flag by list position
};

// A 4-byte copy from global to shared memory that the issuing lane does not wait for.
__device__ __forceinline__ void copy_async4(int *dst, const int32_t *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void copy_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// One block of kIpWarps warps per (subproblem, trial).  SM: the words live in shared memory (at most
// 512 chunks: 16 per lane); otherwise in global memory, with one more level of maxima.
template <typename KT, bool SM>
__global__ void __launch_bounds__(32 * kIpWarps) k_ip_grow(IpArgs a) {
  using W = Word<KT>;
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ int s_nb, s_fj;
  __shared__ long long s_w1;
  __shared__ unsigned long long s_red[kIpWarps];
  __shared__ int32_t s_batch[kSmemBatch];
  __shared__ int s_rs[kSmemBatch], s_re[kSmemBatch];
  __shared__ int s_hist[kBins], s_wsum[2][kIpWarps], s_list[kSmemBatch], s_nlist, s_ncand, s_bin, s_need;
  __shared__ KT s_wmax[kIpWarps], s_cand[kCands], s_rank[kCands], s_tau;
  const int lane = (int)lane_id(), warp = threadIdx.x >> 5;
  const int si = blockIdx.x / a.trials, t = blockIdx.x % a.trials;
  const Sub S = a.subs[si];
  const int cnt = S.count, nch = (cnt + kChunkNodes - 1) / kChunkNodes;
  const int nsup = (nch + 31) / 32;
  const int start = S.start;
  const int64_t tpos = (int64_t)t * a.n + start;  // this trial's place in the [trial][n] arrays
  Words<KT, SM> X, best;
  KT *sup = nullptr;
  uint32_t cv = 0, lx = 0, sadj = 0;  // shared addresses (0: not there) of the node weights (16 bits each), of the
                                      // row bounds from the subproblem's first entry, and of the rows
                                      // (weight << 16 | neighbour)
  const int base = a.lxadj[start];
  if constexpr (SM) {
    const uint32_t dyn0 = (uint32_t)__cvta_generic_to_shared(dyn);
    X.p = dyn0;
    best.p = dyn0 + (uint32_t)sizeof(KT) * cnt;
    int64_t at = (int64_t)sizeof(KT) * (cnt + nch);
    if (a.cv16) {
      uint16_t *c16 = reinterpret_cast<uint16_t *>(dyn + at);
      for (int j = threadIdx.x; j < cnt; j += blockDim.x) c16[j] = (uint16_t)a.cvl[start + j];
      cv = dyn0 + (uint32_t)at;
      at += (2 * (int64_t)cnt + 3) & ~(int64_t)3;
    }
    if (at + 4 * ((int64_t)cnt + 1) <= a.smem_bytes) {
      int32_t *l32 = reinterpret_cast<int32_t *>(dyn + at);
      for (int j = threadIdx.x; j <= cnt; j += blockDim.x) l32[j] = a.lxadj[start + j] - base;
      lx = dyn0 + (uint32_t)at;
      at += 4 * ((int64_t)cnt + 1);
      const int E = a.lxadj[start + cnt] - base;
      if (sizeof(KT) == 4 && at + 4 * (int64_t)E <= a.smem_bytes) {
        uint32_t *ad = reinterpret_cast<uint32_t *>(dyn + at);
        for (int e = threadIdx.x; e < E; e += blockDim.x) {
          const int2 x = a.ladj[base + e];
          ad[e] = ((uint32_t)x.y << 16) | (uint32_t)x.x;
        }
        sadj = dyn0 + (uint32_t)at;
      }
    }
  } else {
    X.p = reinterpret_cast<KT *>(a.gx) + tpos;
    best.p = reinterpret_cast<KT *>(a.gbest) + t * a.bstride + start / kChunkNodes + si;
    sup = reinterpret_cast<KT *>(a.gsup) + t * a.sstride + start / (32 * kChunkNodes) + si;
  }
  const uint64_t kip = stream_key(a.seed, TAG_IP, 0, (uint32_t)S.bid);
  for (int j = threadIdx.x; j < cnt; j += blockDim.x) X.set(j, W::make(-(int64_t)a.dpl[start + j], j) | W::kFree);
  for (int c = threadIdx.x; c < nch; c += blockDim.x) best.set(c, 0);
  if (!SM)
    for (int c = threadIdx.x; c < nsup; c += blockDim.x) sup[c] = 0;
  __syncthreads();

  auto weight = [&](int j) -> int { return cv ? lds_u16(cv + 2 * j) : a.cvl[start + j]; };
  auto entry = [&](int e) -> int2 {  // e counts from the subproblem's first entry
    if (sadj) {
      const uint32_t x = lds_u32(sadj + 4 * e);
      return make_int2((int)(x & 0xFFFFu), (int)(x >> 16));
    }
    return a.ladj[base + e];
  };
  auto row_begin = [&](int j) -> int { return lx ? (int)lds_u32(lx + 4 * j) : a.lxadj[start + j] - base; };
  // largest frontier word of chunk c without node skip (one warp), 0 if none
  auto chunk_max = [&](int c, int skip) -> KT {
    const int j0 = c * kChunkNodes + lane, j1 = j0 + 32;
    KT x0 = j0 < cnt && j0 != skip ? X.get(j0) : 0, x1 = j1 < cnt && j1 != skip ? X.get(j1) : 0;
    x0 = x0 > x1 ? x0 : x1;
    x0 = W::wmax(x0);
    return x0 > kOut ? x0 : 0;
  };
  int nfall = 0, cursor = 0;           // warp 0: fallbacks so far, place in the order
  int bits = 0;                        // buckets: the hash's top bits, at most cnt / kBucketNodes of them
  while ((kBucketNodes << (bits + 1)) <= cnt) bits++;
  const int nbk = 1 << bits;
  int32_t *const place = a.fcur + (int64_t)t * a.hstride + start / kBucketNodes + si;
  uint2 *const order = a.ford + tpos;
  __shared__ int s_free;               // nodes in the order
  auto hash_of = [&](int j) -> uint32_t { return h32(kip, (uint32_t)a.vtx[start + j], (uint32_t)t); };
  // one thread's share of a scan for the free node of smallest (hash, id) that fits
  auto scan_free = [&](int tid, int step, int64_t w1) -> unsigned long long {
    unsigned long long m = ~0ull;
    for (int j = tid; j < cnt; j += step) {
      if (X.get(j) >= 0 || w1 + weight(j) > S.L1) continue;
      const unsigned long long key = ((unsigned long long)hash_of(j) << 32) | (unsigned)j;
      m = key < m ? key : m;
    }
    return m;
  };
  auto bucket_of = [&](uint32_t h) -> int { return (int)((uint64_t)h >> (32 - bits)); };
  // the order of the nodes still free, by one warp or the block (sync: its barrier); warp 0 scans the counts
  auto make_order = [&](int tid, int step, auto sync) {
    for (int b = tid; b < nbk; b += step) place[b] = 0;
    sync();
    for (int j = tid; j < cnt; j += step)
      if (X.get(j) < 0) atomicAdd(&place[bucket_of(hash_of(j))], 1);
    sync();
    if (warp == 0) {
      int run = 0;
      for (int b0 = 0; b0 < nbk; b0 += 32) {
        const int c = b0 + lane < nbk ? *(volatile int32_t *)&place[b0 + lane] : 0;
        int y = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int z = __shfl_up_sync(0xFFFFFFFFu, y, o);
          if (lane >= o) y += z;
        }
        if (b0 + lane < nbk) place[b0 + lane] = run + y - c;
        run += __shfl_sync(0xFFFFFFFFu, y, 31);
      }
      if (lane == 0) s_free = run;
    }
    sync();
    for (int j = tid; j < cnt; j += step) {
      if (X.get(j) >= 0) continue;
      const uint32_t h = hash_of(j);
      order[atomicAdd(&place[bucket_of(h)], 1)] = make_uint2(h, (unsigned)j);
    }
    sync();
  };
  // warp 0: the free node of smallest (hash, id) that fits, from the order; -1 if none.  The first valid
  // node's bucket holds the answer; it may go on past the 32 nodes looked at.
  auto walk_free = [&](int64_t w1) -> int {
    const int total = s_free;
    int bucket = -1;
    unsigned long long best = ~0ull;
    for (int p = cursor; p < total; p += 32) {
      const bool in = p + lane < total;
      const uint2 x = in ? order[p + lane] : make_uint2(0, 0);
      const bool ok = in && X.get((int)x.y) < 0 && w1 + weight((int)x.y) <= S.L1;
      const unsigned m = __ballot_sync(0xFFFFFFFFu, ok);
      if (bucket < 0) {
        if (m == 0) { cursor = p + 32; continue; }
        const int f = __ffs(m) - 1;
        cursor = p + f;
        bucket = bucket_of(__shfl_sync(0xFFFFFFFFu, x.x, f));
      }
      const bool same = in && bucket_of(x.x) == bucket;
      const unsigned long long key = ok && same ? ((unsigned long long)x.x << 32) | x.y : ~0ull;
      const unsigned long long k = wmin_u64(key);
      best = k < best ? k : best;
      if (!__shfl_sync(0xFFFFFFFFu, same, 31)) break;  // the bucket ends within these nodes
    }
    return best == ~0ull ? -1 : (int)(unsigned)best;
  };

  int64_t w1 = 0;
  const int B = 1 + cnt / 1024;  // nodes per growing step
  unsigned long long steps = 0, retired = 0;
  // warp 0: the frontier node next in (gain desc, id asc) order is taken (its id comes back and w1 grows)
  // or, when it no longer fits, retired (-2); -1: no frontier node left.  r: the maxima of the lane's
  // chunks lane, lane + 32, ... (N of them), kept in step with best.
  auto pick = [&](auto &r, auto count) -> int {
    constexpr int N = decltype(count)::value;
    KT m = 0;
    if constexpr (SM) {
#pragma unroll
      for (int i = 0; i < N; i++) m = r[i] > m ? r[i] : m;
    } else {
      for (int c = lane; c < nsup; c += 32) { const KT x = sup[c]; m = x > m ? x : m; }
    }
    m = W::wmax(m);
    if (m <= kOut) return -1;
    const int j = W::node(m), c = j / kChunkNodes;
    const int cj = weight(j);
    const KT nm = chunk_max(c, j);
    const bool fit = w1 + cj <= S.L1;
    if (lane == 0) {
      X.set(j, fit ? kOne : kOut);
      best.set(c, nm);
    }
    __syncwarp();
    if constexpr (SM) {
#pragma unroll
      for (int i = 0; i < N; i++) r[i] = c == lane + 32 * i ? nm : r[i];
    } else {
      const int s0 = (c / 32) * 32;
      KT x = s0 + lane < nch ? best.get(s0 + lane) : 0;
      x = W::wmax(x);
      if (lane == 0) sup[c / 32] = x;
      __syncwarp();
    }
    if (!fit) {
      retired++;
      return -2;
    }
    w1 += cj;
    return j;
  };
  auto load_maxima = [&](auto &r, auto count) {
    if constexpr (SM) {
#pragma unroll
      for (int i = 0; i < decltype(count)::value; i++) r[i] = lane + 32 * i < nch ? best.get(lane + 32 * i) : 0;
    }
  };
  // one warp finds the fallback node; -1: none fits
  auto fallback = [&]() -> int {
    int j;
    if (nfall < kScanFallbacks) {
      const unsigned long long m = wmin_u64(scan_free(lane, 32, w1));
      j = m == ~0ull ? -1 : (int)(unsigned)m;
    } else {
      if (nfall == kScanFallbacks) make_order(lane, 32, [] { __syncwarp(); });
      j = walk_free(w1);
    }
    nfall++;
    return j;
  };

  if (SM && B <= kSoloB) {
    if (warp == 0) {
      constexpr int kN = kSoloB * 1024 / kChunkNodes / 32;  // cnt < kSoloB * 1024
      constexpr IntC<kN> N{};
      KT r[kN];
      while (w1 < S.T1) {
        load_maxima(r, N);
        steps++;
        int nb = 0, rs[kSoloB], re[kSoloB];
        int2 first[kSoloB];  // the first 32 entries of the taken nodes' rows, fetched while others are chosen
#pragma unroll
        for (int q = 0; q < kSoloB; q++) {
          rs[q] = re[q] = 0;
          first[q] = make_int2(-1, 0);
          if (q != nb || q >= B || w1 >= S.T1) continue;
          int j;
          do { j = pick(r, N); } while (j == -2);
          if (j == -1 && q == 0) {  // no frontier node fits
            j = fallback();
            if (j >= 0) {
              w1 += weight(j);
              if (lane == 0) X.set(j, kOne);
              __syncwarp();
              nb = kSoloB;  // the step's only node
            }
          }
          if (j < 0) continue;
          nb++;
          rs[q] = row_begin(j);
          re[q] = row_begin(j + 1);
          if (rs[q] + lane < re[q]) first[q] = entry(rs[q] + lane);
        }
        if (nb == 0) break;
        // neighbours of the step's nodes, row by row (a row has no neighbour twice: no atomic adds)
#pragma unroll
        for (int q = 0; q < kSoloB; q++) {
          if (rs[q] >= re[q]) continue;
          int2 y = first[q];
          for (int f = rs[q];;) {
            if (y.x >= 0) {
              KT x = X.get(y.x);
              if (x < 0 || x > kOut) {
                x = (x & ~W::kFree) + W::delta(y.y);
                X.set(y.x, x);
                best.raise(y.x / kChunkNodes, x);
              }
            }
            f += 32;
            if (f >= re[q]) break;
            y = f + lane < re[q] ? entry(f + lane) : make_int2(-1, 0);
          }
          __syncwarp();
        }
      }
    }
  } else {
    const bool rows_async = SM && !lx && B <= kSmemBatch;
    int32_t *batch = B <= kSmemBatch ? s_batch : a.gbatch + (int64_t)blockIdx.x * a.batch_cap;
    const bool batched = SM && B >= kBatchB && B <= kSmemBatch;
    // One selection of up to `want` nodes by the whole block, appended to batch from nb0 on; returns 0 when no
    // frontier node is left, -1 when they must be picked one by one (gains too far apart, or too many
    // equal ones), else 1; s_nb and s_w1 are the new number and weight (warp 0 keeps w1).
    auto select = [&](int nb0) -> int {
      if constexpr (!SM) {
        return -1;
      } else {
        const int want = B - nb0;
        constexpr int PER = 512 / (32 * kIpWarps);  // chunks per thread
        static_assert(PER >= 1 && PER <= 2, "two chunk maxima a thread at most");
        KT x[PER], mx = 0;
#pragma unroll
        for (int i = 0; i < PER; i++) {
          const int c = (int)threadIdx.x + i * 32 * kIpWarps;
          x[i] = c < nch ? best.get(c) : 0;
          mx = x[i] > mx ? x[i] : mx;
        }
        mx = W::wmax(mx);
        if (lane == 0) s_wmax[warp] = mx;
        for (int t2 = threadIdx.x; t2 < kBins; t2 += blockDim.x) s_hist[t2] = 0;
        if (threadIdx.x == 0) { s_nlist = 0; s_ncand = 0; s_bin = -1; }
        __syncthreads();
        mx = s_wmax[0];
#pragma unroll
        for (int w = 1; w < kIpWarps; w++) mx = s_wmax[w] > mx ? s_wmax[w] : mx;
        if (mx <= kOut) return 0;
        const int64_t top = W::gain(mx);
        int bin[PER];
#pragma unroll
        for (int i = 0; i < PER; i++) {
          const int64_t d = top - W::gain(x[i]);
          bin[i] = x[i] > kOut && d < kBins ? (int)d : kBins;
          if (bin[i] < kBins) atomicAdd(&s_hist[bin[i]], 1);
        }
        const int present = __syncthreads_count(x[0] > kOut) + (PER > 1 ? __syncthreads_count(x[PER - 1] > kOut) : 0);
        const int q = want < present ? want : present;  // chunks that can hold the step's nodes
        // the bin of the q-th largest maximum, and how many of its maxima belong to the q
        if (warp == 0) {
          constexpr int PB = kBins / 32;
          int loc = 0;
#pragma unroll
          for (int i = 0; i < PB; i++) loc += s_hist[lane * PB + i];
          int incl = loc;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (lane >= o) incl += y;
          }
          int run = incl - loc;
          if (run < q && q <= incl) {
#pragma unroll
            for (int i = 0; i < PB; i++) {
              const int h = s_hist[lane * PB + i];
              if (run < q && q <= run + h) { s_bin = lane * PB + i; s_need = q - run; }
              run += h;
            }
          }
        }
        __syncthreads();
        const int cutbin = s_bin, need = s_need;
        if (cutbin < 0) return -1;  // the gains lie further apart than the bins
        // the q largest maxima: those above the cut bin, and the first `need` of it in id order (of equal gains
        // the smaller id goes first).  The smallest of them, tau, is reached by at least q nodes, and all
        // nodes that reach it lie in those q chunks
#pragma unroll
        for (int i = 0; i < PER; i++) {
          const unsigned m = __ballot_sync(0xFFFFFFFFu, bin[i] == cutbin);
          if (lane == 0) s_wsum[i][warp] = __popc(m);
        }
        __syncthreads();
        int before = 0;
#pragma unroll
        for (int i = 0; i < PER; i++) {
          int at = before;
#pragma unroll
          for (int w = 0; w < kIpWarps; w++) {
            const int v = s_wsum[i][w];
            at += w < warp ? v : 0;
            before += v;
          }
          const unsigned m = __ballot_sync(0xFFFFFFFFu, bin[i] == cutbin);
          at += __popc(m & lanemask_lt());
          if (bin[i] < cutbin || (bin[i] == cutbin && at < need))
            s_list[atomicAdd(&s_nlist, 1)] = (int)threadIdx.x + i * 32 * kIpWarps;
          if (bin[i] == cutbin && at == need - 1) s_tau = x[i];
        }
        __syncthreads();
        const KT tau = s_tau;
        const int nl = s_nlist;  // q chunks
        for (int l = warp; l < nl; l += kIpWarps) {
          const int j0 = s_list[l] * kChunkNodes + lane, j1 = j0 + 32;
          const KT a0 = j0 < cnt ? X.get(j0) : 0, a1 = j1 < cnt ? X.get(j1) : 0;
          const bool in0 = a0 >= tau, in1 = a1 >= tau;  // tau > kOut
          const unsigned m0 = __ballot_sync(0xFFFFFFFFu, in0), m1 = __ballot_sync(0xFFFFFFFFu, in1);
          int at = 0;
          if (lane == 0) at = atomicAdd(&s_ncand, __popc(m0) + __popc(m1));
          at = __shfl_sync(0xFFFFFFFFu, at, 0);
          const int p0 = at + __popc(m0 & lanemask_lt()), p1 = at + __popc(m0) + __popc(m1 & lanemask_lt());
          if (in0 && p0 < kCands) s_cand[p0] = a0;
          if (in1 && p1 < kCands) s_cand[p1] = a1;
        }
        __syncthreads();
        const int C = s_ncand;
        if (C > kCands) return -1;
        for (int t2 = threadIdx.x; t2 < C; t2 += blockDim.x) {  // words are distinct: rank = place
          const KT mine = s_cand[t2];
          int r = 0;
#pragma unroll 4
          for (int u = 0; u < C; u++) r += s_cand[u] > mine ? 1 : 0;
          s_rank[r] = mine;
        }
        __syncthreads();
        if (warp == 0) {
          int nb = nb0, i0 = 0;
          while (i0 < C) {
            const int i = i0 + lane;
            const int j = i < C ? W::node(s_rank[i]) : -1;
            const long long c = i < C ? weight(j) : 0;
            long long pre = c;  // weight of lanes 0 .. lane
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
              const long long y = __shfl_up_sync(0xFFFFFFFFu, pre, o);
              if (lane >= o) pre += y;
            }
            // a lane is reached iff every earlier one was taken
            const bool considered = i < C && nb + lane < B && w1 + (pre - c) < S.T1;
            const bool fits = w1 + pre <= S.L1;
            const unsigned bad = __ballot_sync(0xFFFFFFFFu, !(considered && fits));
            const int f = bad ? __ffs(bad) - 1 : 32;
            if (lane < f) {
              X.set(j, kOne);
              batch[nb + lane] = j;
              if (rows_async) {  // the row's bounds come while the chunks are looked over again
                copy_async4(&s_rs[nb + lane], a.lxadj + start + j);
                copy_async4(&s_re[nb + lane], a.lxadj + start + j + 1);
              }
            }
            const long long wf = __shfl_sync(0xFFFFFFFFu, pre, f > 0 ? f - 1 : 0);
            const bool cf = __shfl_sync(0xFFFFFFFFu, considered, f < 32 ? f : 0);
            if (f > 0) w1 += wf;
            nb += f;
            if (f == 32) { i0 += 32; continue; }
            if (i0 + f >= C || !cf) break;  // list used up, or the step is complete
            if (lane == f) X.set(j, kOut);  // reached and does not fit: retired
            retired++;
            i0 += f + 1;
          }
          if (lane == 0) { s_nb = nb; s_w1 = w1; }
        }
        __syncthreads();
        for (int l = warp; l < nl; l += kIpWarps) {  // the listed chunks' maxima again
          const int c = s_list[l];
          const KT nm = chunk_max(c, -1);
          if (lane == 0) best.set(c, nm);
        }
        if (rows_async && warp == 0) copy_async_wait();
        __syncthreads();
        return 1;
      }
    };
    for (;;) {
      int got = 0;     // batched: nodes selected so far
      bool one_by_one = !batched;
      if (batched) {
        if (threadIdx.x == 0) { s_w1 = w1; s_nb = 0; }
        __syncthreads();
        if (s_w1 >= S.T1) break;
        if (warp == 0) steps++;
        while (got < B && s_w1 < S.T1) {
          const int r = select(got);
          if (r <= 0) { one_by_one = r < 0; break; }
          got = s_nb;
        }
      }
      if (one_by_one) {
      if (warp == 0) {
        int nb = -2;  // done
        if (w1 < S.T1) {
          nb = got;
          if (!batched) steps++;
          constexpr int kN = SM ? 16 : 1;
          constexpr IntC<kN> N{};
          KT r[kN];
          load_maxima(r, N);
          while (nb < B && w1 < S.T1) {
            const int j = pick(r, N);
            if (j == -1) break;
            if (j < 0) continue;
            if (lane == 0) {
              batch[nb] = j;
              if (rows_async) {  // the row's bounds come while the next node is chosen
                copy_async4(&s_rs[nb], a.lxadj + start + j);
                copy_async4(&s_re[nb], a.lxadj + start + j + 1);
              }
            }
            nb++;
          }
          if (rows_async) copy_async_wait();
        }
        if (lane == 0) { s_nb = nb; s_w1 = w1; }
      }
      __syncthreads();
      }
      int nb = s_nb;
      if (nb == -2) break;
      bool fell = false;
      if (nb == 0) {  // no frontier node fits
        fell = true;
        w1 = s_w1;
        if (!SM || nfall < kScanFallbacks) {
          const unsigned long long m = wmin_u64(scan_free(threadIdx.x, blockDim.x, w1));
          if (lane == 0) s_red[warp] = m;
          __syncthreads();
          if (threadIdx.x == 0) {
            unsigned long long mm = s_red[0];
            for (int q = 1; q < kIpWarps; q++) mm = s_red[q] < mm ? s_red[q] : mm;
            s_fj = mm == ~0ull ? -1 : (int)(unsigned)mm;
          }
        } else {
          if (nfall == kScanFallbacks) make_order(threadIdx.x, blockDim.x, [] { __syncthreads(); });
          if (warp == 0) {
            const int j = walk_free(w1);
            if (lane == 0) s_fj = j;
          }
        }
        nfall++;
        __syncthreads();
        const int j = s_fj;
        if (j < 0) break;
        w1 += weight(j);  // warp 0's copy goes on from here
        if (threadIdx.x == 0) { X.set(j, kOne); batch[0] = j; }
        nb = 1;
        __syncthreads();
      }
      // neighbours of the step's nodes, over their concatenated local rows (32 nodes at a time),
      // 32 * kUpdUnroll entries per warp and pass
      for (int b0 = 0; b0 < nb; b0 += 32) {
        int r0 = 0, d = 0;
        if (b0 + lane < nb) {
          if (rows_async && !fell) {
            r0 = s_rs[b0 + lane] - base;
            d = s_re[b0 + lane] - base - r0;
          } else {
            const int j = batch[b0 + lane];
            r0 = row_begin(j);
            d = row_begin(j + 1) - r0;
          }
        }
        int incl = d;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
          if (lane >= o) incl += y;
        }
        const int excl = incl - d, total = __shfl_sync(0xFFFFFFFFu, incl, 31);
        for (int f0 = warp * 32 * kUpdUnroll; f0 < total; f0 += kIpWarps * 32 * kUpdUnroll) {
          int idx[kUpdUnroll];
#pragma unroll
          for (int r = 0; r < kUpdUnroll; r++) {
            const int f = f0 + r * 32 + lane;
            int q = 0;
#pragma unroll
            for (int step = 16; step > 0; step >>= 1) {
              const int val = __shfl_sync(0xFFFFFFFFu, incl, q + step - 1);
              if (val <= f) q += step;
            }
            const int sq = __shfl_sync(0xFFFFFFFFu, r0, q), eq = __shfl_sync(0xFFFFFFFFu, excl, q);
            idx[r] = f < total ? sq + (f - eq) : -1;
          }
          int2 e[kUpdUnroll];
#pragma unroll
          for (int r = 0; r < kUpdUnroll; r++) e[r] = idx[r] >= 0 ? entry(idx[r]) : make_int2(-1, 0);
#pragma unroll
          for (int r = 0; r < kUpdUnroll; r++) {
            if (e[r].x < 0) continue;
            const KT x = X.get(e[r].x);
            if (x < 0 || x > kOut) {
              if (x < 0) X.unfree(e[r].x);
              const KT dl = W::delta(e[r].y);
              best.raise(e[r].x / kChunkNodes, X.add(e[r].x, dl) + dl);
            }
          }
        }
      }
      __syncthreads();
      if (!SM) {  // the maxima over 32 chunks again, from the raised chunk maxima (one warp per group)
        for (int sc = warp; sc < nsup; sc += kIpWarps) {
          const int c = sc * 32 + lane;
          const KT x = W::wmax(c < nch ? best.get(c) : 0);
          if (lane == 0) sup[sc] = x;
        }
        __syncthreads();
      }
    }
  }
  __syncthreads();
  if (a.trace && threadIdx.x == 0) {
    atomicAdd(a.trace + 0, steps);
    atomicAdd(a.trace + 1, (unsigned long long)nfall);
    atomicAdd(a.trace + 2, retired);
  }
  // cut of this trial inside the subproblem
  unsigned long long cut = 0;
  for (int j = threadIdx.x; j < cnt; j += blockDim.x) {
    if (X.get(j) != kOne) continue;
    const int e1 = row_begin(j + 1);
    for (int e = row_begin(j); e < e1; e++) {
      const int2 x = entry(e);
      if (X.get(x.x) != kOne) cut += (unsigned long long)x.y;
    }
  }
  cut = warp_sum(cut);
  if (lane == 0) s_red[warp] = cut;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long c = 0;
    for (int q = 0; q < kIpWarps; q++) c += s_red[q];
    a.trial_cut[blockIdx.x] = (int64_t)c;
  }
  uint8_t *fl = a.flags + tpos;
  for (int j = threadIdx.x; j < cnt; j += blockDim.x) fl[j] = X.get(j) == kOne;
}

// Totals of the graph: node weight, heaviest node, largest weighted degree; and the list of depth 0.
struct IpTotals {
  unsigned long long W;
  int cmax;
  int pad;
  unsigned long long dmax;
};

__global__ void k_ip_init(const int32_t *xadj, const int32_t *vwgt, const int32_t *adjwgt, int n, int32_t *vtx,
                          int32_t *cvl, int32_t *sub, int2 *splo, IpTotals *o) {
  const int lane = (int)lane_id();
  const int wid = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nw = (gridDim.x * blockDim.x) >> 5;
  unsigned long long w = 0, dm = 0;
  int cm = 0;
  for (int v = wid; v < n; v += nw) {
    unsigned long long d = 0;
    const int e1 = xadj[v + 1];
    for (int e = xadj[v] + lane; e < e1; e += 32) d += (unsigned)adjwgt[e];
    d = warp_sum(d);
    dm = d > dm ? d : dm;
    if (lane == 0) {
      const int c = vwgt[v];
      w += (unsigned long long)c;
      cm = c > cm ? c : cm;
      vtx[v] = v;
      cvl[v] = c;
      sub[v] = 0;
      splo[v] = make_int2(0, v);
    }
  }
  if (lane == 0) {
    if (w) atomicAdd(&o->W, w);
    if (cm) atomicMax(&o->cmax, cm);
    if (dm) atomicMax(&o->dmax, dm);
  }
}

// deg'(v) (weight to nodes of the same subproblem) and the number of such
// neighbours, one warp per listed node
__global__ void k_sub_dp(const int32_t *xadj, const int32_t *adjncy, const int32_t *adjwgt, const int32_t *vtx,
                         const int32_t *sub, const int2 *splo, int live, int32_t *dpl, int32_t *lcnt) {
  const int lane = (int)lane_id();
  const int wid = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nw = (gridDim.x * blockDim.x) >> 5;
  if (wid == 0 && lane == 0) lcnt[live] = 0;
  for (int p = wid; p < live; p += nw) {
    const int v = vtx[p];
    const int s = sub[p];
    int sum = 0, c = 0;
    const int e1 = xadj[v + 1];
    for (int e = xadj[v] + lane; e < e1; e += 32)
      if (splo[adjncy[e]].x == s) { sum += adjwgt[e]; c++; }
    sum = warp_sum(sum);
    c = warp_sum(c);
    if (lane == 0) { dpl[p] = sum; lcnt[p] = c; }
  }
}

// local rows: (local index, weight) of the internal neighbours of every listed node
__global__ void k_sub_rows(const int32_t *xadj, const int32_t *adjncy, const int32_t *adjwgt, const int32_t *vtx,
                           const int32_t *sub, const int2 *splo, int live, const int32_t *lxadj, int2 *ladj) {
  const int lane = (int)lane_id();
  const int wid = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nw = (gridDim.x * blockDim.x) >> 5;
  for (int p = wid; p < live; p += nw) {
    const int v = vtx[p];
    const int s = sub[p];
    int pos = lxadj[p];
    const int e1 = xadj[v + 1];
    for (int e0 = xadj[v]; e0 < e1; e0 += 32) {
      const int e = e0 + lane;
      int2 sl = make_int2(-1, 0);
      if (e < e1) sl = splo[adjncy[e]];
      const bool in = sl.x == s;
      const unsigned m = __ballot_sync(0xFFFFFFFFu, in);
      if (in) ladj[pos + __popc(m & lanemask_lt())] = make_int2(sl.y, adjwgt[e]);
      pos += __popc(m);
    }
  }
}

// Every subproblem's best trial (smallest cut, then lowest trial): the side of every listed node, and the
// number and weight of its side-1 nodes.  One block per subproblem.
struct Side1 {
  long long count, weight;
};

__global__ void __launch_bounds__(256) k_ip_side(const int64_t *trial_cut, const Sub *subs, int trials, int n,
                                                 const uint8_t *flags, const int32_t *cvl, int32_t *side,
                                                 Side1 *out) {
  __shared__ long long s_c[8], s_w[8];
  const int s = blockIdx.x;
  int bt = 0;
  for (int t = 1; t < trials; t++)
    if (trial_cut[s * trials + t] < trial_cut[s * trials + bt]) bt = t;
  const Sub S = subs[s];
  long long c = 0, w = 0;
  for (int j = threadIdx.x; j < S.count; j += blockDim.x) {
    const int f = flags[(int64_t)bt * n + S.start + j];
    side[S.start + j] = f;
    c += f;
    w += f ? cvl[S.start + j] : 0;
  }
  c = warp_sum(c);
  w = warp_sum(w);
  if (lane_id() == 0) { s_c[threadIdx.x >> 5] = c; s_w[threadIdx.x >> 5] = w; }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int q = 1; q < 8; q++) { c += s_c[q]; w += s_w[q]; }
    out[s].count = c;
    out[s].weight = w;
  }
}

// The next depth's lists, in the same order within each child (so lists stay sorted by id): child[2 s] is
// side 1, child[2 s + 1] side 0; .x = the child's subproblem index, or -(1 + block) when it is final,
// .y = its list start.  rank = number of side-1 nodes at smaller positions.
__global__ void k_ip_split(int live, const int32_t *vtx, const int32_t *cvl, const int32_t *sub, const int32_t *side,
                           const int32_t *rank, const Sub *subs, const int2 *child, int32_t *vtx2, int32_t *cvl2,
                           int32_t *sub2, int2 *splo, int32_t *blocks) {
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < live; p += gridDim.x * blockDim.x) {
    const int v = vtx[p], s = sub[p], st = subs[s].start;
    const int r1 = rank[p] - rank[st];
    const int2 c = child[2 * s + (side[p] ? 0 : 1)];
    if (c.x < 0) {
      blocks[v] = -(c.x + 1);
      splo[v] = make_int2(-1, 0);
      continue;
    }
    const int r = side[p] ? r1 : p - st - r1;
    vtx2[c.y + r] = v;
    cvl2[c.y + r] = cvl[p];
    sub2[c.y + r] = c.x;
    splo[v] = make_int2(c.x, r);
  }
}

int32_t ceil_log2(int64_t k) {
  int32_t b = 0;
  while (((int64_t)1 << b) < k) b++;
  return b;
}

struct HostSub {
  int32_t kk, b0, bid, count;
  int64_t W;
};

template <typename KT, bool SM>
void launch_grow(gp_ctx *ctx, const IpArgs &a, int nblocks, size_t smem) {
  if (SM)
    GP_CUDA(cudaFuncSetAttribute(k_ip_grow<KT, SM>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmemBytes));
  k_ip_grow<KT, SM><<<nblocks, 32 * kIpWarps, smem, ctx->stream>>>(a);
  GP_LAUNCH_CHECK();
}

}  // namespace

void initial_partition(gp_ctx *ctx, const DevGraph &g, int32_t k, int64_t eps_ppm, uint64_t seed,
                       int32_t trials, int32_t *blocks) {
  ProfScope ps(ctx, PROF_IP);
  const int n = g.n;
  GP_REQUIRE(trials >= 1, GP_ERR_INVALID, "ip_trials must be >= 1");
  GP_CUDA(cudaMemsetAsync(blocks, 0, sizeof(int32_t) * (n > 0 ? n : 1), ctx->stream));
  if (k <= 1 || n == 0) return;
  const int grid = grid_for(n, 256, ctx->num_sms * 8);
  const int wgrid = grid_for((int64_t)n * 32, 256, ctx->num_sms * 8);
  // two sets of lists: this depth's and the next one's
  DBuf<int32_t> lists(ctx, (size_t)6 * n), dpl(ctx, (size_t)n), lxadj(ctx, (size_t)n + 1), side(ctx, (size_t)n),
      rank(ctx, (size_t)n);
  int32_t *vtx = lists.get(), *cvl = vtx + n, *sub = cvl + n, *vtx2 = sub + n, *cvl2 = vtx2 + n, *sub2 = cvl2 + n;
  DBuf<int2> ladj(ctx, (size_t)(g.m2 > 0 ? g.m2 : 1));
  DBuf<int2> splo(ctx, (size_t)n);
  DBuf<IpTotals> tot(ctx, 1);
  tot.zero();
  k_ip_init<<<wgrid, 256, 0, ctx->stream>>>(g.xadj, g.vwgt, g.adjwgt, n, vtx, cvl, sub, splo.get(), tot.get());
  GP_LAUNCH_CHECK();
  IpTotals ht;
  read_back(ctx, tot.get(), sizeof(ht), &ht);
  const int64_t eps_l = eps_ppm / ceil_log2(k);
  std::vector<HostSub> subs{{k, 0, 1, n, (int64_t)ht.W}};
  DBuf<uint8_t> flags(ctx, (size_t)trials * n);
  DBuf<uint2> ford;
  DBuf<int32_t> fcur;
  // per depth, at most k subproblems: their records, trial cuts, side totals, children
  DBuf<Sub> dsub(ctx, (size_t)k);
  DBuf<int64_t> tcut(ctx, (size_t)k * trials);
  DBuf<Side1> dside(ctx, (size_t)k);
  DBuf<int2> dchild(ctx, (size_t)2 * k);
  std::vector<Sub> hsub;
  std::vector<Side1> hside;
  std::vector<int2> hchild;
  int live = n;
  const bool trace = getenv("GP_TRACE") != nullptr;
  while (!subs.empty()) {
    const int ns = (int)subs.size();
    hsub.resize((size_t)ns);
    int maxcnt = 0, pos = 0;
    for (int i = 0; i < ns; i++) {
      const int64_t kk = subs[i].kk, k1 = (kk + 1) / 2;
      Sub &s = hsub[(size_t)i];
      s.start = pos;
      s.count = subs[i].count;
      s.bid = subs[i].bid;
      s.pad = 0;
      s.T1 = (subs[i].W * k1 + kk - 1) / kk;
      s.L1 = (int64_t)(((__int128)s.T1 * (1000000 + eps_l)) / 1000000);
      pos += s.count;
      maxcnt = std::max(maxcnt, s.count);
    }
    GP_CUDA(cudaMemcpyAsync(dsub.get(), hsub.data(), sizeof(Sub) * ns, cudaMemcpyHostToDevice, ctx->stream));
    if (live > 0) {
      k_sub_dp<<<grid_for((int64_t)live * 32, 256, ctx->num_sms * 8), 256, 0, ctx->stream>>>(
          g.xadj, g.adjncy, g.adjwgt, vtx, sub, splo.get(), live, dpl.get(), lxadj.get());
      GP_LAUNCH_CHECK();
      scan_exclusive_i32(ctx, lxadj.get(), lxadj.get(), live + 1, nullptr);
      k_sub_rows<<<grid_for((int64_t)live * 32, 256, ctx->num_sms * 8), 256, 0, ctx->stream>>>(
          g.xadj, g.adjncy, g.adjwgt, vtx, sub, splo.get(), live, lxadj.get(), ladj.get());
      GP_LAUNCH_CHECK();
    } else {
      lxadj.zero();
    }
    const int nblocks = ns * trials;
    IpArgs a{};
    a.lxadj = lxadj.get(); a.ladj = ladj.get();
    a.vtx = vtx; a.cvl = cvl; a.dpl = dpl.get();
    a.subs = dsub.get(); a.trials = trials; a.n = n; a.seed = seed;
    a.cv16 = ht.cmax <= 65535 ? 1 : 0;
    a.trial_cut = tcut.get();
    a.flags = flags.get();
    // 32-bit words: |gain| is at most the weighted degree
    const bool narrow = maxcnt < kNarrowNodes && ht.dmax < (unsigned long long)kNarrowGain;
    const int64_t wb = narrow ? 4 : 8;
    const int64_t nch = (maxcnt + kChunkNodes - 1) / kChunkNodes;
    const int64_t need = wb * (maxcnt + nch) + (a.cv16 ? 2 * (int64_t)maxcnt + 4 : 0);
    const bool sm = need <= kMaxSmemBytes && nch <= 512;
    // what the blocks that share an SM leave of its shared memory goes to row bounds and rows
    const int per_sm = std::min(8, (nblocks + ctx->num_sms - 1) / ctx->num_sms);
    const int64_t share = std::min<int64_t>(kMaxSmemBytes, kSmSmem / per_sm - 1024 - kStaticSmem);
    const int64_t smem = sm ? std::max<int64_t>(need, share) : 0;
    a.smem_bytes = (int)smem;
    DBuf<long long> gx, gbest, gsup;
    if (!sm) {
      a.bstride = n / kChunkNodes + ns + 1;
      a.sstride = n / (32 * kChunkNodes) + ns + 1;
      gx.reset(ctx, (size_t)trials * n);
      gbest.reset(ctx, (size_t)trials * a.bstride);
      gsup.reset(ctx, (size_t)trials * a.sstride);
      a.gx = gx.get(); a.gbest = gbest.get(); a.gsup = gsup.get();
    }
    if (sm) {
      a.hstride = n / kBucketNodes + k + 1;
      if (!ford.get()) {
        ford.reset(ctx, (size_t)trials * n);
        fcur.reset(ctx, (size_t)(trials * a.hstride));
      }
      a.ford = ford.get();
      a.fcur = fcur.get();
    }
    a.batch_cap = 1 + maxcnt / 1024;
    DBuf<int32_t> gbatch;
    if (a.batch_cap > kSmemBatch) gbatch.reset(ctx, (size_t)nblocks * a.batch_cap);
    a.gbatch = gbatch.get();
    DBuf<unsigned long long> tr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (trace) {
      tr.reset(ctx, 3);
      tr.zero();
      a.trace = tr.get();
      GP_CUDA(cudaEventCreate(&e0));
      GP_CUDA(cudaEventCreate(&e1));
      GP_CUDA(cudaEventRecord(e0, ctx->stream));
    }
    if (narrow && sm) launch_grow<int32_t, true>(ctx, a, nblocks, (size_t)smem);
    else if (sm) launch_grow<long long, true>(ctx, a, nblocks, (size_t)smem);
    else launch_grow<long long, false>(ctx, a, nblocks, 0);
    if (trace) {
      GP_CUDA(cudaEventRecord(e1, ctx->stream));
      unsigned long long h[3];
      read_back(ctx, tr.get(), sizeof(h), h);
      float ms = 0;
      GP_CUDA(cudaEventElapsedTime(&ms, e0, e1));
      fprintf(stderr,
              "[gp ip] subproblems=%d max_nodes=%d word=%d shared=%lld grow_ms=%.2f steps=%llu fallbacks=%llu "
              "retired=%llu\n",
              ns, maxcnt, narrow && sm ? 32 : 64, (long long)smem, ms, h[0], h[1], h[2]);
      cudaEventDestroy(e0);
      cudaEventDestroy(e1);
    }
    k_ip_side<<<ns, 256, 0, ctx->stream>>>(tcut.get(), dsub.get(), trials, n, flags.get(), cvl, side.get(),
                                           dside.get());
    GP_LAUNCH_CHECK();
    if (live > 0) scan_exclusive_i32(ctx, side.get(), rank.get(), live, nullptr);
    hside.resize((size_t)ns);
    read_back(ctx, dside.get(), sizeof(Side1) * ns, hside.data());
    // children of every subproblem (final when they hold a single block)
    hchild.resize((size_t)2 * ns);
    std::vector<HostSub> next;
    int next_live = 0;
    for (int i = 0; i < ns; i++) {
      const int32_t kk = subs[i].kk, k1 = (kk + 1) / 2, k2 = kk - k1;
      const Side1 &o = hside[(size_t)i];
      const HostSub cs[2] = {{k1, subs[i].b0, 2 * subs[i].bid, (int32_t)o.count, o.weight},
                             {k2, subs[i].b0 + k1, 2 * subs[i].bid + 1, subs[i].count - (int32_t)o.count,
                              subs[i].W - o.weight}};
      for (int q = 0; q < 2; q++) {
        if (cs[q].kk <= 1) {
          hchild[(size_t)(2 * i + q)] = make_int2(-(cs[q].b0 + 1), 0);
        } else {
          hchild[(size_t)(2 * i + q)] = make_int2((int)next.size(), next_live);
          next.push_back(cs[q]);
          next_live += cs[q].count;
        }
      }
    }
    if (live > 0) {
      GP_CUDA(cudaMemcpyAsync(dchild.get(), hchild.data(), sizeof(int2) * 2 * ns, cudaMemcpyHostToDevice,
                              ctx->stream));
      k_ip_split<<<grid, 256, 0, ctx->stream>>>(live, vtx, cvl, sub, side.get(), rank.get(), dsub.get(),
                                                dchild.get(), vtx2, cvl2, sub2, splo.get(), blocks);
      GP_LAUNCH_CHECK();
      std::swap(vtx, vtx2);
      std::swap(cvl, cvl2);
      std::swap(sub, sub2);
    }
    live = next_live;
    GP_CUDA(cudaStreamSynchronize(ctx->stream));  // the host vectors must outlive the copies
    subs.swap(next);
  }
}

// --------------------------------------------------------------- rebalance

namespace {

constexpr int kRbThreads = 1024;

__global__ void __launch_bounds__(kRbThreads) k_rebalance(const int32_t *xadj, const int32_t *adjncy,
                                                          const int32_t *adjwgt, const int32_t *vwgt,
                                                          int n, int k, int64_t Lmax, int32_t *blk,
                                                          int64_t *bw, long long *moves_out) {
  __shared__ int64_t s_d[32];
  __shared__ int s_v[32];
  __shared__ int s_A, s_B, s_best;
  long long moves = 0;
  for (int64_t it = 0; it <= (int64_t)n; it++) {
    if (threadIdx.x == 0) {
      int A = 0, B = 0;
      for (int b = 1; b < k; b++) {
        if (bw[b] > bw[A]) A = b;
        if (bw[b] < bw[B]) B = b;
      }
      s_A = A;
      s_B = B;
    }
    __syncthreads();
    const int A = s_A, B = s_B;
    if (bw[A] <= Lmax || A == B) break;
    int64_t bd = 0;
    int bv = -1;
    for (int v = threadIdx.x; v < n; v += blockDim.x) {
      if (blk[v] != A || bw[B] + vwgt[v] > Lmax) continue;
      int64_t ca = 0, cb = 0;
      for (int e = xadj[v]; e < xadj[v + 1]; e++) {
        const int b = blk[adjncy[e]];
        if (b == A) ca += adjwgt[e];
        else if (b == B) cb += adjwgt[e];
      }
      const int64_t d = ca - cb;
      if (bv < 0 || d < bd || (d == bd && v < bv)) { bd = d; bv = v; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const int64_t d2 = __shfl_xor_sync(0xFFFFFFFFu, bd, o);
      const int v2 = __shfl_xor_sync(0xFFFFFFFFu, bv, o);
      if (v2 >= 0 && (bv < 0 || d2 < bd || (d2 == bd && v2 < bv))) { bd = d2; bv = v2; }
    }
    if (lane_id() == 0) { s_d[threadIdx.x >> 5] = bd; s_v[threadIdx.x >> 5] = bv; }
    __syncthreads();
    if (threadIdx.x == 0) {
      int64_t d = s_d[0];
      int v = s_v[0];
      for (int i = 1; i < kRbThreads / 32; i++)
        if (s_v[i] >= 0 && (v < 0 || s_d[i] < d || (s_d[i] == d && s_v[i] < v))) { d = s_d[i]; v = s_v[i]; }
      s_best = v;
      if (v >= 0) {
        blk[v] = B;
        bw[A] -= vwgt[v];
        bw[B] += vwgt[v];
        moves++;
      }
    }
    __syncthreads();
    if (s_best < 0) break;
  }
  if (threadIdx.x == 0) *moves_out = moves;
}

__global__ void k_block_weights(const int32_t *blk, const int32_t *vwgt, int n, long long *bw) {
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x)
    atomicAdd((unsigned long long *)&bw[blk[v]], (unsigned long long)vwgt[v]);
}

}  // namespace

int64_t rebalance_blocks(gp_ctx *ctx, const DevGraph &g, int32_t k, int64_t Lmax, int32_t *blocks) {
  ProfScope ps(ctx, PROF_REBALANCE);
  if (g.n == 0 || k <= 1) return 0;
  DBuf<long long> bw(ctx, (size_t)k), moves(ctx, 1);
  bw.zero();
  moves.zero();
  k_block_weights<<<grid_for(g.n, 256, ctx->num_sms * 8), 256, 0, ctx->stream>>>(blocks, g.vwgt, g.n, bw.get());
  GP_LAUNCH_CHECK();
  k_rebalance<<<1, kRbThreads, 0, ctx->stream>>>(g.xadj, g.adjncy, g.adjwgt, g.vwgt, g.n, k, Lmax, blocks,
                                                 reinterpret_cast<int64_t *>(bw.get()), moves.get());
  GP_LAUNCH_CHECK();
  return read_scalar(ctx, moves.get());
}

}  // namespace gp
