// modularity.cu -- the modularity of a clustering and Lemma 2's bound
// (Sec. 5): the weight inside clusters, the total weight, and the cluster
// volumes (sums of weighted degrees), from which Q_C = sum_i (e_ii - a_i^2)
// and alpha_C = max_i a_i follow.
#include "gp_internal.cuh"

namespace gp {

namespace {

constexpr unsigned FULL = 0xFFFFFFFFu;

struct ModOut {
  unsigned long long w_internal, w_total, vol_max, vol_sq;
  int bad;  // a label outside [0, nlabels)
};

__device__ __forceinline__ bool in_range(int L, int nl) { return L >= 0 && L < nl; }

// The weight of entries whose endpoints share a label, the total weight, and every row's weight added
// to its node's cluster volume.  Rows and entries are split evenly over the warps (EntryWalk), kModUnroll
// per lane in flight.  Row weights are summed in shared memory (32 bits hold them: the validation
// bounds the total edge weight by 2^31 - 1); with at most kModShared clusters (nsh > 0) the volumes are
// summed per block too, the rows of one cluster in a window added up first: direct adds to a few dozen
// global words were served one after another and took nine tenths of the time (8.4M nodes, 134M
// entries, 64 clusters: 2.2 ms).
constexpr int kModUnroll = 4;
constexpr int kModShared = 2048;

__global__ void __launch_bounds__(256, 6) k_mod_rows(const int32_t *xadj, const int32_t *adjncy,
                                                  const int32_t *adjwgt, const int32_t *label, int n, int nl, int nsh,
                                                  unsigned long long *vol, ModOut *o) {
  __shared__ unsigned s_deg[8][32];
  extern __shared__ unsigned long long s_vol[];
  const int lane = (int)lane_id(), wib = threadIdx.x >> 5;
  const int wid = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int nw = (int)((gridDim.x * blockDim.x) >> 5);
  for (int t = threadIdx.x; t < nsh; t += blockDim.x) s_vol[t] = 0;
  __syncthreads();
  unsigned long long win = 0, wtot = 0;
  int bad = 0;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
    if (!in_range(label[v], nl)) bad = 1;
  for (EntryWalk wk(xadj, n, wid, nw); wk.next();) {
    const int64_t u = wk.u0 + lane;
    const int Lu = u < n ? label[u] : -1;
    const int e1 = wk.e1;
    s_deg[wib][lane] = 0;
    __syncwarp();
    walk_entries<kModUnroll>(wk.e0, e1, [&](auto steps, int f0) {
      constexpr int R = decltype(steps)::value;
      int q[R], Lq[R], w[R], v[R];
#pragma unroll
      for (int r = 0; r < R; r++) {
        q[r] = wk.owner(f0 + r * 32);
        Lq[r] = __shfl_sync(FULL, Lu, q[r]);
      }
#pragma unroll
      for (int r = 0; r < R; r++) {
        const int e = f0 + r * 32 + lane;
        v[r] = e < e1 ? __ldcs(adjncy + e) : -1;
        w[r] = e < e1 ? __ldcs(adjwgt + e) : 0;
      }
#pragma unroll
      for (int r = 0; r < R; r++) {
        if (v[r] < 0) continue;
        const int Lv = label[v[r]];
        if (!in_range(Lv, nl)) bad = 1;
        wtot += (unsigned long long)w[r];
        if (Lv == Lq[r]) win += (unsigned long long)w[r];
        atomicAdd(&s_deg[wib][q[r]], (unsigned)w[r]);
      }
    });
    __syncwarp();
    const unsigned d = s_deg[wib][lane];
    if (nsh > 0) {
      const bool on = d != 0 && in_range(Lu, nl);
      const unsigned act = __ballot_sync(FULL, on);
      if (on) {
        const unsigned peers = __match_any_sync(act, Lu);
        // 32 rows of at most 2^31 - 1 each: the halves are summed apart
        const unsigned lo = __reduce_add_sync(peers, d & 0xFFFFu), hi = __reduce_add_sync(peers, d >> 16);
        if (lane == __ffs(peers) - 1) atomicAdd(&s_vol[Lu], ((unsigned long long)hi << 16) + lo);
      }
    } else if (d != 0 && in_range(Lu, nl)) {
      atomicAdd(&vol[Lu], (unsigned long long)d);
    }
    __syncwarp();
  }
  win = warp_sum(win);
  wtot = warp_sum(wtot);
  bad = __reduce_or_sync(FULL, bad);
  if (lane == 0) {
    if (win) atomicAdd(&o->w_internal, win);
    if (wtot) atomicAdd(&o->w_total, wtot);
    if (bad) atomicOr(&o->bad, 1);
  }
  __syncthreads();
  for (int t = threadIdx.x; t < nsh; t += blockDim.x)
    if (s_vol[t]) atomicAdd(&vol[t], s_vol[t]);
}

__global__ void __launch_bounds__(256) k_mod_volumes(const unsigned long long *vol, int nl, ModOut *o) {
  unsigned long long mx = 0, sq = 0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nl; i += gridDim.x * blockDim.x) {
    const unsigned long long x = vol[i];
    mx = x > mx ? x : mx;
    sq += x * x;
  }
  mx = warp_max(mx);
  sq = warp_sum(sq);
  if (lane_id() == 0) {
    if (mx) atomicMax(&o->vol_max, mx);
    if (sq) atomicAdd(&o->vol_sq, sq);
  }
}

}  // namespace

void modularity(gp_ctx *ctx, const DevGraph &g, const int32_t *labels, int32_t nlabels, gp_modularity_stats *out) {
  GP_REQUIRE(nlabels >= 1, GP_ERR_INVALID, "nlabels must be >= 1");
  GP_REQUIRE(g.n == 0 || labels, GP_ERR_INVALID, "null labels");
  DBuf<unsigned long long> vol(ctx, (size_t)nlabels);
  DBuf<ModOut> o(ctx, 1);
  vol.zero();
  o.zero();
  if (g.n > 0) {
    // per-block volumes pay when a block has several rows a cluster; small graphs add directly
    const int grid = walk_grid(g.n, g.m2, ctx->num_sms, 6);
    const int nsh = nlabels <= kModShared && g.n / grid >= 2 * nlabels ? nlabels : 0;
    k_mod_rows<<<grid, 256, sizeof(unsigned long long) * nsh, ctx->stream>>>(
        g.xadj, g.adjncy, g.adjwgt, labels, g.n, nlabels, nsh, vol.get(), o.get());
    GP_LAUNCH_CHECK();
  }
  k_mod_volumes<<<grid_for(nlabels, 256, ctx->num_sms * 8), 256, 0, ctx->stream>>>(vol.get(), nlabels, o.get());
  GP_LAUNCH_CHECK();
  ModOut h;
  read_back(ctx, o.get(), sizeof(ModOut), &h);
  GP_REQUIRE(!h.bad, GP_ERR_INVALID, "a label lies outside [0, nlabels)");
  out->w_internal = (int64_t)h.w_internal;
  out->w_total = (int64_t)h.w_total;
  out->vol_max = (int64_t)h.vol_max;
  out->vol_sq = h.vol_sq;
  const double W = (double)h.w_total;
  out->inside = W > 0 ? (double)h.w_internal / W : 0.0;
  out->q = W > 0 ? out->inside - (double)h.vol_sq / (W * W) : 0.0;
  out->alpha = W > 0 ? (double)h.vol_max / W : 0.0;
  out->bound = 1.0 - out->q - out->alpha;
}

}  // namespace gp
