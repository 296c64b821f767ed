// engine_tail.cu -- the small end of one graph's hierarchy in one CTA: every level from a few thousand
// nodes down to the coarsest in one launch, and the refinement back up in another.  On the per-level path
// such a level costs about sixty launches, ten host reads and grid-wide barriers, 0.4 to 1 ms whatever its
// size; the batched engine's level code runs it with block barriers alone (a whole 1600-node mesh
// partition 2.45 -> 1.60 ms, ER of 65,536 nodes 10.4 -> 7.9 ms).
#include "engine_dev.cuh"

namespace gp {
namespace eng {

namespace {

constexpr int kTailThreads = 1024;

// What the way up takes from the arena; both ways reserve it, so that a hierarchy is accepted on the way
// down only if the way up will fit.
struct UpScratch {
  int32_t *ba, *bb, *bw;
  ELpScr lp;
};

__device__ void up_scratch(ECtx &c, const TailArgs &a, int levels, UpScratch &u) {
  int nmax = 1, dmax = 0;
  for (int i = 0; i <= levels; i++) {
    if (i > 0 && a.lv[i].g.n > nmax) nmax = a.lv[i].g.n;
    const int d = e_maxdeg(c, a.lv[i].g);
    dmax = d > dmax ? d : dmax;
  }
  u.ba = c.ar.s<int32_t>(nmax);
  u.bb = c.ar.s<int32_t>(nmax);
  u.bw = c.ar.s<int32_t>(a.k);
  lp_scratch(c, a.in.n, a.k, dmax, u.lp);
}

__global__ void __launch_bounds__(kTailThreads) k_tail_down(TailArgs a) {
  extern __shared__ __align__(16) unsigned char esm[];
  __shared__ ESmem s;
  ECtx c;
  e_context(c, esm, s, a.cfg, false);
  c.ar.base = a.arena;
  c.ar.lo = 0;
  c.ar.hi = a.arena_bytes;
  c.ar.fail = false;
  if (threadIdx.x == 0) {
    a.lv[0].g = a.in;
    a.lv[0].cmap = nullptr;
  }
  __syncthreads();
  int L = 0;
  bool ok = e_coarsen(c, a.U, a.k, a.seed, a.level0, a.max_levels, a.lv, a.out->st, L);
  if (ok) {
    UpScratch u;
    up_scratch(c, a, L, u);
    ok = !c.ar.fail;
  }
  if (threadIdx.x == 0) {
    a.out->status = ok ? (int)GP_OK : kERetry;
    a.out->levels = L;
    a.out->coarsest = a.lv[L].g;
    a.out->arena_lo = c.ar.lo;
  }
}

__global__ void __launch_bounds__(kTailThreads) k_tail_up(TailArgs a) {
  extern __shared__ __align__(16) unsigned char esm[];
  __shared__ ESmem s;
  ECtx c;
  e_context(c, esm, s, a.cfg, false);
  c.ar.base = a.arena;
  c.ar.lo = a.out->arena_lo;
  c.ar.hi = a.arena_bytes;
  c.ar.fail = false;
  const int L = a.out->levels;
  UpScratch u;
  up_scratch(c, a, L, u);  // fits: the way down has checked it
  lp_scratch_clear(u.lp);
  __syncthreads();
  int32_t *blk = a.blk;
  e_refine(c, a.lv[L].g, a.k, a.Lmax, a.level0 + L + 1, a.seed, blk, u.bw, u.lp);
  for (int i = L - 1; i >= 0; i--) {
    int32_t *fine = i == 0 ? a.dst : (blk == u.ba ? u.bb : u.ba);
    const int32_t *cm = a.lv[i].cmap;
    for (int v = threadIdx.x; v < a.lv[i].g.n; v += blockDim.x) fine[v] = blk[cm[v]];
    __syncthreads();
    e_refine(c, a.lv[i].g, a.k, a.Lmax, a.level0 + i + 1, a.seed, fine, u.bw, u.lp);
    blk = fine;
  }
  if (L == 0)
    for (int v = threadIdx.x; v < a.in.n; v += blockDim.x) a.dst[v] = blk[v];
}

}  // namespace

void launch_tail_down(cudaStream_t stream, const TailArgs &a) {
  const size_t smem = smem_bytes(kTailThreads);
  GP_CUDA(cudaFuncSetAttribute(k_tail_down, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  k_tail_down<<<1, kTailThreads, smem, stream>>>(a);
  GP_LAUNCH_CHECK();
}

void launch_tail_up(cudaStream_t stream, const TailArgs &a) {
  const size_t smem = smem_bytes(kTailThreads);
  GP_CUDA(cudaFuncSetAttribute(k_tail_up, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  k_tail_up<<<1, kTailThreads, smem, stream>>>(a);
  GP_LAUNCH_CHECK();
}

}  // namespace eng
}  // namespace gp
