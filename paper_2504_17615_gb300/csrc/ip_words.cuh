// ip_words.cuh -- the node words of the growing trials of the initial partition, for the per-graph path (ip.cu)
// and the batched engine (engine_dev.cuh).
#pragma once
#include "gp_internal.cuh"

namespace gp {

namespace {

constexpr int kChunkNodes = 64;        // nodes per chunk maximum
constexpr int kNarrowNodes = 1 << 15;  // 32-bit words: subproblems below this many nodes ...
constexpr int kNarrowGain = 1 << 15;   // ... and weighted degrees below this
constexpr int kScanFallbacks = 8;      // fallbacks found by a scan over all nodes before the order is made
constexpr int kBucketNodes = 4;        // nodes per hash bucket of that order at least, on average

// The node words.  Frontier nodes: (gain, -id), positive and above kOut; free nodes (not connected to
// side 1): the same with the sign bit set; kOne: in side 1; kOut: retired (can never fit again).
template <typename T> struct Word;
template <> struct Word<int32_t> {
  static constexpr int32_t kFree = INT32_MIN;
  __device__ static int32_t make(int64_t gain, int j) {
    return ((int32_t)(gain + kNarrowGain) << 15) | (kNarrowNodes - 1 - j);
  }
  __device__ static int64_t gain(int32_t x) { return x >> 15; }  // plus a constant
  __device__ static int node(int32_t x) { return kNarrowNodes - 1 - (x & (kNarrowNodes - 1)); }
  __device__ static int32_t delta(int w) { return (int32_t)((uint32_t)(2 * w) << 15); }  // connection + w
  __device__ static int32_t wmax(int32_t x) { return __reduce_max_sync(0xFFFFFFFFu, x); }
};
template <> struct Word<long long> {
  static constexpr long long kFree = INT64_MIN;
  __device__ static long long make(int64_t gain, int j) {
    return ((gain + 2147483648ll) << 31) | (2147483647 - j);
  }
  __device__ static int64_t gain(long long x) { return x >> 31; }
  __device__ static int node(long long x) { return 2147483647 - (int)(x & 2147483647ll); }
  __device__ static long long delta(int w) { return (long long)w << 32; }
  __device__ static long long wmax(long long x) {
    const int hi = (int)(x >> 32);
    const int mh = __reduce_max_sync(0xFFFFFFFFu, hi);
    const unsigned ml = __reduce_max_sync(0xFFFFFFFFu, hi == mh ? (unsigned)x : 0u);
    return ((long long)mh << 32) | ml;
  }
};
constexpr int kOne = 0, kOut = 1;
constexpr int kStep = 2;  // taken in the current step (within a step's update only)

// An array of node words: shared memory by its 32-bit address (so that every access is a shared-memory
// instruction and none a generic one), or global memory.
template <typename T, bool SM> struct Words;
template <> struct Words<int32_t, true> {
  uint32_t p;
  __device__ int32_t get(int i) const {
    int32_t x;
    asm volatile("ld.shared.s32 %0, [%1];" : "=r"(x) : "r"(p + 4 * i) : "memory");
    return x;
  }
  __device__ void set(int i, int32_t x) const { asm volatile("st.shared.s32 [%0], %1;" ::"r"(p + 4 * i), "r"(x) : "memory"); }
  __device__ int32_t add(int i, int32_t d) const {
    int32_t x;
    asm volatile("atom.shared.add.s32 %0, [%1], %2;" : "=r"(x) : "r"(p + 4 * i), "r"(d) : "memory");
    return x;
  }
  __device__ void unfree(int i) const { asm volatile("red.shared.and.b32 [%0], %1;" ::"r"(p + 4 * i), "r"(INT32_MAX) : "memory"); }
  __device__ void raise(int i, int32_t x) const { asm volatile("red.shared.max.s32 [%0], %1;" ::"r"(p + 4 * i), "r"(x) : "memory"); }
};
template <> struct Words<long long, true> {
  uint32_t p;
  __device__ long long get(int i) const {
    long long x;
    asm volatile("ld.shared.s64 %0, [%1];" : "=l"(x) : "r"(p + 8 * i) : "memory");
    return x;
  }
  __device__ void set(int i, long long x) const { asm volatile("st.shared.s64 [%0], %1;" ::"r"(p + 8 * i), "l"(x) : "memory"); }
  __device__ long long add(int i, long long d) const {
    long long x;
    asm volatile("atom.shared.add.u64 %0, [%1], %2;" : "=l"(x) : "r"(p + 8 * i), "l"(d) : "memory");
    return x;
  }
  __device__ void unfree(int i) const { asm volatile("red.shared.and.b64 [%0], %1;" ::"r"(p + 8 * i), "l"(INT64_MAX) : "memory"); }
  __device__ void raise(int i, long long x) const { asm volatile("red.shared.max.s64 [%0], %1;" ::"r"(p + 8 * i), "l"(x) : "memory"); }
};
template <typename T> struct Words<T, false> {
  T *p;
  __device__ T get(int i) const { return *(volatile T *)(p + i); }
  __device__ void set(int i, T x) const { *(volatile T *)(p + i) = x; }
  __device__ T add(int i, T d) const { return (T)atomicAdd((unsigned long long *)(p + i), (unsigned long long)d); }
  __device__ void unfree(int i) const { atomicAnd((unsigned long long *)(p + i), (unsigned long long)INT64_MAX); }
  __device__ void raise(int i, T x) const { atomicMax(p + i, x); }
};
__device__ __forceinline__ unsigned long long wmin_u64(unsigned long long x) {
  const unsigned hi = (unsigned)(x >> 32);
  const unsigned mh = __reduce_min_sync(0xFFFFFFFFu, hi);
  const unsigned ml = __reduce_min_sync(0xFFFFFFFFu, hi == mh ? (unsigned)x : 0xFFFFFFFFu);
  return ((unsigned long long)mh << 32) | ml;
}

}  // namespace

}  // namespace gp
