// tables.cuh -- sizes of the hash tables that label propagation and contraction build, for up to 2^31 - 1 keys
// (a row, or a segment of a contraction, may hold every entry of a graph).
#pragma once
#include <stdint.h>

namespace gp {

// Bits (at least `least`, at most 31) of a power-of-two table of at least two slots per key; beyond 2^30 keys
// of more slots than keys.
__host__ __device__ __forceinline__ int table_bits(int keys, int least) {
  int bits = least;
  while (bits < 31 && ((int64_t)1 << bits) < 2 * (int64_t)keys) bits++;
  return bits;
}

// Slots of a table for `keys` keys, q4 quarters of a slot each: more than the keys (q4 > 4), so that no table
// fills, and little enough that a place in it plus a few thousand still fits an int.
__host__ __device__ __forceinline__ int tab_slots(int keys, int q4) {
  const int64_t s = (int64_t)keys * q4 / 4 + 1;
  return s > 0x7FFF0000 ? 0x7FFF0000 : (int)s;
}

// Steps of `step` entries that cover `count` of them.
__host__ __device__ __forceinline__ int chunks_of(int count, int step) {
  return (int)(((int64_t)count + step - 1) / step);
}

// Blocks that get a private global hash table of `slots` int pairs, at most
// `want`: the tables together stay within `bytes` (8 per CSR entry plus 16 MiB,
// Limits), so scratch memory grows with the graph, not with its largest degree.
inline int table_blocks(int64_t bytes, int64_t slots, int want) {
  int64_t b = bytes / (slots * 8);
  if (b > want) b = want;
  return b < 1 ? 1 : (int)b;
}

}  // namespace gp
