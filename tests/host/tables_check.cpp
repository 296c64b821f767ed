// Table sizes on the CPU, up to the largest counts an int holds.
#include <stdint.h>
#include <stdio.h>

#include <initializer_list>

#define __device__
#define __host__
#define __forceinline__ inline
#include "tables.cuh"

int main() {
  int bad = 0;
  const int64_t M = 0x7FFFFFFF;
  const int64_t at[] = {0, 1, 16, 17, 128, 2048, 2049, 18432, 1 << 28, (1 << 29) - 1, 1 << 29, (1 << 29) + 1,
                        805306368, (1 << 30) - 1, 1 << 30, (1 << 30) + 1, M - 0x10000, M - 1, M};
  for (int64_t k : at) {
    for (int least : {1, 5}) {
      const int b = gp::table_bits((int)k, least);
      const int64_t slots = (int64_t)1 << b;
      if (b < least || b > 31 || slots <= k) bad |= 1;             // never fills
      if (k <= 1 << 30 && slots < 2 * k) bad |= 2;                 // two slots a key where they exist
      if (b > least && slots / 2 >= 2 * k) bad |= 4;               // and no more than needed
    }
    for (int q4 = 5; q4 <= 12; q4++) {
      const int64_t s = gp::tab_slots((int)k, q4), want = k * q4 / 4 + 1;
      if (s != want && (want <= M - 0x10000 || s < 0x7FFF0000)) bad |= 8;
      if (k < 0x7FFF0000 && s <= k) bad |= 16;
      if (s + 8192 > M) bad |= 32;                                 // a place and a few thousand fit an int
    }
    for (int step : {2048, 4096}) {
      const int64_t c = gp::chunks_of((int)k, step);
      if (c * step < k || (c - 1) * step >= k + (k == 0)) bad |= 64;
    }
  }
  for (int64_t bytes : {(int64_t)0, (int64_t)24000000, 8 * M})
    for (int b : {13, 30, 31}) {
      const int n = gp::table_blocks(bytes, (int64_t)1 << b, 608);
      if (n < 1 || n > 608 || (n > 1 && ((int64_t)n << b) * 8 > bytes)) bad |= 128;
    }
  printf("bad=%d\n", bad);
  return bad != 0;
}
