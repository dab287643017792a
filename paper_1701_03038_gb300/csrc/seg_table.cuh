// seg_table.cuh -- the size of the (symbol, state) table.
#pragma once

#include <stdint.h>

namespace fstgpu {

constexpr int64_t SEG_BUCKET_BYTES = 64, SEG_BUCKET_SLOTS = 2;

// Buckets for nseg segments with free_bytes of device memory free: three
// slots a segment (96 bytes; about 3% of the buckets spill), or, where that
// table would take more than a third of the free memory, two (64), one and a
// half (48) or at least nine eighths (36 bytes, 11% of the slots empty: the
// lookups read on more often, and FSTs of over a billion arcs still fit).
inline int64_t seg_buckets(int64_t nseg, int64_t free_bytes) {
  const int64_t most = ((int64_t)1 << 31) - 1;  // (slots are numbered in 32 bits)
  int64_t b = 0;
  for (int64_t sixteenths : {24, 16, 12, 9}) {
    b = 1 + (nseg > 0 ? nseg : 1) * sixteenths / 16;
    if (b <= most && b * SEG_BUCKET_BYTES <= free_bytes / 3) break;
  }
  return b < most ? b : most;
}

}  // namespace fstgpu
