// Ranges of the pool that holds the whitening components' matrix entries (k_solve.cu).
// The pool of an N-observation catalog has up to 4 N entries and more, beyond 2^31
// for N above 2^29, so its cursor and a slice's first entry count grains of four
// entries, and positions inside a slice are relative to its first entry.
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define SPIDER_HD __host__ __device__
#else
#define SPIDER_HD
#endif

namespace spider {

constexpr int kPoolGrain = 4;

// The layout of a slice of 32 rows with `rest` entries in `steps` steps (a multiple
// of four): every row padded to `steps`, unless that would more than double the
// entries; positions stay below 2^30 padded and below rest otherwise.
SPIDER_HD constexpr bool pool_padded(int steps, int rest) {
  return rest < (1 << 29) && 32 * (int64_t)steps <= 2 * (int64_t)rest;
}

// grains that a slice takes
SPIDER_HD constexpr int32_t pool_grains(int steps, int rest) {
  return pool_padded(steps, rest) ? 32 / kPoolGrain * steps : rest / kPoolGrain + (rest % kPoolGrain != 0);
}

// first entry of a slice; the complement marks one that is not padded
SPIDER_HD constexpr int64_t pool_first(int32_t gb) { return (int64_t)kPoolGrain * (gb >= 0 ? gb : ~gb); }

// Entries of the largest step: two per observation, at most as many again for
// padding or for the last grain.  Only a slice of a single entry takes more than
// twice what it holds (four for one); every row has an entry, so it is the last of
// a component of more than 32 of the P rows, and there is one such slice a component.
SPIDER_HD constexpr int64_t pool_entries(int64_t N, int64_t P) { return 4 * N + P / 16 / kPoolGrain * kPoolGrain + 64; }

}  // namespace spider

#undef SPIDER_HD
