// sort.cuh -- device-wide radix sort.
#pragma once

#include "gp_internal.cuh"

namespace gp {

// Stable LSD radix sort of n (key, value) pairs by the low `bits` key bits. The sorted pairs end in
// (keys_tmp, vals_tmp) when *result_in_tmp is true on return, else in (keys, vals).
int radix_sort_pairs(unsigned long long *keys, unsigned long long *vals, unsigned long long *keys_tmp,
                     unsigned long long *vals_tmp, int64_t n, int bits, bool *result_in_tmp, Workspace &ws);

// A pass takes the digit (key >> shift) & (2^bits - 1) of at most kSortBits bits; a tile is kSortTile consecutive
// items.
constexpr int kSortBits = 9;
constexpr int kSortThreads = 512;
constexpr int kSortItems = 8;  // items per thread
constexpr int64_t kSortTile = (int64_t)kSortThreads * kSortItems;

__host__ __device__ inline int64_t sort_tiles(int64_t n) { return (n + kSortTile - 1) / kSortTile; }
// Digits for `bits` key bits: as few passes as kSortBits allows, of equal width (narrow digits leave longer
// runs per tile).
__host__ __device__ inline int sort_passes(int bits) { return bits <= 0 ? 1 : (bits + kSortBits - 1) / kSortBits; }

}  // namespace gp
