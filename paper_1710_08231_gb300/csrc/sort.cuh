// sort.cuh -- device-wide radix sort.
#pragma once

#include "gp_internal.cuh"

namespace gp {

// Stable LSD radix sort of n (key, value) pairs by the low `bits` key bits. The sorted pairs end in
// (keys_tmp, vals_tmp) when *result_in_tmp is true on return, else in (keys, vals).
int radix_sort_pairs(unsigned long long *keys, unsigned long long *vals, unsigned long long *keys_tmp,
                     unsigned long long *vals_tmp, int64_t n, int bits, bool *result_in_tmp, Workspace &ws);

// The parts of the sort, for callers that count the first digit while they write the keys.
//
// A tile is kSortTile consecutive items. One pass over digit (key >> shift) & (2^bits - 1), bits <= kSortBits:
// counts hist[digit * ntiles + tile] (radix_hist, or the caller's kernel), radix_offsets (counts to first
// positions, in place; the item count to hist[ntiles << bits]), radix_scatter.
constexpr int kSortBits = 9;
constexpr int kSortThreads = 512;
constexpr int kSortItems = 8;  // items per thread
constexpr int64_t kSortTile = (int64_t)kSortThreads * kSortItems;
constexpr unsigned long long kSortDropped = ~0ull;  // key of an item that a scatter with `drop` leaves out

inline int64_t sort_tiles(int64_t n) { return (n + kSortTile - 1) / kSortTile; }
// Digits for `bits` key bits: as few passes as kSortBits allows, of equal width (narrow digits leave longer
// runs per tile).
inline int sort_passes(int bits) { return bits <= 0 ? 1 : (bits + kSortBits - 1) / kSortBits; }

// n_max bounds the item count; n_dev (device, may be NULL) holds it when the host does not know it.
// val_bytes: 0 (no values), 4 or 8.
int radix_hist(const unsigned long long *keys, const int64_t *n_dev, int64_t n_max, int shift, int bits, int64_t *hist,
               cudaStream_t s);
int radix_offsets(int64_t *hist, int64_t n_max, int bits, Workspace &ws);
int radix_scatter(const unsigned long long *kin, const void *vin, unsigned long long *kout, void *vout, int val_bytes,
                  const int64_t *n_dev, int64_t n_max, int shift, int bits, const int64_t *offs, bool drop,
                  cudaStream_t s);

}  // namespace gp
