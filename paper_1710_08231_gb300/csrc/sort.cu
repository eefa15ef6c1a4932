// sort.cu -- device-wide stable LSD radix sort of (uint64 key, uint64 value) pairs.
//
// Each pass takes up to nine key bits with three kernels: per-tile digit counts (digit-major), an exclusive scan
// of the counts, and a stable scatter in which every tile ranks its items per digit in order (one vote per
// digit bit and 32 items, per-warp counts), stages them in shared memory in digit order and writes each digit's run
// contiguously. Used for vertex orders; the contraction runs the same tiles in its own kernel.
#include <algorithm>

#include "sort_tile.cuh"

namespace gp {

namespace {

__global__ void __launch_bounds__(kSortThreads) k_radix_hist(const unsigned long long *keys, int64_t n, int shift,
                                                             int bits, int64_t ntiles, int64_t *hist) {
  __shared__ unsigned h[kMaxDigits];
  radix_tile_hist(keys, (int64_t)blockIdx.x * kSortTile, n, shift, bits, hist + blockIdx.x, ntiles, h);
}

__global__ void __launch_bounds__(kSortThreads, 2) k_radix_scatter(const unsigned long long *kin,
                                                                   const unsigned long long *vin,
                                                                   unsigned long long *kout, unsigned long long *vout,
                                                                   int64_t n, int shift, int bits, int64_t ntiles,
                                                                   const int64_t *offs) {
  extern __shared__ unsigned long long s_key[];
  __shared__ RadixSmem sm;
  const int64_t base = (int64_t)blockIdx.x * kSortTile;
  radix_tile_scatter<unsigned long long>(kin, vin, kout, vout, base, (int)min(kSortTile, n - base), shift, bits,
                                         offs + blockIdx.x, ntiles, s_key, sm);
}

}  // namespace

int radix_sort_pairs(unsigned long long *keys, unsigned long long *vals, unsigned long long *keys_tmp,
                     unsigned long long *vals_tmp, int64_t n, int bits, bool *result_in_tmp, Workspace &ws) {
  cudaStream_t s = ws.stream();
  *result_in_tmp = false;
  if (n <= 1 || bits <= 0) return GP_OK;
  int per_sm = 0;
  GP_TRY(kernel_blocks_per_sm((const void *)k_radix_scatter, kSortThreads, kSortSmem<unsigned long long>,
                              kSortSmem<unsigned long long>, &per_sm));
  const int passes = sort_passes(bits), width = (bits + passes - 1) / passes;
  const int64_t ntiles = sort_tiles(n);
  int64_t *hist;
  GP_TRY(ws.get(&hist, (size_t)((ntiles << width) + 1)));
  unsigned long long *ks = keys, *vs = vals, *kd = keys_tmp, *vd = vals_tmp;
  for (int shift = 0; shift < bits; shift += width) {
    const int w = std::min(width, bits - shift);
    (::gp::count_launch(),
     k_radix_hist<<<(unsigned)ntiles, kSortThreads, 0, s>>>(ks, n, shift, w, ntiles, hist));
    GP_TRY(scan_excl_i64(hist, hist, ntiles << w, hist + (ntiles << w), ws));
    (::gp::count_launch(), k_radix_scatter<<<(unsigned)ntiles, kSortThreads, kSortSmem<unsigned long long>, s>>>(
                               ks, vs, kd, vd, n, shift, w, ntiles, hist));
    GP_LAUNCH_CHECK();
    std::swap(ks, kd);
    std::swap(vs, vd);
    *result_in_tmp = !*result_in_tmp;
  }
  return GP_OK;
}

}  // namespace gp
