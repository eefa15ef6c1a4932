// sort.cu -- device-wide stable LSD radix sort of (uint64 key, value) pairs.
//
// Each pass takes up to nine key bits with three kernels: per-tile digit counts (digit-major), an exclusive scan
// of the counts, and a stable scatter in which every tile ranks its items per digit in order (one warp match
// per 32 items, per-warp counts), stages them in shared memory in digit order and writes each digit's run
// contiguously. Used where many independent rows must be sorted at once (contraction) and for vertex orders.
#include <algorithm>
#include <type_traits>

#include "sort.cuh"

namespace gp {

namespace {

constexpr int kSortWarps = kSortThreads / 32;
constexpr int kMaxDigits = 1 << kSortBits;
static_assert(kSortThreads == kMaxDigits, "one thread per digit");

__global__ void __launch_bounds__(kSortThreads) k_radix_hist(const unsigned long long *keys, const int64_t *n_dev,
                                                             int64_t n_max, int shift, int bits, int64_t ntiles,
                                                             int64_t *hist) {
  __shared__ unsigned h[kMaxDigits];
  const int64_t n = n_dev ? *n_dev : n_max;
  const int64_t base = (int64_t)blockIdx.x * kSortTile;
  const unsigned mask = (1u << bits) - 1u;
  h[threadIdx.x] = 0;
  __syncthreads();
  if (base < n) {
    unsigned long long key[kSortItems];
#pragma unroll
    for (int k = 0; k < kSortItems; k++) {
      const int64_t i = base + (int64_t)k * kSortThreads + threadIdx.x;
      key[k] = i < n ? keys[i] : 0;
    }
#pragma unroll
    for (int k = 0; k < kSortItems; k++)
      if (base + (int64_t)k * kSortThreads + threadIdx.x < n) atomicAdd(&h[(unsigned)(key[k] >> shift) & mask], 1u);
  }
  __syncthreads();
  if (threadIdx.x <= mask) hist[(int64_t)threadIdx.x * ntiles + blockIdx.x] = h[threadIdx.x];
}

// Stable scatter of one pass. Warp w of a tile owns its items [w, w + 1) * 32 kSortItems (the tile's order is
// warp, then round, then lane). Bound by memory: an item is read once and written once; its key stays in a
// register between ranking and staging. Two blocks per SM hold 8192 items of 16 bytes in shared memory.
struct NoVal {};

template <class V>
__global__ void __launch_bounds__(kSortThreads, 2) k_radix_scatter(const unsigned long long *kin, const V *vin,
                                                                   unsigned long long *kout, V *vout,
                                                                   const int64_t *n_dev, int64_t n_max, int shift,
                                                                   int bits, int64_t ntiles, const int64_t *offs,
                                                                   bool drop) {
  constexpr bool kVals = !std::is_same<V, NoVal>::value;
  extern __shared__ unsigned long long s_key[];  // kSortTile keys, then kSortTile values
  V *const s_val = reinterpret_cast<V *>(s_key + kSortTile);
  __shared__ unsigned short wcnt[kSortWarps][kMaxDigits];
  __shared__ unsigned loc[kMaxDigits];
  __shared__ int64_t gbase[kMaxDigits];
  __shared__ unsigned wsum[kSortWarps];
  const int64_t n = n_dev ? *n_dev : n_max;
  const int64_t tbase = (int64_t)blockIdx.x * kSortTile;
  if (tbase >= n) return;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const unsigned mask = (1u << bits) - 1u;
  const int64_t wbase = tbase + (int64_t)wid * (32 * kSortItems) + lane;
  unsigned long long key[kSortItems];
#pragma unroll
  for (int k = 0; k < kSortItems; k++) key[k] = wbase + 32 * k < n ? kin[wbase + 32 * k] : kSortDropped;
  // this thread's digit's first output position (loaded while the items are ranked)
  const int64_t first = threadIdx.x <= mask ? offs[(int64_t)threadIdx.x * ntiles + blockIdx.x] : 0;
  V val[kVals ? kSortItems : 1];
  if constexpr (kVals) {
#pragma unroll
    for (int k = 0; k < kSortItems; k++) val[k] = wbase + 32 * k < n ? vin[wbase + 32 * k] : (V)0;
  }
  for (int t = threadIdx.x; t < kSortWarps * kMaxDigits / 2; t += kSortThreads) reinterpret_cast<unsigned *>(wcnt)[t] = 0;
  __syncthreads();
  unsigned live = 0;
  unsigned short rank[kSortItems];
#pragma unroll
  for (int k = 0; k < kSortItems; k++) {
    const bool on = wbase + 32 * k < n && !(drop && key[k] == kSortDropped);
    const unsigned dg = on ? (unsigned)(key[k] >> shift) & mask : (unsigned)kMaxDigits;
    const unsigned peers = __match_any_sync(kFull, dg);
    const unsigned lt = (unsigned)__popc(peers & lanemask_lt());
    unsigned old = 0;
    if (on) {
      old = wcnt[wid][dg];
      live |= 1u << k;
    }
    __syncwarp();
    if (on && lt == 0) wcnt[wid][dg] = (unsigned short)(old + __popc(peers));
    __syncwarp();
    rank[k] = (unsigned short)(old + lt);
  }
  __syncthreads();
  {
    // thread d: the warps' starts inside digit d's run, and the run's start in the tile
    const int d = threadIdx.x;
    unsigned tot = 0;
#pragma unroll
    for (int w = 0; w < kSortWarps; w++) {
      const unsigned c = wcnt[w][d];
      wcnt[w][d] = (unsigned short)tot;
      tot += c;
    }
    unsigned x = tot;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned y = __shfl_up_sync(kFull, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) wsum[wid] = x;
    __syncthreads();
    unsigned run = x - tot;
    for (int w = 0; w < wid; w++) run += wsum[w];
    loc[d] = run;
    gbase[d] = first - (int64_t)run;
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < kSortItems; k++) {
    if (live >> k & 1u) {
      const unsigned dg = (unsigned)(key[k] >> shift) & mask;
      const unsigned p = loc[dg] + wcnt[wid][dg] + rank[k];
      s_key[p] = key[k];
      if constexpr (kVals) s_val[p] = val[k];
    }
  }
  __syncthreads();
  unsigned tn = 0;
#pragma unroll
  for (int w = 0; w < kSortWarps; w++) tn += wsum[w];
  for (unsigned p = threadIdx.x; p < tn; p += kSortThreads) {
    const unsigned long long x = s_key[p];
    const int64_t out = gbase[(unsigned)(x >> shift) & mask] + (int64_t)p;
    kout[out] = x;
    if constexpr (kVals) vout[out] = s_val[p];
  }
}

template <class V>
int scatter_as(const unsigned long long *kin, const void *vin, unsigned long long *kout, void *vout,
               const int64_t *n_dev, int64_t n_max, int shift, int bits, const int64_t *offs, bool drop,
               cudaStream_t s) {
  constexpr int kBytes = (int)(kSortTile * (8 + (std::is_same<V, NoVal>::value ? 0 : sizeof(V))));
  static const cudaError_t attr =
      cudaFuncSetAttribute(k_radix_scatter<V>, cudaFuncAttributeMaxDynamicSharedMemorySize, kBytes);
  GP_CUDA(attr);
  const int64_t ntiles = sort_tiles(n_max);
  (::gp::count_launch(), k_radix_scatter<V><<<(unsigned)ntiles, kSortThreads, kBytes, s>>>(
                             kin, static_cast<const V *>(vin), kout, static_cast<V *>(vout), n_dev, n_max, shift, bits,
                             ntiles, offs, drop));
  GP_LAUNCH_CHECK();
  return GP_OK;
}

}  // namespace

int radix_hist(const unsigned long long *keys, const int64_t *n_dev, int64_t n_max, int shift, int bits, int64_t *hist,
               cudaStream_t s) {
  const int64_t ntiles = sort_tiles(n_max);
  (::gp::count_launch(),
   k_radix_hist<<<(unsigned)ntiles, kSortThreads, 0, s>>>(keys, n_dev, n_max, shift, bits, ntiles, hist));
  GP_LAUNCH_CHECK();
  return GP_OK;
}

int radix_offsets(int64_t *hist, int64_t n_max, int bits, Workspace &ws) {
  const int64_t cells = sort_tiles(n_max) << bits;
  return scan_excl_i64(hist, hist, cells, hist + cells, ws);
}

int radix_scatter(const unsigned long long *kin, const void *vin, unsigned long long *kout, void *vout, int val_bytes,
                  const int64_t *n_dev, int64_t n_max, int shift, int bits, const int64_t *offs, bool drop,
                  cudaStream_t s) {
  if (val_bytes == 0) return scatter_as<NoVal>(kin, vin, kout, vout, n_dev, n_max, shift, bits, offs, drop, s);
  if (val_bytes == 4) return scatter_as<unsigned>(kin, vin, kout, vout, n_dev, n_max, shift, bits, offs, drop, s);
  return scatter_as<unsigned long long>(kin, vin, kout, vout, n_dev, n_max, shift, bits, offs, drop, s);
}

int radix_sort_pairs(unsigned long long *keys, unsigned long long *vals, unsigned long long *keys_tmp,
                     unsigned long long *vals_tmp, int64_t n, int bits, bool *result_in_tmp, Workspace &ws) {
  cudaStream_t s = ws.stream();
  *result_in_tmp = false;
  if (n <= 1 || bits <= 0) return GP_OK;
  const int passes = sort_passes(bits), width = (bits + passes - 1) / passes;
  int64_t *hist;
  GP_TRY(ws.get(&hist, (size_t)((sort_tiles(n) << width) + 1)));
  unsigned long long *ks = keys, *vs = vals, *kd = keys_tmp, *vd = vals_tmp;
  for (int shift = 0; shift < bits; shift += width) {
    const int w = std::min(width, bits - shift);
    GP_TRY(radix_hist(ks, nullptr, n, shift, w, hist, s));
    GP_TRY(radix_offsets(hist, n, w, ws));
    GP_TRY(radix_scatter(ks, vs, kd, vd, 8, nullptr, n, shift, w, hist, false, s));
    std::swap(ks, kd);
    std::swap(vs, vd);
    *result_in_tmp = !*result_in_tmp;
  }
  return GP_OK;
}

}  // namespace gp
