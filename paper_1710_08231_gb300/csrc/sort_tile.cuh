// sort_tile.cuh -- one tile of a radix pass, for the sort's own kernels and for kernels that run several passes.
#pragma once

#include <type_traits>

#include "sort.cuh"

namespace gp {

constexpr int kSortWarps = kSortThreads / 32;
constexpr int kMaxDigits = 1 << kSortBits;
static_assert(kSortThreads == kMaxDigits, "one thread per digit");

struct NoVal {};
template <class V>
constexpr int kSortValBytes = std::is_same<V, NoVal>::value ? 0 : (int)sizeof(V);
template <class V>
constexpr int kSortSmem = (int)kSortTile * (8 + kSortValBytes<V>);  // dynamic shared memory of a scatter

// The lanes with the caller's digit: one vote per digit bit. (__match_any_sync takes a step per distinct value:
// 29 ns per warp and SM for 32 different digits against 5 ns for eight votes.) Lanes that are off match nobody.
__device__ __forceinline__ unsigned digit_peers(unsigned dg, int bits, bool on) {
  unsigned peers = __ballot_sync(kFull, on);
  for (int b = 0; b < bits; b++) {
    const unsigned m = __ballot_sync(kFull, dg >> b & 1u);
    peers &= dg >> b & 1u ? m : ~m;
  }
  return on ? peers : 0u;
}

struct RadixSmem {
  unsigned short wcnt[kSortWarps][kMaxDigits];
  unsigned loc[kMaxDigits];
  int64_t gbase[kMaxDigits];
  unsigned wsum[kSortWarps];
};

// Counts of one tile's digits (cnt[digit * stride]); h: kMaxDigits words of shared memory.
__device__ __forceinline__ void radix_tile_hist(const unsigned long long *keys, int64_t base, int64_t n, int shift,
                                                int bits, int64_t *cnt, int64_t stride, unsigned *h) {
  const unsigned mask = (1u << bits) - 1u;
  __syncthreads();
  h[threadIdx.x] = 0;
  __syncthreads();
  unsigned long long key[kSortItems];
#pragma unroll
  for (int k = 0; k < kSortItems; k++) {
    const int64_t i = base + (int64_t)k * kSortThreads + threadIdx.x;
    key[k] = i < n ? keys[i] : 0;
  }
#pragma unroll
  for (int k = 0; k < kSortItems; k++)
    if (base + (int64_t)k * kSortThreads + threadIdx.x < n) atomicAdd(&h[(unsigned)(key[k] >> shift) & mask], 1u);
  __syncthreads();
  if (threadIdx.x <= mask) cnt[(int64_t)threadIdx.x * stride] = h[threadIdx.x];
}

// Stable scatter of the tile's items [base, base + tn), tn <= kSortTile; offs[digit * stride] is the tile's first
// output position for the digit. Warp w of a tile owns its items [w, w + 1) * 32 kSortItems (the tile's order is
// warp, then round, then lane). Bound by memory once the ranking is by votes: an item is read once and written once, its key stays in a
// register between ranking and staging, and the staged items leave run by run.
template <class V>
__device__ __forceinline__ void radix_tile_scatter(const unsigned long long *kin, const V *vin,
                                                   unsigned long long *kout, V *vout, int64_t base, int tn, int shift,
                                                   int bits, const int64_t *offs, int64_t stride,
                                                   unsigned long long *s_key, RadixSmem &sm) {
  constexpr bool kVals = !std::is_same<V, NoVal>::value;
  V *const s_val = reinterpret_cast<V *>(s_key + kSortTile);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const unsigned mask = (1u << bits) - 1u;
  const int at = wid * (32 * kSortItems) + lane;
  unsigned long long key[kSortItems];
#pragma unroll
  for (int k = 0; k < kSortItems; k++) key[k] = at + 32 * k < tn ? kin[base + at + 32 * k] : 0;
  // this thread's digit's first output position (loaded while the items are ranked)
  const int64_t first = threadIdx.x <= mask ? offs[(int64_t)threadIdx.x * stride] : 0;
  V val[kVals ? kSortItems : 1];
  if constexpr (kVals) {
#pragma unroll
    for (int k = 0; k < kSortItems; k++) val[k] = at + 32 * k < tn ? vin[base + at + 32 * k] : (V)0;
  }
  __syncthreads();  // (the shared state of an earlier tile is read no more)
  for (int t = threadIdx.x; t < kSortWarps * kMaxDigits / 2; t += kSortThreads) reinterpret_cast<unsigned *>(sm.wcnt)[t] = 0;
  __syncthreads();
  unsigned short rank[kSortItems];
#pragma unroll
  for (int k = 0; k < kSortItems; k++) {
    const bool on = at + 32 * k < tn;
    const unsigned dg = (unsigned)(key[k] >> shift) & mask;
    const unsigned peers = digit_peers(dg, bits, on);
    const unsigned lt = (unsigned)__popc(peers & lanemask_lt());
    const unsigned old = on ? sm.wcnt[wid][dg] : 0u;
    __syncwarp();
    if (on && lt == 0) sm.wcnt[wid][dg] = (unsigned short)(old + __popc(peers));
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
      const unsigned c = sm.wcnt[w][d];
      sm.wcnt[w][d] = (unsigned short)tot;
      tot += c;
    }
    unsigned x = tot;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned y = __shfl_up_sync(kFull, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) sm.wsum[wid] = x;
    __syncthreads();
    unsigned run = x - tot;
    for (int w = 0; w < wid; w++) run += sm.wsum[w];
    sm.loc[d] = run;
    sm.gbase[d] = first - (int64_t)run;
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < kSortItems; k++) {
    if (at + 32 * k < tn) {
      const unsigned dg = (unsigned)(key[k] >> shift) & mask;
      const unsigned p = sm.loc[dg] + sm.wcnt[wid][dg] + rank[k];
      s_key[p] = key[k];
      if constexpr (kVals) s_val[p] = val[k];
    }
  }
  __syncthreads();
  for (int p = threadIdx.x; p < tn; p += kSortThreads) {
    const unsigned long long x = s_key[p];
    const int64_t out = sm.gbase[(unsigned)(x >> shift) & mask] + (int64_t)p;
    kout[out] = x;
    if constexpr (kVals) vout[out] = s_val[p];
  }
}

}  // namespace gp
