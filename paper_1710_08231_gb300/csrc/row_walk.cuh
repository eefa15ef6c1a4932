// row_walk.cuh -- CSR entries in segments: a warp takes consecutive entries, whatever rows they belong to.
#pragma once

#include <algorithm>

#include "gp_internal.cuh"

namespace gp {

// The longest rows of a power-law graph are spread over as many warps as they have segments. A segment starts with a
// search for its row (and what the row needs), so a large graph takes 256 entries; a smaller one down to 32, so that
// every warp of the chip has about four and the last ones end together. Scoring with four against one per warp: R-MAT
// 14 159 and 210 us, 260000 points 439 and 465, 50000 points 144 and 126 (151 with a half-warp per vertex); 12,000
// entries in segments of 256 took 145 us, in segments of 32 they take 54.
inline int row_segment(int64_t m) {
  const int64_t warps = (int64_t)num_sms() * 32 * 4;  // (four blocks of eight are resident per SM)
  return (int)std::max<int64_t>(32, std::min<int64_t>(256, (m / warps + 31) / 32 * 32));
}

// The largest v with off[v] <= x (0 <= x < m), found by the whole warp: 32 pivots per step.
__device__ __forceinline__ int64_t warp_row_of(const DGraph &g, int64_t x) {
  const int lane = threadIdx.x & 31;
  int64_t lo = 0, hi = g.n;  // off[lo] <= x < off[hi]
  while (hi - lo > 1) {
    const int64_t step = (hi - lo + 31) / 32;
    const int64_t p = lo + (lane + 1) * step;
    const unsigned below = __ballot_sync(kFull, p < hi && g.row_begin(p) <= x);  // (a prefix of the lanes)
    const int c = __popc(below);
    const int64_t base = lo;
    lo = base + c * step;
    hi = min(hi, base + (c + 1) * step);
  }
  return lo;
}

// The rows of a segment, in order; lane l holds the end of row base + l.
struct RowWindow {
  int64_t base, first, ends;  // first: begin of row `base`
  __device__ __forceinline__ void load(const DGraph &g, int64_t v) {
    base = v;
    first = g.row_begin(v);
    const int64_t x = v + 1 + (threadIdx.x & 31);
    ends = g.row_begin(x < g.n ? x : g.n);
  }
  // the row that holds entry e (at or after the window's start) and its bounds
  __device__ __forceinline__ int64_t seek(const DGraph &g, int64_t e, int64_t *beg, int64_t *end) {
    unsigned m;
    while ((m = __ballot_sync(kFull, ends > e)) == 0) load(g, base + 32);
    const int f = __ffs(m) - 1;
    *end = __shfl_sync(kFull, ends, f);
    const int64_t b = __shfl_sync(kFull, ends, f > 0 ? f - 1 : 0);
    *beg = f > 0 ? b : first;
    return base + f;
  }
};

}  // namespace gp
