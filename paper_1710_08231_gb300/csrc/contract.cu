// contract.cu -- contraction of a clustering into the weighted quotient graph on the GPU.
//
// Method (Section III-A; Section IV-A "Parallel Contraction"): cluster ids are remapped to
// [0, n') by a prefix sum over an array holding ones at the used ids; each coarse vertex weighs the
// sum of its members; each coarse edge (a, b), a != b, weighs the sum of the fine edges between
// clusters a and b.
//
// GPU design: instead of the paper's concurrent hash table, one stable sort of the (cv, cu, omega) pairs and a
// segmented sum. Fine vertices are bucketed by coarse id (a counting sort). Walking their rows in that order
// lists the pairs in ascending order of the walking side cu; because the graph is symmetric, each entry can
// stand for its reverse, row = the cluster of its other end cv, so only a stable sort by cv is left: two or
// three radix passes over the bits of n' where sorting by (cv, cu) would take twice as many. Pairs inside a
// cluster are dropped before the first pass. The sorted pairs are the coarse rows, sorted by neighbour id;
// equal pairs are adjacent and summed. Rows of every length take the same path, so neither a hub row nor the
// mix of lengths decides the time.
#include <algorithm>
#include <memory>
#include <new>
#include <vector>

#include "contract.cuh"
#include "lp.cuh"
#include "sort_tile.cuh"

namespace gp {

namespace {

constexpr int kMaxContractBlocks = 1024;  // (per-block partial sums)

// Edge-weight values that travel with the pairs: none (unit weights), 32 or 64 bits.
template <int EW>
struct PairVal {
  using T = NoVal;
};
template <>
struct PairVal<1> {
  using T = unsigned;
};
template <>
struct PairVal<2> {
  using T = unsigned long long;
};

constexpr int kThreads = kSortThreads;
constexpr int64_t kSegment = 32 * kSortItems;  // positions of the walk that a warp takes at a time
constexpr int64_t kOwnedRow = 16 * kSegment;   // longest row whose segments the thread that places it records
constexpr int kHeadThreads = 256;
constexpr int kHeadItems = 8;  // per lane
constexpr int64_t kHeadTile = (int64_t)kHeadThreads * kHeadItems;

// What the host reads back.
struct ContractHead {
  int64_t nc, mc, pairs;
  unsigned long long maxcw;
  unsigned long long classes[kLpClassWords];
  int bad, err;
};

struct ContractArgs {
  DGraph g;
  const int32_t *labels;
  int64_t nl;
  uint32_t *used;    // zeroed (used, cnt, cw, rowcnt, head, bar)
  int32_t *newid, *f2c, *members;
  int64_t *cnt, *mstart, *cw, *mpre, *hist, *tile_heads, *rowcnt, *off, *part;
  unsigned long long *k0, *k1;
  void *v0, *v1;
  int *tile_n;
  int32_t *seg_owner;  // the row that holds the first position of each of the walk's segments, -1: a long one
  int64_t segments;
  ContractHead *head;
  unsigned *bar;
  unsigned wait_us;
  int want_classes, deg_warp, deg_cta;
  int walk_only;  // up to step 5: the caller sorts the pairs in parts (contract_in_parts)
};

struct ContractSmem {
  RadixSmem radix;
  unsigned h[kMaxDigits];
  unsigned wbase[kSortWarps + 1];
  long long tmp[32], tot;
  unsigned heads[2];
};

// The largest i with pre[i] <= x (0 <= x < pre[n]), found by the whole warp: 32 pivots per step.
__device__ __forceinline__ int64_t warp_owner(const int64_t *pre, int64_t n, int64_t x) {
  const int lane = threadIdx.x & 31;
  int64_t lo = 0, hi = n;
  while (hi - lo > 1) {
    const int64_t step = (hi - lo + 31) / 32;
    const int64_t p = lo + (lane + 1) * step;
    const int c = __popc(__ballot_sync(kFull, p < hi && pre[p] <= x));  // (a prefix of the lanes)
    hi = min(hi, lo + (c + 1) * step);
    lo += c * step;
  }
  return lo;
}

// A scan over all blocks in two halves with a meeting between them: every block sums a contiguous chunk (the sum
// goes to part[block]); then it adds up the chunks before its own and writes its exclusive sums. Four
// consecutive items per thread.
__device__ __forceinline__ int64_t scan_chunk(int64_t n) {
  const int64_t step = 4 * kThreads;
  return ((n + gridDim.x - 1) / gridDim.x + step - 1) / step * step;
}

template <class In>
__device__ __forceinline__ void scan_sums(int64_t n, In in, int64_t *part, ContractSmem &sm) {
  const int64_t per = scan_chunk(n), lo = min(n, (int64_t)blockIdx.x * per), hi = min(n, lo + per);
  long long s = 0;
  for (int64_t i = lo + threadIdx.x; i < hi; i += kThreads) s += in(i);
  block_excl_scan64(s, sm.tmp, &sm.tot);
  if (threadIdx.x == 0) part[blockIdx.x] = sm.tot;
}

// Returns the sum of all items. out(i, sum of the items before i, item i) may overwrite item i.
template <class In, class Out>
__device__ __forceinline__ int64_t scan_write(int64_t n, In in, Out out, const int64_t *part, ContractSmem &sm) {
  const int64_t per = scan_chunk(n), lo = min(n, (int64_t)blockIdx.x * per), hi = min(n, lo + per);
  __syncthreads();
  long long before = 0, all = 0;
  for (unsigned x = threadIdx.x; x < gridDim.x; x += kThreads) {
    const long long p = part[x];
    all += p;
    if (x < blockIdx.x) before += p;
  }
  block_excl_scan64(all, sm.tmp, &sm.tot);
  const long long total = sm.tot;
  block_excl_scan64(before, sm.tmp, &sm.tot);
  long long run = sm.tot;
  for (int64_t base = lo; base < hi; base += 4 * kThreads) {
    const int64_t i = base + 4 * (int64_t)threadIdx.x;
    long long x[4], s = 0;
#pragma unroll
    for (int k = 0; k < 4; k++) {
      x[k] = i + k < hi ? (long long)in(i + k) : 0;
      s += x[k];
    }
    long long at = run + block_excl_scan64(s, sm.tmp, &sm.tot);
    run += sm.tot;
#pragma unroll
    for (int k = 0; k < 4; k++) {
      if (i + k < hi) out(i + k, at, x[k]);
      at += x[k];
    }
  }
  return total;
}

// The pairs of tile `tile` of the walk, keys (cv << 32 | cu) and values omega, compacted to the tile's front, and
// the digit counts of the sort's first pass. Position p of the walk belongs to the member row with
// mpre[i] <= p < mpre[i + 1]; a warp takes 256 consecutive positions, eight per lane, whatever rows they lie in:
// 32 rows at a time are held by the lanes and searched by shuffles. All positions are resolved first, then
// their adjacency entries are loaded, then the coarse ids of those are gathered, so that eight gathers per lane
// are in flight: the gathers bound it.
template <int EW>
__device__ __forceinline__ void pairs_tile(const ContractArgs &a, int64_t tile, int64_t m, int bits, int64_t ntiles,
                                           ContractSmem &sm) {
  using V = typename PairVal<EW>::T;
  const DGraph &g = a.g;
  const int64_t *const mpre = a.mpre;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const unsigned mask = (1u << bits) - 1u;
  const int64_t s0 = tile * kSortTile + (int64_t)wid * kSegment;
  __syncthreads();
  sm.h[threadIdx.x] = 0;
  int64_t x[kSortItems];
  int cu[kSortItems], cv[kSortItems];
#pragma unroll
  for (int k = 0; k < kSortItems; k++) x[k] = -1;
  if (s0 < m) {
    int64_t base = 0, ends = 0, delta = 0;
    int own = 0;
    auto window = [&](int64_t i0) {  // lane l: row i0 + l (rows past the last one end where the walk ends)
      base = i0;
      const int64_t i = i0 + lane;
      ends = mpre[i < g.n ? i + 1 : g.n];
      if (i < g.n) {
        const int v = a.members[i];
        delta = g.row_begin(v) - mpre[i];
        own = a.f2c[v];
      }
    };
    const int owner = a.seg_owner[s0 / kSegment];
    window(owner >= 0 ? owner : warp_owner(mpre, g.n, s0));
#pragma unroll
    for (int k = 0; k < kSortItems; k++) {
      const int64_t p = s0 + 32 * k + lane;
      bool open = p < m;
      cu[k] = 0;
      while (true) {
        int j = 0;  // rows of the window that end at or before p (31 at most)
#pragma unroll
        for (int step = 16; step > 0; step >>= 1)
          if (__shfl_sync(kFull, ends, j + step - 1) <= p) j += step;
        const int64_t ej = __shfl_sync(kFull, ends, j), dj = __shfl_sync(kFull, delta, j);
        const int cj = __shfl_sync(kFull, own, j);
        if (open && ej > p) {
          x[k] = p + dj;
          cu[k] = cj;
          open = false;
        }
        const unsigned left = __ballot_sync(kFull, open);
        if (!left) break;
        // the next 32 rows, or past a stretch without entries the first open position's row
        const int64_t want = s0 + 32 * k + (__ffs(left) - 1);
        const int64_t after = mpre[base + 64 < g.n ? base + 64 : g.n];
        window(after > want ? base + 32 : warp_owner(mpre, g.n, want));
      }
    }
  }
#pragma unroll
  for (int k = 0; k < kSortItems; k++) cv[k] = x[k] >= 0 ? __ldg(g.adj + x[k]) : -1;
#pragma unroll
  for (int k = 0; k < kSortItems; k++) cv[k] = x[k] >= 0 ? a.f2c[cv[k]] : -1;
  unsigned kept = 0;
#pragma unroll
  for (int k = 0; k < kSortItems; k++) kept += (unsigned)__popc(__ballot_sync(kFull, x[k] >= 0 && cv[k] != cu[k]));
  if (lane == 0) sm.wbase[wid] = kept;
  __syncthreads();
  int64_t at = tile * kSortTile;
  unsigned all = 0;
#pragma unroll
  for (int w = 0; w < kSortWarps; w++) {
    if (w < wid) at += sm.wbase[w];
    all += sm.wbase[w];
  }
#pragma unroll
  for (int k = 0; k < kSortItems; k++) {
    const bool out = x[k] >= 0 && cv[k] != cu[k];
    const unsigned outs = __ballot_sync(kFull, out);
    if (out) {
      const int64_t to = at + __popc(outs & lanemask_lt());
      a.k0[to] = ((unsigned long long)(unsigned)cv[k] << 32) | (unsigned)cu[k];
      if constexpr (EW != 0) static_cast<V *>(a.v0)[to] = __ldg(static_cast<const V *>(g.ew) + x[k]);
      atomicAdd(&sm.h[(unsigned)cv[k] & mask], 1u);
    }
    at += __popc(outs);
  }
  __syncthreads();
  if (threadIdx.x <= mask) a.hist[(int64_t)threadIdx.x * ntiles + tile] = sm.h[threadIdx.x];
  if (threadIdx.x == 0) a.tile_n[tile] = (int)all;
}

// Heads (first of equal sorted pairs) of two head tiles, half a block each, and per coarse row.
__device__ __forceinline__ void heads_tiles(const unsigned long long *keys, int64_t n, int64_t pair, int64_t *tile_heads,
                                            int64_t htiles, int64_t *rowcnt, ContractSmem &sm) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, half = wid / (kHeadThreads / 32);
  const int64_t base = 2 * pair * kHeadTile + (int64_t)wid * (32 * kHeadItems);
  __syncthreads();
  if (threadIdx.x < 2) sm.heads[threadIdx.x] = 0;
  __syncthreads();
  if (base < n) {
    unsigned long long key[kHeadItems];
#pragma unroll
    for (int k = 0; k < kHeadItems; k++) {
      const int64_t i = base + 32 * k + lane;
      key[k] = i < n ? keys[i] : ~0ull;
    }
    unsigned long long before = base > 0 ? keys[base - 1] : ~0ull;
    unsigned total = 0;
#pragma unroll
    for (int k = 0; k < kHeadItems; k++) {
      unsigned long long prev = __shfl_up_sync(kFull, key[k], 1);
      if (lane == 0) prev = before;
      before = __shfl_sync(kFull, key[k], 31);
      const bool head = base + 32 * k + lane < n && key[k] != prev;
      const unsigned heads = __ballot_sync(kFull, head);
      total += (unsigned)__popc(heads);
      const int row = (int)(key[k] >> 32);
      const unsigned peers = __match_any_sync(kFull, head ? row : -1);
      if (head && lane == __ffs(peers) - 1)
        atomicAdd(reinterpret_cast<unsigned long long *>(&rowcnt[row]), (unsigned long long)__popc(peers));
    }
    if (lane == 0) atomicAdd(&sm.heads[half], total);
  }
  __syncthreads();
  if (threadIdx.x < 2 && 2 * pair + threadIdx.x < htiles) tile_heads[2 * pair + threadIdx.x] = sm.heads[threadIdx.x];
}

// Everything up to the coarse offsets in one cooperative launch: the steps follow one another by grid meetings
// (about 2 us each) instead of kernel launches, and the sizes that the later steps need (n', the number of pairs)
// never go to the host. Small levels are bound by these steps one after another: 17 launches and 9 memsets took
// 250 us for a few thousand vertices, against 140 us now. Large ones are bound by the walk's gathers and the sort's
// passes over memory (R-MAT 22 with weights, 128 M entries: 34.2 ms with hash tables per row, 6.3 ms so; 2^20
// points: 0.62 and 0.42 ms).
template <int EW>
__global__ void __launch_bounds__(kThreads, 2) k_contract(ContractArgs a) {
  using V = typename PairVal<EW>::T;
  extern __shared__ unsigned long long dsm[];
  __shared__ ContractSmem sm;
  const GridBarrier bar{a.bar, &a.head->err, gridDim.x, blockIdx.x, a.wait_us};
  unsigned met = 0;
#define MEET() \
  if (!grid_meet(bar, met)) return
  const DGraph &g = a.g;
  const int64_t n = g.n;
  const int lane = threadIdx.x & 31;
  const int64_t tid = (int64_t)blockIdx.x * kThreads + threadIdx.x, stride = (int64_t)gridDim.x * kThreads;
  // 1. used labels (a label outside [0, nl) is an error of the call: nothing more is done)
  for (int64_t y = tid; y < a.segments; y += stride) a.seg_owner[y] = -1;
  for (int64_t v = tid; v < n; v += stride) {
    const int L = a.labels[v];
    if (L < 0 || L >= a.nl) atomicExch(&a.head->bad, 1);
    else a.used[L] = 1;
  }
  MEET();
  if (*(volatile int *)&a.head->bad) return;
  // 2. new ids by a prefix sum
  scan_sums(a.nl, [&](int64_t i) { return (long long)a.used[i]; }, a.part, sm);
  MEET();
  const int64_t nc = scan_write(a.nl, [&](int64_t i) { return (long long)a.used[i]; },
                                [&](int64_t i, long long x, long long) { a.newid[i] = (int32_t)x; }, a.part, sm);
  MEET();
  // 3. fine -> coarse map and, per coarse vertex, member count and weight. Members of one cluster are mostly
  // neighbours in id order, so the warp combines equal coarse ids before its atomics.
  for (int64_t v0 = (int64_t)blockIdx.x * kThreads; v0 < n; v0 += stride) {
    const int64_t v = v0 + threadIdx.x;
    const bool ok = v < n;
    int cv = -1;
    long long c = 0;
    if (ok) {
      cv = a.newid[a.labels[v]];
      a.f2c[v] = cv;
      c = g.vweight(v);
    }
    const unsigned peers = __match_any_sync(kFull, cv);
    if (!ok) continue;
    long long cs = 0;
    for (unsigned m = peers; m; m &= m - 1) cs += __shfl_sync(peers, c, __ffs(m) - 1);
    if (lane == __ffs(peers) - 1) {
      atomicAdd(reinterpret_cast<unsigned long long *>(&a.cnt[cv]), (unsigned long long)__popc(peers));
      atomicAdd(reinterpret_cast<unsigned long long *>(&a.cw[cv]), (unsigned long long)cs);
    }
  }
  MEET();
  // 4. members bucketed by coarse id (in any order within a cluster) with their degrees; largest coarse weight
  scan_sums(nc, [&](int64_t i) { return (long long)a.cnt[i]; }, a.part, sm);
  MEET();
  scan_write(nc, [&](int64_t i) { return (long long)a.cnt[i]; }, [&](int64_t i, long long x, long long) { a.mstart[i] = x; }, a.part,
             sm);
  {
    unsigned long long m = 0;
    for (int64_t i = tid; i < nc; i += stride) m = max(m, (unsigned long long)a.cw[i]);
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(kFull, m, o));
    if (lane == 0 && m) atomicMax(&a.head->maxcw, m);
  }
  MEET();
  for (int64_t v = tid; v < n; v += stride) {
    const int cv = a.f2c[v];
    const int64_t pos =
        a.mstart[cv] + (int64_t)atomicAdd(reinterpret_cast<unsigned long long *>(&a.cnt[cv]), ~0ull) - 1;
    a.members[pos] = (int32_t)v;
    a.mpre[pos] = g.row_begin(v + 1) - g.row_begin(v);
  }
  MEET();
  // 5. where the members' rows start in the walk over them
  scan_sums(n, [&](int64_t i) { return (long long)a.mpre[i]; }, a.part, sm);
  MEET();
  const int64_t m = min(g.m, scan_write(n, [&](int64_t i) { return (long long)a.mpre[i]; },
                                        [&](int64_t i, long long x, long long d) {
                                          a.mpre[i] = x;
                                          // the segments of the walk that begin in this row (a long row's are
                                          // left to a search)
                                          if (d <= kOwnedRow)
                                            for (int64_t y = (x + kSegment - 1) / kSegment; y * kSegment < x + d; y++)
                                              if (y < a.segments) a.seg_owner[y] = (int32_t)i;
                                        },
                                        a.part, sm));
  if (tid == 0) {
    a.mpre[n] = m;
    a.head->nc = nc;
  }
  if (a.walk_only) return;
  MEET();
  // 6. pairs, sorted by row
  int kb = 0;
  while (kb < 31 && ((int64_t)1 << kb) < nc) kb++;
  const int passes = sort_passes(kb), width = max(1, (kb + passes - 1) / passes);
  int64_t ntiles = sort_tiles(m);
  for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) pairs_tile<EW>(a, t, m, width, ntiles, sm);
  MEET();
  unsigned long long *ki = a.k0, *ko = a.k1;
  V *vi = static_cast<V *>(a.v0), *vo = static_cast<V *>(a.v1);
  int64_t pairs = 0;
  for (int p = 0; p < passes; p++) {
    const int shift = 32 + p * width, w = max(1, min(width, kb - p * width));
    if (p > 0) {
      ntiles = sort_tiles(pairs);
      for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x)
        radix_tile_hist(ki, t * kSortTile, pairs, shift, w, a.hist + t, ntiles, sm.h);
      MEET();
    }
    const int64_t cells = ntiles << w;
    scan_sums(cells, [&](int64_t i) { return (long long)a.hist[i]; }, a.part, sm);
    MEET();
    pairs = scan_write(cells, [&](int64_t i) { return (long long)a.hist[i]; },
                       [&](int64_t i, long long x, long long) { a.hist[i] = x; }, a.part, sm);
    MEET();
    for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
      const int tn = p == 0 ? a.tile_n[t] : (int)min(kSortTile, pairs - t * kSortTile);
      radix_tile_scatter<V>(ki, vi, ko, vo, t * kSortTile, tn, shift, w, a.hist + t, ntiles, dsm, sm.radix);
    }
    MEET();
    unsigned long long *tk = ki;
    ki = ko;
    ko = tk;
    V *tv = vi;
    vi = vo;
    vo = tv;
  }
  // 7. heads, coarse offsets
  const int64_t htiles = (pairs + kHeadTile - 1) / kHeadTile;
  for (int64_t t = blockIdx.x; 2 * t < htiles; t += gridDim.x)
    heads_tiles(ki, pairs, t, a.tile_heads, htiles, a.rowcnt, sm);
  MEET();
  scan_sums(htiles, [&](int64_t i) { return (long long)a.tile_heads[i]; }, a.part, sm);
  scan_sums(nc, [&](int64_t i) { return (long long)a.rowcnt[i]; }, a.part + gridDim.x, sm);
  MEET();
  const int64_t mc = scan_write(htiles, [&](int64_t i) { return (long long)a.tile_heads[i]; },
                                [&](int64_t i, long long x, long long) { a.tile_heads[i] = x; }, a.part, sm);
  scan_write(nc, [&](int64_t i) { return (long long)a.rowcnt[i]; }, [&](int64_t i, long long x, long long) { a.off[i] = x; },
             a.part + gridDim.x, sm);
  if (tid == 0) {
    a.off[nc] = mc;
    a.head->mc = mc;
    a.head->pairs = pairs;
  }
  // 8. LP degree classes of the coarse graph, from the row lengths (words as lp_classes_from reads them)
  if (a.want_classes) {
    unsigned *const cls = sm.h;
    __syncthreads();
    if (threadIdx.x < 16) cls[threadIdx.x] = 0;
    __syncthreads();
    unsigned long long ent = 0, hub_max = 0, hub_sum = 0, wide = 0;
    for (int64_t c = tid; c < nc; c += stride) {
      const int64_t d = a.rowcnt[c];
      if (d == 0) continue;
      const int b = lp_bin_of(d, a.deg_warp, a.deg_cta);
      atomicAdd(&cls[b], 1u);
      ent += (unsigned long long)d;
      if (b == 6) {
        hub_max = max(hub_max, (unsigned long long)hub_cap(d));
        hub_sum += (unsigned long long)hub_cap(d);
      }
      if (d > kWideDeg) wide++;
    }
    for (int o = 16; o > 0; o >>= 1) {
      ent += __shfl_xor_sync(kFull, ent, o);
      hub_max = max(hub_max, __shfl_xor_sync(kFull, hub_max, o));
      hub_sum += __shfl_xor_sync(kFull, hub_sum, o);
      wide += __shfl_xor_sync(kFull, wide, o);
    }
    unsigned long long *const words = a.head->classes;
    if (lane == 0 && ent) {
      atomicAdd(&words[5], ent);
      if (hub_max) atomicMax(&words[6], hub_max);
      if (hub_sum) atomicAdd(&words[7], hub_sum);
      if (wide) atomicAdd(&words[8], wide);
    }
    __syncthreads();
    if (threadIdx.x < 9 && cls[threadIdx.x]) atomicAdd(reinterpret_cast<unsigned *>(words) + threadIdx.x, cls[threadIdx.x]);
  }
#undef MEET
}

// Sorted pairs to coarse entries: a run of equal pairs becomes one entry at the run's rank, written by its last
// lane. A run inside one step of 32 is stored; the parts of a run that crosses steps are added (ew must be zero on
// entry). Bound by memory: the pairs are read once and the entries written once (the run sums are five shuffle
// steps; a reduction per run of a step took four times as long on rows of distinct neighbours). Also copies the
// coarse offsets and vertex weights.
template <int EW>
__global__ void __launch_bounds__(kHeadThreads) k_entries(const unsigned long long *keys, const void *vals, int64_t n,
                                                          const int64_t *tile_first, int32_t *adj, int64_t *ew,
                                                          int64_t nc, const int64_t *off_in, int64_t *off,
                                                          const int64_t *vw_in, int64_t *vw) {
  __shared__ unsigned s_warp[kHeadThreads / 32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int64_t i = (int64_t)blockIdx.x * kHeadThreads + threadIdx.x; i <= nc; i += (int64_t)gridDim.x * kHeadThreads) {
    off[i] = off_in[i];
    if (i < nc) vw[i] = vw_in[i];
  }
  const int64_t tbase = (int64_t)blockIdx.x * kHeadTile;
  if (tbase >= n) return;
  const int64_t base = tbase + (int64_t)wid * (32 * kHeadItems);
  unsigned long long key[kHeadItems], before = ~0ull, after = ~0ull;
  long long w[kHeadItems];
#pragma unroll
  for (int k = 0; k < kHeadItems; k++) {
    const int64_t i = base + 32 * k + lane;
    key[k] = i < n ? keys[i] : ~0ull;
    w[k] = 0;
    if (i < n) w[k] = EW == 0 ? 1 : EW == 1 ? (long long)static_cast<const int32_t *>(vals)[i] : static_cast<const long long *>(vals)[i];
  }
  if (base < n && base > 0) before = keys[base - 1];
  if (base + 32 * kHeadItems < n) after = keys[base + 32 * kHeadItems];
  unsigned heads[kHeadItems], total = 0;
#pragma unroll
  for (int k = 0; k < kHeadItems; k++) {
    unsigned long long prev = __shfl_up_sync(kFull, key[k], 1);
    if (lane == 0) prev = before;
    before = __shfl_sync(kFull, key[k], 31);
    heads[k] = __ballot_sync(kFull, base + 32 * k + lane < n && key[k] != prev);
    total += (unsigned)__popc(heads[k]);
  }
  if (lane == 0) s_warp[wid] = total;
  __syncthreads();
  int64_t at = tile_first[blockIdx.x] - 1;  // rank of the run open before the warp's first item
  for (int x = 0; x < wid; x++) at += s_warp[x];
#pragma unroll
  for (int k = 0; k < kHeadItems; k++) {
    if (base + 32 * k >= n) break;  // (uniform over the warp)
    const bool on = base + 32 * k + lane < n;
    const unsigned upto = heads[k] & (lanemask_lt() | 1u << lane);
    const int64_t run = at + __popc(upto);
    const int first = upto ? 31 - __clz(upto) : 0;  // the run's first lane in this step
    const unsigned long long next = k + 1 < kHeadItems ? __shfl_sync(kFull, key[k + 1 < kHeadItems ? k + 1 : k], 0) : after;
    unsigned long long mine_next = __shfl_down_sync(kFull, key[k], 1);
    if (lane == 31) mine_next = next;
    long long sum;
    if (EW == 0) {
      sum = on ? lane - first + 1 : 0;
    } else if (!__any_sync(kFull, w[k] >= (1ll << 26) || w[k] < 0)) {  // (32 of them fit 32 bits)
      unsigned x = (unsigned)w[k];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(kFull, x, o);
        if (lane - o >= first) x += y;
      }
      sum = x;
    } else {
      sum = w[k];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const long long y = __shfl_up_sync(kFull, sum, o);
        if (lane - o >= first) sum += y;
      }
    }
    const bool ends = mine_next != key[k];  // the run ends with this lane (past n the keys differ from any pair)
    if (on && (ends || lane == 31)) {
      const bool starts = upto != 0;
      if (starts) adj[run] = (int32_t)(key[k] & 0xffffffffull);
      if (starts && ends) ew[run] = sum;
      else atomicAdd(reinterpret_cast<unsigned long long *>(&ew[run]), (unsigned long long)sum);
    }
    at += __popc(heads[k]);
  }
}

template <int EW>
int launch_contract(ContractArgs &a, cudaStream_t s) {
  using V = typename PairVal<EW>::T;
  int per_sm = 0;
  GP_TRY(kernel_blocks_per_sm((const void *)k_contract<EW>, kThreads, kSortSmem<V>, kSortSmem<V>, &per_sm));
  // a block per sort tile or per 2048 vertices, up to what is resident: fewer blocks meet sooner
  const int64_t want = std::max<int64_t>(sort_tiles(a.g.m), (std::max(a.g.n, a.nl) + 2047) / 2048);
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(want, std::min<int64_t>((int64_t)per_sm * num_sms(), kMaxContractBlocks)));
  count_launch();
  void *args[] = {(void *)&a};
  GP_CUDA(cudaLaunchCooperativeKernel((void *)k_contract<EW>, grid, kThreads, args, kSortSmem<V>, s));
  return GP_OK;
}

// ------------------------------------------------------------------------------------------ in parts
// The pairs of a contraction take 17 (unit weights) to 33 bytes per entry while they are sorted. Where the allocator
// cannot give that, or not the coarse graph beside them, the coarse rows are made in parts of about an eighth of the
// entries, whose pairs (row, neighbour) are sorted by both halves of the key with 33 bytes per entry of the part: once
// for the row lengths and, with the coarse graph allocated, once more for the rows. Slower (a launch per step, two to
// three times the passes, two read backs per part), with the same coarse graph.
constexpr int64_t kParts = 8;

// starts[c]: where coarse row c starts in the walk over the members' rows (starts[nc]: its end)
__global__ void k_walk_starts(const int64_t *mstart, const int64_t *mpre, int64_t n, int64_t nc, int64_t *starts) {
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c <= nc; c += (int64_t)gridDim.x * blockDim.x)
    starts[c] = mpre[c < nc ? mstart[c] : n];
}

// Keys ((cu - c0) << 32 | cv) and weights of the entries of coarse rows [c0, c1), whose walk starts at w0; entries inside
// a cluster get a row behind the others. *kept += the entries between clusters. A warp per member row.
template <int EW>
__global__ void k_part_pairs(DGraph g, const int32_t *members, const int32_t *f2c, const int64_t *mstart,
                             const int64_t *mpre, int64_t nc, int64_t c0, int64_t c1, int64_t w0,
                             unsigned long long *keys, unsigned long long *vals, unsigned long long *kept) {
  const int lane = threadIdx.x & 31;
  const int64_t i0 = mstart[c0], i1 = c1 < nc ? mstart[c1] : g.n;
  const int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5, nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  unsigned long long out = 0;
  for (int64_t i = i0 + gw; i < i1; i += nw) {
    const int v = members[i], cu = f2c[v];
    const int64_t beg = g.row_begin(v), end = g.row_begin(v + 1), at = mpre[i] - w0 - beg;
    for (int64_t x = beg + lane; x < end; x += 32) {
      const int cv = f2c[__ldg(g.adj + x)];
      keys[at + x] = (unsigned long long)(cv == cu ? c1 - c0 : (int64_t)cu - c0) << 32 | (unsigned)cv;
      vals[at + x] = (unsigned long long)load_ew<EW>(g.ew, x);
      out += cv != cu;
    }
  }
  out = (unsigned long long)warp_sum64((int64_t)out);
  if (lane == 0 && out) atomicAdd(kept, out);
}

__global__ void __launch_bounds__(kThreads) k_part_heads(const unsigned long long *keys, int64_t n, int64_t *tile_heads,
                                                         int64_t htiles, int64_t *rowcnt) {
  __shared__ ContractSmem sm;
  for (int64_t t = blockIdx.x; 2 * t < htiles; t += gridDim.x) heads_tiles(keys, n, t, tile_heads, htiles, rowcnt, sm);
}

}  // namespace

int alloc_graph(OwnedGraph *g, int64_t n, int64_t m, cudaStream_t s) {
  g->n = n;
  g->m = m;
  g->off_bytes = sizeof(int64_t) * (size_t)(n + 1);
  g->adj_bytes = sizeof(int32_t) * (size_t)std::max<int64_t>(m, 1);
  g->vw_bytes = sizeof(int64_t) * (size_t)std::max<int64_t>(n, 1);
  g->ew_bytes = sizeof(int64_t) * (size_t)std::max<int64_t>(m, 1);
  g->off = (int64_t *)dev_alloc(g->off_bytes, s);
  g->adj = (int32_t *)dev_alloc(g->adj_bytes, s);
  g->vw = (int64_t *)dev_alloc(g->vw_bytes, s);
  g->ew = (int64_t *)dev_alloc(g->ew_bytes, s);
  if (!g->off || !g->adj || !g->vw || !g->ew) {
    g->release(s);
    set_error("device allocation for a coarse graph failed");
    return GP_ERR_OOM;
  }
  return GP_OK;
}

// The coarse graph of a walk that k_contract has prepared, part by part: first the row lengths, unless they are known
// already (counted), then the rows.
static int contract_in_parts(const ContractArgs &a, const ContractHead &h, bool counted, OwnedGraph *out, cudaStream_t s,
                             const LpConfig *cfg, LpClassInfo *cls) {
  Workspace ws(s);
  const DGraph &g = a.g;
  const int64_t nc = h.nc;
  auto grid_n = [](int64_t items) {
    return (int)std::max<int64_t>(1, std::min<int64_t>((items + 255) / 256, (int64_t)num_sms() * 8));
  };
  const std::unique_ptr<int64_t[]> starts(new (std::nothrow) int64_t[(size_t)nc + 1]);
  if (!starts) {
    set_error("contraction: host allocation failed");
    return GP_ERR_OOM;
  }
  {
    int64_t *d;
    GP_TRY(ws.get(&d, (size_t)nc + 1));
    (::gp::count_launch(), k_walk_starts<<<grid_n(nc + 1), 256, 0, s>>>(a.mstart, a.mpre, g.n, nc, d));
    GP_LAUNCH_CHECK();
    GP_CUDA(cudaMemcpyAsync(starts.get(), d, sizeof(int64_t) * ((size_t)nc + 1), cudaMemcpyDeviceToHost, s));
    GP_CUDA(cudaStreamSynchronize(s));
    ws.release();
  }
  const int64_t per = std::max<int64_t>(1, starts[(size_t)nc] / kParts);
  int64_t mc = h.mc;
  for (int write = counted ? 1 : 0; write < 2; write++) {
    if (write) GP_TRY(alloc_graph(out, nc, mc, s));
    if (write && mc > 0) GP_CUDA(cudaMemsetAsync(out->ew, 0, sizeof(int64_t) * (size_t)mc, s));
    int64_t at = 0;  // coarse entries of the rows before
    for (int64_t c0 = 0, c1 = 0; c0 < nc; c0 = c1) {
      // rows c0 .. c1 - 1: as many as stay within the part, one at least
      const int64_t w0 = starts[(size_t)c0];
      c1 = std::upper_bound(starts.get() + c0 + 1, starts.get() + nc + 1, w0 + per) - starts.get() - 1;
      c1 = std::max(c0 + 1, std::min(c1, nc));
      const int64_t np = starts[(size_t)c1] - w0;
      if (np <= 0) continue;
      Workspace part(s);
      unsigned long long *k0, *v0, *k1, *v1;
      int64_t *sizes, hs[2] = {0, 0};  // pairs between clusters, coarse entries
      GP_TRY(part.get(&k0, (size_t)np));
      GP_TRY(part.get(&v0, (size_t)np));
      GP_TRY(part.get(&k1, (size_t)np));
      GP_TRY(part.get(&v1, (size_t)np));
      GP_TRY(part.zeros(&sizes, 2));
      auto pairs_of = [&](auto kernel) {
        (::gp::count_launch(), kernel<<<grid_n(np), 256, 0, s>>>(g, a.members, a.f2c, a.mstart, a.mpre, nc, c0, c1, w0, k0,
                                                                 v0, reinterpret_cast<unsigned long long *>(sizes)));
      };
      if (g.ew_mode() == 0) pairs_of(k_part_pairs<0>);
      else if (g.ew_mode() == 1) pairs_of(k_part_pairs<1>);
      else pairs_of(k_part_pairs<2>);
      GP_LAUNCH_CHECK();
      GP_CUDA(cudaMemcpyAsync(hs, sizes, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
      GP_CUDA(cudaStreamSynchronize(s));
      if (hs[0] == 0) continue;
      int bits = 32;
      while (((int64_t)1 << (bits - 32)) <= c1 - c0) bits++;
      bool in_tmp = false;
      GP_TRY(radix_sort_pairs(k0, v0, k1, v1, np, bits, &in_tmp, part));
      const unsigned long long *keys = in_tmp ? k1 : k0, *vals = in_tmp ? v1 : v0;
      const int64_t htiles = (hs[0] + kHeadTile - 1) / kHeadTile;
      int64_t *tile_heads;
      GP_TRY(part.get(&tile_heads, (size_t)htiles));
      // (the row lengths are read no more once the rows are written)
      (::gp::count_launch(), k_part_heads<<<(unsigned)std::min<int64_t>((htiles + 1) / 2, (int64_t)num_sms() * 4), kThreads,
                                            0, s>>>(keys, hs[0], tile_heads, htiles, a.rowcnt + c0));
      GP_TRY(scan_excl_i64(tile_heads, tile_heads, htiles, sizes + 1, part));
      GP_CUDA(cudaMemcpyAsync(hs + 1, sizes + 1, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
      GP_CUDA(cudaStreamSynchronize(s));
      if (write) {
        (::gp::count_launch(), k_entries<2><<<(unsigned)htiles, kHeadThreads, 0, s>>>(
                                   keys, vals, hs[0], tile_heads, out->adj + at, out->ew + at, -1, nullptr, nullptr, nullptr, nullptr));
        GP_LAUNCH_CHECK();
      }
      at += hs[1];
    }
    if (!write) {
      mc = at;
      GP_TRY(scan_excl_i64(a.rowcnt, a.off, nc, a.off + nc, ws));
      ws.release();
    }
  }
  out->max_vw = (int64_t)h.maxcw;
  GP_CUDA(cudaMemcpyAsync(out->off, a.off, sizeof(int64_t) * ((size_t)nc + 1), cudaMemcpyDeviceToDevice, s));
  GP_CUDA(cudaMemcpyAsync(out->vw, a.cw, sizeof(int64_t) * (size_t)nc, cudaMemcpyDeviceToDevice, s));
  if (cfg && cls) {
    unsigned long long *words, hw[kLpStatWords];
    GP_TRY(ws.get(&words, (size_t)kLpStatWords));
    GP_TRY(lp_stats_launch(out->view(), *cfg, words, s));
    Readback rb;
    rb.add(hw, words, sizeof(hw));
    GP_TRY(rb.run(s));
    lp_classes_from(hw, *cfg, cls);
  }
  return GP_OK;
}

int contract_graph(const DGraph &g, const int32_t *labels, int64_t nl, OwnedGraph *out, int32_t *f2c_user,
                   cudaStream_t s, const LpConfig *cfg, LpClassInfo *cls) {
  Workspace ws(s);
  const int64_t n = g.n;
  if (n == 0) {
    GP_TRY(alloc_graph(out, 0, 0, s));
    GP_CUDA(cudaMemsetAsync(out->off, 0, sizeof(int64_t), s));
    return GP_OK;
  }
  // Arrays indexed by coarse vertex are sized for the bound min(n, nl); what must start at zero is one
  // allocation and one memset.
  const size_t ncb = (size_t)std::max<int64_t>(1, std::min<int64_t>(n, nl)), m = (size_t)g.m;
  const int ew = g.ew_mode();
  ContractArgs a;
  a.g = g;
  a.labels = labels;
  a.nl = nl;
  {
    auto up = [](size_t x) { return (x + 255) & ~size_t(255); };
    const size_t b_head = up(sizeof(ContractHead)), b_bar = up(sizeof(unsigned) * kBarrierStride),
                 b_used = up(sizeof(uint32_t) * (size_t)nl), b_cnt = up(sizeof(int64_t) * (ncb + 1));
    unsigned char *z;
    GP_TRY(ws.zeros(&z, b_head + b_bar + b_used + 3 * b_cnt));
    a.head = reinterpret_cast<ContractHead *>(z);
    a.bar = reinterpret_cast<unsigned *>(z + b_head);
    a.used = reinterpret_cast<uint32_t *>(z + b_head + b_bar);
    z += b_head + b_bar + b_used;
    a.cnt = reinterpret_cast<int64_t *>(z);
    a.cw = reinterpret_cast<int64_t *>(z + b_cnt);
    a.rowcnt = reinterpret_cast<int64_t *>(z + 2 * b_cnt);
  }
  GP_TRY(ws.get(&a.newid, (size_t)nl));
  a.f2c = f2c_user;
  if (!a.f2c) GP_TRY(ws.get(&a.f2c, (size_t)n));
  GP_TRY(ws.get(&a.members, (size_t)n));
  GP_TRY(ws.get(&a.mstart, ncb + 1));
  GP_TRY(ws.get(&a.mpre, (size_t)n + 1));
  GP_TRY(ws.get(&a.off, ncb + 1));
  GP_TRY(ws.get(&a.part, (size_t)2 * kMaxContractBlocks));
  Workspace pairs(s);  // what is sized by the entries
  auto get_pairs = [&]() -> int {
    GP_TRY(pairs.get(&a.k0, m));
    GP_TRY(pairs.get(&a.k1, m));
    const size_t vb = ew == 0 ? 0 : ew == 1 ? 4 : 8;
    unsigned char *v0 = nullptr, *v1 = nullptr;
    if (vb) {
      GP_TRY(pairs.get(&v0, m * vb));
      GP_TRY(pairs.get(&v1, m * vb));
    }
    a.v0 = v0;
    a.v1 = v1;
    const size_t ntiles = (size_t)sort_tiles(g.m);
    int kbound = 0;  // bits of the largest n' possible: the widest digit the kernel can choose
    while (kbound < 31 && ((int64_t)1 << kbound) < (int64_t)ncb) kbound++;
    GP_TRY(pairs.get(&a.tile_n, ntiles));
    a.segments = (int64_t)ntiles * (kSortTile / kSegment);
    GP_TRY(pairs.get(&a.seg_owner, (size_t)a.segments));
    GP_TRY(pairs.get(&a.hist, ntiles << std::min(std::max(kbound, 1), kSortBits)));
    GP_TRY(pairs.get(&a.tile_heads, m / (size_t)kHeadTile + 1));
    return GP_OK;
  };
  const int got = get_pairs();
  if (got != GP_OK && got != GP_ERR_OOM) return got;
  a.walk_only = got == GP_ERR_OOM;
  if (a.walk_only) {
    pairs.release();
    a.k0 = a.k1 = nullptr;
    a.v0 = a.v1 = nullptr;
    a.tile_n = nullptr;
    a.seg_owner = nullptr;
    a.segments = 0;
    a.hist = a.tile_heads = nullptr;
  }
  a.wait_us = (unsigned)std::min<unsigned long long>(wait_limit_ns() / 1000, 0xffffffffull);
  a.want_classes = cfg && cls && !a.walk_only;
  a.deg_warp = cfg ? cfg->deg_warp : 0;
  a.deg_cta = cfg ? cfg->deg_cta : 0;
  {
    ProfScope ps("contract_rows", s);
    GP_TRY(ew == 0 ? launch_contract<0>(a, s) : ew == 1 ? launch_contract<1>(a, s) : launch_contract<2>(a, s));
  }
  ContractHead h;
  {
    Readback rb;
    rb.add(&h, a.head, sizeof(h));
    GP_TRY(rb.run(s));
  }
  if (h.bad) {
    set_error("contract: a label is outside [0, n)");
    return GP_ERR_INVALID_ARG;
  }
  if (h.err) {
    set_error("contraction: a bounded device barrier gave up");
    return GP_ERR_TIMEOUT;
  }
  const int room = a.walk_only ? GP_ERR_OOM : alloc_graph(out, h.nc, h.mc, s);
  if (room != GP_OK) {
    pairs.release();
    const int st = contract_in_parts(a, h, !a.walk_only, out, s, cfg, cls);
    if (st != GP_OK) out->release(s);
    return st;
  }
  if (cfg && cls) lp_classes_from(h.classes, *cfg, cls);
  out->max_vw = (int64_t)h.maxcw;
  {
    // equal pairs summed into the coarse entries; the sorted pairs lie where the last pass left them
    int kb = 0;
    while (kb < 31 && ((int64_t)1 << kb) < h.nc) kb++;
    const bool odd = sort_passes(kb) & 1;
    const unsigned long long *keys = odd ? a.k1 : a.k0;
    const void *vals = odd ? a.v1 : a.v0;
    ProfScope ps("contract_compact", s);
    if (h.mc > 0) GP_CUDA(cudaMemsetAsync(out->ew, 0, sizeof(int64_t) * (size_t)h.mc, s));
    const unsigned grid = (unsigned)std::max<int64_t>((h.pairs + kHeadTile - 1) / kHeadTile,
                                                      std::min<int64_t>(h.nc / kHeadThreads + 1, (int64_t)num_sms() * 8));
    auto run = [&](auto kernel) {
      (::gp::count_launch(), kernel<<<grid, kHeadThreads, 0, s>>>(keys, vals, h.pairs, a.tile_heads, out->adj, out->ew,
                                                                  h.nc, a.off, out->off, a.cw, out->vw));
    };
    if (ew == 0) run(k_entries<0>);
    else if (ew == 1) run(k_entries<1>);
    else run(k_entries<2>);
    GP_LAUNCH_CHECK();
  }
  if (profiling()) {
    const int64_t rb = n * 2 * g.offset_bytes() + g.m * (4 + g.ew_bytes()) + g.m * 4;
    prof_add_counts("contract_rows", h.nc, g.m, rb);
    prof_add_counts("contract_compact", h.nc, h.mc, h.mc * 12 + h.nc * 8);
  }
  return GP_OK;  // stream-ordered: the temporary buffers are released on s after the kernels
}

}  // namespace gp
