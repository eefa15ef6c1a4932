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

#include "contract.cuh"
#include "lp.cuh"
#include "sort.cuh"

namespace gp {

namespace {

__global__ void k_mark_used(const int32_t *labels, int64_t n, int64_t nl, uint32_t *used, int *bad) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    const int L = labels[v];
    if (L < 0 || L >= nl) {
      atomicExch(bad, 1);
      continue;
    }
    used[L] = 1;
  }
}

// Fine -> coarse map and, per coarse vertex, member count and weight. Members of one cluster are mostly
// neighbours in id order, so the warp combines equal coarse ids before its atomics.
// A label outside [0, nl) sets *bad and maps its vertex to 0 (the caller reports the error).
__global__ void k_f2c(DGraph g, const int32_t *labels, int64_t nl, const int32_t *newid, int32_t *f2c, int64_t *cnt,
                      int64_t *cw, int *bad) {
  const int lane = threadIdx.x & 31;
  for (int64_t v0 = blockIdx.x * (int64_t)blockDim.x; v0 < g.n; v0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t v = v0 + threadIdx.x;
    bool ok = v < g.n;
    int cv = 0;
    long long c = 0;
    if (ok) {
      const int L = labels[v];
      if (L < 0 || L >= nl) {
        atomicExch(bad, 1);
        f2c[v] = 0;
        ok = false;
      } else {
        cv = newid[L];
        f2c[v] = cv;
        c = g.vweight(v);
      }
    }
    const unsigned peers = __match_any_sync(kFull, ok ? cv : -1);
    if (!ok) continue;
    long long cs = 0;
    for (unsigned m = peers; m; m &= m - 1) cs += __shfl_sync(peers, c, __ffs(m) - 1);
    if (lane == __ffs(peers) - 1) {
      atomicAdd(reinterpret_cast<unsigned long long *>(&cnt[cv]), (unsigned long long)__popc(peers));
      atomicAdd(reinterpret_cast<unsigned long long *>(&cw[cv]), (unsigned long long)cs);
    }
  }
}

// Members bucketed by coarse id (in any order within a cluster) with their degrees; largest coarse weight.
__global__ void k_members(DGraph g, const int32_t *f2c, const int64_t *mstart, unsigned *fill, int32_t *members,
                          int64_t *mdeg, const int64_t *cw, int64_t ncb, unsigned long long *maxcw) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < g.n; v += (int64_t)gridDim.x * blockDim.x) {
    const int cv = f2c[v];
    const int64_t pos = mstart[cv] + atomicAdd(&fill[cv], 1u);
    members[pos] = (int32_t)v;
    mdeg[pos] = g.row_begin(v + 1) - g.row_begin(v);
  }
  unsigned long long m = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < ncb; i += (int64_t)gridDim.x * blockDim.x)
    m = max(m, (unsigned long long)cw[i]);
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(kFull, m, o));
  if ((threadIdx.x & 31) == 0 && m) atomicMax(maxcw, m);
}

// Edge-weight values that travel with the pairs: none (unit weights), 32 or 64 bits.
template <int EW>
constexpr int kValBytes = EW == 0 ? 0 : (EW == 1 ? 4 : 8);

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

// The pairs in walking order, keys (cv << 32 | cu) and values omega, and the digit counts of the sort's first
// pass. Position p of the walk belongs to the member row with mpre[i] <= p < mpre[i + 1]; a warp takes 256
// consecutive positions, eight per lane, whatever rows they lie in: 32 rows at a time are held by the lanes
// and searched by shuffles. All positions are resolved first, then their adjacency entries are loaded, then
// the coarse ids of those are gathered, so that eight gathers per lane are in flight: the gathers bound it.
template <int EW>
__global__ void __launch_bounds__(kSortThreads) k_pairs(DGraph g, const int32_t *members, const int64_t *mpre,
                                                        const int32_t *f2c, unsigned long long *keys, void *vals,
                                                        int bits, int64_t ntiles, int64_t *hist) {
  __shared__ unsigned h[1 << kSortBits];
  static_assert(kSortThreads == 1 << kSortBits, "one thread per digit");
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const unsigned mask = (1u << bits) - 1u;
  const int64_t m = mpre[g.n];
  h[threadIdx.x] = 0;
  __syncthreads();
  const int64_t s0 = (int64_t)blockIdx.x * kSortTile + (int64_t)wid * (32 * kSortItems);
  if (s0 < m) {
    int64_t x[kSortItems];
    int cu[kSortItems];
    int64_t base = 0, ends = 0, delta = 0;
    int own = 0;
    auto window = [&](int64_t i0) {  // lane l: row i0 + l (rows past the last one end where the walk ends)
      base = i0;
      const int64_t i = i0 + lane;
      ends = mpre[i < g.n ? i + 1 : g.n];
      if (i < g.n) {
        const int v = members[i];
        delta = g.row_begin(v) - mpre[i];
        own = f2c[v];
      }
    };
    window(warp_owner(mpre, g.n, s0));
#pragma unroll
    for (int k = 0; k < kSortItems; k++) {
      const int64_t p = s0 + 32 * k + lane;
      bool open = p < m;
      x[k] = -1;
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
        const int64_t after = base + 64 < g.n ? mpre[base + 64] : mpre[g.n];
        window(after > want ? base + 32 : warp_owner(mpre, g.n, want));
      }
    }
    int cv[kSortItems];
#pragma unroll
    for (int k = 0; k < kSortItems; k++) cv[k] = x[k] >= 0 ? __ldg(g.adj + x[k]) : 0;
#pragma unroll
    for (int k = 0; k < kSortItems; k++) cv[k] = x[k] >= 0 ? f2c[cv[k]] : 0;
#pragma unroll
    for (int k = 0; k < kSortItems; k++) {
      if (x[k] < 0) continue;
      const int64_t p = s0 + 32 * k + lane;
      const bool out = cv[k] != cu[k];
      keys[p] = out ? ((unsigned long long)(unsigned)cv[k] << 32) | (unsigned)cu[k] : kSortDropped;
      if (EW == 1) static_cast<int32_t *>(vals)[p] = __ldg(static_cast<const int32_t *>(g.ew) + x[k]);
      if (EW == 2) static_cast<long long *>(vals)[p] = __ldg(static_cast<const long long *>(g.ew) + x[k]);
      if (out) atomicAdd(&h[(unsigned)cv[k] & mask], 1u);
    }
  }
  __syncthreads();
  if (threadIdx.x <= mask) hist[(int64_t)threadIdx.x * ntiles + blockIdx.x] = h[threadIdx.x];
}

// Sorted pairs: the first of equal ones is a head. Heads per tile and per coarse row.
constexpr int kHeadThreads = 256;
constexpr int kHeadItems = 8;  // per lane
constexpr int64_t kHeadTile = (int64_t)kHeadThreads * kHeadItems;

__global__ void __launch_bounds__(kHeadThreads) k_heads(const unsigned long long *keys, const int64_t *n_dev,
                                                        int64_t *tile_heads, int64_t *rowcnt) {
  __shared__ unsigned s_heads;
  const int64_t n = *n_dev;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t base = (int64_t)blockIdx.x * kHeadTile + (int64_t)wid * (32 * kHeadItems);
  if (threadIdx.x == 0) s_heads = 0;
  __syncthreads();
  if (base < n) {
    unsigned long long key[kHeadItems];
#pragma unroll
    for (int k = 0; k < kHeadItems; k++) {
      const int64_t i = base + 32 * k + lane;
      key[k] = i < n ? keys[i] : kSortDropped;
    }
    unsigned long long before = base > 0 ? keys[base - 1] : kSortDropped;
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
    if (lane == 0) atomicAdd(&s_heads, total);
  }
  __syncthreads();
  if (threadIdx.x == 0) tile_heads[blockIdx.x] = s_heads;
}

// Sorted pairs to coarse entries: a run of equal pairs becomes one entry at the run's rank. A run inside one
// step of 32 is stored; the parts of a run that crosses steps are added (ew must be zero on entry).
template <int EW>
__global__ void __launch_bounds__(kHeadThreads) k_entries(const unsigned long long *keys, const void *vals,
                                                          const int64_t *n_dev, const int64_t *tile_first, int32_t *adj,
                                                          int64_t *ew) {
  __shared__ unsigned s_warp[kHeadThreads / 32];
  const int64_t n = *n_dev;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t tbase = (int64_t)blockIdx.x * kHeadTile;
  if (tbase >= n) return;
  const int64_t base = tbase + (int64_t)wid * (32 * kHeadItems);
  unsigned long long key[kHeadItems], before = kSortDropped, after = kSortDropped;
  long long w[kHeadItems];
#pragma unroll
  for (int k = 0; k < kHeadItems; k++) {
    const int64_t i = base + 32 * k + lane;
    key[k] = i < n ? keys[i] : kSortDropped;
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
    const int64_t run = at + __popc(heads[k] & (lanemask_lt() | 1u << lane));
    const unsigned long long next = k + 1 < kHeadItems ? __shfl_sync(kFull, key[k + 1 < kHeadItems ? k + 1 : k], 0) : after;
    const unsigned peers = __match_any_sync(kFull, on ? (unsigned)(run - at) : 64u);
    long long sum = EW == 0 ? (long long)__popc(peers) : 0;
    if (EW) {
      // weights below 2^26 sum exactly in 32 bits over at most 32 lanes: one warp reduction
      if (!__any_sync(kFull, w[k] >= (1ll << 26) || w[k] < 0)) {
        sum = (long long)__reduce_add_sync(peers, (unsigned)w[k]);
      } else {
        for (unsigned pm = peers; pm; pm &= pm - 1) sum += __shfl_sync(peers, w[k], __ffs(pm) - 1);
      }
    }
    if (on && lane == __ffs(peers) - 1) {
      const bool starts = heads[k] >> lane & 1u;
      const int last = 31 - __clz(peers);
      const bool ends = last < 31 || next != key[k];
      if (starts) adj[run] = (int32_t)(key[k] & 0xffffffffull);
      if (starts && ends) ew[run] = sum;
      else atomicAdd(reinterpret_cast<unsigned long long *>(&ew[run]), (unsigned long long)sum);
    }
    at += __popc(heads[k]);
  }
}

// The pairs of g, sorted by (cv, cu): keys and values end in *keys_out / *vals_out, their number on the device at
// *count_out.
template <int EW>
int sorted_pairs(const DGraph &g, const int32_t *members, const int64_t *mpre, const int32_t *f2c, int kb,
                 unsigned long long **keys_out, void **vals_out, int64_t **count_out, Workspace &ws) {
  cudaStream_t s = ws.stream();
  const size_t m = (size_t)g.m;
  unsigned long long *k0, *k1;
  unsigned char *v0 = nullptr, *v1 = nullptr;
  GP_TRY(ws.get(&k0, m));
  GP_TRY(ws.get(&k1, m));
  if (kValBytes<EW>) {
    GP_TRY(ws.get(&v0, m * kValBytes<EW>));
    GP_TRY(ws.get(&v1, m * kValBytes<EW>));
  }
  const int passes = sort_passes(kb), width = std::max(1, (kb + passes - 1) / passes);
  const int64_t ntiles = sort_tiles(g.m), cells = ntiles << width;
  int64_t *hist, *count;
  GP_TRY(ws.get(&hist, (size_t)cells + 1));
  GP_TRY(ws.get(&count, 1));
  ProfScope ps("contract_rows", s);
  (::gp::count_launch(), k_pairs<EW><<<(unsigned)ntiles, kSortThreads, 0, s>>>(g, members, mpre, f2c, k0, v0, width, ntiles, hist));
  GP_LAUNCH_CHECK();
  for (int p = 0; p < passes; p++) {
    const int shift = 32 + p * width, w = std::max(1, std::min(width, kb - p * width));
    if (p > 0) GP_TRY(radix_hist(k0, count, g.m, shift, w, hist, s));
    GP_TRY(radix_offsets(hist, g.m, w, ws));
    if (p == 0)  // the number of pairs that are not inside a cluster
      GP_CUDA(cudaMemcpyAsync(count, hist + (ntiles << w), sizeof(int64_t), cudaMemcpyDeviceToDevice, s));
    GP_TRY(radix_scatter(k0, v0, k1, v1, kValBytes<EW>, p > 0 ? count : mpre + g.n, g.m, shift, w, hist, p == 0, s));
    std::swap(k0, k1);
    std::swap(v0, v1);
  }
  *keys_out = k0;
  *vals_out = v0;
  *count_out = count;
  return GP_OK;
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

int contract_graph(const DGraph &g, const int32_t *labels, int64_t nl, OwnedGraph *out, int32_t *f2c_user,
                   cudaStream_t s, const LpConfig *cfg, LpClassInfo *cls) {
  Workspace ws(s);
  const int nsm = num_sms();
  const int64_t n = g.n;
  auto grid_n = [&](int64_t items) {
    return (int)std::max<int64_t>(1, std::min<int64_t>((items + 255) / 256, nsm * 8));
  };
  if (n == 0) {
    GP_TRY(alloc_graph(out, 0, 0, s));
    GP_CUDA(cudaMemsetAsync(out->off, 0, sizeof(int64_t), s));
    return GP_OK;
  }
  // 1. used flags -> new ids by an exclusive prefix sum
  uint32_t *used;
  int32_t *newid;
  int *bad;
  int64_t *hdr;  // [0] = n', [1] = m'
  GP_TRY(ws.zeros(&used, (size_t)nl));
  GP_TRY(ws.get(&newid, (size_t)nl));
  GP_TRY(ws.zeros(&bad, 1));
  GP_TRY(ws.zeros(&hdr, 4));
  (::gp::count_launch(), k_mark_used<<<grid_n(n), 256, 0, s>>>(labels, n, nl, used, bad));
  GP_LAUNCH_CHECK();
  GP_TRY(scan_excl_u32(used, newid, nl, hdr, ws));
  // The coarse vertex count nc = hdr[0] stays on the device until the read back after step 4: the
  // arrays indexed by coarse vertex are sized for the bound min(n, nl) (zero beyond nc, so the scans
  // over the bound equal the scans over nc) and the row classification reads nc on the device.
  const int64_t ncb = std::max<int64_t>(1, std::min<int64_t>(n, nl));
  // 2. fine -> coarse map, member counts, coarse vertex weights
  int32_t *f2c = f2c_user;
  if (!f2c) GP_TRY(ws.get(&f2c, (size_t)n));
  int64_t *cnt, *mstart, *cw;
  GP_TRY(ws.zeros(&cnt, (size_t)ncb + 1));
  GP_TRY(ws.zeros(&cw, (size_t)ncb));
  GP_TRY(ws.get(&mstart, (size_t)ncb + 1));
  (::gp::count_launch(), k_f2c<<<grid_n(n), 256, 0, s>>>(g, labels, nl, newid, f2c, cnt, cw, bad));
  GP_LAUNCH_CHECK();
  GP_TRY(scan_excl_i64(cnt, mstart, ncb, mstart + ncb, ws));
  // 3. members bucketed by coarse id, and where their rows start in the walk over them
  unsigned *fill;
  int32_t *members;
  int64_t *mpre;
  unsigned long long *maxvw_dev;
  GP_TRY(ws.zeros(&fill, (size_t)ncb));
  GP_TRY(ws.get(&members, (size_t)n));
  GP_TRY(ws.get(&mpre, (size_t)n + 1));
  GP_TRY(ws.zeros(&maxvw_dev, 1));
  (::gp::count_launch(),
   k_members<<<grid_n(n), 256, 0, s>>>(g, f2c, mstart, fill, members, mpre, cw, ncb, maxvw_dev));
  GP_LAUNCH_CHECK();
  GP_TRY(scan_excl_i64(mpre, mpre, n, mpre + n, ws));
  unsigned long long maxvw = 0;
  int64_t hh[4];
  int hbad = 0;
  {
    Readback rb;
    rb.add(hh, hdr, sizeof(hh));
    rb.add(&hbad, bad, sizeof(int));
    rb.add(&maxvw, maxvw_dev, sizeof(maxvw));
    GP_TRY(rb.run(s));
  }
  if (hbad) {
    set_error("contract: a label is outside [0, n)");
    return GP_ERR_INVALID_ARG;
  }
  const int64_t nc = hh[0];
  int kb = 0;
  while (kb < 31 && ((int64_t)1 << kb) < nc) kb++;
  // 4. sorted pairs, heads per coarse row, coarse offsets
  const int ew = g.ew_mode();
  unsigned long long *keys = nullptr;
  void *vals = nullptr;
  int64_t *npairs = nullptr, *rowcnt, *off_tmp, *tile_heads = nullptr;
  GP_TRY(ws.zeros(&rowcnt, (size_t)nc + 1));
  GP_TRY(ws.get(&off_tmp, (size_t)nc + 1));
  const int64_t htiles = (g.m + kHeadTile - 1) / kHeadTile;
  if (g.m > 0) {
    GP_TRY(ew == 0   ? sorted_pairs<0>(g, members, mpre, f2c, kb, &keys, &vals, &npairs, ws)
           : ew == 1 ? sorted_pairs<1>(g, members, mpre, f2c, kb, &keys, &vals, &npairs, ws)
                     : sorted_pairs<2>(g, members, mpre, f2c, kb, &keys, &vals, &npairs, ws));
    GP_TRY(ws.get(&tile_heads, (size_t)htiles));
    (::gp::count_launch(), k_heads<<<(unsigned)htiles, kHeadThreads, 0, s>>>(keys, npairs, tile_heads, rowcnt));
    GP_LAUNCH_CHECK();
    GP_TRY(scan_excl_i64(tile_heads, tile_heads, htiles, nullptr, ws));
  }
  int64_t mc = 0;
  GP_TRY(scan_excl_i64(rowcnt, off_tmp, nc, off_tmp + nc, ws));
  // the next level's LP degree classes need only the coarse offsets: computed here and read back
  // with the coarse entry count
  unsigned long long *cls_dev = nullptr;
  unsigned long long cls_words[kLpClassWords];
  if (cfg && cls) {
    GP_TRY(ws.get(&cls_dev, (size_t)kLpClassWords));
    DGraph cg;
    cg.n = nc;
    cg.off = off_tmp;
    cg.off64 = 1;
    GP_TRY(lp_classes_launch(cg, *cfg, cls_dev, ws));
  }
  {
    Readback rb;
    rb.add(&mc, off_tmp + nc, sizeof(int64_t));
    if (cls_dev) rb.add(cls_words, cls_dev, sizeof(cls_words));
    GP_TRY(rb.run(s));
  }
  if (cls_dev) lp_classes_from(cls_words, *cfg, cls);
  GP_TRY(alloc_graph(out, nc, mc, s));
  out->max_vw = (int64_t)maxvw;
  GP_CUDA(cudaMemcpyAsync(out->off, off_tmp, sizeof(int64_t) * (size_t)(nc + 1), cudaMemcpyDeviceToDevice, s));
  GP_CUDA(cudaMemcpyAsync(out->vw, cw, sizeof(int64_t) * (size_t)nc, cudaMemcpyDeviceToDevice, s));
  // 5. equal pairs summed into the coarse entries
  if (mc > 0) {
    ProfScope ps("contract_compact", s);
    GP_CUDA(cudaMemsetAsync(out->ew, 0, sizeof(int64_t) * (size_t)mc, s));
    if (ew == 0)
      (::gp::count_launch(), k_entries<0><<<(unsigned)htiles, kHeadThreads, 0, s>>>(keys, vals, npairs, tile_heads, out->adj, out->ew));
    else if (ew == 1)
      (::gp::count_launch(), k_entries<1><<<(unsigned)htiles, kHeadThreads, 0, s>>>(keys, vals, npairs, tile_heads, out->adj, out->ew));
    else
      (::gp::count_launch(), k_entries<2><<<(unsigned)htiles, kHeadThreads, 0, s>>>(keys, vals, npairs, tile_heads, out->adj, out->ew));
    GP_LAUNCH_CHECK();
  }
  if (profiling()) {
    const int64_t rb = n * 2 * g.offset_bytes() + g.m * (4 + g.ew_bytes()) + g.m * 4;
    prof_add_counts("contract_rows", nc, g.m, rb);
    prof_add_counts("contract_compact", nc, mc, mc * 12 + nc * 8);
  }
  return GP_OK;  // stream-ordered: the temporary buffers are released on s after the kernels
}

}  // namespace gp
