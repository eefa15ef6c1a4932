// mls.cu -- multi-try k-way local search (MLS) on the GPU, after label-propagation refinement.
//
// Section III-C: localized k-way searches, each started from a single boundary vertex of a todo list,
// move the vertex of largest gain from a priority queue seeded with the start vertex and its
// neighbours, queue the neighbours of moved vertices, respect the balance bound and keep the best
// prefix of their moves. Section IV-C, Algorithm 1 (PerformMoves / ApplyMoves): searches run in
// parallel on the partition of the local iteration's start and only record their moves; the recorded
// sequences are then applied one after another with every gain recomputed on the current partition,
// each sequence up to its best prefix. Local iterations repeat on the moved vertices while their gain
// exceeds alpha of the global iteration's gain; global iterations restart from all boundary vertices.
//
// GPU form:
//   * PerformMoves: one warp per search, all searches of a local iteration in one launch. A warp keeps
//     its whole search state in shared memory: the queue (an unsorted array; the maximum is found by a
//     warp reduction over (gain, H(s, w, 0), -w)), its moves and a small hash map of the blocks they
//     changed (the search's view of the partition), its copy of the block weights, and connection arrays.
//     The neighbours of a moved vertex are taken 32 at a time, a lane each: a lane finds its vertex in the
//     queue and computes its gain with connections of its own, since neither depends on what the others do.
//     (All searches of a partition of 262144 points, k = 4: 11.0 ms with a vertex per warp, 5.2 ms so.)
//     Each search writes its best prefix to its own slot range, so the sequences keep the todo order.
//   * ApplyMoves: one CTA walks the sequences in todo order (the non-empty ones found 256 at a time by a
//     block scan), recomputes each move's gain with a block-wide sum over the vertex's row, and applies
//     the best prefix; block weights live in shared memory. The vertices it moved are the next todo list.
//   * Todo lists are ordered by (H(s, v, 1), v) -- the order the oracle uses: every vertex counts the ones
//     before it (lists of up to kRankMax), or a radix sort. (Ordering 30 lists: 2.4 ms by sorts alone, 0.35 ms.)
// The readings the paper leaves open (fixed search bounds instead of the adaptive stopping rule, no
// global moved bitmap during a local iteration, the degree bound, the hash orders) are those of the
// CPU oracle; results are bit-identical to it.
#include <algorithm>
#include <climits>
#include <type_traits>
#include <vector>

#include "gp_internal.cuh"
#include "mls.cuh"
#include "sort.cuh"

namespace gp {
namespace {

constexpr int kMlsWarps = 4;
constexpr int kMlsThreads = kMlsWarps * 32;
constexpr int kMaxMoves = 64;
constexpr int kQCap = 256;  // (even: the queue is searched by pairs)
constexpr int kMaxK = 256;
constexpr int kMovedSlots = 128;  // hash map of moved vertices (at most kMaxMoves entries)
constexpr int kApplyThreads = 256;

struct WarpState {
  long long qg[kQCap];
  unsigned long long qh[kQCap];
  long long bw[kMaxK];
  int qv[kQCap];
  int mv[kMaxMoves], mto[kMaxMoves], mfrom[kMaxMoves];
  int hk[kMovedSlots], hb[kMovedSlots];
  int qn, nm;
};

// Per-warp connection arrays behind the WarpStates: k sums per lane (a vertex per lane), or k 64-bit sums shared by
// the lanes (a vertex per warp). More blocks than kLaneK leave no room for the former. Where rows are long, many lanes
// wait for the longest and what counts is how many searches are resident: there the arrays of a warp are at most
// kLaneBytes, half of its state (R-MAT 18 with weights, k = 64: 2.92 s with 16 KB a warp, 1.61 s with a vertex per
// warp; R-MAT 14, k = 24 / 32 / 48: unit 873 / 843 / 992 against 798 / 748 / 753 ms, weighted 986 / 1060 / - against
// 732 / 765 / -). With rows of up to kLaneMean entries on average lanes are faster (50000 points of degree 12, k = 32 /
// 48 / 64: 195 / 220 / 208 against 221 / 241 / 223 ms).
template <int EW>
using ConnT = typename std::conditional<EW == 0, unsigned, long long>::type;
constexpr int kLaneK = 64;
constexpr int kLaneRow = 64;  // longest row that a lane walks alone
constexpr int64_t kLaneMean = 16;
constexpr size_t kLaneBytes = 4096;
template <int EW>
bool lane_conn(const DGraph &g, int k) {
  return k <= kLaneK && (g.m <= kLaneMean * g.n || (size_t)k * 32 * sizeof(ConnT<EW>) <= kLaneBytes);
}
template <int EW>
size_t conn_bytes(const DGraph &g, int k) {
  return lane_conn<EW>(g, k) ? (size_t)k * 32 * sizeof(ConnT<EW>) : (size_t)k * sizeof(long long);
}
constexpr size_t kConnMost = (size_t)kLaneK * 32 * sizeof(long long);
static_assert(kConnMost >= kMaxK * sizeof(long long), "the largest connection arrays are those of the lanes");

struct MlsArgs {
  DGraph g;
  const int32_t *part;
  const int64_t *bw;  // block weights at the local iteration's start
  int k;
  int64_t lmax;
  uint64_t smix;  // mix64(s)
  int max_moves, fruitless, queue_cap, max_degree;
  unsigned conn_bytes;  // per warp
  int lane_conn;
};

__device__ __forceinline__ uint64_t hkey(uint64_t smix, uint64_t a, uint64_t b) { return mix64(mix64(smix ^ a) ^ b); }

__device__ __forceinline__ int moved_block(const WarpState &W, int u) {
  unsigned sl = mix32((unsigned)u) & (kMovedSlots - 1);
  while (true) {
    const int key = W.hk[sl];
    if (key == u) return W.hb[sl];
    if (key < 0) return -1;
    sl = (sl + 1) & (kMovedSlots - 1);
  }
}

__device__ __forceinline__ int view_block(const MlsArgs &A, const WarpState &W, int u) {
  const int b = W.nm ? moved_block(W, u) : -1;
  return b >= 0 ? b : A.part[u];
}

__device__ __forceinline__ int64_t degree_of(const DGraph &g, int v) { return g.row_begin(v + 1) - g.row_begin(v); }

// Best move of x in the warp's view (all lanes call; results are uniform). Returns movable.
template <int EW>
__device__ bool gain_of(const MlsArgs &A, WarpState &W, long long *conn, int x, int *to_out, long long *gain_out) {
  const int lane = threadIdx.x & 31;
  for (int b = lane; b < A.k; b += 32) conn[b] = 0;
  __syncwarp();
  const int64_t rb = A.g.row_begin(x), re = A.g.row_begin(x + 1);
  for (int64_t e = rb + lane; e < re; e += 32) {
    const int u = __ldg(A.g.adj + e);
    atomicAdd(reinterpret_cast<unsigned long long *>(&conn[view_block(A, W, u)]),
              (unsigned long long)load_ew<EW>(A.g.ew, e));
  }
  __syncwarp();
  const int a = view_block(A, W, x);
  const long long cx = A.g.vweight(x);
  const uint64_t hx = mix64(A.smix ^ (uint64_t)(uint32_t)x);
  long long bc = -1;
  uint64_t bh = 0;
  int bb = -1;
  for (int b = lane; b < A.k; b += 32) {
    const long long c = conn[b];
    if (b == a || c <= 0 || W.bw[b] + cx > A.lmax) continue;
    const uint64_t h = mix64(hx ^ (uint64_t)b);
    if (bb < 0 || c > bc || (c == bc && (h > bh || (h == bh && b < bb)))) {
      bc = c;
      bh = h;
      bb = b;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const long long c2 = __shfl_xor_sync(kFull, bc, o);
    const uint64_t h2 = __shfl_xor_sync(kFull, bh, o);
    const int b2 = __shfl_xor_sync(kFull, bb, o);
    if (b2 >= 0 && (bb < 0 || c2 > bc || (c2 == bc && (h2 > bh || (h2 == bh && b2 < bb))))) {
      bc = c2;
      bh = h2;
      bb = b2;
    }
  }
  const long long own = conn[a];
  __syncwarp();
  if (bb < 0) return false;
  *to_out = bb;
  *gain_out = bc - own;
  return true;
}

__device__ __forceinline__ int queue_find(const WarpState &W, int x) {
  int at = -1;
  for (int base = 0; base < W.qn; base += 32) {
    const int i = base + (threadIdx.x & 31);
    const unsigned m = __ballot_sync(kFull, i < W.qn && W.qv[i] == x);
    if (m) {
      at = base + __ffs(m) - 1;
      break;
    }
  }
  return at;
}

__device__ __forceinline__ void queue_remove(WarpState &W, int i) {
  __syncwarp();
  if ((threadIdx.x & 31) == 0) {
    const int last = W.qn - 1;
    W.qv[i] = W.qv[last];
    W.qg[i] = W.qg[last];
    W.qh[i] = W.qh[last];
    W.qn = last;
  }
  __syncwarp();
}

// Best move of the lane's vertex u (u < 0: none) in the warp's view, with connections conn[b * 32 + lane]. Bound by
// the chain row -> neighbour -> its block, which 32 vertices share (one vertex at a time, by the whole warp, took
// about 3 us each); four neighbours of a lane are in flight.
template <int EW>
__device__ bool lane_gain(const MlsArgs &A, const WarpState &W, ConnT<EW> *conn, int u, int *to_out,
                          long long *gain_out) {
  if (u < 0) return false;
  const int lane = threadIdx.x & 31;
  const int64_t rb = A.g.row_begin(u), re = A.g.row_begin(u + 1);
  const int a = view_block(A, W, u);
  const long long cu = A.g.vweight(u);
  for (int b = 0; b < A.k; b++) conn[b * 32 + lane] = 0;
  for (int64_t e = rb; e < re; e += 4) {
    int x[4], p[4];
    long long w[4];
#pragma unroll
    for (int y = 0; y < 4; y++) {
      x[y] = e + y < re ? __ldg(A.g.adj + e + y) : -1;
      w[y] = e + y < re ? load_ew<EW>(A.g.ew, e + y) : 0;
    }
#pragma unroll
    for (int y = 0; y < 4; y++) p[y] = x[y] >= 0 ? A.part[x[y]] : 0;
#pragma unroll
    for (int y = 0; y < 4; y++) {
      if (x[y] < 0) continue;
      const int moved = W.nm ? moved_block(W, x[y]) : -1;
      conn[(moved >= 0 ? moved : p[y]) * 32 + lane] += (ConnT<EW>)w[y];
    }
  }
  const uint64_t hu = mix64(A.smix ^ (uint64_t)(uint32_t)u);
  long long bc = 0;
  uint64_t bh = 0;
  int bb = -1;
  for (int b = 0; b < A.k; b++) {
    const long long c = (long long)conn[b * 32 + lane];
    if (b == a || c <= 0 || c < bc || W.bw[b] + cu > A.lmax) continue;
    const uint64_t h = mix64(hu ^ (uint64_t)b);
    if (c > bc || h > bh) {  // (blocks in ascending order: the smaller one stays on equal hashes)
      bc = c;
      bh = h;
      bb = b;
    }
  }
  if (bb < 0) return false;
  *to_out = bb;
  *gain_out = bc - (long long)conn[a * 32 + lane];
  return true;
}

__device__ __forceinline__ void queue_append(const MlsArgs &A, WarpState &W, int at, int x, long long gain) {
  W.qv[at] = x;
  W.qg[at] = gain;
  W.qh[at] = hkey(A.smix, (uint64_t)(uint32_t)x, 0);
}

// The lanes' vertices (u < 0: none; distinct, in lane order) are queued, or their keys recomputed: a vertex that is in
// the queue gets its gain anew or leaves, another is inserted if it is movable and the queue has room. Vertices above
// the degree bound and moved ones are left out. All lanes call.
template <int EW>
__device__ void touch(const MlsArgs &A, WarpState &W, unsigned char *conn_raw, int u) {
  const int lane = threadIdx.x & 31;
  const int64_t d = u >= 0 ? degree_of(A.g, u) : 0;
  if (u >= 0 && (d > A.max_degree || (W.nm && moved_block(W, u) >= 0))) u = -1;
  int at = -1;
  const int qn0 = W.qn;
#pragma unroll 4
  for (int i = 0; i < qn0; i += 2) {
    const int2 x = *reinterpret_cast<const int2 *>(&W.qv[i]);
    if (x.x == u) at = i;
    if (x.y == u && i + 1 < qn0) at = i + 1;
  }
  if (u < 0) at = -1;
  const unsigned queued = __ballot_sync(kFull, at >= 0), fresh = __ballot_sync(kFull, u >= 0) & ~queued;
  const unsigned shorts = __ballot_sync(kFull, A.lane_conn && d <= kLaneRow);
  int to = 0;
  long long gain = 0;
  bool movable = false;
  // The gains of vertices that a full queue has no room for are not computed (on dense graphs most neighbours are
  // such): then the vertices in the queue come first and, in lane order, those that find room left by a leaving vertex
  // come in a second step. Vertices of a lane each come in the first one unless the queue is full already, the others
  // only if all fit.
  int room = A.queue_cap - W.qn;
  unsigned now = queued | fresh, later = 0, leave = 0;
  if (__popc(fresh) > room) {
    later = room > 0 ? fresh & ~shorts : fresh;
    now &= ~later;
  }
#pragma unroll 1
  for (int step = 0;; step++) {
    const unsigned lanes = now & shorts;
    if (lanes) {
      const bool on = lanes >> lane & 1u;
      if (lane_gain<EW>(A, W, reinterpret_cast<ConnT<EW> *>(conn_raw), on ? u : -1, &to, &gain)) movable = true;
      __syncwarp();
    }
    unsigned o = now & ~lanes;
    if (o) {
      const unsigned enter = step ? fresh & __ballot_sync(kFull, movable) : 0;
      if (step) o |= leave | enter;
      for (; o; o &= o - 1) {
        const int src = __ffs(o) - 1;
        if (step) {
          if (leave >> src & 1u) {
            room++;
            continue;
          }
          if (room <= 0) continue;
          room--;
          if (enter >> src & 1u) continue;
        }
        int t1 = 0;
        long long g1 = 0;
        const bool m1 = gain_of<EW>(A, W, reinterpret_cast<long long *>(conn_raw), __shfl_sync(kFull, u, src), &t1, &g1);
        if (lane == src) {
          movable = m1;
          to = t1;
          gain = g1;
        }
        if (step && !m1) room++;
      }
    }
    if (!later) break;
    leave = queued & ~__ballot_sync(kFull, movable);
    now = later & (room > 0 ? kFull : leave ? ~(2u * (leave & (0u - leave)) - 1u) : 0u);
    later = 0;
    if (!now) break;
  }
  if (at >= 0 && movable) W.qg[at] = gain;
  const unsigned moving = __ballot_sync(kFull, movable);
  const unsigned out = queued & ~moving, in = fresh & moving;
  __syncwarp();
  if (W.qn + __popc(in) <= A.queue_cap) {
    // every insertion finds room whatever the order
    const int qn = W.qn;
    if (in >> lane & 1u) queue_append(A, W, qn + __popc(in & lanemask_lt()), u, gain);
    __syncwarp();
    if (lane == 0) W.qn = qn + __popc(in);
    __syncwarp();
    for (unsigned o = out; o; o &= o - 1) queue_remove(W, queue_find(W, __shfl_sync(kFull, u, __ffs(o) - 1)));
  } else {
    for (unsigned o = out | in; o; o &= o - 1) {
      const int src = __ffs(o) - 1;
      const int us = __shfl_sync(kFull, u, src);
      const long long gs = __shfl_sync(kFull, gain, src);
      if (out >> src & 1u) {
        queue_remove(W, queue_find(W, us));
      } else if (W.qn < A.queue_cap) {
        __syncwarp();
        if (lane == 0) {
          queue_append(A, W, W.qn, us, gs);
          W.qn += 1;
        }
        __syncwarp();
      }
    }
  }
}

// PerformMoves: one warp per todo vertex; seq[i * max_moves + j] = (vertex, from, to) of the best prefix,
// len[i] its length.
template <int EW>
__global__ void __launch_bounds__(kMlsThreads) k_mls_search(MlsArgs A, const int32_t *todo, int64_t m, int3 *seq,
                                                            int32_t *len) {
  extern __shared__ __align__(16) unsigned char smem[];
  WarpState &W = reinterpret_cast<WarpState *>(smem)[threadIdx.x >> 5];
  unsigned char *const conn = smem + kMlsWarps * sizeof(WarpState) + (threadIdx.x >> 5) * A.conn_bytes;
  const int lane = threadIdx.x & 31;
  const int64_t gw = (int64_t)blockIdx.x * kMlsWarps + (threadIdx.x >> 5);
  const int64_t nw = (int64_t)gridDim.x * kMlsWarps;
  for (int64_t i = gw; i < m; i += nw) {
    const int v = todo[i];
    const int64_t dv = degree_of(A.g, v);
    if (dv == 0 || dv > A.max_degree) {
      if (lane == 0) len[i] = 0;
      continue;
    }
    for (int b = lane; b < A.k; b += 32) W.bw[b] = A.bw[b];
    for (int t = lane; t < kMovedSlots; t += 32) W.hk[t] = -1;
    if (lane == 0) {
      W.qn = 0;
      W.nm = 0;
    }
    __syncwarp();
    {
      // the start vertex, then its neighbours in row order
      const int64_t rb = A.g.row_begin(v);
      for (int64_t y0 = 0; y0 <= dv; y0 += 32) {
        const int64_t y = y0 + lane;
        touch<EW>(A, W, conn, y == 0 ? v : y <= dv ? __ldg(A.g.adj + rb + y - 1) : -1);
      }
    }
    long long cum = 0, best = 0;
    int best_len = 0, fruitless = 0;
    while (W.qn > 0 && W.nm < A.max_moves) {
      // the queue's maximum by (gain, hash, -vertex)
      long long bg = 0;
      uint64_t bh = 0;
      int bx = -1, bi = -1;
      for (int j = lane; j < W.qn; j += 32) {
        const long long gq = W.qg[j];
        const uint64_t hq = W.qh[j];
        const int xq = W.qv[j];
        if (bi < 0 || gq > bg || (gq == bg && (hq > bh || (hq == bh && xq < bx)))) {
          bg = gq;
          bh = hq;
          bx = xq;
          bi = j;
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const long long g2 = __shfl_xor_sync(kFull, bg, o);
        const uint64_t h2 = __shfl_xor_sync(kFull, bh, o);
        const int x2 = __shfl_xor_sync(kFull, bx, o);
        const int i2 = __shfl_xor_sync(kFull, bi, o);
        if (i2 >= 0 && (bi < 0 || g2 > bg || (g2 == bg && (h2 > bh || (h2 == bh && x2 < bx))))) {
          bg = g2;
          bh = h2;
          bx = x2;
          bi = i2;
        }
      }
      const int x = bx;
      queue_remove(W, bi);
      int to;
      long long gain;
      if (!gain_of<EW>(A, W, reinterpret_cast<long long *>(conn), x, &to, &gain)) continue;
      const int a = view_block(A, W, x);
      const long long cx = A.g.vweight(x);
      __syncwarp();
      if (lane == 0) {
        const int j = W.nm;
        W.mv[j] = x;
        W.mfrom[j] = a;
        W.mto[j] = to;
        unsigned sl = mix32((unsigned)x) & (kMovedSlots - 1);
        while (W.hk[sl] >= 0) sl = (sl + 1) & (kMovedSlots - 1);
        W.hk[sl] = x;
        W.hb[sl] = to;
        W.bw[a] -= cx;
        W.bw[to] += cx;
        W.nm = j + 1;
      }
      __syncwarp();
      cum += gain;
      if (cum > best) {
        best = cum;
        best_len = W.nm;
        fruitless = 0;
      } else if (++fruitless >= A.fruitless) {
        break;
      }
      const int64_t re = A.g.row_begin(x + 1);
      for (int64_t e0 = A.g.row_begin(x); e0 < re; e0 += 32)
        touch<EW>(A, W, conn, e0 + lane < re ? __ldg(A.g.adj + e0 + lane) : -1);
    }
    const int L = best > 0 ? best_len : 0;
    for (int j = lane; j < L; j += 32) seq[i * A.max_moves + j] = make_int3(W.mv[j], W.mfrom[j], W.mto[j]);
    if (lane == 0) len[i] = L;
    __syncwarp();
  }
}

__device__ __forceinline__ long long block_sum_ll(long long x, long long *red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x;
  __syncthreads();
  long long t = 0;
  for (int w = 0; w < kApplyThreads / 32; w++) t += red[w];
  __syncthreads();
  return t;
}

// ApplyMoves: one CTA, sequences in todo order. out[0] += gain, out[1] += applied moves, whose vertices (each once) go
// to moved_list.
template <int EW>
__global__ void __launch_bounds__(kApplyThreads) k_mls_apply(DGraph g, int32_t *part, int64_t *bw_g, int k,
                                                             int64_t lmax, const int3 *seq, const int32_t *len,
                                                             int64_t m, int max_moves, uint32_t *moved,
                                                             int32_t *moved_list, long long *out) {
  __shared__ long long bw[kMaxK];
  __shared__ long long red[kApplyThreads / 32];
  __shared__ int idx[kApplyThreads];
  __shared__ int nidx;
  __shared__ int ok;
  __shared__ long long cum, best, gain_total, moves_total;
  __shared__ int best_len, napplied;
  for (int b = threadIdx.x; b < k; b += kApplyThreads) bw[b] = bw_g[b];
  if (threadIdx.x == 0) {
    gain_total = 0;
    moves_total = 0;
  }
  __syncthreads();
  for (int64_t base = 0; base < m; base += kApplyThreads) {
    const int64_t i = base + threadIdx.x;
    const bool ne = i < m && len[i] > 0;
    if (threadIdx.x == 0) nidx = 0;
    __syncthreads();
    // the non-empty sequences of this tile, in order
    const unsigned bal = __ballot_sync(kFull, ne);
    __shared__ int wbase[kApplyThreads / 32];
    if ((threadIdx.x & 31) == 0) wbase[threadIdx.x >> 5] = __popc(bal);
    __syncthreads();
    if (threadIdx.x == 0) {
      int s = 0;
      for (int w = 0; w < kApplyThreads / 32; w++) {
        const int c = wbase[w];
        wbase[w] = s;
        s += c;
      }
      nidx = s;
    }
    __syncthreads();
    if (ne) idx[wbase[threadIdx.x >> 5] + __popc(bal & lanemask_lt())] = (int)threadIdx.x;
    __syncthreads();
    for (int q = 0; q < nidx; q++) {
      const int64_t si = base + idx[q];
      const int L = len[si];
      if (threadIdx.x == 0) {
        cum = 0;
        best = 0;
        best_len = 0;
        napplied = 0;
      }
      __syncthreads();
      for (int j = 0; j < L; j++) {
        const int3 mvj = seq[si * max_moves + j];
        const int w = mvj.x, from = mvj.y, to = mvj.z;
        const long long cw = g.vweight(w);
        if (threadIdx.x == 0) ok = !(moved[w] || part[w] != from || bw[to] + cw > lmax);
        __syncthreads();
        if (!ok) break;
        long long gsum = 0;
        for (int64_t e = g.row_begin(w) + threadIdx.x; e < g.row_begin(w + 1); e += kApplyThreads) {
          const int b = part[__ldg(g.adj + e)];
          const long long we = load_ew<EW>(g.ew, e);
          if (b == to) gsum += we;
          if (b == from) gsum -= we;
        }
        gsum = block_sum_ll(gsum, red);
        if (threadIdx.x == 0) {
          part[w] = to;
          bw[from] -= cw;
          bw[to] += cw;
          napplied = j + 1;
          cum += gsum;
          if (cum > best) {
            best = cum;
            best_len = j + 1;
          }
        }
        __syncthreads();
      }
      // roll back the moves after the best prefix, mark the applied ones
      if (threadIdx.x == 0) {
        for (int j = napplied - 1; j >= best_len; j--) {
          const int3 mvj = seq[si * max_moves + j];
          const long long cw = g.vweight(mvj.x);
          part[mvj.x] = mvj.y;
          bw[mvj.z] -= cw;
          bw[mvj.y] += cw;
        }
        for (int j = 0; j < best_len; j++) {
          const int w = seq[si * max_moves + j].x;
          moved[w] = 1;
          moved_list[moves_total + j] = w;
        }
        gain_total += best;
        moves_total += best_len;
      }
      __syncthreads();
    }
  }
  for (int b = threadIdx.x; b < k; b += kApplyThreads) bw_g[b] = bw[b];
  if (threadIdx.x == 0) {
    out[0] += gain_total;
    out[1] += moves_total;
  }
}

// Boundary vertices within the degree bound, in any order: list[0 .. *count).
__global__ void k_boundary_list(DGraph g, const int32_t *part, int max_degree, int32_t *list, unsigned long long *count) {
  for (int64_t v0 = (int64_t)blockIdx.x * blockDim.x; v0 < g.n; v0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t v = v0 + threadIdx.x;
    bool f = false;
    if (v < g.n) {
      const int64_t rb = g.row_begin(v), re = g.row_begin(v + 1);
      if (re - rb <= max_degree) {
        const int a = part[v];
        for (int64_t e = rb; e < re && !f; e += 4) {
          int p[4];
#pragma unroll
          for (int y = 0; y < 4; y++) p[y] = e + y < re ? __ldg(g.adj + e + y) : -1;
#pragma unroll
          for (int y = 0; y < 4; y++) p[y] = p[y] >= 0 ? part[p[y]] : a;
          f = p[0] != a || p[1] != a || p[2] != a || p[3] != a;
        }
      }
    }
    const unsigned m = __ballot_sync(kFull, f);
    if (!m) continue;
    unsigned long long base = 0;
    if ((threadIdx.x & 31) == 0) base = atomicAdd(count, (unsigned long long)__popc(m));
    base = __shfl_sync(kFull, base, 0);
    if (f) list[base + __popc(m & lanemask_lt())] = (int32_t)v;
  }
}

// todo = list ordered by (H(s, v, 1), v). Short lists: every vertex counts those before it, a tile of keys at a time
// (m^2 compares of a launch that takes a few microseconds, where a radix sort of 64 bits takes two dozen launches).
constexpr int64_t kRankMax = 8192;
constexpr int kRankThreads = 256;

__global__ void __launch_bounds__(kRankThreads) k_todo_rank(const int32_t *list, int m, uint64_t smix, int32_t *todo) {
  __shared__ unsigned long long s_key[kRankThreads];
  __shared__ int s_v[kRankThreads];
  // a warp of eight lanes per vertex: 32 vertices per block
  const int i = blockIdx.x * (kRankThreads / 8) + (int)threadIdx.x / 8, part = threadIdx.x & 7;
  const int v = i < m ? list[i] : 0;
  const unsigned long long key = hkey(smix, (uint64_t)(uint32_t)v, 1);
  int before = 0;
  for (int t0 = 0; t0 < m; t0 += kRankThreads) {
    __syncthreads();
    if (t0 + (int)threadIdx.x < m) {
      const int x = list[t0 + threadIdx.x];
      s_v[threadIdx.x] = x;
      s_key[threadIdx.x] = hkey(smix, (uint64_t)(uint32_t)x, 1);
    }
    __syncthreads();
    const int cnt = min(kRankThreads, m - t0);
    for (int y = part; y < cnt; y += 8) before += s_key[y] < key || (s_key[y] == key && s_v[y] < v);
  }
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) before += __shfl_xor_sync(kFull, before, o, 8);
  if (part == 0 && i < m) todo[before] = v;
}

// Longer lists: radix sort of the keys, then runs of equal keys by vertex.
__global__ void k_todo_keys(const int32_t *list, int64_t m, uint64_t smix, unsigned long long *keys,
                            unsigned long long *vals) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
    keys[i] = hkey(smix, (uint64_t)(uint32_t)list[i], 1);
    vals[i] = (unsigned long long)(unsigned)list[i];
  }
}

__global__ void k_todo_out(const unsigned long long *keys, const unsigned long long *vals, int64_t m, int32_t *out) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
    const unsigned long long k = keys[i], v = vals[i];
    int64_t lo = i, hi = i + 1;  // the run of equal keys
    while (lo > 0 && keys[lo - 1] == k) lo--;
    while (hi < m && keys[hi] == k) hi++;
    int64_t at = lo;
    for (int64_t y = lo; y < hi; y++) at += vals[y] < v;
    out[at] = (int32_t)v;
  }
}

__global__ void k_mls_block_weights(DGraph g, const int32_t *part, int64_t *bw) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < g.n; v += (int64_t)gridDim.x * blockDim.x)
    atomicAdd(reinterpret_cast<unsigned long long *>(&bw[part[v]]), (unsigned long long)g.vweight(v));
}

int grid_of(int64_t items, int threads) {
  return (int)std::max<int64_t>(1, std::min<int64_t>((items + threads - 1) / threads, (int64_t)num_sms() * 8));
}

struct TodoBuffers {
  unsigned long long *k0, *v0, *k1, *v1;  // long lists only
  bool ready = false;
};

// todo = the m vertices of list (distinct, any order) ordered by (H(s, v, 1), v)
int order_todo(const int32_t *list, int64_t m, int64_t n, uint64_t s, int32_t *todo, TodoBuffers &B, Workspace &ws) {
  cudaStream_t st = ws.stream();
  if (m <= 0) return GP_OK;
  if (m <= kRankMax) {
    (count_launch(), k_todo_rank<<<(unsigned)((m + kRankThreads / 8 - 1) / (kRankThreads / 8)), kRankThreads, 0, st>>>(
                         list, (int)m, mix64(s), todo));
    GP_LAUNCH_CHECK();
    return GP_OK;
  }
  if (!B.ready) {
    GP_TRY(ws.get(&B.k0, (size_t)n));
    GP_TRY(ws.get(&B.v0, (size_t)n));
    GP_TRY(ws.get(&B.k1, (size_t)n));
    GP_TRY(ws.get(&B.v1, (size_t)n));
    B.ready = true;
  }
  (count_launch(), k_todo_keys<<<grid_of(m, 256), 256, 0, st>>>(list, m, mix64(s), B.k0, B.v0));
  GP_LAUNCH_CHECK();
  bool in_tmp = false;
  Workspace sort_ws(st);
  GP_TRY(radix_sort_pairs(B.k0, B.v0, B.k1, B.v1, m, 64, &in_tmp, sort_ws));
  (count_launch(), k_todo_out<<<grid_of(m, 256), 256, 0, st>>>(in_tmp ? B.k1 : B.k0, in_tmp ? B.v1 : B.v0, m, todo));
  GP_LAUNCH_CHECK();
  return GP_OK;
}

}  // namespace

void mls_default_params(MlsParams *p) {
  p->global_iters = 3;
  p->alpha_pct = 10;
  p->max_local = 16;
  p->max_moves = 64;
  p->fruitless = 16;
  p->queue_cap = 256;
  p->max_degree = 1024;
}

int run_mls(const DGraph &g, int k, int64_t lmax, uint64_t seed, const MlsParams &p, int32_t *part, MlsStats *out,
            cudaStream_t s) {
  if (out) *out = MlsStats();
  if (g.n <= 0 || p.global_iters <= 0) return GP_OK;
  if (k > kMaxK || p.max_moves < 1 || p.max_moves > kMaxMoves || p.queue_cap < 1 || p.queue_cap > kQCap ||
      p.fruitless < 1 || p.max_degree < 0) {
    set_error("multi-try local search: k <= 256, 1 <= max_moves <= 64, 1 <= queue_cap <= 256, fruitless >= 1");
    return GP_ERR_UNSUPPORTED;
  }
  Workspace ws(s);
  const int64_t n = g.n;
  uint32_t *flags;
  int32_t *list, *todo, *len;
  int64_t *bw;
  unsigned long long *acc;  // gain, moves of a local iteration; boundary vertices of a global one
  int3 *seq;
  TodoBuffers tb;
  GP_TRY(ws.get(&flags, (size_t)n));
  GP_TRY(ws.get(&list, (size_t)n));
  GP_TRY(ws.get(&todo, (size_t)n));
  GP_TRY(ws.get(&len, (size_t)n));
  GP_TRY(ws.zeros(&bw, (size_t)k));
  GP_TRY(ws.get(&acc, 3));
  const int gn = grid_of(n, 256);
  (count_launch(), k_mls_block_weights<<<gn, 256, 0, s>>>(g, part, bw));
  GP_LAUNCH_CHECK();
  const int ew = g.ew_mode();
  MlsArgs A;
  A.g = g;
  A.part = part;
  A.bw = bw;
  A.k = k;
  A.lmax = lmax;
  A.max_moves = (int)p.max_moves;
  A.fruitless = (int)p.fruitless;
  A.queue_cap = (int)p.queue_cap;
  A.max_degree = (int)p.max_degree;
  A.conn_bytes = (unsigned)(ew == 0 ? conn_bytes<0>(g, k) : conn_bytes<1>(g, k));
  A.lane_conn = ew == 0 ? lane_conn<0>(g, k) : lane_conn<1>(g, k);
  const size_t smem = (sizeof(WarpState) + A.conn_bytes) * kMlsWarps;
  {
    const int most = (int)((sizeof(WarpState) + kConnMost) * kMlsWarps);
    const void *const kernel = ew == 0   ? (const void *)k_mls_search<0>
                               : ew == 1 ? (const void *)k_mls_search<1>
                                         : (const void *)k_mls_search<2>;
    int per_sm = 0;
    GP_TRY(kernel_blocks_per_sm(kernel, kMlsThreads, smem, most, &per_sm));
  }
  MlsStats st;
  size_t seq_cap = 0;
  for (int gi = 0; gi < p.global_iters; gi++) {
    uint64_t sl = hash3(seed, (uint64_t)gi, 5);
    GP_CUDA(cudaMemsetAsync(acc, 0, sizeof(unsigned long long) * 3, s));
    (count_launch(), k_boundary_list<<<gn, 256, 0, s>>>(g, part, (int)p.max_degree, list, acc + 2));
    GP_LAUNCH_CHECK();
    unsigned long long h[3];
    {
      Readback rb;
      rb.add(h, acc, sizeof(h));
      GP_TRY(rb.run(s));
    }
    int64_t m = (int64_t)h[2];
    GP_TRY(order_todo(list, m, n, sl, todo, tb, ws));
    int64_t total = 0;
    for (int li = 0; li < p.max_local && m > 0; li++) {
      if ((size_t)m * p.max_moves > seq_cap) {
        seq_cap = (size_t)m * p.max_moves;
        GP_TRY(ws.get(&seq, seq_cap));
      }
      A.smix = mix64(sl);
      const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((m + kMlsWarps - 1) / kMlsWarps,
                                                                    (int64_t)num_sms() * 8));
      {
        ProfScope ps("mls_search", s);
        if (ew == 0) (count_launch(), k_mls_search<0><<<grid, kMlsThreads, smem, s>>>(A, todo, m, seq, len));
        else if (ew == 1) (count_launch(), k_mls_search<1><<<grid, kMlsThreads, smem, s>>>(A, todo, m, seq, len));
        else (count_launch(), k_mls_search<2><<<grid, kMlsThreads, smem, s>>>(A, todo, m, seq, len));
        GP_LAUNCH_CHECK();
      }
      GP_CUDA(cudaMemsetAsync(flags, 0, sizeof(uint32_t) * (size_t)n, s));  // moved in this local iteration
      GP_CUDA(cudaMemsetAsync(acc, 0, sizeof(unsigned long long) * 2, s));
      {
        ProfScope ps("mls_apply", s);
        long long *out = reinterpret_cast<long long *>(acc);
        if (ew == 0) (count_launch(), k_mls_apply<0><<<1, kApplyThreads, 0, s>>>(g, part, bw, k, lmax, seq, len, m, (int)p.max_moves, flags, list, out));
        else if (ew == 1) (count_launch(), k_mls_apply<1><<<1, kApplyThreads, 0, s>>>(g, part, bw, k, lmax, seq, len, m, (int)p.max_moves, flags, list, out));
        else (count_launch(), k_mls_apply<2><<<1, kApplyThreads, 0, s>>>(g, part, bw, k, lmax, seq, len, m, (int)p.max_moves, flags, list, out));
        GP_LAUNCH_CHECK();
      }
      {
        Readback rb;
        rb.add(h, acc, sizeof(h));
        GP_TRY(rb.run(s));
      }
      st.searches += m;
      st.moves += (int64_t)h[1];
      st.local_iters += 1;
      const int64_t gain = (int64_t)h[0];
      const bool more = gain > 0 && 100 * gain > p.alpha_pct * total;
      total += gain;
      if (!more) break;
      sl = hash3(sl, (uint64_t)li + 1, 6);
      m = (int64_t)h[1];  // the moved vertices, which the application listed
      GP_TRY(order_todo(list, m, n, sl, todo, tb, ws));
    }
    st.gain += total;
  }
  if (out) *out = st;
  return GP_OK;
}

}  // namespace gp
