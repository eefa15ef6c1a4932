// ip.cu -- initial partitioning of the coarsest graph, evaluation, projection and degree-0 vertices.
//
// Initial partitioning (Section III-B, Section IV-B): the coarsest graph is partitioned several
// times independently and the best result is kept; each try is a recursive bisection into
// ceil(k/2) and floor(k/2) blocks. KaHIP's bisection with local search and flows is external to the
// paper; this library's bisection is deterministic: BFS from the vertex of minimum
// H(s_try, depth, v), a second BFS from the farthest vertex found (ties: smaller id), vertices
// ordered by (distance, id) with unreachable ones last, side 0 the shortest prefix whose weight
// reaches ceil(k/2)/k of the set. All sets of one recursion depth are split together (their BFS
// runs are one multi-source BFS restricted to each set), one CTA per try, tries in parallel.
// A balance repair then moves vertices out of overloaded blocks (Section II-A: a block is
// overloaded when heavier than Lmax).
// Projection (Section III-C): a fine vertex takes the block of its coarse representative.
#include <algorithm>
#include <climits>
#include <vector>

#include "block_sort.cuh"
#include "ip.cuh"
#include "lp.cuh"
#include "row_walk.cuh"

namespace gp {

namespace {

constexpr int kIpThreads = 1024;

// One graph of an initial-partitioning launch: a local view (offsets and vertex weights shifted to its
// first vertex; adjacency holds global ids, minus vbase gives local ids), its parameters and where its
// tries' partitions and scratch live.
struct IpGraph {
  DGraph g;
  int64_t vbase;
  int k;
  int level;
  int64_t lmax;
  uint64_t seed;
  int32_t *parts;     // tries * n
  int64_t ns;         // per-try stride of n-sized scratch: max(n, k)
  int64_t scr_off;    // offset of this graph's n-sized scratch (tries * ns)
  int64_t kscr_off;   // offset of this graph's k-sized scratch (tries * k)
  int64_t conn_off;   // offset of this graph's repair connection scratch (tries * kIpThreads * k)
};

struct IpArgs {
  const IpGraph *graphs;
  const int *block_graph;
  const int *block_try;
  int repair_rounds;
  int32_t *gk;               // n-sized scratch arrays
  int32_t *dist;
  int32_t *qa, *qb;
  unsigned long long *ka, *kb;
  int32_t *va, *vb;
  int32_t *mv_t;
  long long *mv_g;
  uint8_t *flag;
  int64_t smem_ns;           // > 0: the bisection keeps part, gk, dist and both BFS queues of every try
                             // in dynamic shared memory (every graph of the launch has ns <= smem_ns)
  int smem_sort;             // with smem_ns: the sort's key and value arrays are in shared memory too
  long long *gws;            // k-sized scratch arrays
  unsigned long long *gminh;
  int *gstart;
  unsigned long long *gfar;
  long long *bw;
  long long *conn;
  int *err;
};

// Multi-source BFS restricted to same-set vertices (part equal, set still being split). All sources start at
// distance 0 together, so a step finds the vertices of one distance. On graphs of long rows a frontier of more than an
// eighth of the vertices is taken from the other side: every vertex still without a distance looks for a neighbour in
// the frontier and stops at the first 32 entries that hold one, instead of every frontier vertex walking its whole row
// (on the coarsest level of an R-MAT graph, one CTA per try, the two or three large steps of each search: 8.6 -> 7.2
// ms). Rows of up to 32 entries cost a step from either side, and the frontier has the fewer of them. The distances
// are the same.
__device__ void set_bfs(const DGraph &g, int64_t vbase, int32_t *part, int32_t *gk, int32_t *dist, int32_t *qa,
                        int32_t *qb, int nf) {
  __shared__ int s_next;
  const int n = (int)g.n;
  const bool long_rows = g.row_begin(n) - g.row_begin(0) > 32 * (int64_t)n;
  for (int level = 0; nf > 0; level++) {
    if (threadIdx.x == 0) s_next = 0;
    __syncthreads();
    // one warp per frontier vertex, lanes over its row
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (long_rows && 8 * (int64_t)nf > n) {
      for (int u0 = wid * 32; u0 < n; u0 += nw * 32) {
        const int mine = u0 + lane;
        unsigned open = __ballot_sync(kFull, mine < n && gk[mine] > 1 && dist[mine] == -1);
        for (; open; open &= open - 1) {
          const int u = u0 + __ffs(open) - 1;
          const int pu = part[u];
          const int64_t b = g.row_begin(u), e = g.row_begin(u + 1);
          for (int64_t j = b; j < e; j += 32) {
            bool hit = false;
            if (j + lane < e) {
              const int x = (int)(g.adj[j + lane] - vbase);
              hit = *(volatile int32_t *)&dist[x] == level && part[x] == pu;
            }
            if (__any_sync(kFull, hit)) {  // (a vertex found in this step has distance level + 1)
              if (lane == 0) {
                dist[u] = level + 1;
                qb[atomicAdd(&s_next, 1)] = u;
              }
              break;
            }
          }
        }
      }
    } else for (int i = wid; i < nf; i += nw) {
      const int x = qa[i];
      const int px = part[x];
      const int dx = dist[x];
      const int64_t b = g.row_begin(x), e = g.row_begin(x + 1);
      for (int64_t j = b + lane; j < e; j += 32) {
        const int u = (int)(g.adj[j] - vbase);
        if (gk[u] <= 1 || part[u] != px) continue;
        if (atomicCAS(&dist[u], -1, dx + 1) == -1) qb[atomicAdd(&s_next, 1)] = u;
      }
    }
    __syncthreads();
    nf = s_next;
    int32_t *t = qa;
    qa = qb;
    qb = t;
    __syncthreads();
  }
}

// Per-vertex state of a bisection in shared memory: 5 arrays of ns int32 (part, gk, dist, qa, qb), and
// for ns <= kIpSmemSortNs also the sort's keys and values (2 x ns uint64 + 2 x ns int32) after them.
constexpr int64_t kIpSmemMaxNs = 8192;
constexpr int64_t kIpSmemSortNs = 4096;
constexpr size_t ip_state_bytes(int64_t ns) { return ((size_t)ns * 5 * sizeof(int32_t) + 15) & ~size_t(15); }
constexpr size_t ip_smem_bytes(int64_t ns, bool sort) {
  return ip_state_bytes(ns) + (sort ? (size_t)ns * (2 * sizeof(unsigned long long) + 2 * sizeof(int32_t)) : 0);
}

__global__ void __launch_bounds__(kIpThreads, 2) k_bisect(IpArgs a) {
  extern __shared__ __align__(16) unsigned char ip_dsm[];
  __shared__ BlockSortSmem sm;
  __shared__ int s_any, s_maxd;
  const IpGraph &G = a.graphs[a.block_graph[blockIdx.x]];
  const int t = a.block_try[blockIdx.x];
  const DGraph g = G.g;
  const int n = (int)g.n, k = G.k;
  const size_t ns = (size_t)G.ns;
  const size_t so = (size_t)G.scr_off + (size_t)t * ns, ko = (size_t)G.kscr_off + (size_t)t * k;
  int32_t *const part_out = G.parts + (size_t)t * n;
  int32_t *part = part_out, *gk = a.gk + so, *dist = a.dist + so;
  int32_t *qa = a.qa + so, *qb = a.qb + so;
  if (a.smem_ns > 0) {
    // small coarsest graphs: the BFS state lives in shared memory (the partition is copied out at
    // the end)
    int32_t *sp = reinterpret_cast<int32_t *>(ip_dsm);
    part = sp;
    gk = sp + ns;
    dist = sp + 2 * ns;
    qa = sp + 3 * ns;
    qb = sp + 4 * ns;
  }
  unsigned long long *ka = a.ka + so, *kb = a.kb + so;
  int32_t *va = a.va + so, *vb = a.vb + so;
  if (a.smem_sort) {
    unsigned char *sb = ip_dsm + ip_state_bytes((int64_t)ns);
    ka = reinterpret_cast<unsigned long long *>(sb);
    kb = ka + ns;
    va = reinterpret_cast<int32_t *>(kb + ns);
    vb = va + ns;
  }
  long long *gws = a.gws + ko;
  unsigned long long *gminh = a.gminh + ko, *gfar = a.gfar + ko;
  int *gstart = a.gstart + ko;
  const uint64_t s_try = hash3(G.seed, (uint64_t)G.level, (uint64_t)(4 + t));
  for (int v = threadIdx.x; v < n; v += blockDim.x) {
    part[v] = 0;
    gk[v] = k;
  }
  __syncthreads();
  for (int depth = 0; depth < 64; depth++) {
    if (threadIdx.x == 0) {
      s_any = 0;
      s_maxd = 0;
    }
    __syncthreads();
    for (int v = threadIdx.x; v < n; v += blockDim.x)
      if (gk[v] > 1) s_any = 1;
    __syncthreads();
    if (!s_any) break;
    for (int b = threadIdx.x; b < k; b += blockDim.x) {
      gws[b] = 0;
      gminh[b] = ~0ull;
      gstart[b] = INT_MAX;
      gfar[b] = 0;
    }
    __syncthreads();
    const uint64_t hd = mix64(mix64(s_try) ^ (uint64_t)depth);
    for (int v = threadIdx.x; v < n; v += blockDim.x) {
      if (gk[v] <= 1) continue;
      const int b = part[v];
      atomicAdd(reinterpret_cast<unsigned long long *>(&gws[b]), (unsigned long long)g.vweight(v));
      atomicMin(&gminh[b], (unsigned long long)mix64(hd ^ (uint64_t)v));
      dist[v] = -1;
    }
    __syncthreads();
    for (int v = threadIdx.x; v < n; v += blockDim.x) {
      if (gk[v] <= 1) continue;
      const int b = part[v];
      if (mix64(hd ^ (uint64_t)v) == gminh[b]) atomicMin(&gstart[b], v);
    }
    __syncthreads();
    // BFS 1 from the start vertex of every set
    int nf = block_compact(k, [&](int b) { return gstart[b] != INT_MAX; }, qa, sm);
    for (int i = threadIdx.x; i < nf; i += blockDim.x) {
      const int v = gstart[qa[i]];
      qa[i] = v;
      dist[v] = 0;
    }
    __syncthreads();
    set_bfs(g, G.vbase, part, gk, dist, qa, qb, nf);
    // farthest vertex per set, ties by smaller id
    for (int v = threadIdx.x; v < n; v += blockDim.x) {
      if (gk[v] <= 1 || dist[v] < 0) continue;
      atomicMax(&gfar[part[v]], ((unsigned long long)dist[v] << 32) | (unsigned long long)(0x7fffffff - v));
    }
    __syncthreads();
    for (int v = threadIdx.x; v < n; v += blockDim.x)
      if (gk[v] > 1) dist[v] = -1;
    __syncthreads();
    nf = block_compact(k, [&](int b) { return gfar[b] != 0; }, qa, sm);
    for (int i = threadIdx.x; i < nf; i += blockDim.x) {
      const int v = 0x7fffffff - (int)(gfar[qa[i]] & 0xffffffffull);
      qa[i] = v;
      dist[v] = 0;
    }
    __syncthreads();
    set_bfs(g, G.vbase, part, gk, dist, qa, qb, nf);
    // order the vertices of every set by (set, unreachable, distance), stable in id order
    const int na = block_compact(n, [&](int v) { return gk[v] > 1; }, va, sm);
    for (int i = threadIdx.x; i < na; i += blockDim.x) atomicMax(&s_maxd, dist[va[i]]);
    __syncthreads();
    const int db = bits_of((unsigned long long)s_maxd + 1);
    const int kbits = bits_of((unsigned long long)(k > 1 ? k - 1 : 0));
    for (int i = threadIdx.x; i < na; i += blockDim.x) {
      const int v = va[i];
      const int dv = dist[v];
      const unsigned long long unreach = dv < 0 ? 1ull : 0ull;
      ka[i] = ((unsigned long long)part[v] << (db + 1)) | (unreach << db) | (unsigned long long)(dv < 0 ? 0 : dv);
    }
    __syncthreads();
    const bool in_b = block_radix_sort(ka, va, kb, vb, na, kbits + db + 1, sm);
    unsigned long long *ks = in_b ? kb : ka;
    int32_t *vs = in_b ? vb : va;
    // side 0: shortest prefix of the set whose weight reaches ceil(kS/2)/kS of the set
    block_seg_scan(
        na, [&](int p) { return (int)(ks[p] >> (db + 1)); },
        [&](int p) { return g.vweight(vs[p]); },
        [&](int p, long long excl, long long) {
          const int v = vs[p];
          const int base = (int)(ks[p] >> (db + 1));
          const int kS = gk[v];
          const int k0 = (kS + 1) / 2, k1 = kS / 2;
          const __int128 lhs = (__int128)excl * kS, rhs = (__int128)gws[base] * k0;
          if (lhs < rhs) {
            gk[v] = k0;
          } else {
            part[v] = base + k0;
            gk[v] = k1;
          }
        },
        sm);
    __syncthreads();
  }
  if (a.smem_ns > 0) {
    __syncthreads();
    for (int v = threadIdx.x; v < n; v += blockDim.x) part_out[v] = part[v];
  }
}

// Balance repair (one CTA per try).
__global__ void __launch_bounds__(kIpThreads) k_repair(IpArgs a) {
  __shared__ BlockSortSmem sm;
  __shared__ int s_over, s_light, s_applied;
  __shared__ long long s_gmin, s_gmax;
  const IpGraph &G = a.graphs[a.block_graph[blockIdx.x]];
  const int t = a.block_try[blockIdx.x];
  const DGraph g = G.g;
  const int n = (int)g.n, k = G.k;
  const int64_t lmax = G.lmax, vbase = G.vbase;
  const size_t ns = (size_t)G.ns;
  const size_t so = (size_t)G.scr_off + (size_t)t * ns, ko = (size_t)G.kscr_off + (size_t)t * k;
  int32_t *part = G.parts + (size_t)t * n;
  unsigned long long *ka = a.ka + so, *kb = a.kb + so;
  int32_t *va = a.va + so, *vb = a.vb + so;
  int32_t *mv_t = a.mv_t + so;
  long long *mv_g = a.mv_g + so;
  uint8_t *flag = a.flag + so;
  int32_t *list2 = a.qa + so;
  long long *bw = a.bw + ko;
  long long *conn = a.conn + (size_t)G.conn_off + ((size_t)t * blockDim.x + threadIdx.x) * (size_t)k;
  const int kbits = bits_of((unsigned long long)(k > 1 ? k - 1 : 0));
  for (int b = 0; b < k; b++) conn[b] = 0;
  for (int rr = 0; rr < a.repair_rounds; rr++) {
    for (int b = threadIdx.x; b < k; b += blockDim.x) bw[b] = 0;
    __syncthreads();
    for (int v = threadIdx.x; v < n; v += blockDim.x)
      atomicAdd(reinterpret_cast<unsigned long long *>(&bw[part[v]]), (unsigned long long)g.vweight(v));
    __syncthreads();
    if (threadIdx.x == 0) {
      int over = 0, light = 0;
      for (int b = 0; b < k; b++) {
        if (bw[b] > lmax) over = 1;
        if (bw[b] < bw[light]) light = b;
      }
      s_over = over;
      s_light = light;
      s_applied = 0;
      s_gmin = LLONG_MAX;
      s_gmax = LLONG_MIN;
    }
    __syncthreads();
    if (!s_over) break;
    // per vertex of an overloaded block: target and gain
    for (int v = threadIdx.x; v < n; v += blockDim.x) {
      mv_t[v] = -1;
      const int P = part[v];
      if (bw[P] <= lmax) continue;
      const long long cv = g.vweight(v);
      const int64_t b = g.row_begin(v), e = g.row_begin(v + 1);
      for (int64_t j = b; j < e; j++) conn[part[g.adj[j] - vbase]] += g.eweight(j);
      int best = -1;
      for (int64_t j = b; j < e; j++) {
        const int B = part[g.adj[j] - vbase];
        if (B == P || conn[B] <= 0 || bw[B] + cv > lmax) continue;
        if (best < 0 || conn[B] > conn[best] || (conn[B] == conn[best] && B < best)) best = B;
      }
      if (best < 0 && s_light != P && bw[s_light] + cv <= lmax) best = s_light;
      if (best >= 0) {
        mv_t[v] = best;
        mv_g[v] = conn[best] - conn[P];
        atomicMin(&s_gmin, mv_g[v]);
        atomicMax(&s_gmax, mv_g[v]);
      }
      for (int64_t j = b; j < e; j++) conn[part[g.adj[j] - vbase]] = 0;
    }
    __syncthreads();
    const int nm = block_compact(n, [&](int v) { return mv_t[v] >= 0; }, va, sm);
    if (nm == 0) break;
    const unsigned long long grange = (unsigned long long)(s_gmax - s_gmin);
    const int gb = bits_of(grange);
    if (kbits + gb > 64) {
      if (threadIdx.x == 0) atomicExch(a.err, GP_ERR_UNSUPPORTED);
      return;
    }
    // per target: (gain desc, id asc) -- input is in id order, the sort is stable
    for (int i = threadIdx.x; i < nm; i += blockDim.x) {
      const int v = va[i];
      ka[i] = ((unsigned long long)mv_t[v] << gb) | (unsigned long long)(s_gmax - mv_g[v]);
    }
    __syncthreads();
    bool in_b = block_radix_sort(ka, va, kb, vb, nm, kbits + gb, sm);
    unsigned long long *ks = in_b ? kb : ka;
    int32_t *vs = in_b ? vb : va;
    for (int v = threadIdx.x; v < n; v += blockDim.x) flag[v] = 0;
    __syncthreads();
    block_seg_scan(
        nm, [&](int p) { return (int)(ks[p] >> gb); }, [&](int p) { return g.vweight(vs[p]); },
        [&](int p, long long, long long incl) {
          const int v = vs[p];
          if (bw[mv_t[v]] + incl <= lmax) flag[v] = 1;
        },
        sm);
    __syncthreads();
    // per source: take movers while the source is still overloaded
    const int na = block_compact(n, [&](int v) { return flag[v] != 0; }, list2, sm);
    for (int i = threadIdx.x; i < na; i += blockDim.x) {
      const int v = list2[i];
      ka[i] = ((unsigned long long)part[v] << gb) | (unsigned long long)(s_gmax - mv_g[v]);
      va[i] = v;
    }
    __syncthreads();
    in_b = block_radix_sort(ka, va, kb, vb, na, kbits + gb, sm);
    ks = in_b ? kb : ka;
    vs = in_b ? vb : va;
    block_seg_scan(
        na, [&](int p) { return (int)(ks[p] >> gb); }, [&](int p) { return g.vweight(vs[p]); },
        [&](int p, long long excl, long long) {
          const int v = vs[p];
          const int P = (int)(ks[p] >> gb);
          flag[v] = (bw[P] - excl > lmax) ? 2 : 0;
        },
        sm);
    __syncthreads();
    for (int v = threadIdx.x; v < n; v += blockDim.x)
      if (flag[v] == 2) {
        part[v] = mv_t[v];
        s_applied = 1;
      }
    __syncthreads();
    if (!s_applied) break;
  }
}

// Doubled cuts of up to T partitions of g (parts: one after another, g.n each): acc[t] += weight of each entry whose
// ends lie in different blocks of partition t. The adjacency is read once for all of them, in segments, so that the
// rows of millions of entries that power-law graphs have do not decide the time (128 M entries: 1.27 ms, a pass over
// the adjacency and its weights takes 0.2 ms; the parts gathered by neighbour bound it. The tries' cuts on R-MAT 22's
// coarsest graph, a vertex per thread and a launch per try: 2.2 ms; so: 0.02 ms).
template <int T>
__global__ void __launch_bounds__(256) k_cut(DGraph g, int seg, const int32_t *parts, int tries,
                                             unsigned long long *acc) {
  __shared__ unsigned long long s_acc[T];
  if (threadIdx.x < T) s_acc[threadIdx.x] = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int64_t m = min(g.m, g.row_begin(g.n)), nseg = (m + seg - 1) / seg;
  const int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5, nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  unsigned long long c[T];
#pragma unroll
  for (int t = 0; t < T; t++) c[t] = 0;
  for (int64_t sg = gw; sg < nseg; sg += nw) {
    const int64_t s1 = min(m, (sg + 1) * seg);
    RowWindow W;
    W.load(g, warp_row_of(g, sg * seg));
    for (int64_t e = sg * seg; e < s1;) {
      int64_t beg, end;
      const int64_t v = W.seek(g, e, &beg, &end);
      const int64_t stop = min(end, s1);
      for (int64_t x = e + lane; x < stop; x += 32) {
        const int a = __ldg(g.adj + x);
        const unsigned long long w = (unsigned long long)g.eweight(x);
#pragma unroll
        for (int t = 0; t < T; t++) {
          if (T > 1 && t >= tries) break;
          const int32_t *p = parts + (size_t)t * g.n;
          if (p[a] != p[v]) c[t] += w;
        }
      }
      e = stop;
    }
  }
#pragma unroll
  for (int t = 0; t < T; t++) {
    const unsigned long long x = (unsigned long long)warp_sum64((int64_t)c[t]);
    if (lane == 0 && x) atomicAdd(&s_acc[t], x);
  }
  __syncthreads();
  if (threadIdx.x < T && s_acc[threadIdx.x]) atomicAdd(&acc[threadIdx.x], s_acc[threadIdx.x]);
}

__global__ void k_project(const int32_t *coarse, const int32_t *f2c, int64_t n, int32_t *fine) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
    fine[v] = coarse[f2c[v]];
}

__global__ void k_vw_stats(DGraph g, unsigned long long *mx, unsigned long long *sum) {
  unsigned long long m = 0, s = 0;
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < g.n; v += (int64_t)gridDim.x * blockDim.x) {
    const unsigned long long c = (unsigned long long)g.vweight(v);
    m = max(m, c);
    s += c;
  }
  for (int o = 16; o > 0; o >>= 1) {
    m = max(m, __shfl_xor_sync(kFull, m, o));
    s += __shfl_xor_sync(kFull, s, o);
  }
  if ((threadIdx.x & 31) == 0) {
    atomicMax(mx, m);
    atomicAdd(sum, s);
  }
}

// Keep flags (degree > 0).
__global__ void k_deg_flags(DGraph g, uint32_t *keep) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < g.n; v += (int64_t)gridDim.x * blockDim.x)
    keep[v] = g.row_begin(v + 1) - g.row_begin(v) > 0 ? 1u : 0u;
}

// Degree-0 vertices own no CSR entries, so the kept vertices' rows keep their entries in the same
// order: the stripped offsets are the kept vertices' offsets, the stripped adjacency is the renamed
// adjacency and the edge weights are unchanged.
__global__ void k_strip_rows(DGraph g, const int32_t *rank, const uint32_t *keep, int64_t n0, int64_t *off0,
                             void *vw0) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < g.n; v += (int64_t)gridDim.x * blockDim.x) {
    if (!keep[v]) continue;
    const int r = rank[v];
    off0[r] = g.row_begin(v);
    if (vw0) {
      if (g.vw64) static_cast<int64_t *>(vw0)[r] = static_cast<const int64_t *>(g.vw)[v];
      else static_cast<int32_t *>(vw0)[r] = static_cast<const int32_t *>(g.vw)[v];
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) off0[n0] = g.row_begin(g.n);
}

__global__ void k_strip_adj(const int32_t *adj, int64_t m, const int32_t *rank, int32_t *adj0) {
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < m; j += (int64_t)gridDim.x * blockDim.x)
    adj0[j] = rank[adj[j]];
}

// Degree-0 vertex placement with unit weights, closed form of the greedy rule: at water level x
// every block of weight <= x receives one vertex, blocks in id order. F(x) = sum_b max(0, x - bw_b)
// vertices are placed before level x; vertex j (0-based, ascending id) is placed at the level x with
// F(x) <= j < F(x+1), into the (j - F(x))-th block (by id) among those with bw_b <= x. With the block weights sorted
// (in shared memory, k <= kPlaceK) and their prefix sums, the c lowest blocks are the ones below level x and
// F(x) = c x - prefix(c): a search for c replaces a search for x over sums of k terms (2 M vertices, k = 64:
// 2.0 -> 0.15 ms).
constexpr int kPlaceK = 1024;

__global__ void __launch_bounds__(256) k_place_unit(DGraph g, const int32_t *rank, const int32_t *part0,
                                                    const int64_t *iso_idx, const long long *bw, int k,
                                                    int32_t *part_full) {
  __shared__ long long s_bw[kPlaceK], s_sorted[kPlaceK], s_pre[kPlaceK + 1];
  for (int b = threadIdx.x; b < k; b += blockDim.x) s_bw[b] = bw[b];
  __syncthreads();
  for (int b = threadIdx.x; b < k; b += blockDim.x) {
    int at = 0;
    for (int x = 0; x < k; x++) at += s_bw[x] < s_bw[b] || (s_bw[x] == s_bw[b] && x < b);
    s_sorted[at] = s_bw[b];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    long long run = 0;
    for (int b = 0; b < k; b++) {
      s_pre[b] = run;
      run += s_sorted[b];
    }
    s_pre[k] = run;
  }
  __syncthreads();
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < g.n; v += (int64_t)gridDim.x * blockDim.x) {
    const int r = rank[v];
    if (r >= 0) {
      part_full[v] = part0[r];
      continue;
    }
    const long long j = iso_idx[v];
    int lo = 0, hi = k;  // the largest c with F(sorted[c]) <= j
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (mid * s_sorted[mid] - s_pre[mid] <= j) lo = mid;
      else hi = mid;
    }
    const int c = lo + 1;
    const long long x = (j + s_pre[c]) / c;
    long long rem = j - (c * x - s_pre[c]);
    int pick = (int)rem;
    if (c < k) {
      for (pick = 0; pick < k; pick++) {
        if (s_bw[pick] <= x && rem-- == 0) break;
      }
    }
    part_full[v] = pick;
  }
}

// The same for any k, searching the level by sums over the blocks.
__global__ void k_place_unit_any(DGraph g, const int32_t *rank, const int32_t *part0, const int64_t *iso_idx,
                                 const long long *bw, int64_t k, int32_t *part_full) {
  long long bmin = LLONG_MAX;
  for (int64_t b = 0; b < k; b++) bmin = min(bmin, bw[b]);
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < g.n; v += (int64_t)gridDim.x * blockDim.x) {
    const int r = rank[v];
    if (r >= 0) {
      part_full[v] = part0[r];
      continue;
    }
    const long long j = iso_idx[v];
    long long lo = bmin, hi = bmin + j + 1;  // F(lo) = 0 <= j; F(hi) > j
    auto F = [&](long long x) {
      long long s = 0;
      for (int64_t b = 0; b < k; b++) s += x > bw[b] ? x - bw[b] : 0;
      return s;
    };
    while (hi - lo > 1) {
      const long long mid = lo + (hi - lo) / 2;
      if (F(mid) <= j) lo = mid;
      else hi = mid;
    }
    long long rem = j - F(lo);
    int pick = 0;
    for (int64_t b = 0; b < k; b++)
      if (bw[b] <= lo) {
        if (rem == 0) {
          pick = (int)b;
          break;
        }
        rem--;
      }
    part_full[v] = pick;
  }
}

// Degree-0 vertices with general weights, part 1: kept vertices take their blocks, the others are listed in id order.
__global__ void k_place_list(DGraph g, const int32_t *rank, const int32_t *part0, const int64_t *iso_idx, int32_t *iso,
                             int32_t *part_full) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < g.n; v += (int64_t)gridDim.x * blockDim.x) {
    const int r = rank[v];
    if (r >= 0) part_full[v] = part0[r];
    else iso[iso_idx[v]] = (int32_t)v;
  }
}

// Part 2: one warp applies the greedy rule in id order. Lane l owns the blocks l, l + 32, ... and keeps the lightest
// of them; a vertex costs one warp minimum (a thread going through all blocks took about a microsecond).
__global__ void k_place_seq(DGraph g, const int32_t *iso, int64_t n_iso, long long *bw, int64_t k, int32_t *part_full) {
  const int lane = threadIdx.x;
  auto lightest = [&](long long *w) {
    int best = -1;
    long long bwt = LLONG_MAX;
    for (int64_t b = lane; b < k; b += 32) {
      const long long x = bw[b];
      if (best < 0 || x < bwt) {
        bwt = x;
        best = (int)b;
      }
    }
    *w = bwt;
    return best;
  };
  long long w;
  int b = lightest(&w);
  for (int64_t i0 = 0; i0 < n_iso; i0 += 32) {
    const int v = i0 + lane < n_iso ? iso[i0 + lane] : 0;
    const long long c = i0 + lane < n_iso ? g.vweight(v) : 0;
    const int cnt = (int)min((int64_t)32, n_iso - i0);
    int mine = 0;
    for (int y = 0; y < cnt; y++) {
      const long long cy = __shfl_sync(kFull, c, y);
      long long wm = b >= 0 ? w : LLONG_MAX;
      int bm = b >= 0 ? b : INT_MAX;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const long long w2 = __shfl_xor_sync(kFull, wm, o);
        const int b2 = __shfl_xor_sync(kFull, bm, o);
        if (w2 < wm || (w2 == wm && b2 < bm)) {
          wm = w2;
          bm = b2;
        }
      }
      if (lane == y) mine = bm;
      if (b == bm) {
        bw[b] = wm + cy;
        b = lightest(&w);
      }
    }
    if (lane < cnt) part_full[v] = mine;
  }
}

// rank_out[v] = rank[v] for vertices with neighbours, -1 otherwise; iso_idx[v] = v - rank[v]
// (the number of degree-0 vertices before v, since rank counts the kept vertices before v).
__global__ void k_mark_rank(DGraph g, const int32_t *rank, int32_t *rank_out, int64_t *iso_idx) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < g.n; v += (int64_t)gridDim.x * blockDim.x) {
    const int64_t d = g.row_begin(v + 1) - g.row_begin(v);
    rank_out[v] = d > 0 ? rank[v] : -1;
    iso_idx[v] = v - rank[v];
  }
}

int grid_for_n(int64_t n) {
  return (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, (int64_t)num_sms() * 8));
}

}  // namespace

int initial_partition_multi(const IpJob *jobs, int njobs, int tries, int repair_rounds, cudaStream_t s,
                            int *err_dev) {
  if (njobs <= 0) return GP_OK;
  Workspace ws(s);
  std::vector<IpGraph> hg(njobs);
  std::vector<int> bgraph, btry;
  int64_t scr = 0, kscr = 0, cscr = 0;
  for (int j = 0; j < njobs; j++) {
    const IpJob &jb = jobs[j];
    if (jb.g.n >= (1 << 30)) {
      set_error("initial partitioning supports coarsest graphs below 2^30 vertices");
      return GP_ERR_UNSUPPORTED;
    }
    IpGraph &G = hg[j];
    G.g = jb.g;
    G.vbase = jb.vbase;
    G.k = jb.k;
    G.level = jb.level;
    G.lmax = jb.lmax;
    G.seed = jb.seed;
    G.parts = jb.parts;
    G.ns = std::max<int64_t>(std::max<int64_t>(jb.g.n, jb.k), 1);
    G.scr_off = scr;
    G.kscr_off = kscr;
    G.conn_off = cscr;
    scr += (int64_t)tries * G.ns;
    kscr += (int64_t)tries * jb.k;
    cscr += (int64_t)tries * kIpThreads * jb.k;
    for (int t = 0; t < tries; t++) {
      bgraph.push_back(j);
      btry.push_back(t);
    }
  }
  IpArgs a;
  a.repair_rounds = repair_rounds;
  GP_TRY(ws.get(&a.gk, (size_t)scr));
  GP_TRY(ws.get(&a.dist, (size_t)scr));
  GP_TRY(ws.get(&a.qa, (size_t)scr));
  GP_TRY(ws.get(&a.qb, (size_t)scr));
  GP_TRY(ws.get(&a.ka, (size_t)scr));
  GP_TRY(ws.get(&a.kb, (size_t)scr));
  GP_TRY(ws.get(&a.va, (size_t)scr));
  GP_TRY(ws.get(&a.vb, (size_t)scr));
  GP_TRY(ws.get(&a.mv_t, (size_t)scr));
  GP_TRY(ws.get(&a.mv_g, (size_t)scr));
  GP_TRY(ws.get(&a.flag, (size_t)scr));
  GP_TRY(ws.get(&a.gws, (size_t)kscr));
  GP_TRY(ws.get(&a.gminh, (size_t)kscr));
  GP_TRY(ws.get(&a.gstart, (size_t)kscr));
  GP_TRY(ws.get(&a.gfar, (size_t)kscr));
  GP_TRY(ws.get(&a.bw, (size_t)kscr));
  GP_TRY(ws.get(&a.conn, (size_t)cscr));
  GP_TRY(ws.zeros(&a.err, 1));
  IpGraph *graphs_dev;
  int *bg_dev, *bt_dev;
  GP_TRY(ws.get(&graphs_dev, hg.size()));
  GP_TRY(ws.get(&bg_dev, bgraph.size()));
  GP_TRY(ws.get(&bt_dev, btry.size()));
  GP_CUDA(cudaMemcpyAsync(graphs_dev, hg.data(), sizeof(IpGraph) * hg.size(), cudaMemcpyHostToDevice, s));
  GP_CUDA(cudaMemcpyAsync(bg_dev, bgraph.data(), sizeof(int) * bgraph.size(), cudaMemcpyHostToDevice, s));
  GP_CUDA(cudaMemcpyAsync(bt_dev, btry.data(), sizeof(int) * btry.size(), cudaMemcpyHostToDevice, s));
  a.graphs = graphs_dev;
  a.block_graph = bg_dev;
  a.block_try = bt_dev;
  const int grid = (int)bgraph.size();
  int64_t max_ns = 0;
  for (const IpGraph &G : hg) max_ns = std::max<int64_t>(max_ns, G.ns);
  a.smem_ns = max_ns <= kIpSmemMaxNs ? max_ns : 0;
  a.smem_sort = max_ns <= kIpSmemSortNs ? 1 : 0;
  const size_t dsm = a.smem_ns > 0 ? ip_smem_bytes(a.smem_ns, a.smem_sort != 0) : 0;
  if (dsm > 0) {  // (per call: the attribute belongs to the current device)
    const size_t cap = std::max(ip_smem_bytes(kIpSmemMaxNs, false), ip_smem_bytes(kIpSmemSortNs, true));
    GP_CUDA(cudaFuncSetAttribute(k_bisect, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cap));
  }
  (::gp::count_launch(), k_bisect<<<grid, kIpThreads, dsm, s>>>(a));
  GP_LAUNCH_CHECK();
  (::gp::count_launch(), k_repair<<<grid, kIpThreads, 0, s>>>(a));
  GP_LAUNCH_CHECK();
  if (err_dev) {
    GP_CUDA(cudaMemcpyAsync(err_dev, a.err, sizeof(int), cudaMemcpyDeviceToDevice, s));
    return GP_OK;
  }
  int err = 0;
  GP_CUDA(cudaMemcpyAsync(&err, a.err, sizeof(int), cudaMemcpyDeviceToHost, s));
  GP_CUDA(cudaStreamSynchronize(s));
  if (err) {
    set_error("initial partitioning: gain range too wide for the repair sort keys");
    return err;
  }
  return GP_OK;
}

int initial_partition(const DGraph &g, int k, int64_t lmax, uint64_t seed, int level, int tries, int repair_rounds,
                      int32_t *parts, cudaStream_t s, int *err_dev) {
  IpJob j;
  j.g = g;
  j.vbase = 0;
  j.k = k;
  j.lmax = lmax;
  j.seed = seed;
  j.level = level;
  j.parts = parts;
  return initial_partition_multi(&j, 1, tries, repair_rounds, s, err_dev);
}

int cuts_launch(const DGraph &g, const int32_t *parts, int tries, unsigned long long *acc_dev, cudaStream_t s) {
  GP_CUDA(cudaMemsetAsync(acc_dev, 0, sizeof(unsigned long long) * (size_t)tries, s));
  if (g.n == 0 || g.m == 0) return GP_OK;
  const int seg = row_segment(g.m);
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(((g.m + seg - 1) / seg + 7) / 8, (int64_t)num_sms() * 8));
  auto run = [&](auto kernel) { (::gp::count_launch(), kernel<<<grid, 256, 0, s>>>(g, seg, parts, tries, acc_dev)); };
  if (tries == 1) run(k_cut<1>);
  else if (tries <= 4) run(k_cut<4>);
  else run(k_cut<16>);
  GP_LAUNCH_CHECK();
  return GP_OK;
}

int eval_cut_launch(const DGraph &g, const int32_t *part, int64_t k, unsigned long long *acc_dev, int64_t *bw_dev,
                    cudaStream_t s) {
  GP_TRY(cuts_launch(g, part, 1, acc_dev, s));
  if (bw_dev) GP_TRY(block_weights(g, part, k, bw_dev, nullptr, s));
  return GP_OK;
}

int eval_cut(const DGraph &g, const int32_t *part, int64_t k, int64_t *cut_host, int64_t *bw_dev, cudaStream_t s) {
  Workspace ws(s);
  unsigned long long *acc;
  GP_TRY(ws.get(&acc, 1));
  GP_TRY(eval_cut_launch(g, part, k, acc, bw_dev, s));
  unsigned long long h = 0;
  GP_CUDA(cudaMemcpyAsync(&h, acc, sizeof(h), cudaMemcpyDeviceToHost, s));
  GP_CUDA(cudaStreamSynchronize(s));
  *cut_host = (int64_t)(h / 2);
  return GP_OK;
}

int project(const int32_t *coarse, const int32_t *f2c, int64_t n, int32_t *fine, cudaStream_t s) {
  if (n == 0) return GP_OK;
  (::gp::count_launch(), k_project<<<grid_for_n(n), 256, 0, s>>>(coarse, f2c, n, fine));
  GP_LAUNCH_CHECK();
  return GP_OK;
}

int vertex_weight_stats(const DGraph &g, int64_t *maxc, int64_t *total, cudaStream_t s) {
  Workspace ws(s);
  unsigned long long *d;
  GP_TRY(ws.zeros(&d, 2));
  if (g.n > 0) {
    (::gp::count_launch(), k_vw_stats<<<grid_for_n(g.n), 256, 0, s>>>(g, d, d + 1));
    GP_LAUNCH_CHECK();
  }
  unsigned long long h[2];
  GP_CUDA(cudaMemcpyAsync(h, d, sizeof(h), cudaMemcpyDeviceToHost, s));
  GP_CUDA(cudaStreamSynchronize(s));
  if (maxc) *maxc = (int64_t)h[0];
  if (total) *total = (int64_t)h[1];
  return GP_OK;
}

int strip_isolated(const DGraph &g, Stripped *out, Workspace &ws, cudaStream_t s, int64_t *W_out,
                   int64_t *maxc_kept_out, const LpConfig *cfg, LpClassInfo *cls) {
  out->g0 = g;
  out->n0 = g.n;
  out->n_iso = 0;
  out->rank = nullptr;
  if (W_out) *W_out = 0;
  if (maxc_kept_out) *maxc_kept_out = 0;
  if (g.n == 0) return GP_OK;
  // one kernel and one read back for the degree classes (valid for the level-0 graph when no vertex is stripped), the
  // kept vertices and the weights
  unsigned long long *words, hw[kLpStatWords];
  GP_TRY(ws.get(&words, (size_t)kLpStatWords));
  GP_TRY(lp_stats_launch(g, cfg ? *cfg : LpConfig(), words, s));
  {
    Readback rb;
    rb.add(hw, words, sizeof(hw));
    GP_TRY(rb.run(s));
  }
  const int64_t n0 = (int64_t)hw[kStatKept];
  if (maxc_kept_out) *maxc_kept_out = (int64_t)hw[kStatMaxKept];
  if (W_out) *W_out = (int64_t)hw[kStatTotal];
  if (cfg && cls && n0 == g.n) lp_classes_from(hw, *cfg, cls);
  if (n0 == g.n) return GP_OK;
  uint32_t *keep;
  int32_t *rank;
  GP_TRY(ws.get(&keep, (size_t)g.n));
  GP_TRY(ws.get(&rank, (size_t)g.n));
  (::gp::count_launch(), k_deg_flags<<<grid_for_n(g.n), 256, 0, s>>>(g, keep));
  GP_LAUNCH_CHECK();
  GP_TRY(scan_excl_u32(keep, rank, g.n, nullptr, ws));
  out->n0 = n0;
  out->n_iso = g.n - n0;
  out->rank = rank;
  // rank of kept vertices = exclusive count of kept before v; degree-0 ones are marked -1 later
  int64_t *off0;
  GP_TRY(ws.get(&off0, (size_t)n0 + 1));
  void *vw0 = nullptr;
  if (g.vw) {
    if (g.vw64) {
      int64_t *p;
      GP_TRY(ws.get(&p, (size_t)std::max<int64_t>(n0, 1)));
      vw0 = p;
    } else {
      int32_t *p;
      GP_TRY(ws.get(&p, (size_t)std::max<int64_t>(n0, 1)));
      vw0 = p;
    }
  }
  int32_t *adj0;
  GP_TRY(ws.get(&adj0, (size_t)std::max<int64_t>(g.m, 1)));
  (::gp::count_launch(), k_strip_rows<<<grid_for_n(g.n), 256, 0, s>>>(g, rank, keep, n0, off0, vw0));
  if (g.m > 0) (::gp::count_launch(), k_strip_adj<<<grid_for_n(g.m), 256, 0, s>>>(g.adj, g.m, rank, adj0));
  GP_LAUNCH_CHECK();
  DGraph d;
  d.n = n0;
  d.m = g.m;
  d.off = off0;
  d.off64 = 1;
  d.adj = adj0;
  d.vw = vw0;
  d.vw64 = g.vw64;
  d.ew = g.ew;  // same entries in the same order
  d.ew64 = g.ew64;
  out->g0 = d;
  return GP_OK;
}

int place_isolated(const DGraph &g, const Stripped &st, const int32_t *part0, int64_t k, int32_t *part_full,
                   cudaStream_t s) {
  Workspace ws(s);
  if (st.n_iso == 0) {
    if (g.n) GP_CUDA(cudaMemcpyAsync(part_full, part0, sizeof(int32_t) * (size_t)g.n, cudaMemcpyDeviceToDevice, s));
    return GP_OK;
  }
  // block weights of the kept vertices
  long long *bw;
  GP_TRY(ws.zeros(&bw, (size_t)k));
  GP_TRY(block_weights(st.g0, part0, k, reinterpret_cast<int64_t *>(bw), nullptr, s));
  // rank[v] becomes -1 for degree-0 vertices; iso_idx[v] = number of degree-0 vertices before v
  int32_t *rank;
  int64_t *iso_idx;
  GP_TRY(ws.get(&rank, (size_t)g.n));
  GP_TRY(ws.get(&iso_idx, (size_t)g.n));
  (::gp::count_launch(), k_mark_rank<<<grid_for_n(g.n), 256, 0, s>>>(g, st.rank, rank, iso_idx));
  GP_LAUNCH_CHECK();
  if (!g.vw && k <= kPlaceK) {
    (::gp::count_launch(), k_place_unit<<<grid_for_n(g.n), 256, 0, s>>>(g, rank, part0, iso_idx, bw, (int)k, part_full));
  } else if (!g.vw) {
    (::gp::count_launch(), k_place_unit_any<<<grid_for_n(g.n), 256, 0, s>>>(g, rank, part0, iso_idx, bw, k, part_full));
  } else {
    int32_t *iso;
    GP_TRY(ws.get(&iso, (size_t)st.n_iso));
    (::gp::count_launch(), k_place_list<<<grid_for_n(g.n), 256, 0, s>>>(g, rank, part0, iso_idx, iso, part_full));
    (::gp::count_launch(), k_place_seq<<<1, 32, 0, s>>>(g, iso, st.n_iso, bw, k, part_full));
  }
  GP_LAUNCH_CHECK();
  return GP_OK;
}

}  // namespace gp
