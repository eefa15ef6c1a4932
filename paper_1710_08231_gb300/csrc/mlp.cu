// mlp.cu -- learned edge scorer: per-edge features, BF16 tensor-core inference, training kernels.
//
// The paper has no learned component. This scorer guides label propagation during coarsening: its
// quantised score q = round-half-even(s * 2^15) of each CSR entry breaks ties between equally
// connected labels (larger score sum first) and orders admission after the gain.
//
// Features of entry (v,u), symmetric in v and u:
//   0 log2(1 + min(d(v), d(u)))        1 log2(1 + max(d(v), d(u)))
//   2 log2(1 + omega(v,u))             3 log2(1 + min(c(v), c(u)))
//   4 log2(1 + max(c(v), c(u)))
//   5 |first64(N(v)) intersect first64(N(u))| / 64
//   6 omega(v,u) / max(wdeg(v), wdeg(u))
//   7 level / 16
// Network: h = relu(W1 x + b1) (32 hidden), s = sigmoid(w2 . h + b2). Inference multiplies BF16
// features by BF16 W1 on the tensor cores (mma.sync m16n8k16, FP32 accumulation), rounds the hidden
// activations to BF16 and finishes the second layer in FP32. Training runs full-batch Adam on FP32
// master weights; its forward pass uses the BF16-rounded weights that inference uses.
#include <cuda_bf16.h>

#include <algorithm>
#include <cstring>
#include <vector>

#include "mlp.cuh"
#include "row_walk.cuh"

namespace gp {

namespace {

constexpr int kIn = 8, kHid = 32, kParams = kHid * kIn + kHid + kHid + 1;  // 321

__device__ __forceinline__ int64_t gp_min64(int64_t a, int64_t b) { return a < b ? a : b; }

__device__ __forceinline__ float bf16_to_float(uint16_t b) {
  return __uint_as_float(((unsigned)b) << 16);
}

__device__ __forceinline__ uint16_t float_to_bf16(float f) {
  const __nv_bfloat16 h = __float2bfloat16_rn(f);
  return *reinterpret_cast<const uint16_t *>(&h);
}

__device__ __forceinline__ unsigned pack2(uint16_t lo, uint16_t hi) { return (unsigned)lo | ((unsigned)hi << 16); }

// Weighted degrees (graphs with edge weights; without, the degree serves). Exact integer sums: a row
// inside one segment is stored, the parts of a row that spans segments are added (wsum is zero on entry).
__global__ void __launch_bounds__(256) k_wdeg(DGraph g, int seg, unsigned long long *wsum) {
  const int lane = threadIdx.x & 31;
  const int64_t m = gp_min64(g.m, g.row_begin(g.n)), nseg = (m + seg - 1) / seg;
  const int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t sg = gw; sg < nseg; sg += nw) {
    const int64_t s1 = gp_min64(m, (sg + 1) * seg);
    RowWindow W;
    W.load(g, warp_row_of(g, sg * seg));
    for (int64_t e = sg * seg; e < s1;) {
      int64_t beg, end;
      const int64_t v = W.seek(g, e, &beg, &end);
      const int64_t stop = gp_min64(end, s1);
      long long s = 0;
      for (int64_t x = e + lane; x < stop; x += 32) s += g.eweight(x);
      s = warp_sum64(s);
      if (lane == 0) {
        if (beg >= sg * seg && end <= s1) wsum[v] = (unsigned long long)s;
        else atomicAdd(&wsum[v], (unsigned long long)s);
      }
      e = stop;
    }
  }
}

__device__ __forceinline__ void mma_16816(float c[4], const unsigned a[4], const unsigned b[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// Features of every entry (SCORE false: written as floats) or their scores (SCORE true: the features go
// straight into the network and never to memory).
//
// What bounds it: the shared-neighbour counts look up to 64 neighbours of u up for every entry (v,u), from
// rows scattered over the adjacency. A warp takes a segment of entries; for each of its rows the set of
// v's first 64 neighbours is a table in the warp's shared memory (kTab slots and no probing: the keys whose
// slot was taken, two on average for a full set, are compared one by one), and lane l owns one entry of 32.
// The neighbours of two entries are looked up together, each by a half-warp that reads them contiguously, up
// to 64 per entry, with the loads of four entries issued before the first lookup. Half-warps serve short
// lists (mesh rows of 12 entries take one step) and long ones (four steps) alike. A lane per entry, walking its list alone, read 32 separate rows per load and
// waited for the warp's longest list and probe: 22.4 ms a call on an R-MAT graph of scale 19 with edge
// weights (15.5 M entries) against 2.1 ms now, at the same bits.
//
// Scores: the entries of a segment are staged in shared memory and scored 32 at a time, whatever rows they lie
// in (a step per row left most lanes of the network idle on meshes: a grid of 2000 x 2000 took 3.81 ms a call
// so, 2.97 now, R-MAT 19 2.57 and 2.13). 16 entries per tensor-core step, A = 16 entries x 16 features (8
// used, 8 zero), B = W1^T in four 16x8 slices (32 hidden units). Thread (g = lane/4, t = lane%4) holds features 2t, 2t+1 of rows g and
// g+8, and C elements (rows g, g+8; hidden units 8nb + 2t, 8nb + 2t + 1).
constexpr int kTab = 1024;
constexpr int kEdgeWarps = 8;
__device__ __forceinline__ unsigned tab_slot(int x) { return ((unsigned)x * 0x9E3779B1u) >> 22; }
static_assert(kTab == 1 << 10, "tab_slot keeps ten bits");

template <bool SCORE>
__global__ void __launch_bounds__(kEdgeWarps * 32, 4) k_edges(DGraph g, int seg, int level, const unsigned long long *wsum,
                                                           float *fout, const gp_mlp *mlp, float *s_out,
                                                           int32_t *q_out) {
  __shared__ int s_tab[kEdgeWarps][kTab], s_over[kEdgeWarps][64];
  __shared__ uint4 s_x[SCORE ? kEdgeWarps : 1][SCORE ? 64 : 1];
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31, half = lane >> 4, hl = lane & 15;
  const int gq = lane >> 2, t = lane & 3;
  int *tab = s_tab[wid], *over = s_over[wid];
  for (int x = lane; x < kTab; x += 32) tab[x] = -1;
  // The network's operands: W1^T by lane, and (bias, bias, w2, w2) by lane % 4 and slice. In registers they made
  // the lookups spill.
  __shared__ uint4 s_w1[SCORE ? 32 : 1];
  __shared__ float4 s_bw[SCORE ? 4 : 1][4];
  if (SCORE) {
    if (wid == 0) {
      unsigned w[4];
#pragma unroll
      for (int nb = 0; nb < 4; nb++) w[nb] = pack2(mlp->w1[(nb * 8 + gq) * kIn + 2 * t], mlp->w1[(nb * 8 + gq) * kIn + 2 * t + 1]);
      s_w1[SCORE ? lane : 0] = make_uint4(w[0], w[1], w[2], w[3]);
      if (lane < 16) {
        const int j = (lane >> 2) * 8 + 2 * t;
        s_bw[SCORE ? t : 0][lane >> 2] = make_float4(mlp->b1[j], mlp->b1[j + 1], bf16_to_float(mlp->w2[j]), bf16_to_float(mlp->w2[j + 1]));
      }
    }
    __syncthreads();
  }
  // Scores of the staged entries b .. b + cnt - 1 (b: a multiple of 32 entries after the segment's first).
  int64_t first = 0;
  auto score = [&](int64_t b, int cnt) {
    const unsigned *xw = reinterpret_cast<const unsigned *>(s_x[SCORE ? wid : 0]) + ((b - first) & 63) * 4;
    const uint4 w1 = s_w1[SCORE ? lane : 0];
    const unsigned bfrag[4] = {w1.x, w1.y, w1.z, w1.w};
    const float b2 = mlp->b2;
    float zmine = 0.f;
#pragma unroll
    for (int tile = 0; tile < 2; tile++) {
      if (tile * 16 >= cnt) break;
      const int r0 = tile * 16 + gq, r1 = r0 + 8;
      const unsigned a[4] = {r0 < cnt ? xw[r0 * 4 + t] : 0u, r1 < cnt ? xw[r1 * 4 + t] : 0u, 0u, 0u};
      float z0 = 0.f, z1 = 0.f;
#pragma unroll
      for (int nb = 0; nb < 4; nb++) {
        const float4 bw = s_bw[SCORE ? t : 0][nb];
        float c[4] = {bw.x, bw.y, bw.x, bw.y};
        const unsigned bf[2] = {bfrag[nb], 0u};  // (features 8..15 are zero)
        mma_16816(c, a, bf);
        // hidden activations are rounded to BF16 before the second layer
        const float h0 = bf16_to_float(float_to_bf16(fmaxf(c[0], 0.f)));
        const float h1 = bf16_to_float(float_to_bf16(fmaxf(c[1], 0.f)));
        const float h2 = bf16_to_float(float_to_bf16(fmaxf(c[2], 0.f)));
        const float h3 = bf16_to_float(float_to_bf16(fmaxf(c[3], 0.f)));
        z0 = fmaf(h0, bw.z, fmaf(h1, bw.w, z0));
        z1 = fmaf(h2, bw.z, fmaf(h3, bw.w, z1));
      }
      z0 += __shfl_xor_sync(kFull, z0, 1);
      z0 += __shfl_xor_sync(kFull, z0, 2);
      z1 += __shfl_xor_sync(kFull, z1, 1);
      z1 += __shfl_xor_sync(kFull, z1, 2);
      // back to the entries' lanes: entry 16 tile + x comes from lane 4 (x mod 8)
      const float a0 = __shfl_sync(kFull, z0, (lane & 7) * 4), a1 = __shfl_sync(kFull, z1, (lane & 7) * 4);
      if (half == tile) zmine = lane & 8 ? a1 : a0;
    }
    if (lane < cnt) {
      const float s = 1.0f / (1.0f + expf(-(zmine + b2)));
      if (s_out) s_out[b + lane] = s;
      if (q_out) q_out[b + lane] = __float2int_rn(s * 32768.0f);
    }
  };
  const float flevel = (float)level / 16.0f;
  const int64_t m = gp_min64(g.m, g.row_begin(g.n)), nseg = (m + seg - 1) / seg;
  const int64_t gw = blockIdx.x * (int64_t)kEdgeWarps + wid, nw = (int64_t)gridDim.x * kEdgeWarps;
  for (int64_t sg = gw; sg < nseg; sg += nw) {
    const int64_t s1 = gp_min64(m, (sg + 1) * seg);
    RowWindow W;
    W.load(g, warp_row_of(g, sg * seg));
    first = sg * seg;
    int64_t staged = first;  // the first entry that waits for its score
    for (int64_t e0 = first; e0 < s1;) {
      int64_t beg, end;
      const int64_t v = W.seek(g, e0, &beg, &end);
      const int64_t stop = gp_min64(end, s1), dv = end - beg;
      // v's first 64 neighbours (two per lane; the ids of a row are distinct) enter the table; a key whose
      // slot is taken goes to the list instead
      int own[2], nover = 0;
#pragma unroll
      for (int h = 0; h < 2; h++) {
        own[h] = -1;
        bool put = false;
        int x = 0;
        if (lane + 32 * h < dv) {
          x = __ldg(g.adj + beg + lane + 32 * h);
          const unsigned sl = tab_slot(x);
          if (atomicCAS(&tab[sl], -1, x) == -1) own[h] = (int)sl;
          else put = true;
        }
        const unsigned m = __ballot_sync(kFull, put);
        if (put) over[nover + __popc(m & lanemask_lt())] = x;
        nover += __popc(m);
      }
      __syncwarp();
      const float cv = (float)g.vweight(v);
      const float wv = wsum ? (float)(double)wsum[v] : (float)dv;
      for (; e0 < stop; e0 += 32) {
        const int64_t e = e0 + lane;
        const bool has = e < stop;
        const int u = has ? __ldg(g.adj + e) : 0;
        const int64_t bu = has ? g.row_begin(u) : 0;
        const int64_t du64 = has ? g.row_begin(u + 1) - bu : 0;
        const int lenu = (int)gp_min64(du64, 64);
        const float cu = has ? (float)g.vweight(u) : 0.0f;
        const float wu = has ? (wsum ? (float)(double)wsum[u] : (float)du64) : 0.0f;
        const float w = has ? (float)g.eweight(e) : 0.0f;
        const int cnt = (int)gp_min64(stop - e0, 32);
        int mine = 0;
        if (!__any_sync(kFull, lenu > 16)) {
          // (meshes: every list is one step of a half-warp)
          for (int p = 0; p < cnt; p += 4) {
            int xs[2];
#pragma unroll
            for (int y = 0; y < 2; y++) {
              const int64_t b = __shfl_sync(kFull, bu, p + 2 * y + half);
              const int len = __shfl_sync(kFull, lenu, p + 2 * y + half);
              xs[y] = hl < len ? __ldg(g.adj + b + hl) : -2;
            }
#pragma unroll
            for (int y = 0; y < 2; y++) {
              unsigned hits = tab[tab_slot(xs[y])] == xs[y];
              for (int o = 0; o < nover; o++) hits += over[o] == xs[y];
              const unsigned c = __reduce_add_sync(kFull, hits << (16 * half));
              if (lane == p + 2 * y) mine = (int)(c & 0xffffu);
              if (lane == p + 2 * y + 1) mine = (int)(c >> 16);
            }
          }
        } else
        for (int p = 0; p < cnt; p += 4) {
          // entries p, p + 2 (lower half-warp) and p + 1, p + 3 (upper)
          int xs[2][4], most[2];
#pragma unroll
          for (int y = 0; y < 2; y++) {
            const int64_t b = __shfl_sync(kFull, bu, p + 2 * y + half);
            const int len = __shfl_sync(kFull, lenu, p + 2 * y + half);
            most[y] = max(len, __shfl_xor_sync(kFull, len, 16));
#pragma unroll
            for (int q = 0; q < 4; q++) xs[y][q] = hl + 16 * q < len ? __ldg(g.adj + b + hl + 16 * q) : -2;
          }
#pragma unroll
          for (int y = 0; y < 2; y++) {
            unsigned hits = 0;
#pragma unroll
            for (int q = 0; q < 4; q++)
              if (16 * q < most[y]) hits += tab[tab_slot(xs[y][q])] == xs[y][q];
            for (int o = 0; o < nover; o++) {
              const int k = over[o];
#pragma unroll
              for (int q = 0; q < 4; q++) hits += k == xs[y][q];
            }
            const unsigned c = __reduce_add_sync(kFull, hits << (16 * half));  // both half-warps' counts
            if (lane == p + 2 * y) mine = (int)(c & 0xffffu);
            if (lane == p + 2 * y + 1) mine = (int)(c >> 16);
          }
        }
        const float du = (float)du64, dvf = (float)dv;
        float f[kIn];
        f[0] = log2f(1.0f + fminf(dvf, du));
        f[1] = log2f(1.0f + fmaxf(dvf, du));
        f[2] = log2f(1.0f + w);
        f[3] = log2f(1.0f + fminf(cv, cu));
        f[4] = log2f(1.0f + fmaxf(cv, cu));
        f[5] = (float)mine / 64.0f;
        f[6] = w / fmaxf(wv, wu);
        f[7] = flevel;
        if (!SCORE) {
          if (has) {
#pragma unroll
            for (int i = 0; i < kIn; i++) fout[e * kIn + i] = f[i];
          }
          continue;
        }
        uint4 pk;
        pk.x = pack2(float_to_bf16(f[0]), float_to_bf16(f[1]));
        pk.y = pack2(float_to_bf16(f[2]), float_to_bf16(f[3]));
        pk.z = pack2(float_to_bf16(f[4]), float_to_bf16(f[5]));
        pk.w = pack2(float_to_bf16(f[6]), float_to_bf16(f[7]));
        // the step's entries join the ones staged before (entry e at slot (e - first) mod 64)
        if (has) s_x[SCORE ? wid : 0][(e - first) & 63] = pk;
        const int64_t upto = e0 + cnt;
        __syncwarp();
        while (upto - staged >= 32 || (upto == s1 && staged < s1)) {
          const int c = (int)gp_min64(upto - staged, 32);
          score(staged, c);
          staged += c;
        }
        __syncwarp();
      }
      e0 = stop;
      __syncwarp();
#pragma unroll
      for (int h = 0; h < 2; h++)
        if (own[h] >= 0) tab[own[h]] = -1;
      __syncwarp();
    }
  }
}

// ------------------------------------------------------------------------------------------ training
struct TrainWeights {
  float w1[kHid * kIn];
  float b1[kHid];
  float w2[kHid];
  float b2;
};

// Loss and gradient partial sums of one block (FP32), forward with the given weights; block b leaves
// parameter p's sum at partials[p * gridDim.x + b].
//
// Bound by FP32 arithmetic: about 30 multiply-adds per entry and hidden unit. A warp takes 32 entries.
// First lane l runs the whole forward pass of entry l (weights broadcast from shared memory) up to the
// loss and dz; then lane j owns hidden unit j, with its weights and ten gradient sums in registers, and
// walks the 32 entries (features and dz broadcast from shared memory). No value crosses lanes, against one
// warp reduction per parameter and group of entries before: 568 us for a million entries then, 65 us now.
// Each sum is over m / (8 blocks) entries per lane (290 at a million entries, 27,000 at 10^8: the grid is at
// most three blocks per SM), then over the warps and the blocks (in 64 bits). RMS error of the gradient against
// 64 bits: 4.4e-8 of its size at 10^6 entries, 3.6e-8 at 2 10^7, 4.4e-8 at 10^8 (with the reductions 4.4, 3.5
// and 4.8e-8).
constexpr int kGradWarps = 8;

__global__ void __launch_bounds__(kGradWarps * 32) k_grad(const float *x, const float *y, int64_t m,
                                                          const TrainWeights *W, float *partials) {
  __shared__ __align__(16) TrainWeights sw;
  __shared__ __align__(16) float s_x[kGradWarps][32][kIn];
  __shared__ __align__(16) float s_dz[kGradWarps][32];
  __shared__ float s_acc[kGradWarps][kHid][kIn + 2], s_tail[kGradWarps][2];
  for (int p = threadIdx.x; p < (int)(sizeof(TrainWeights) / 4); p += blockDim.x)
    reinterpret_cast<float *>(&sw)[p] = reinterpret_cast<const float *>(W)[p];
  __syncthreads();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const float inv_m = 1.0f / (float)m;
  float wj[kIn], acc[kIn + 2], sum_dz = 0.f, sum_loss = 0.f;
#pragma unroll
  for (int i = 0; i < kIn; i++) wj[i] = sw.w1[lane * kIn + i];
  const float bj = sw.b1[lane], vj = sw.w2[lane];
#pragma unroll
  for (int i = 0; i < kIn + 2; i++) acc[i] = 0.f;
  const int64_t gw = blockIdx.x * (int64_t)kGradWarps + wid, nw = (int64_t)gridDim.x * kGradWarps;
  for (int64_t base = gw * 32; base < m; base += nw * 32) {
    const int64_t e = base + lane;
    const bool valid = e < m;
    float xi[kIn];
#pragma unroll
    for (int i = 0; i < kIn; i++) xi[i] = valid ? x[e * kIn + i] : 0.f;
    const float ye = valid ? y[e] : 0.f;
    float z = sw.b2;
#pragma unroll
    for (int j = 0; j < kHid; j++) {
      float a = sw.b1[j];
#pragma unroll
      for (int i = 0; i < kIn; i++) a = fmaf(sw.w1[j * kIn + i], xi[i], a);
      z = fmaf(sw.w2[j], fmaxf(a, 0.f), z);
    }
    const float s = 1.0f / (1.0f + expf(-z));
    const float loss = valid ? (fmaxf(z, 0.f) - ye * z + log1pf(expf(-fabsf(z)))) : 0.f;
    const float dz = valid ? (s - ye) * inv_m : 0.f;
    sum_dz += dz;
    sum_loss += loss * inv_m;
    __syncwarp();
#pragma unroll
    for (int i = 0; i < kIn; i++) s_x[wid][lane][i] = xi[i];
    s_dz[wid][lane] = dz;
    __syncwarp();
#pragma unroll 8
    for (int r = 0; r < 32; r++) {
      float xr[kIn], a = bj;
#pragma unroll
      for (int i = 0; i < kIn; i++) xr[i] = s_x[wid][r][i];
#pragma unroll
      for (int i = 0; i < kIn; i++) a = fmaf(wj[i], xr[i], a);
      const float d = s_dz[wid][r];
      const float dh = a > 0.f ? d * vj : 0.f;
#pragma unroll
      for (int i = 0; i < kIn; i++) acc[i] = fmaf(dh, xr[i], acc[i]);
      acc[kIn] += dh;
      acc[kIn + 1] = fmaf(d, fmaxf(a, 0.f), acc[kIn + 1]);
    }
  }
#pragma unroll
  for (int i = 0; i < kIn + 2; i++) s_acc[wid][lane][i] = acc[i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    sum_dz += __shfl_xor_sync(kFull, sum_dz, o);
    sum_loss += __shfl_xor_sync(kFull, sum_loss, o);
  }
  if (lane == 0) {
    s_tail[wid][0] = sum_dz;
    s_tail[wid][1] = sum_loss;
  }
  __syncthreads();
  for (int p = threadIdx.x; p < kParams + 1; p += blockDim.x) {
    float s = 0.f;
    for (int w = 0; w < kGradWarps; w++)
      s += p < kHid * kIn          ? s_acc[w][p / kIn][p % kIn]
           : p < kHid * kIn + 2 * kHid ? s_acc[w][(p - kHid * kIn) % kHid][kIn + (p - kHid * kIn) / kHid]
                                   : s_tail[w][p - (kHid * kIn + 2 * kHid)];
    partials[(size_t)p * gridDim.x + blockIdx.x] = s;
  }
}

// The blocks' partial sums of parameter p, in 64 bits, by one warp (all lanes get the sum).
__device__ __forceinline__ float grad_total(const float *partials, int nblocks, int p) {
  double s = 0;
  for (int b = threadIdx.x & 31; b < nblocks; b += 32) s += partials[(size_t)p * nblocks + b];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
  return (float)s;
}

// One warp per parameter (one block summing every parameter's partials in turn took 120 us).
__global__ void k_grad_sum(const float *partials, int nblocks, float *out) {
  const int p = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  if (p > kParams) return;
  const float s = grad_total(partials, nblocks, p);
  if ((threadIdx.x & 31) == 0) out[p] = s;
}

// Gradient sums and the Adam step on the FP32 master weights, one warp per parameter; writes the BF16
// weights used by inference and the next forward pass. Warp kParams logs the loss.
__global__ void k_adam(const float *partials, int nblocks, TrainWeights *master, TrainWeights *fwd, float *mom,
                       float *vel, int step, float lr, gp_mlp *mlp, float *loss_log) {
  const int p = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  if (p > kParams) return;
  const float g = grad_total(partials, nblocks, p);
  if (threadIdx.x & 31) return;
  if (p == kParams) {
    if (loss_log) loss_log[step - 1] = g;
    return;
  }
  const float beta1 = 0.9f, beta2 = 0.999f, epsv = 1e-8f;
  const float c1 = 1.0f - powf(beta1, (float)step), c2 = 1.0f - powf(beta2, (float)step);
  float *wm = reinterpret_cast<float *>(master);
  float *wf = reinterpret_cast<float *>(fwd);
  mom[p] = beta1 * mom[p] + (1.f - beta1) * g;
  vel[p] = beta2 * vel[p] + (1.f - beta2) * g * g;
  wm[p] -= lr * (mom[p] / c1) / (sqrtf(vel[p] / c2) + epsv);
  if (p < kHid * kIn) {
    const uint16_t b = float_to_bf16(wm[p]);
    mlp->w1[p] = b;
    wf[p] = bf16_to_float(b);
  } else if (p < kHid * kIn + kHid) {
    mlp->b1[p - kHid * kIn] = wm[p];
    wf[p] = wm[p];
  } else if (p < kHid * kIn + 2 * kHid) {
    const uint16_t b = float_to_bf16(wm[p]);
    mlp->w2[p - kHid * kIn - kHid] = b;
    wf[p] = bf16_to_float(b);
  } else {
    mlp->b2 = wm[p];
    wf[p] = wm[p];
  }
}

// Master/forward weights from the gp_mlp (BF16 weights become exact FP32 values).
__global__ void k_weights_from(const gp_mlp *mlp, TrainWeights *master, TrainWeights *fwd) {
  float *wm = reinterpret_cast<float *>(master);
  float *wf = reinterpret_cast<float *>(fwd);
  for (int p = threadIdx.x; p < kParams; p += blockDim.x) {
    float v;
    if (p < kHid * kIn) v = bf16_to_float(mlp->w1[p]);
    else if (p < kHid * kIn + kHid) v = mlp->b1[p - kHid * kIn];
    else if (p < kHid * kIn + 2 * kHid) v = bf16_to_float(mlp->w2[p - kHid * kIn - kHid]);
    else v = mlp->b2;
    wm[p] = v;
    wf[p] = v;
  }
}

int grid_for(int64_t items, int per_block, int limit) {
  return (int)std::max<int64_t>(1, std::min<int64_t>((items + per_block - 1) / per_block, limit));
}

// The entry kernel of features (fout) or scores (mlp, s_out, q_out) after the weighted degrees.
int run_edges(const DGraph &g, int level, float *fout, const gp_mlp *mlp, float *s_out, int32_t *q_out, cudaStream_t s) {
  if (g.m == 0) return GP_OK;
  Workspace ws(s);
  const int nsm = num_sms();
  const int seg = row_segment(g.m);
  const int64_t warps = (g.m + seg - 1) / seg;
  unsigned long long *wsum = nullptr;
  if (g.ew) {
    GP_TRY(ws.zeros(&wsum, (size_t)g.n));
    (::gp::count_launch(), k_wdeg<<<grid_for(warps, 8, nsm * 8), 256, 0, s>>>(g, seg, wsum));
  }
  {
    ProfScope ps(fout ? "mlp_features" : "mlp_score_mma", s);
    const int grid = grid_for(warps, kEdgeWarps, nsm * 16);
    if (fout)
      (::gp::count_launch(), k_edges<false><<<grid, kEdgeWarps * 32, 0, s>>>(g, seg, level, wsum, fout, nullptr, nullptr, nullptr));
    else
      (::gp::count_launch(), k_edges<true><<<grid, kEdgeWarps * 32, 0, s>>>(g, seg, level, wsum, nullptr, mlp, s_out, q_out));
  }
  GP_LAUNCH_CHECK();
  return GP_OK;
}

}  // namespace

int mlp_score(const DGraph &g, int level, const gp_mlp *mlp, float *s_out, int32_t *q_out, cudaStream_t s) {
  if (g.m == 0) return GP_OK;
  GP_TRY(run_edges(g, level, nullptr, mlp, s_out, q_out, s));
  prof_add_counts("mlp_score_mma", g.m, g.m, g.m * (4 + g.ew_bytes() + (q_out ? 4 : 0) + (s_out ? 4 : 0)));
  return GP_OK;
}

int mlp_train(const float *x, const float *y, int64_t m, gp_mlp *mlp, int steps, float lr, float *loss_host,
              float *grad_host, cudaStream_t s) {
  Workspace ws(s);
  TrainWeights *master, *fwd;
  float *partials;
  GP_TRY(ws.get(&master, 1));
  GP_TRY(ws.get(&fwd, 1));
  // a few groups of 32 entries per warp; a smaller set gets fewer blocks, not emptier ones
  const int nb = grid_for(m, kGradWarps * 32, num_sms() * 3);
  const int nbp = (kParams + 1 + 7) / 8;  // one warp per parameter and the loss
  GP_TRY(ws.get(&partials, (size_t)nb * (kParams + 1)));
  (::gp::count_launch(), k_weights_from<<<1, 352, 0, s>>>(mlp, master, fwd));
  if (steps <= 0) {
    // gradient only
    float *grad;
    GP_TRY(ws.get(&grad, kParams + 1));
    (::gp::count_launch(), k_grad<<<nb, kGradWarps * 32, 0, s>>>(x, y, m, fwd, partials));
    (::gp::count_launch(), k_grad_sum<<<nbp, 256, 0, s>>>(partials, nb, grad));
    GP_LAUNCH_CHECK();
    if (!grad_host) {
      GP_CUDA(cudaStreamSynchronize(s));
      return GP_OK;
    }
    Readback rb;
    rb.add(grad_host, grad, sizeof(float) * (kParams + 1));
    return rb.run(s);
  }
  float *mom, *vel, *losses;
  GP_TRY(ws.zeros(&mom, kParams));
  GP_TRY(ws.zeros(&vel, kParams));
  GP_TRY(ws.get(&losses, (size_t)steps));
  for (int st = 1; st <= steps; st++) {
    (::gp::count_launch(), k_grad<<<nb, kGradWarps * 32, 0, s>>>(x, y, m, fwd, partials));
    (::gp::count_launch(), k_adam<<<nbp, 256, 0, s>>>(partials, nb, master, fwd, mom, vel, st, lr, mlp, losses));
  }
  GP_LAUNCH_CHECK();
  if (loss_host) GP_CUDA(cudaMemcpyAsync(loss_host, losses, sizeof(float) * steps, cudaMemcpyDeviceToHost, s));
  GP_CUDA(cudaStreamSynchronize(s));
  return GP_OK;
}

}  // namespace gp

using namespace gp;

extern "C" {

int gp_mlp_score(const gp_graph *g, int32_t level, const gp_mlp *mlp, float *s_out, int32_t *q_out, gp_stream stream) {
  if (!g || !mlp || g->n < 0 || g->m_dir < 0) {
    set_error("gp_mlp_score: graph and mlp are required");
    return GP_ERR_INVALID_ARG;
  }
  cudaStream_t s = (cudaStream_t)stream;
  GP_TRY(mlp_score(make_dgraph(g), level, mlp, s_out, q_out, s));
  GP_CUDA(cudaStreamSynchronize(s));
  return GP_OK;
}

int gp_edge_features(const gp_graph *g, int32_t level, float *feat_out, gp_stream stream) {
  if (!g || !feat_out || g->n < 0 || g->m_dir < 0) {
    set_error("gp_edge_features: graph and output are required");
    return GP_ERR_INVALID_ARG;
  }
  cudaStream_t s = (cudaStream_t)stream;
  GP_TRY(run_edges(make_dgraph(g), level, feat_out, nullptr, nullptr, nullptr, s));
  GP_CUDA(cudaStreamSynchronize(s));
  return GP_OK;
}

int gp_mlp_train(const float *feat, const float *y, int64_t m, gp_mlp *mlp, int32_t steps, float lr, float *loss_out,
                 gp_stream stream) {
  if (!feat || !y || m <= 0 || !mlp || steps < 1) {
    set_error("gp_mlp_train: feat, y, m > 0, mlp and steps >= 1 are required");
    return GP_ERR_INVALID_ARG;
  }
  return mlp_train(feat, y, m, mlp, steps, lr, loss_out, nullptr, (cudaStream_t)stream);
}

int gp_mlp_grad(const float *feat, const float *y, int64_t m, const gp_mlp *mlp, float *loss_out, float *grad_out,
                gp_stream stream) {
  if (!feat || !y || m <= 0 || !mlp) {
    set_error("gp_mlp_grad: feat, y, m > 0 and mlp are required");
    return GP_ERR_INVALID_ARG;
  }
  std::vector<float> g(kParams + 1);
  GP_TRY(mlp_train(feat, y, m, const_cast<gp_mlp *>(mlp), 0, 0.f, nullptr, g.data(), (cudaStream_t)stream));
  if (grad_out) std::memcpy(grad_out, g.data(), sizeof(float) * kParams);
  if (loss_out) *loss_out = g[kParams];
  return GP_OK;
}

}  // extern "C"
