// Learned seed proposer: training and batched inference kernels.
//
// The paper bipartitions a coarsest graph by repeating simple algorithms
// several times and keeping the best (Section 4.2).  Here a small
// message-passing network (kmp_mpnn.cuh) scores the nodes; the score order
// seeds one extra bipartition in the bipartitioner, which goes through the
// same 2-way FM and the same feasible/lower-cut selection as the portfolio.
//
// A batch is one disjoint union of graphs in CSR form (union node ids) plus
// the node offset of each graph: layers are node-parallel over the union,
// features and loss work per graph.  Training keeps fp32 master weights and
// Adam moments and uses a BF16 copy of the weights in every kernel.
#include <algorithm>
#include <cmath>
#include <vector>

#include "kmp_mpnn.cuh"

struct kmp_mpnn {
  float *master = nullptr;
  __nv_bfloat16 *wbf = nullptr;
  float *am = nullptr, *av = nullptr, *grad = nullptr;
  int64_t step = 0;
};

static_assert(kmp::P_TOTAL == KMP_MPNN_PARAMS, "parameter layout of kmp.h");

namespace kmp {

static Proposer g_proposer;
Proposer &proposer() { return g_proposer; }
static SampleSink g_sink;
SampleSink &sample_sink() { return g_sink; }

static void sink_release() {
  SampleSink &K = g_sink;
  for (void *p : {(void *)K.counters, (void *)K.rec, (void *)K.deg, (void *)K.vw, (void *)K.side,
                  (void *)K.adj, (void *)K.ew})
    if (p) dfree(p);
  K = SampleSink{};
}

struct Batch {
  int32_t ng = 0, N = 0;
  int32_t max_n = 0;  // nodes of the largest graph
  int64_t E = 0;
  DBuf<int32_t> noff, adj, vw, ew, side;
  DBuf<int64_t> xadj;
  DBuf<uint64_t> keys;
};

// ---------------------------------------------------------------- kernels
// One CTA per graph.  The hop counts live in shared memory when the batch's
// largest graph fits (MP_FEAT_SMEM_N nodes), else in d1, d2: a hop level scans
// them once, and with 512 threads a level of a 4000-node mesh is eight reads a
// thread and a barrier.  256 graphs of 200..4000 nodes (325,000 in all):
// 2.15 ms with sweeps over all entries in global memory, 0.67 ms now.
constexpr int MP_FEAT_T = 512;
constexpr int MP_FEAT_SMEM_N = 12288;  // 96 KB of hop counts: two CTAs per SM
__global__ void __launch_bounds__(MP_FEAT_T) k_mp_features(int32_t ng, const int32_t *noff, const int64_t *xadj,
                                                           const int32_t *adj, const int32_t *vw,
                                                           const int32_t *ew, const uint64_t *keys, float *X,
                                                           int32_t *d1, int32_t *d2, int32_t smem_n) {
  extern __shared__ int32_t mp_hops[];
  for (int32_t g = blockIdx.x; g < ng; g += gridDim.x) {
    int32_t v0 = noff[g];
    GView<int64_t> G{noff[g + 1] - v0, xadj + v0, adj, v0, vw ? vw + v0 : nullptr, ew};
    const bool in_smem = G.n <= smem_n;
    mp_features(G, keys[g], X + (int64_t)v0 * MF, in_smem ? mp_hops : d1 + v0, in_smem ? mp_hops + smem_n : d2 + v0);
  }
}

// four consecutive channels of a neighbour sum: s = fma(w, h, s) in CSR order
__device__ __forceinline__ void fma4(float4 &s, float w, const float4 &h) {
  s.x = __fmaf_rn(w, h.x, s.x);
  s.y = __fmaf_rn(w, h.y, s.y);
  s.z = __fmaf_rn(w, h.z, s.z);
  s.w = __fmaf_rn(w, h.w, s.w);
}

// Neighbour mean over the union, D channels a node, four channels a thread
// (16 lanes read a neighbour's 64 channels as one 256-byte row); the loads of
// four entries are issued before their sums, which stay in CSR order.  Bound by
// the L2 traffic of the rows (64 channels, 3.3 M entries: 0.85 GB).
template <int D>
__global__ void __launch_bounds__(256) k_mp_nbr(int32_t N, const int64_t *__restrict__ xadj,
                                                const int32_t *__restrict__ adj,
                                                const int32_t *__restrict__ ew,
                                                const float *__restrict__ Hin, float *__restrict__ M) {
  constexpr int LN = D / 4;  // lanes per node
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < (int64_t)N * LN;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int32_t v = (int32_t)(t / LN), c = 4 * (int)(t % LN);
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    float ws = 0.f;
    int64_t e = xadj[v];
    const int64_t e1 = xadj[v + 1];
    for (; e + 4 <= e1; e += 4) {
      float w[4];
      float4 h[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        w[q] = ew ? (float)ew[e + q] : 1.f;
        h[q] = *reinterpret_cast<const float4 *>(Hin + (int64_t)adj[e + q] * D + c);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        ws += w[q];
        fma4(s, w[q], h[q]);
      }
    }
    for (; e < e1; ++e) {
      const float w = ew ? (float)ew[e] : 1.f;
      ws += w;
      fma4(s, w, *reinterpret_cast<const float4 *>(Hin + (int64_t)adj[e] * D + c));
    }
    float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
    if (ws > 0.f) r = make_float4(s.x / ws, s.y / ws, s.z / ws, s.w / ws);
    *reinterpret_cast<float4 *>(M + (int64_t)v * D + c) = r;
  }
}

// Tiles of the layer kernels: MP_TILE nodes x 64 channels, 256 threads of 4 x 4
// values each.  A shared row holds 64 channels and four words of padding, so the
// two rows that a warp reads together lie on different banks.
constexpr int MP_TILE = 64;
constexpr int MP_T = 256;
constexpr int MP_LD = MH + 4;

// rows [base, base + cnt) of a [N][D] array into shared rows of D + 4 words
// (missing rows as zeros)
template <int D>
__device__ __forceinline__ void mp_load_tile(float *dst, const float *__restrict__ src, int64_t base, int cnt) {
  constexpr int Q = D / 4;
  for (int t = threadIdx.x; t < MP_TILE * Q; t += MP_T) {
    const int r = t / Q, c = 4 * (t % Q);
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
    if (r < cnt) x = *reinterpret_cast<const float4 *>(src + (base + r) * D + c);
    *reinterpret_cast<float4 *>(dst + r * (D + 4) + c) = x;
  }
}

// One layer over the union, H = relu(b + W_self h + W_nbr m), every output's
// fused multiply-adds in the fixed order of mp_preact.  The weights sit in
// shared memory as floats, input-major, for the whole launch; a thread keeps a
// 4 x 4 block of outputs in registers, so 32 multiply-adds take six 16-byte
// shared reads instead of a global read each.  READOUT: the scores of the
// tile's nodes as well, from the tile in shared memory.  Bound by
// latency: layer 2 of 325,000 nodes, 5.3 GFLOP in 0.21 ms, keeps the FMA pipe 34 % busy
// and issues in 42 % of cycles; the eight warps of each of two CTAs an SM wait for the
// tile's global loads and for shared reads.  Both layers with the read-out: 8.9 ms with
// one output a thread and strided weight reads, 0.24 ms now.
template <int DIN, bool READOUT>
constexpr size_t mp_layer_smem() {
  return sizeof(float) * (2 * DIN * MH + 2 * MP_TILE * (DIN + 4) + (READOUT ? MP_TILE * MP_LD : 0));
}
template <int DIN, bool READOUT>
__global__ void __launch_bounds__(MP_T) k_mp_layer(int32_t N, const __nv_bfloat16 *__restrict__ W, int ws, int wn,
                                                   int b, const float *__restrict__ Hin,
                                                   const float *__restrict__ M, float *__restrict__ H,
                                                   float *__restrict__ S) {
  extern __shared__ __align__(16) float mp_sm[];
  float *Ws = mp_sm, *Wn = Ws + DIN * MH;                  // [i][o]
  float *sh = Wn + DIN * MH, *sm = sh + MP_TILE * (DIN + 4);
  float *so = sm + MP_TILE * (DIN + 4);                    // output tile (READOUT)
  for (int t = threadIdx.x; t < DIN * MH; t += MP_T) {
    const int o = t / DIN, i = t % DIN;
    Ws[i * MH + o] = wbf(W, ws + t);
    Wn[i * MH + o] = wbf(W, wn + t);
  }
  const int o0 = 4 * (threadIdx.x & 15), r0 = 4 * (threadIdx.x >> 4);
  float bias[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) bias[j] = wbf(W, b + o0 + j);
  for (int64_t base = (int64_t)blockIdx.x * MP_TILE; base < N; base += (int64_t)gridDim.x * MP_TILE) {
    const int cnt = (int)(N - base < MP_TILE ? N - base : MP_TILE);
    __syncthreads();  // the previous tile's readers are done
    mp_load_tile<DIN>(sh, Hin, base, cnt);
    mp_load_tile<DIN>(sm, M, base, cnt);
    __syncthreads();
    float a[4][4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int j = 0; j < 4; ++j) a[q][j] = bias[j];
#pragma unroll 2
    for (int i = 0; i < DIN; i += 4) {
      float4 h[4], m[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        h[q] = *reinterpret_cast<const float4 *>(sh + (r0 + q) * (DIN + 4) + i);
        m[q] = *reinterpret_cast<const float4 *>(sm + (r0 + q) * (DIN + 4) + i);
      }
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        const float4 u = *reinterpret_cast<const float4 *>(Ws + (i + x) * MH + o0);
        const float4 n = *reinterpret_cast<const float4 *>(Wn + (i + x) * MH + o0);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float hv = x == 0 ? h[q].x : x == 1 ? h[q].y : x == 2 ? h[q].z : h[q].w;
          const float mv = x == 0 ? m[q].x : x == 1 ? m[q].y : x == 2 ? m[q].z : m[q].w;
          a[q][0] = __fmaf_rn(n.x, mv, __fmaf_rn(u.x, hv, a[q][0]));
          a[q][1] = __fmaf_rn(n.y, mv, __fmaf_rn(u.y, hv, a[q][1]));
          a[q][2] = __fmaf_rn(n.z, mv, __fmaf_rn(u.z, hv, a[q][2]));
          a[q][3] = __fmaf_rn(n.w, mv, __fmaf_rn(u.w, hv, a[q][3]));
        }
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float4 r = make_float4(a[q][0] > 0.f ? a[q][0] : 0.f, a[q][1] > 0.f ? a[q][1] : 0.f,
                                   a[q][2] > 0.f ? a[q][2] : 0.f, a[q][3] > 0.f ? a[q][3] : 0.f);
      if (r0 + q < cnt) *reinterpret_cast<float4 *>(H + (base + r0 + q) * MH + o0) = r;
      if (READOUT) *reinterpret_cast<float4 *>(so + (r0 + q) * MP_LD + o0) = r;
    }
    if (READOUT) {
      __syncthreads();
      if ((int)threadIdx.x < cnt) S[base + threadIdx.x] = mp_readout(W, so + threadIdx.x * MP_LD);
    }
  }
}

__device__ __forceinline__ float softplusf(float z) { return z > 0.f ? z + log1pf(expf(-z)) : log1pf(expf(z)); }

// per graph: orientation-symmetric BCE, gS = dL/ds with L = mean over graphs;
// lossg[g] = graph g's share of L (summed on the host in graph order)
__global__ void k_mp_loss(int32_t ng, const int32_t *noff, const float *S, const int32_t *side, float *gS,
                          float *lossg) {
  __shared__ float r0[32], r1[32];
  for (int32_t g = blockIdx.x; g < ng; g += gridDim.x) {
    int32_t v0 = noff[g], n = noff[g + 1] - v0;
    float l0 = 0, l1 = 0;
    for (int32_t v = threadIdx.x; v < n; v += blockDim.x) {
      float s = S[v0 + v], y = side[v0 + v] == 0 ? 1.f : 0.f, sp = softplusf(s);
      l0 += sp - y * s;
      l1 += sp - (1.f - y) * s;
    }
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) {
      l0 += __shfl_xor_sync(0xFFFFFFFFu, l0, m);
      l1 += __shfl_xor_sync(0xFFFFFFFFu, l1, m);
    }
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) {
      r0[w] = l0;
      r1[w] = l1;
    }
    __syncthreads();
    float t0 = 0, t1 = 0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) {
      t0 += r0[i];
      t1 += r1[i];
    }
    bool flip = t1 < t0;
    float scale = 1.f / ((float)(n > 0 ? n : 1) * (float)ng);
    for (int32_t v = threadIdx.x; v < n; v += blockDim.x) {
      float y = side[v0 + v] == 0 ? 1.f : 0.f;
      if (flip) y = 1.f - y;
      float p = 1.f / (1.f + expf(-S[v0 + v]));
      gS[v0 + v] = (p - y) * scale;
    }
    if (threadIdx.x == 0) lossg[g] = (flip ? t1 : t0) * scale;
    __syncthreads();
  }
}

// Weight gradients without atomics, so training is deterministic: CTA c of a
// fixed number sums tiles c, c + G, c + 2G, ... of MP_TILE nodes in order and
// writes its partial sums of dW_self[o][i] = sum_v gA[v][o] Hin[v][i], dW_nbr
// (with M) and db[o] = sum_v gA[v][o] to part[c][...]; k_mp_reduce adds the G
// partials in order.
//
// Backward of the read-out and of layer 2 in one pass over the tiles:
// gA2 = relu'(h2) gS w_o in shared memory only; the read-out's and layer 2's
// weight gradients; and the layer's input gradients gH1[v][i] = sum_o
// W2s[o][i] gA2[v][o], gM1 likewise with W2n.  Threads hold 4 x 4 blocks as in
// k_mp_layer.  Bound by latency too (325,000 nodes, 10.6 GFLOP: FMA pipe 40 %, issue
// 52 % of cycles; waits for the tile's loads); 1.8 ms as five kernels with gA2 in
// global memory, 0.41 ms now.
constexpr size_t MP_BW2_SMEM = sizeof(float) * (4 * MP_TILE * MP_LD + 2 * MH * MH + MP_TILE + MH);
__global__ void __launch_bounds__(MP_T) k_mp_bw2(int32_t N, const __nv_bfloat16 *__restrict__ W,
                                                 const float *__restrict__ gS, const float *__restrict__ H2,
                                                 const float *__restrict__ H1, const float *__restrict__ M1,
                                                 float *__restrict__ gH1, float *__restrict__ gM1,
                                                 float *__restrict__ part) {
  extern __shared__ __align__(16) float mp_sm[];
  float *sg = mp_sm, *s2 = sg + MP_TILE * MP_LD, *sh = s2 + MP_TILE * MP_LD, *sm = sh + MP_TILE * MP_LD;
  float *Ws = sm + MP_TILE * MP_LD, *Wn = Ws + MH * MH;  // [o][i]
  float *sS = Wn + MH * MH, *swo = sS + MP_TILE;
  for (int t = threadIdx.x; t < MH * MH; t += MP_T) {
    Ws[t] = wbf(W, P_W2S + t);
    Wn[t] = wbf(W, P_W2N + t);
  }
  if (threadIdx.x < MH) swo[threadIdx.x] = wbf(W, P_WO + threadIdx.x);
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  float ds[4][4], dn[4][4];  // dW2[4 ty + q][4 tx + j]
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int j = 0; j < 4; ++j) ds[q][j] = dn[q][j] = 0.f;
  float accb = 0.f, accw = 0.f, accs = 0.f;  // threads < 64: db2, dw_o; thread 0: db_o
  for (int64_t base = (int64_t)blockIdx.x * MP_TILE; base < N; base += (int64_t)gridDim.x * MP_TILE) {
    const int cnt = (int)(N - base < MP_TILE ? N - base : MP_TILE);
    __syncthreads();
    mp_load_tile<MH>(s2, H2, base, cnt);
    mp_load_tile<MH>(sh, H1, base, cnt);
    mp_load_tile<MH>(sm, M1, base, cnt);
    if (threadIdx.x < MP_TILE) sS[threadIdx.x] = (int)threadIdx.x < cnt ? gS[base + threadIdx.x] : 0.f;
    __syncthreads();
    for (int t = threadIdx.x; t < MP_TILE * MH; t += MP_T) {
      const int r = t / MH, o = t % MH;
      sg[r * MP_LD + o] = s2[r * MP_LD + o] > 0.f ? sS[r] * swo[o] : 0.f;
    }
    __syncthreads();
    // weight gradients: the tile's nodes in order
    for (int r = 0; r < cnt; ++r) {
      const float4 g = *reinterpret_cast<const float4 *>(sg + r * MP_LD + 4 * ty);
      const float4 h = *reinterpret_cast<const float4 *>(sh + r * MP_LD + 4 * tx);
      const float4 m = *reinterpret_cast<const float4 *>(sm + r * MP_LD + 4 * tx);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float gv = q == 0 ? g.x : q == 1 ? g.y : q == 2 ? g.z : g.w;
        ds[q][0] = __fmaf_rn(gv, h.x, ds[q][0]);
        ds[q][1] = __fmaf_rn(gv, h.y, ds[q][1]);
        ds[q][2] = __fmaf_rn(gv, h.z, ds[q][2]);
        ds[q][3] = __fmaf_rn(gv, h.w, ds[q][3]);
        dn[q][0] = __fmaf_rn(gv, m.x, dn[q][0]);
        dn[q][1] = __fmaf_rn(gv, m.y, dn[q][1]);
        dn[q][2] = __fmaf_rn(gv, m.z, dn[q][2]);
        dn[q][3] = __fmaf_rn(gv, m.w, dn[q][3]);
      }
    }
    if (threadIdx.x < MH) {
      for (int r = 0; r < cnt; ++r) {
        accb += sg[r * MP_LD + threadIdx.x];
        accw = __fmaf_rn(sS[r], s2[r * MP_LD + threadIdx.x], accw);
      }
      if (threadIdx.x == 0)
        for (int r = 0; r < cnt; ++r) accs += sS[r];
    }
    // input gradients: nodes 4 ty .. 4 ty + 3, inputs 4 tx .. 4 tx + 3, o in order
    float a[4][4], c[4][4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int j = 0; j < 4; ++j) a[q][j] = c[q][j] = 0.f;
    for (int o = 0; o < MH; ++o) {
      const float4 u = *reinterpret_cast<const float4 *>(Ws + o * MH + 4 * tx);
      const float4 n = *reinterpret_cast<const float4 *>(Wn + o * MH + 4 * tx);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float gv = sg[(4 * ty + q) * MP_LD + o];
        a[q][0] = __fmaf_rn(u.x, gv, a[q][0]);
        a[q][1] = __fmaf_rn(u.y, gv, a[q][1]);
        a[q][2] = __fmaf_rn(u.z, gv, a[q][2]);
        a[q][3] = __fmaf_rn(u.w, gv, a[q][3]);
        c[q][0] = __fmaf_rn(n.x, gv, c[q][0]);
        c[q][1] = __fmaf_rn(n.y, gv, c[q][1]);
        c[q][2] = __fmaf_rn(n.z, gv, c[q][2]);
        c[q][3] = __fmaf_rn(n.w, gv, c[q][3]);
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (4 * ty + q < cnt) {
        const int64_t at = (base + 4 * ty + q) * MH + 4 * tx;
        *reinterpret_cast<float4 *>(gH1 + at) = make_float4(a[q][0], a[q][1], a[q][2], a[q][3]);
        *reinterpret_cast<float4 *>(gM1 + at) = make_float4(c[q][0], c[q][1], c[q][2], c[q][3]);
      }
  }
  float *pc = part + (int64_t)blockIdx.x * P_TOTAL;
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int pr = (4 * ty + q) * MH + 4 * tx + j;
      pc[P_W2S + pr] = ds[q][j];
      pc[P_W2N + pr] = dn[q][j];
    }
  if (threadIdx.x < MH) {
    pc[P_B2 + threadIdx.x] = accb;
    pc[P_WO + threadIdx.x] = accw;
  }
  if (threadIdx.x == 0) pc[P_BO] = accs;
}

// layer 1's weight gradients (8 inputs): thread t sums outputs t / 4 with inputs
// 2 (t % 4) and the next, over the same tiles in the same order
__global__ void __launch_bounds__(MP_T) k_mp_wgrad1(int32_t N, const float *__restrict__ gA,
                                                    const float *__restrict__ X, const float *__restrict__ M,
                                                    float *__restrict__ part) {
  static_assert(MH * MF == 2 * MP_T, "two weights of each kind a thread");
  __shared__ __align__(16) float sg[MP_TILE * MP_LD], sh[MP_TILE * (MF + 4)], sm[MP_TILE * (MF + 4)];
  const int o = threadIdx.x >> 2, i = 2 * (threadIdx.x & 3);
  float s0 = 0.f, s1 = 0.f, n0 = 0.f, n1 = 0.f, accb = 0.f;
  for (int64_t base = (int64_t)blockIdx.x * MP_TILE; base < N; base += (int64_t)gridDim.x * MP_TILE) {
    const int cnt = (int)(N - base < MP_TILE ? N - base : MP_TILE);
    __syncthreads();
    mp_load_tile<MH>(sg, gA, base, cnt);
    mp_load_tile<MF>(sh, X, base, cnt);
    mp_load_tile<MF>(sm, M, base, cnt);
    __syncthreads();
#pragma unroll 4
    for (int r = 0; r < cnt; ++r) {
      const float g = sg[r * MP_LD + o];
      const float2 h = *reinterpret_cast<const float2 *>(sh + r * (MF + 4) + i);
      const float2 m = *reinterpret_cast<const float2 *>(sm + r * (MF + 4) + i);
      s0 = __fmaf_rn(g, h.x, s0);
      s1 = __fmaf_rn(g, h.y, s1);
      n0 = __fmaf_rn(g, m.x, n0);
      n1 = __fmaf_rn(g, m.y, n1);
      accb += g;
    }
  }
  float *pc = part + (int64_t)blockIdx.x * P_TOTAL;
  pc[P_W1S + o * MF + i] = s0;
  pc[P_W1S + o * MF + i + 1] = s1;
  pc[P_W1N + o * MF + i] = n0;
  pc[P_W1N + o * MF + i + 1] = n1;
  if (i == 0) pc[P_B1 + o] = accb;
}

__global__ void k_mp_reduce(int32_t G, const float *part, float *grad) {
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < P_TOTAL; p += gridDim.x * blockDim.x) {
    float s = 0.f;
    for (int32_t c = 0; c < G; ++c) s += part[(int64_t)c * P_TOTAL + p];
    grad[p] = s;
  }
}

// gA1[u][i] = relu'(h1) * (gH1[u][i] + sum_{v in N(u)} w(u,v)/wdeg(v) gM1[v][i]),
// four channels a thread as in k_mp_nbr
__global__ void __launch_bounds__(256) k_mp_bw_agg(int32_t N, const int64_t *__restrict__ xadj,
                                                   const int32_t *__restrict__ adj,
                                                   const int32_t *__restrict__ ew,
                                                   const float *__restrict__ wdeg,
                                                   const float *__restrict__ gH1,
                                                   const float *__restrict__ gM1,
                                                   const float *__restrict__ H1, float *__restrict__ gA1) {
  constexpr int LN = MH / 4;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < (int64_t)N * LN;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int32_t u = (int32_t)(t / LN);
    const int64_t at = 4 * t;
    float4 s = *reinterpret_cast<const float4 *>(gH1 + at);
    const float4 h = *reinterpret_cast<const float4 *>(H1 + at);
    const int c = 4 * (int)(t % LN);
    int64_t e = xadj[u];
    const int64_t e1 = xadj[u + 1];
    for (; e + 4 <= e1; e += 4) {
      float w[4], d[4];
      float4 g[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int32_t v = adj[e + q];
        w[q] = ew ? (float)ew[e + q] : 1.f;
        d[q] = wdeg[v];
        g[q] = *reinterpret_cast<const float4 *>(gM1 + (int64_t)v * MH + c);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (d[q] > 0.f) fma4(s, w[q] / d[q], g[q]);
    }
    for (; e < e1; ++e) {
      const int32_t v = adj[e];
      const float w = ew ? (float)ew[e] : 1.f, d = wdeg[v];
      if (d > 0.f) fma4(s, w / d, *reinterpret_cast<const float4 *>(gM1 + (int64_t)v * MH + c));
    }
    *reinterpret_cast<float4 *>(gA1 + at) = make_float4(h.x > 0.f ? s.x : 0.f, h.y > 0.f ? s.y : 0.f,
                                                        h.z > 0.f ? s.z : 0.f, h.w > 0.f ? s.w : 0.f);
  }
}

__global__ void k_mp_wdeg(int32_t N, const int64_t *xadj, const int32_t *ew, float *wdeg) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < N;
       v += (int64_t)gridDim.x * blockDim.x) {
    float s = 0;
    for (int64_t e = xadj[v]; e < xadj[v + 1]; ++e) s += ew ? (float)ew[e] : 1.f;
    wdeg[v] = s;
  }
}

__global__ void k_mp_adam(int32_t P, float *master, float *grad, float *am, float *av, __nv_bfloat16 *wbfo,
                          float lr, float b1, float b2, float epsa, float c1, float c2) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < P; i += gridDim.x * blockDim.x) {
    float g = grad[i];
    float m = b1 * am[i] + (1.f - b1) * g;
    float v = b2 * av[i] + (1.f - b2) * g * g;
    am[i] = m;
    av[i] = v;
    float w = master[i] - lr * (m / c1) / (sqrtf(v / c2) + epsa);
    master[i] = w;
    wbfo[i] = __float2bfloat16(w);
    grad[i] = 0.f;
  }
}

__global__ void k_mp_tobf(int32_t P, const float *master, __nv_bfloat16 *wbfo) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < P; i += gridDim.x * blockDim.x)
    wbfo[i] = __float2bfloat16(master[i]);
}

__global__ void k_mp_frombf(int32_t P, const __nv_bfloat16 *w, float *out) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < P; i += gridDim.x * blockDim.x)
    out[i] = __bfloat162float(w[i]);
}

// ------------------------------------------------------------------ host
static void upload_batch(Batch &b, int32_t ng, const int32_t *noff, const int64_t *xadj, const int32_t *adj,
                         const int32_t *vw, const int32_t *ew, const uint64_t *keys, const int32_t *side) {
  b.ng = ng;
  b.N = noff[ng];
  for (int32_t g = 0; g < ng; ++g) b.max_n = std::max(b.max_n, noff[g + 1] - noff[g]);
  b.E = xadj[b.N];
  b.noff.alloc(ng + 1);
  to_dev(b.noff.p, noff, ng + 1);
  b.xadj.alloc(b.N + 1);
  to_dev(b.xadj.p, xadj, b.N + 1);
  b.adj.alloc(b.E);
  to_dev(b.adj.p, adj, b.E);
  if (vw) {
    b.vw.alloc(b.N);
    to_dev(b.vw.p, vw, b.N);
  }
  if (ew) {
    b.ew.alloc(b.E);
    to_dev(b.ew.p, ew, b.E);
  }
  b.keys.alloc(ng);
  to_dev(b.keys.p, keys, ng);
  if (side) {
    b.side.alloc(b.N);
    to_dev(b.side.p, side, b.N);
  }
}

struct Acts {
  DBuf<float> X, M0, H1, M1, H2, S, wdeg;
  DBuf<int32_t> d1, d2;
};

template <class K>
static void mp_smem(K kernel, size_t bytes) {
  KMP_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
}

static void forward(const kmp_mpnn *m, const Batch &b, Acts &a) {
  cudaStream_t s = ctx().stream;
  int32_t N = b.N;
  a.X.alloc((int64_t)N * MF);
  a.M0.alloc((int64_t)N * MF);
  a.H1.alloc((int64_t)N * MH);
  a.M1.alloc((int64_t)N * MH);
  a.H2.alloc((int64_t)N * MH);
  a.S.alloc(N);
  a.d1.alloc(N);
  a.d2.alloc(N);
  const int32_t *vw = b.vw.p, *ew = b.ew.p;
  // hop counts in shared memory for the graphs that fit: sized by the largest of those
  int32_t hop_n = std::min(b.max_n, MP_FEAT_SMEM_N);
  const size_t hop_bytes = 2 * (size_t)hop_n * sizeof(int32_t);
  mp_smem(k_mp_features, 2 * (size_t)MP_FEAT_SMEM_N * sizeof(int32_t));
  k_mp_features<<<grid_for(b.ng, 1, 4), MP_FEAT_T, hop_bytes, s>>>(b.ng, b.noff, b.xadj, b.adj, vw, ew, b.keys,
                                                                  a.X, a.d1, a.d2, hop_n);
  KMP_LAUNCHED("mp_features");
  const int tiles = (int)ceil_div(std::max(N, 1), MP_TILE);
  k_mp_nbr<MF><<<grid_for((int64_t)N * (MF / 4), 256, 8), 256, 0, s>>>(N, b.xadj, b.adj, ew, a.X, a.M0);
  KMP_LAUNCHED("mp_nbr");
  constexpr size_t l1 = mp_layer_smem<MF, false>(), l2 = mp_layer_smem<MH, true>();
  mp_smem(k_mp_layer<MF, false>, l1);
  mp_smem(k_mp_layer<MH, true>, l2);
  k_mp_layer<MF, false><<<grid_for(tiles, 1, 8), MP_T, l1, s>>>(N, m->wbf, P_W1S, P_W1N, P_B1, a.X, a.M0, a.H1,
                                                               nullptr);
  KMP_LAUNCHED("mp_layer");
  k_mp_nbr<MH><<<grid_for((int64_t)N * (MH / 4), 256, 8), 256, 0, s>>>(N, b.xadj, b.adj, ew, a.H1, a.M1);
  KMP_LAUNCHED("mp_nbr");
  k_mp_layer<MH, true><<<grid_for(tiles, 1, 2), MP_T, l2, s>>>(N, m->wbf, P_W2S, P_W2N, P_B2, a.H1, a.M1, a.H2,
                                                              a.S);
  KMP_LAUNCHED("mp_layer");
}

// loss and its gradient (written to m->grad); returns the loss
static float backward(kmp_mpnn *m, const Batch &b, Acts &a) {
  cudaStream_t s = ctx().stream;
  int32_t N = b.N;
  DBuf<float> gS(N), lossg(b.ng), gH1((int64_t)N * MH), gM1((int64_t)N * MH), gA1((int64_t)N * MH);
  a.wdeg.alloc(N);
  const int32_t *ew = b.ew.p;
  k_mp_loss<<<grid_for(b.ng, 1, 8), 256, 0, s>>>(b.ng, b.noff, a.S, b.side, gS, lossg);
  KMP_LAUNCHED("mp_loss");
  // a fixed number of partial sums (not tied to the GPU) keeps results identical everywhere
  int32_t G = (int32_t)std::min<int64_t>(ceil_div(std::max(N, 1), MP_TILE), 256);
  DBuf<float> part((int64_t)G * P_TOTAL);
  mp_smem(k_mp_bw2, MP_BW2_SMEM);
  k_mp_bw2<<<G, MP_T, MP_BW2_SMEM, s>>>(N, m->wbf, gS, a.H2, a.H1, a.M1, gH1, gM1, part);
  KMP_LAUNCHED("mp_bw2");
  k_mp_wdeg<<<grid_for(N, 256), 256, 0, s>>>(N, b.xadj, ew, a.wdeg);
  KMP_LAUNCHED("mp_wdeg");
  k_mp_bw_agg<<<grid_for((int64_t)N * (MH / 4), 256, 8), 256, 0, s>>>(N, b.xadj, b.adj, ew, a.wdeg, gH1, gM1,
                                                                     a.H1, gA1);
  KMP_LAUNCHED("mp_bw_agg");
  k_mp_wgrad1<<<G, MP_T, 0, s>>>(N, gA1, a.X, a.M0, part);
  KMP_LAUNCHED("mp_wgrad1");
  k_mp_reduce<<<grid_for(P_TOTAL, 32), 32, 0, s>>>(G, part, m->grad);
  KMP_LAUNCHED("mp_reduce");
  std::vector<float> hl(b.ng);
  to_host(hl.data(), lossg.p, b.ng);
  float l = 0.f;
  for (float x : hl) l += x;
  return l;
}

template <class F>
static int guarded_mp(F &&f) {
  try {
    ensure_init();
    set_last_error("");
    f();
    return KMP_OK;
  } catch (const Error &e) {
    set_last_error(e.msg);
    return e.code;
  } catch (...) {
    set_last_error("unknown error");
    return KMP_ERR_CUDA;
  }
}

static void check_batch(int32_t ng, const int32_t *noff, const int64_t *xadj) {
  if (ng < 1 || !noff || !xadj) fail(KMP_ERR_ARG, "invalid batch");
  if (noff[0] != 0) fail(KMP_ERR_ARG, "noff[0] != 0");
  for (int32_t g = 0; g < ng; ++g)
    if (noff[g + 1] < noff[g]) fail(KMP_ERR_ARG, "noff must be non-decreasing");
}

}  // namespace kmp

using namespace kmp;

extern "C" {

int kmp_mpnn_num_params(void) { return P_TOTAL; }

int kmp_mpnn_create(uint64_t seed, kmp_mpnn **out) {
  return guarded_mp([&] {
    if (!out) fail(KMP_ERR_ARG, "out is NULL");
    kmp_mpnn *m = new kmp_mpnn;
    m->master = static_cast<float *>(dmalloc(P_TOTAL * sizeof(float)));
    m->wbf = static_cast<__nv_bfloat16 *>(dmalloc(P_TOTAL * sizeof(__nv_bfloat16)));
    m->am = static_cast<float *>(dmalloc(P_TOTAL * sizeof(float)));
    m->av = static_cast<float *>(dmalloc(P_TOTAL * sizeof(float)));
    m->grad = static_cast<float *>(dmalloc(P_TOTAL * sizeof(float)));
    // He-style uniform initialisation from the counter-based generator
    std::vector<float> h(P_TOTAL, 0.f);
    auto uni = [&](int i) {
      return (double)(key_step(mix64(seed + 0x9E3779B97F4A7C15ull), (uint64_t)i) >> 11) * 0x1.0p-53 * 2.0 - 1.0;
    };
    for (int i = 0; i < MH * MF; ++i) {
      h[P_W1S + i] = (float)(uni(P_W1S + i) * std::sqrt(6.0 / (2 * MF)));
      h[P_W1N + i] = (float)(uni(P_W1N + i) * std::sqrt(6.0 / (2 * MF)));
    }
    for (int i = 0; i < MH * MH; ++i) {
      h[P_W2S + i] = (float)(uni(P_W2S + i) * std::sqrt(6.0 / (2 * MH)));
      h[P_W2N + i] = (float)(uni(P_W2N + i) * std::sqrt(6.0 / (2 * MH)));
    }
    for (int i = 0; i < MH; ++i) h[P_WO + i] = (float)(uni(P_WO + i) * std::sqrt(6.0 / MH));
    to_dev(m->master, h.data(), P_TOTAL);
    KMP_CUDA(cudaMemsetAsync(m->am, 0, P_TOTAL * sizeof(float), ctx().stream));
    KMP_CUDA(cudaMemsetAsync(m->av, 0, P_TOTAL * sizeof(float), ctx().stream));
    KMP_CUDA(cudaMemsetAsync(m->grad, 0, P_TOTAL * sizeof(float), ctx().stream));
    k_mp_tobf<<<grid_for(P_TOTAL, 256), 256, 0, ctx().stream>>>(P_TOTAL, m->master, m->wbf);
    KMP_LAUNCHED("mp_tobf");
    sync_and_check("mpnn_create");
    *out = m;
  });
}

int kmp_mpnn_free(kmp_mpnn *m) {
  return guarded_mp([&] {
    if (!m) return;
    if (proposer().W == m->wbf) proposer().W = nullptr;
    dfree(m->master);
    dfree(m->wbf);
    dfree(m->am);
    dfree(m->av);
    dfree(m->grad);
    KMP_CUDA(cudaStreamSynchronize(ctx().stream));
    delete m;
  });
}

int kmp_mpnn_get_params(const kmp_mpnn *m, float *params) {
  return guarded_mp([&] {
    if (!m || !params) fail(KMP_ERR_ARG, "NULL argument");
    DBuf<float> t(P_TOTAL);
    k_mp_frombf<<<grid_for(P_TOTAL, 256), 256, 0, ctx().stream>>>(P_TOTAL, m->wbf, t);
    KMP_LAUNCHED("mp_frombf");
    to_host(params, t.p, P_TOTAL);
  });
}

int kmp_mpnn_set_params(kmp_mpnn *m, const float *params) {
  return guarded_mp([&] {
    if (!m || !params) fail(KMP_ERR_ARG, "NULL argument");
    to_dev(m->master, params, P_TOTAL);
    k_mp_tobf<<<grid_for(P_TOTAL, 256), 256, 0, ctx().stream>>>(P_TOTAL, m->master, m->wbf);
    KMP_LAUNCHED("mp_tobf");
    sync_and_check("mpnn_set_params");
  });
}

int kmp_mpnn_forward(kmp_mpnn *m, int32_t ng, const int32_t *noff, const int64_t *xadj, const int32_t *adj,
                     const int32_t *vw, const int32_t *ew, const uint64_t *keys, float *scores,
                     float *features) {
  return guarded_mp([&] {
    if (!m || !scores) fail(KMP_ERR_ARG, "NULL argument");
    check_batch(ng, noff, xadj);
    Batch b;
    upload_batch(b, ng, noff, xadj, adj, vw, ew, keys, nullptr);
    Acts a;
    forward(m, b, a);
    to_host(scores, a.S.p, b.N);
    if (features) to_host(features, a.X.p, (size_t)b.N * MF);
    sync_and_check("mpnn_forward");
  });
}

int kmp_mpnn_gradients(kmp_mpnn *m, int32_t ng, const int32_t *noff, const int64_t *xadj, const int32_t *adj,
                       const int32_t *vw, const int32_t *ew, const uint64_t *keys, const int32_t *side,
                       float *loss_out, float *grad_out) {
  return guarded_mp([&] {
    if (!m || !side) fail(KMP_ERR_ARG, "NULL argument");
    check_batch(ng, noff, xadj);
    Batch b;
    upload_batch(b, ng, noff, xadj, adj, vw, ew, keys, side);
    Acts a;
    forward(m, b, a);
    KMP_CUDA(cudaMemsetAsync(m->grad, 0, P_TOTAL * sizeof(float), ctx().stream));
    float l = backward(m, b, a);
    if (grad_out) to_host(grad_out, m->grad, P_TOTAL);
    KMP_CUDA(cudaMemsetAsync(m->grad, 0, P_TOTAL * sizeof(float), ctx().stream));
    sync_and_check("mpnn_gradients");
    if (loss_out) *loss_out = l;
  });
}

int kmp_mpnn_train(kmp_mpnn *m, int32_t ng, const int32_t *noff, const int64_t *xadj, const int32_t *adj,
                   const int32_t *vw, const int32_t *ew, const uint64_t *keys, const int32_t *side,
                   int32_t epochs, float lr, float *loss_per_epoch) {
  return guarded_mp([&] {
    if (!m || !side || epochs < 0 || !(lr > 0.f)) fail(KMP_ERR_ARG, "invalid arguments");
    check_batch(ng, noff, xadj);
    Batch b;
    upload_batch(b, ng, noff, xadj, adj, vw, ew, keys, side);
    for (int32_t ep = 0; ep < epochs; ++ep) {
      Acts a;
      forward(m, b, a);
      float l = backward(m, b, a);
      m->step += 1;
      const float b1 = 0.9f, b2 = 0.999f;
      float c1 = 1.f - std::pow(b1, (float)m->step), c2 = 1.f - std::pow(b2, (float)m->step);
      k_mp_adam<<<grid_for(P_TOTAL, 256), 256, 0, ctx().stream>>>(P_TOTAL, m->master, m->grad, m->am, m->av,
                                                                 m->wbf, lr, b1, b2, 1e-8f, c1, c2);
      KMP_LAUNCHED("mp_adam");
      if (loss_per_epoch) loss_per_epoch[ep] = l;
    }
    sync_and_check("mpnn_train");
  });
}

int kmp_set_proposer(const kmp_mpnn *m) {
  return guarded_mp([&] { proposer().W = m ? m->wbf : nullptr; });
}

int kmp_sample_sink_level(int32_t item_level) {
  return guarded_mp([&] {
    if (item_level < 0 || item_level > 1) fail(KMP_ERR_ARG, "sink level must be 0 or 1");
    sample_sink().item_level = item_level;
  });
}

int kmp_sample_sink_open(int32_t max_graphs, int64_t max_nodes, int64_t max_entries) {
  return guarded_mp([&] {
    if (max_graphs < 1 || max_nodes < 1 || max_entries < 0) fail(KMP_ERR_ARG, "invalid sink capacity");
    sink_release();
    SampleSink &K = sample_sink();
    cudaStream_t s = ctx().stream;
    K.max_graphs = max_graphs;
    K.max_nodes = max_nodes;
    K.max_entries = max_entries;
    K.counters = static_cast<unsigned long long *>(dmalloc(4 * sizeof(unsigned long long)));
    K.rec = static_cast<int64_t *>(dmalloc((size_t)max_graphs * 5 * sizeof(int64_t)));
    K.deg = static_cast<int32_t *>(dmalloc((size_t)max_nodes * sizeof(int32_t)));
    K.vw = static_cast<int32_t *>(dmalloc((size_t)max_nodes * sizeof(int32_t)));
    K.side = static_cast<int32_t *>(dmalloc((size_t)max_nodes * sizeof(int32_t)));
    K.adj = static_cast<int32_t *>(dmalloc((size_t)std::max<int64_t>(max_entries, 1) * sizeof(int32_t)));
    K.ew = static_cast<int32_t *>(dmalloc((size_t)std::max<int64_t>(max_entries, 1) * sizeof(int32_t)));
    KMP_CUDA(cudaMemsetAsync(K.counters, 0, 4 * sizeof(unsigned long long), s));
    KMP_CUDA(cudaMemsetAsync(K.rec, 0xFF, (size_t)max_graphs * 5 * sizeof(int64_t), s));
    sync_and_check("sample_sink_open");
  });
}

int kmp_sample_sink_count(int32_t *graphs, int64_t *nodes, int64_t *entries, int64_t *dropped) {
  return guarded_mp([&] {
    SampleSink &K = sample_sink();
    if (!K.counters) fail(KMP_ERR_ARG, "no sample sink is open");
    unsigned long long c[4];
    to_host(c, K.counters, 4);
    int64_t kept = (int64_t)c[0] - (int64_t)c[3];
    // kept records sit at reservation indices below max_graphs; their node
    // and entry totals are summed from the records themselves
    std::vector<int64_t> rec((size_t)K.max_graphs * 5);
    to_host(rec.data(), K.rec, rec.size());
    int64_t nn = 0, ne = 0;
    int32_t ng = 0;
    for (int32_t g = 0; g < K.max_graphs; ++g)
      if (rec[5 * g + 1] >= 0) {
        ++ng;
        nn += rec[5 * g + 1];
        ne += rec[5 * g + 3];
      }
    if (ng != kept) fail(KMP_ERR_CUDA, "sample sink records inconsistent");
    if (graphs) *graphs = ng;
    if (nodes) *nodes = nn;
    if (entries) *entries = ne;
    if (dropped) *dropped = (int64_t)c[3];
  });
}

int kmp_sample_sink_read(int32_t *noff, int64_t *xadj, int32_t *adj, int32_t *vw, int32_t *ew,
                         uint64_t *keys, int32_t *side) {
  return guarded_mp([&] {
    SampleSink &K = sample_sink();
    if (!K.counters) fail(KMP_ERR_ARG, "no sample sink is open");
    if (!noff || !xadj || !adj || !vw || !ew || !keys || !side) fail(KMP_ERR_ARG, "NULL argument");
    std::vector<int64_t> rec((size_t)K.max_graphs * 5);
    to_host(rec.data(), K.rec, rec.size());
    std::vector<int32_t> idx;
    for (int32_t g = 0; g < K.max_graphs; ++g)
      if (rec[5 * g + 1] >= 0) idx.push_back(g);
    // deterministic order: by item key (unique per item and round), then size
    std::sort(idx.begin(), idx.end(), [&](int32_t a, int32_t b) {
      uint64_t ka = (uint64_t)rec[5 * a + 4], kb = (uint64_t)rec[5 * b + 4];
      if (ka != kb) return ka < kb;
      return rec[5 * a + 1] < rec[5 * b + 1];
    });
    int64_t nmax = 0, emax = 0;
    for (int32_t g : idx) {
      nmax = std::max(nmax, rec[5 * g] + rec[5 * g + 1]);
      emax = std::max(emax, rec[5 * g + 2] + rec[5 * g + 3]);
    }
    std::vector<int32_t> hdeg(nmax), hvw(nmax), hside(nmax), hadj(emax), hew(emax);
    to_host(hdeg.data(), K.deg, nmax);
    to_host(hvw.data(), K.vw, nmax);
    to_host(hside.data(), K.side, nmax);
    to_host(hadj.data(), K.adj, emax);
    to_host(hew.data(), K.ew, emax);
    int64_t nb = 0, eb = 0;
    noff[0] = 0;
    xadj[0] = 0;
    for (size_t i = 0; i < idx.size(); ++i) {
      const int64_t *r = &rec[5 * idx[i]];
      int64_t n0 = r[0], n = r[1], e0 = r[2], m = r[3];
      keys[i] = (uint64_t)r[4];
      for (int64_t v = 0; v < n; ++v) {
        xadj[nb + v + 1] = xadj[nb + v] + hdeg[n0 + v];
        vw[nb + v] = hvw[n0 + v];
        side[nb + v] = hside[n0 + v];
      }
      for (int64_t e = 0; e < m; ++e) {
        adj[eb + e] = (int32_t)(hadj[e0 + e] + nb);
        ew[eb + e] = hew[e0 + e];
      }
      nb += n;
      eb += m;
      noff[i + 1] = (int32_t)nb;
    }
  });
}

int kmp_sample_sink_close(void) {
  return guarded_mp([&] {
    KMP_CUDA(cudaStreamSynchronize(ctx().stream));
    sink_release();
  });
}

}  // extern "C"
