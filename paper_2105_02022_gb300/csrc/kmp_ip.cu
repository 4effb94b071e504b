// Batched multilevel initial bipartitioning (Section 4.2) for Algorithm 2
// (bipartitionBlocks): every block that must be split becomes one work item;
// all items of a split round run in ONE persistent launch whose CTAs take
// items from a device work queue (largest first).  Per item, one CTA:
//   1. coarsens the induced subgraph G[B] with the deterministic sub-round LP
//      (CTA-parallel rating with per-warp hash tables, commit by a bitonic
//      sort of (target, gain desc, node) keys and a segmented prefix sum),
//      packs isolated nodes, and contracts (sort of (cu, cv) pairs, run sums),
//      level after level until nothing contracts or the shrink stalls;
//   2. runs the portfolio -- random, BFS and greedy graph growing starts, each
//      refined by 2-way FM -- with one warp per repetition; in learned mode
//      the CTA first scores the coarsest graph with the message-passing
//      network (kmp_mpnn.cuh) and its score order is one more start, ahead of
//      a reduced portfolio; the rest of the portfolio runs only if the best so
//      far is infeasible;
//   3. projects the best bipartition up the item's hierarchy and runs 2-way FM
//      (one warp) on every level.
// Scratch comes from a region per CTA through a bump allocator, reset for every
// item; if a region is too small the launch reports it and the host repeats the
// round with larger regions, so results never depend on scratch sizes.
#include <algorithm>
#include <cmath>

#include "kmp_internal.cuh"
#include "kmp_mpnn.cuh"
#include "kmp_plan.h"

#ifndef KMP_IP_MULTI
#define KMP_IP_MULTI 0
#endif

namespace kmp {

constexpr int IPT = 256;
constexpr int IPW = IPT / 32;
constexpr int IP_MAXL = 63;
constexpr int32_t IP_MAX_N = 65535;
constexpr uint16_t IP_NONE = 0xFFFF;  // no node: ids are below IP_MAX_N
// Dynamic shared memory of a bipartitioner CTA: the working state of the item's
// phases (dyn_words) and behind it a hash table per warp (wtab slots of key and
// weight: rows up to wtab / 2 entries).  An item's time is latency, so what counts
// is how many an SM works on.  A round with more items than SMs: 67 KB in all,
// three CTAs an SM (with 80 registers a thread).  That holds items of up to 2300
// nodes; larger ones work in their scratch, which is still faster than two CTAs an
// SM that hold 3350 nodes (4096 items of 200..4000 nodes: 32.4 against 38.2 ms).
// Otherwise the items are on the critical path: one CTA an SM with what it offers.
// The tables take what the largest item's state leaves, from 256 to 2048 slots:
// coarse R-MAT items of 300 nodes have rows of 300 entries, and a row beyond its
// warp's table is aggregated in the item's scratch (partition of R-MAT 2^22, k = 4096:
// 372.0 -> 368.4 ms).
constexpr int32_t IP_WORDS3 = 16896, IP_WORDS1 = 53192, IP_WTAB_MIN = 256, IP_WTAB_MAX = 2048;

struct ItemDesc {
  int64_t vbase;  // first member position
  int64_t ebase;  // first induced edge
  uint64_t key;
  int32_t n, m;
  int32_t t0, t1, L0, L1;
  int32_t pad0, pad1;
};

struct IPArgs {
  const ItemDesc *items;
  const int32_t *order;   // item processing order
  int32_t nitems;
  int32_t *queue;         // items taken beyond the CTAs' first ones
  int32_t *oom;           // set when a scratch region was too small
  const int64_t *gx;      // induced CSR offsets over all members (n+1)
  const uint16_t *sadj;   // local neighbour ids (an item has at most IP_MAX_N nodes)
  const int32_t *sew;     // null: unit weights
  const int32_t *svw;
  int32_t *side_out;      // per member position
  int32_t *scratch;       // CTA b's region, reused by its items: [region[b], region[b + 1])
  const int64_t *region;
  // configuration
  int32_t S, ip_C, ip_lp_rounds, rep_random, rep_bfs, rep_ggg, fm_passes, fm_stop;
  int32_t conv_num, conv_den;
  // learned mode: proposer weights (null: plain portfolio) and reduced repetitions
  const __nv_bfloat16 *W;
  int32_t lrep_random, lrep_bfs, lrep_ggg;
  int32_t adaptive;  // adaptive portfolio (plain mode only)
  int32_t learned_item;  // learned item mode (W set): start on the item graph, FM there
  SampleSink sink;  // counters null: no recording
  int32_t wtab;       // slots of a warp's shared hash table
  int32_t dyn_words;  // words of the phases' working state in shared memory
};

#if KMP_IP_MULTI
namespace multi {
#endif

// A level of an item.  Neighbour ids take 16 bits and unit weights are not
// stored, so the 2048-node items of a degree-16 mesh take 64 KB each instead of
// 250: what the resident items read again and again stays in L2.
struct LG {
  int32_t n, m;
  int32_t *xadj;
  uint16_t *adj;
  int32_t *ew;  // null: unit weights
  int32_t *vw;
  int32_t maxdeg, maxc;
};
__device__ __forceinline__ int32_t lg_w(const LG &g, int32_t q) { return g.ew ? g.ew[q] : 1; }

// The CTA's scratch region: base and words, in shared memory, so that a take holds no
// registers for them (4096 items of 200..4000 nodes: 32.3 ms with both in registers,
// 560 bytes of spill loads a thread; 30.4 like this, 288)
struct Region {
  int32_t *base;
  int64_t cap;
};
__device__ __forceinline__ Region &region() {
  __shared__ Region r;
  return r;
}
struct Bump {
  int64_t top;
  bool oom;
  __device__ int32_t *take(int64_t cnt) {
    int64_t t = (top + 1) & ~1ll;
    if (oom || t + cnt > region().cap) {
      oom = true;
      return region().base;  // never dereferenced: callers check oom
    }
    top = t + cnt;
    return region().base + t;
  }
};

// ------------------------------------------------------- block helpers
__device__ int64_t block_sum64(int64_t v) {
  __shared__ int64_t red[IPW];
  v = warp_sum64(v);
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) red[w] = v;
  __syncthreads();
  int64_t s = 0;
  for (int i = 0; i < IPW; ++i) s += red[i];
  __syncthreads();
  return s;
}

__device__ int32_t block_max32(int32_t v) {
  __shared__ int32_t red[IPW];
#pragma unroll
  for (int m = 16; m > 0; m >>= 1) v = max(v, __shfl_xor_sync(0xFFFFFFFFu, v, m));
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) red[w] = v;
  __syncthreads();
  int32_t s = red[0];
  for (int i = 1; i < IPW; ++i) s = max(s, red[i]);
  __syncthreads();
  return s;
}

// exclusive scan of in[0..n) into out (may alias), returns total
template <class T>
__device__ T block_scan_excl(const T *in, T *out, int32_t n) {
  __shared__ T wsum[IPW];
  __shared__ T carry;
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int32_t base = 0; base < n; base += IPT) {
    int32_t i = base + threadIdx.x;
    T v = i < n ? in[i] : T(0);
    T x = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      T y = __shfl_up_sync(0xFFFFFFFFu, x, d);
      if (lane >= d) x += y;
    }
    if (lane == 31) wsum[w] = x;
    __syncthreads();
    T pre = carry;
    for (int k = 0; k < w; ++k) pre += wsum[k];
    T tot = 0;
    for (int k = 0; k < IPW; ++k) tot += wsum[k];
    if (i < n) out[i] = pre + x - v;
    __syncthreads();
    if (threadIdx.x == 0) carry += tot;
    __syncthreads();
  }
  T r = carry;
  __syncthreads();
  return r;
}

// bitonic sort of P (power of two) keys ascending, optional values; block-wide
__device__ void block_bitonic(uint64_t *key, int32_t *val, int32_t P) {
  for (int32_t k = 2; k <= P; k <<= 1)
    for (int32_t j = k >> 1; j > 0; j >>= 1) {
      for (int32_t i = threadIdx.x; i < P; i += IPT) {
        int32_t l = i ^ j;
        if (l > i) {
          uint64_t x = key[i], y = key[l];
          bool up = (i & k) == 0;
          if ((x > y) == up) {
            key[i] = y;
            key[l] = x;
            if (val) {
              int32_t t = val[i];
              val[i] = val[l];
              val[l] = t;
            }
          }
        }
      }
      __syncthreads();
    }
}

// warp bitonic of P pairs (h, v) ascending by (h, v)
__device__ void warp_bitonic_hv(uint64_t *h, int32_t *v, int32_t P) {
  int lane = threadIdx.x & 31;
  for (int32_t k = 2; k <= P; k <<= 1)
    for (int32_t j = k >> 1; j > 0; j >>= 1) {
      for (int32_t i = lane; i < P; i += 32) {
        int32_t l = i ^ j;
        if (l > i) {
          uint64_t a = h[i], b = h[l];
          int32_t va = v[i], vb = v[l];
          bool gt = a > b || (a == b && va > vb);
          bool up = (i & k) == 0;
          if (gt == up) {
            h[i] = b; h[l] = a;
            v[i] = vb; v[l] = va;
          }
        }
      }
      __syncwarp();
    }
}

// warp bitonic of P (power of two) 64-bit keys ascending
__device__ void warp_bitonic_u64(uint64_t *a, int32_t P) {
  int lane = threadIdx.x & 31;
  for (int32_t k = 2; k <= P; k <<= 1)
    for (int32_t j = k >> 1; j > 0; j >>= 1) {
      for (int32_t i = lane; i < P; i += 32) {
        int32_t l = i ^ j;
        if (l > i) {
          uint64_t x = a[i], y = a[l];
          if ((x > y) == ((i & k) == 0)) {
            a[i] = y;
            a[l] = x;
          }
        }
      }
      __syncwarp();
    }
}

__device__ __forceinline__ int32_t pow2_at_least(int32_t x) {
  int32_t p = 1;
  while (p < x) p <<= 1;
  return p;
}

// ------------------------------------------------------ item clustering
// rating of node u by one warp; returns (via lane 0) proposal target or -1
__device__ void item_rate(const LG &g, int32_t u, const uint16_t *label, const int32_t *wt, int32_t U,
                          uint32_t rk_hi, uint32_t wtab, int32_t *skeys, int32_t *svals, int32_t *gkeys,
                          int32_t *gvals, uint16_t *out_t, int32_t *out_g) {
  int lane = threadIdx.x & 31;
  int32_t b = g.xadj[u], e = g.xadj[u + 1], deg = e - b;
  uint32_t cap = 32;
  while ((int64_t)cap < 2ll * deg) cap <<= 1;
  uint32_t mask = cap - 1;
  // shared-memory table unless this node's table does not fit there
  int32_t *keys = cap <= wtab ? skeys : gkeys;
  int32_t *vals = cap <= wtab ? svals : gvals;
  for (uint32_t i = lane; i < cap; i += 32) {
    keys[i] = HT_EMPTY;
    vals[i] = 0;
  }
  __syncwarp();
  for (int32_t q = b + lane; q < e; q += 32) ht_add(keys, vals, mask, label[g.adj[q]], lg_w(g, q));
  __syncwarp();
  int32_t own = label[u], cu = g.vw[u];
  int32_t rown = ht_get(keys, vals, mask, own);
  uint64_t kc = 0;
  int32_t lc = -1;
  for (uint32_t i = lane; i < cap; i += 32) {
    int32_t K = keys[i];
    if (K == HT_EMPTY || K == own) continue;
    if ((int64_t)wt[K] + cu > U) continue;
    uint64_t k = ((uint64_t)(uint32_t)vals[i] << 32) | (uint64_t)(0xFFFFFFFFu - perm32(rk_hi, K));
    if (k > kc) { kc = k; lc = K; }
  }
  uint64_t mc = group_max64<32>(kc);
  unsigned bc = __ballot_sync(0xFFFFFFFFu, mc != 0 && kc == mc);
  lc = __shfl_sync(0xFFFFFFFFu, lc, bc ? __ffs(bc) - 1 : 0);
  if (lane == 0) {
    int32_t rc = (int32_t)(mc >> 32);
    if (mc != 0 && rc > rown) {
      *out_t = (uint16_t)lc;
      *out_g = rc - rown;
    } else {
      *out_t = IP_NONE;
    }
  }
  __syncwarp();
}

// inputs of one group node: neighbour label and edge weight of this lane, own
// label and node weight (u < 0: no node)
struct GroupIn {
  int32_t l, x, own, cu;
};

// rating of 32 / G nodes by one warp, G lanes per node (degree <= G, one
// neighbour per lane): lanes of a group holding the same label form a peer
// set whose weight sum is that label's rating.  Same decision as item_rate.
template <int G>
__device__ __forceinline__ void item_group_rate(const GroupIn &in, bool unit, int32_t u, const int32_t *wt, int32_t U,
                                                uint32_t rk_hi, uint16_t *pt, int32_t *pg) {
  const int lane = threadIdx.x & 31, gl = lane & (G - 1);
  const unsigned gmask = (G == 32) ? 0xFFFFFFFFu : (((1u << G) - 1u) << (lane & ~(G - 1)));
  const int32_t l = in.l;
  // as k_rate's groups: the set's size with unit weights, else its peers' weights, one by
  // one here (an item's sets are small: 4096 items 30.33 ms, 30.47 with peer_sum)
  const unsigned peers = __match_any_sync(0xFFFFFFFFu, l) & gmask;
  int32_t r;
  if (unit) {
    r = __popc(peers);
  } else {
    r = in.x;
    unsigned rest = l < 0 ? 0 : peers & ~(1u << lane);
    while (__any_sync(0xFFFFFFFFu, rest != 0)) {
      const int32_t t = __shfl_sync(0xFFFFFFFFu, in.x, rest ? __ffs(rest) - 1 : lane);
      if (rest) r += t;
      rest &= rest - 1;
    }
  }
  unsigned bown = __ballot_sync(0xFFFFFFFFu, l >= 0 && l == in.own) & gmask;
  int32_t rown = __shfl_sync(0xFFFFFFFFu, r, bown ? __ffs(bown) - 1 : lane);
  if (!bown) rown = 0;
  bool adm = l >= 0 && l != in.own && (int64_t)wt[l] + in.cu <= U;
  uint64_t k = adm ? ((uint64_t)(uint32_t)r << 32) | (uint64_t)(0xFFFFFFFFu - perm32(rk_hi, l)) : 0ull;
  uint64_t mc = group_max64<G>(k);
  unsigned bc = __ballot_sync(0xFFFFFFFFu, mc != 0 && k == mc) & gmask;
  int32_t lc = __shfl_sync(0xFFFFFFFFu, l, bc ? __ffs(bc) - 1 : lane);
  if (gl == 0 && u >= 0) {
    int32_t rc = (int32_t)(mc >> 32);
    if (mc != 0 && rc > rown) {
      pt[u] = (uint16_t)lc;
      pg[u] = rc - rown;
    } else {
      pt[u] = IP_NONE;
    }
  }
}

// the nodes sl[lo..hi) rated 32 / G per warp step
template <int G>
__device__ __forceinline__ void item_rate_groups(const LG &g, const uint16_t *sl, int32_t lo, int32_t hi,
                                                 const uint16_t *label, const int32_t *wt, int32_t U,
                                                 uint32_t rk_hi, uint16_t *pt, int32_t *pg) {
  constexpr int per = 32 / G;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, gl = lane & (G - 1);
  for (int32_t i0 = lo + per * w; i0 < hi; i0 += per * IPW) {
    const int32_t i = i0 + lane / G, u = i < hi ? sl[i] : -1;
    GroupIn a{-1, 0, -1, 0};
    if (u >= 0) {
      const int32_t b = g.xadj[u], deg = g.xadj[u + 1] - b;
      a.own = label[u];
      a.cu = g.vw[u];
      if (gl < deg) {
        a.l = label[g.adj[b + gl]];
        a.x = lg_w(g, b + gl);
      }
    }
    item_group_rate<G>(a, g.ew == nullptr, u, wt, U, rk_hi, pt, pg);
  }
}

// degree class of a node for the item rating schedule: 0 (<= 16, two nodes
// per warp), 1 (<= 32, one node per warp, no table), 2 (table)
__device__ __forceinline__ int32_t item_deg_class(int32_t deg) { return deg <= 16 ? 0 : (deg <= 32 ? 1 : 2); }

// segmented inclusive scan in shared memory (one element per thread)
__device__ int64_t block_seg_scan(int64_t x, bool head) {
  __shared__ int64_t sv[IPT];
  __shared__ int32_t sf[IPT];
  int t = threadIdx.x;
  sv[t] = x;
  sf[t] = head ? 1 : 0;
  __syncthreads();
  for (int d = 1; d < IPT; d <<= 1) {
    int64_t v = sv[t];
    int32_t f = sf[t];
    if (t >= d && !f) {
      v += sv[t - d];
      f |= sf[t - d];
    }
    __syncthreads();
    sv[t] = v;
    sf[t] = f;
    __syncthreads();
  }
  int64_t r = sv[t];
  __syncthreads();
  return r;
}

// LP clustering of one item level + isolated packing; returns #clusters
__device__ int32_t item_cluster(const IPArgs &A, const LG &g, int32_t U, uint64_t basekey,
                                int32_t *label, Bump &B, int32_t *wkeys, int32_t *wvals, int32_t *dyn,
                                int32_t dyn_words) {
  __shared__ int32_t s_cnt, s_fast;
  __shared__ int32_t s_moved;
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int32_t n = g.n;
  int64_t mark = B.top;
  int32_t P = pow2_at_least(n > 1 ? n : 2);
  // working arrays: in shared memory when the level fits (every phase of a
  // sub-round reads them), else in the item's scratch; labels are written
  // to `label` at the end either way.  The sort space of contested proposals
  // sits in shared memory behind them when a sub-round's proposals fit
  // there, else in the scratch (pl_g, always reserved).
  int32_t *wt, *pg, *tsum;  // tsum: proposed weight per target (kept zero between uses)
  uint16_t *lab, *pt, *sl, *fl;  // sl: the round's nodes by sub-round; fl: accepted
                                 // proposals of uncontested targets
  uint8_t *act, *act2;           // active flags
  uint64_t *pl_s = nullptr;
  int32_t pl_cap = 0;   // entries of pl_s
  uint64_t *pl_g = reinterpret_cast<uint64_t *>(B.take(2ll * P));
  const int32_t id_words = (n + 1) / 2, flag_words = (n + 3) / 4;
  const int64_t lp_words = 3ll * n + 4ll * id_words + 2ll * flag_words;
  const bool fast = lp_words + 2 + 128 <= dyn_words;
  {
    int32_t *q = fast ? dyn : B.take(lp_words);
    wt = q; q += n;
    pg = q; q += n;
    tsum = q; q += n;
    lab = reinterpret_cast<uint16_t *>(q); q += id_words;
    pt = reinterpret_cast<uint16_t *>(q); q += id_words;
    sl = reinterpret_cast<uint16_t *>(q); q += id_words;
    fl = reinterpret_cast<uint16_t *>(q); q += id_words;
    act = reinterpret_cast<uint8_t *>(q); q += flag_words;
    act2 = reinterpret_cast<uint8_t *>(q); q += flag_words;
    if (fast) {
      q += (q - dyn) & 1;  // 8-byte alignment
      pl_s = reinterpret_cast<uint64_t *>(q);
      pl_cap = (int32_t)((dyn_words - (q - dyn)) / 2);
    }
  }
  int32_t *gtab = nullptr;
  uint32_t gcap = 0;
  if (g.maxdeg > A.wtab / 2) {
    gcap = 32;
    while ((int64_t)gcap < 2ll * g.maxdeg) gcap <<= 1;
    gtab = B.take(2ll * gcap * IPW);
  }
  if (B.oom) return -1;
  for (int32_t v = threadIdx.x; v < n; v += IPT) {
    lab[v] = (uint16_t)v;
    wt[v] = g.vw[v];
    act[v] = 1;
    tsum[v] = 0;
  }
  __syncthreads();
  int32_t *mk = wkeys + w * A.wtab, *mv = wvals + w * A.wtab;
  int32_t *gk = nullptr, *gv = nullptr;
  if (gtab) {
    gk = gtab + (int64_t)w * 2 * gcap;
    gv = gk + gcap;
  }
  for (int32_t r = 0; r < A.ip_lp_rounds; ++r) {
    uint64_t rk = key_step(basekey, (uint64_t)r);
    uint32_t rk_hi = (uint32_t)(rk >> 32);
    // the round's active nodes (with edges) bucketed by sub-round and, inside
    // a sub-round, by degree class (the rating schedule; any order inside a
    // sub-round gives the same result)
    __shared__ int32_t s_soff[3 * 8 + 1], s_fill[3 * 8];
    if (threadIdx.x < 3 * 8) s_fill[threadIdx.x] = 0;
    if (threadIdx.x == 0) s_moved = 0;
    __syncthreads();
    for (int32_t v = threadIdx.x; v < n; v += IPT) {
      act2[v] = 0;
      int32_t d = g.xadj[v + 1] - g.xadj[v];
      if (act[v] && d > 0)
        atomicAdd(&s_fill[3 * (int32_t)(key_step(rk, (uint64_t)(uint32_t)v) & (uint64_t)(A.S - 1)) +
                          item_deg_class(d)],
                  1);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      s_soff[0] = 0;
      for (int32_t x = 0; x < 3 * A.S; ++x) {
        s_soff[x + 1] = s_soff[x] + s_fill[x];
        s_fill[x] = 0;
      }
    }
    __syncthreads();
    for (int32_t v = threadIdx.x; v < n; v += IPT) {
      int32_t d = g.xadj[v + 1] - g.xadj[v];
      if (act[v] && d > 0) {
        int32_t x = 3 * (int32_t)(key_step(rk, (uint64_t)(uint32_t)v) & (uint64_t)(A.S - 1)) + item_deg_class(d);
        sl[s_soff[x] + atomicAdd(&s_fill[x], 1)] = (uint16_t)v;
      }
    }
    __syncthreads();
    for (int32_t s = 0; s < A.S; ++s) {
      const int32_t lo = s_soff[3 * s], hi = s_soff[3 * s + 3];
      const int32_t m1 = s_soff[3 * s + 1], m2 = s_soff[3 * s + 2];
      // contested proposals are at most the sub-round's nodes
      uint64_t *pl = pow2_at_least(hi - lo > 1 ? hi - lo : 2) <= pl_cap ? pl_s : pl_g;
      // rating: two nodes per warp, then one per warp without a table, then
      // one per warp with a table
      item_rate_groups<16>(g, sl, lo, m1, lab, wt, U, rk_hi, pt, pg);
      item_rate_groups<32>(g, sl, m1, m2, lab, wt, U, rk_hi, pt, pg);
      for (int32_t i = m2 + w; i < hi; i += IPW) {
        int32_t u = sl[i];
        item_rate(g, u, lab, wt, U, rk_hi, (uint32_t)A.wtab, mk, mv, gk, gv, &pt[u], &pg[u]);
      }
      if (threadIdx.x == 0) {
        s_cnt = 0;
        s_fast = 0;
      }
      __syncthreads();
      // proposed weight per target
      for (int32_t i = lo + threadIdx.x; i < hi; i += IPT) {
        int32_t u = sl[i], T = pt[u];
        if (T != IP_NONE) atomicAdd(&tsum[T], g.vw[u]);
      }
      __syncthreads();
      // a target whose proposals all fit takes them all; only the proposals
      // of contested targets need the (target, gain desc, node) order
      for (int32_t i = lo + threadIdx.x; i < hi; i += IPT) {
        int32_t u = sl[i], T = pt[u];
        if (T == IP_NONE) continue;
        if ((int64_t)wt[T] + tsum[T] <= U) {
          fl[atomicAdd(&s_fast, 1)] = (uint16_t)u;
        } else {
          int32_t p = atomicAdd(&s_cnt, 1);
          pl[p] = ((uint64_t)(uint32_t)T << 47) | ((uint64_t)(uint32_t)(0x7FFFFFFF - pg[u]) << 16) |
                  (uint64_t)(uint32_t)u;
        }
      }
      __syncthreads();
      for (int32_t i = lo + threadIdx.x; i < hi; i += IPT) {
        int32_t T = pt[sl[i]];
        if (T != IP_NONE) tsum[T] = 0;  // every reader is past the barrier above
      }
      int32_t np = s_cnt, nf = s_fast;
      if (np > 0) {
        int32_t Pp = pow2_at_least(np);
        for (int32_t i = np + threadIdx.x; i < Pp; i += IPT) pl[i] = ~0ull;
        __syncthreads();
        block_bitonic(pl, nullptr, Pp);
        // accepted prefix per target: start weight + segmented prefix <= U
        __shared__ int64_t carry;
        __shared__ int32_t carryT;
        if (threadIdx.x == 0) { carry = 0; carryT = -1; }
        __syncthreads();
        for (int32_t base = 0; base < np; base += IPT) {
          int32_t i = base + threadIdx.x;
          bool ok = i < np;
          uint64_t k = ok ? pl[i] : 0;
          int32_t T = ok ? (int32_t)(k >> 47) : -1;
          int32_t u = ok ? (int32_t)(k & 0xFFFF) : 0;
          // only threads holding a proposal look at their predecessor (i - 1 < np)
          int32_t Tprev = (!ok || i == 0) ? -1 : (int32_t)((pl[i - 1] >> 47) & 0xFFFF);
          bool head = !ok || i == 0 || T != Tprev;
          int64_t c = ok ? g.vw[u] : 0;
          int64_t pre = block_seg_scan(c, head || threadIdx.x == 0);
          // the chunk's first segment continues the previous chunk's last one
          bool cont = ok && base > 0 && T == carryT;
          __shared__ int32_t firsthead;
          if (threadIdx.x == 0) firsthead = IPT;
          __syncthreads();
          if (ok && threadIdx.x > 0 && head) atomicMin(&firsthead, (int32_t)threadIdx.x);
          __syncthreads();
          if (cont && (int32_t)threadIdx.x < firsthead) pre += carry;
          if (ok) {
            bool acc = (int64_t)wt[T] + pre <= U;
            if (acc) pl[i] = k | (1ull << 63);
          }
          __syncthreads();
          int32_t last = min(IPT, np - base) - 1;
          if ((int32_t)threadIdx.x == last) {
            carry = pre;
            carryT = T;
          }
          __syncthreads();
        }
      }
      // apply: every warp takes its share of the accepted moves, a lane each, and
      // then walks the moved nodes' rows together, an entry per lane, to mark the
      // neighbours active for the next round (a warp per move cost the latency of
      // its row 30 times over: 40,000 cycles in the first sub-rounds of a
      // 2048-node item)
      int32_t mv_local = 0;
      const int32_t share = (nf + np + IPW - 1) / IPW;
      const int32_t mend = min((w + 1) * share, nf + np);
      for (int32_t i0 = w * share; i0 < mend; i0 += 32) {
        const int32_t i = i0 + lane;
        int32_t u = -1, T = 0, deg = 0, beg = 0;
        if (i < mend) {
          if (i < nf) {
            u = fl[i];
            T = pt[u];
          } else {
            const uint64_t k = pl[i - nf];
            if (k >> 63) {
              T = (int32_t)((k >> 47) & 0xFFFF);
              u = (int32_t)(k & 0xFFFF);
            }
          }
        }
        if (u >= 0) {
          const int32_t own = lab[u], c = g.vw[u];
          lab[u] = (uint16_t)T;
          atomicAdd(&wt[T], c);
          atomicSub(&wt[own], c);
          ++mv_local;
          beg = g.xadj[u];
          deg = g.xadj[u + 1] - beg;
        }
        int32_t inc = deg;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int32_t t = __shfl_up_sync(0xFFFFFFFFu, inc, o);
          if (lane >= o) inc += t;
        }
        const int32_t tot = __shfl_sync(0xFFFFFFFFu, inc, 31), shift = beg - (inc - deg);
        for (int32_t e0 = 0; e0 < tot; e0 += 32) {
          const int32_t e = e0 + lane;
          int32_t j = 0;  // moves whose rows end at or before entry e
#pragma unroll
          for (int st = 16; st > 0; st >>= 1) {
            const int32_t t = __shfl_sync(0xFFFFFFFFu, inc, j + st - 1);
            if (t <= e) j += st;
          }
          const int32_t q = __shfl_sync(0xFFFFFFFFu, shift, j & 31) + e;
          if (e < tot) act2[g.adj[q]] = 1;
        }
      }
      mv_local = warp_sum32(mv_local);
      if (lane == 0 && mv_local) atomicAdd(&s_moved, mv_local);
      __syncthreads();
    }
    int32_t moved = s_moved;
    uint8_t *t = act;
    act = act2;
    act2 = t;
    __syncthreads();
    if (moved == 0) break;
  }
  // isolated packing in id order
  int32_t *iw = pg;  // reuse: weights of isolated nodes, then prefix
  for (int32_t v = threadIdx.x; v < n; v += IPT) iw[v] = (g.xadj[v + 1] == g.xadj[v]) ? g.vw[v] : 0;
  __syncthreads();
  block_scan_excl<int32_t>(iw, iw, n);
  int32_t *first = tsum;
  for (int32_t v = threadIdx.x; v < n; v += IPT) first[v] = INT32_MAX;
  __syncthreads();
  for (int32_t v = threadIdx.x; v < n; v += IPT) {
    if (g.xadj[v + 1] != g.xadj[v]) continue;
    int64_t P0 = iw[v], c = g.vw[v];
    int64_t q = P0 / U, qe = (P0 + c - 1) / U;
    if (q == qe) atomicMin(&first[q], (int32_t)lab[v]);
  }
  __syncthreads();
  for (int32_t v = threadIdx.x; v < n; v += IPT) {
    if (g.xadj[v + 1] != g.xadj[v]) continue;
    int64_t P0 = iw[v], c = g.vw[v];
    int64_t q = P0 / U, qe = (P0 + c - 1) / U;
    if (q == qe) lab[v] = (uint16_t)first[q];
  }
  __syncthreads();
  // count clusters
  uint16_t *used = pt;
  for (int32_t v = threadIdx.x; v < n; v += IPT) used[v] = 0;
  __syncthreads();
  for (int32_t v = threadIdx.x; v < n; v += IPT) used[lab[v]] = 1;
  __syncthreads();
  int64_t c = 0;
  for (int32_t v = threadIdx.x; v < n; v += IPT) c += used[v];
  int32_t nc = (int32_t)block_sum64(c);
  for (int32_t v = threadIdx.x; v < n; v += IPT) label[v] = lab[v];
  __syncthreads();
  B.top = mark;
  return nc;
}

// contraction of one item level; fills *out (arrays allocated from B)
__device__ void item_contract(const LG &g, const int32_t *label, int32_t *map, LG *out, Bump &B, int32_t wtab,
                              int32_t *wkeys, int32_t *wvals) {
  int32_t n = g.n;
  int32_t *cid = B.take(n + 1);
  if (B.oom) return;
  for (int32_t v = threadIdx.x; v < n; v += IPT) cid[v] = 0;
  __syncthreads();
  for (int32_t v = threadIdx.x; v < n; v += IPT) cid[label[v]] = 1;
  __syncthreads();
  int32_t nc = block_scan_excl<int32_t>(cid, cid, n);
  for (int32_t v = threadIdx.x; v < n; v += IPT) map[v] = cid[label[v]];
  __syncthreads();
  // coarse arrays (kept); rows hold at most the cross entries of the level
  int32_t *cvw = B.take(nc);
  int32_t *cx = B.take(nc + 1);
  int64_t cnt = 0;
  for (int32_t v = threadIdx.x; v < n; v += IPT)
    for (int32_t q = g.xadj[v]; q < g.xadj[v + 1]; ++q) cnt += (map[v] != map[g.adj[q]]);
  int32_t np = (int32_t)block_sum64(cnt);
  uint16_t *cadj = reinterpret_cast<uint16_t *>(B.take((np + 1) / 2));
  int32_t *cew = B.take(np);
  int64_t mark = B.top;
  // members grouped by coarse node; members' total degree per coarse node
  int32_t *moff = B.take(nc + 1), *mcur = B.take(nc), *members = B.take(n);
  int32_t *ub = B.take(nc + 1), *toff = B.take(nc + 1), *rowlen = B.take(nc + 1);
  uint16_t *tadj = reinterpret_cast<uint16_t *>(B.take((g.m + 2) / 2));
  int32_t *tw = B.take(g.m > 0 ? g.m : 1);
  if (B.oom) return;
  for (int32_t x = threadIdx.x; x <= nc; x += IPT) {
    if (x < nc) {
      cvw[x] = 0;
      mcur[x] = 0;
    }
    moff[x] = 0;
    ub[x] = 0;
  }
  __syncthreads();
  for (int32_t v = threadIdx.x; v < n; v += IPT) {
    int32_t x = map[v];
    atomicAdd(&cvw[x], g.vw[v]);
    atomicAdd(&moff[x], 1);
    atomicAdd(&ub[x], g.xadj[v + 1] - g.xadj[v]);
  }
  __syncthreads();
  block_scan_excl<int32_t>(moff, moff, nc + 1);
  int32_t maxub = 0;
  for (int32_t x = threadIdx.x; x < nc; x += IPT) maxub = max(maxub, ub[x]);
  maxub = block_max32(maxub);
  block_scan_excl<int32_t>(ub, toff, nc + 1);
  for (int32_t v = threadIdx.x; v < n; v += IPT) {
    int32_t x = map[v];
    members[moff[x] + atomicAdd(&mcur[x], 1)] = v;
  }
  // per-warp global table and sort list for rows that do not fit shared memory
  int32_t dmax = maxub < nc ? maxub : nc;
  int32_t gcap = 32;
  while (gcap < 2 * dmax) gcap <<= 1;
  int32_t lcap = pow2_at_least(dmax > 1 ? dmax : 2);
  int32_t *gtab = gcap > wtab ? B.take(2ll * gcap * IPW) : nullptr;
  uint64_t *lbuf = reinterpret_cast<uint64_t *>(B.take(2ll * lcap * IPW));
  __syncthreads();
  if (B.oom) return;
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint64_t *L = lbuf + (int64_t)w * lcap;
  // one warp per coarse node: aggregate, compact, sort by neighbour, write the row
  for (int32_t x = w; x < nc; x += IPW) {
    int32_t d = ub[x] < nc ? ub[x] : nc;
    uint32_t cap = 32;
    while ((int32_t)cap < 2 * d) cap <<= 1;
    int32_t *K = cap <= (uint32_t)wtab ? wkeys + w * wtab : gtab + (int64_t)w * 2 * gcap;
    int32_t *V = cap <= (uint32_t)wtab ? wvals + w * wtab : K + gcap;
    for (uint32_t i = lane; i < cap; i += 32) {
      K[i] = HT_EMPTY;
      V[i] = 0;
    }
    __syncwarp();
    // up to 32 members at a time spread their edges over the lanes: a warp
    // prefix of their degrees, and each lane finds the member of its edge
    for (int32_t c0 = moff[x]; c0 < moff[x + 1]; c0 += 32) {
      int32_t d = 0, b = 0;
      if (c0 + lane < moff[x + 1]) {
        int32_t v = members[c0 + lane];
        b = g.xadj[v];
        d = g.xadj[v + 1] - b;
      }
      int32_t inc = d;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        int32_t t = __shfl_up_sync(0xFFFFFFFFu, inc, o);
        if (lane >= o) inc += t;
      }
      const int32_t tot = __shfl_sync(0xFFFFFFFFu, inc, 31);
      for (int32_t e0 = 0; e0 < tot; e0 += 32) {
        const int32_t e = e0 + lane;
        int32_t j = 0;  // members before the owner of edge e
#pragma unroll
        for (int st = 16; st > 0; st >>= 1) {
          int32_t t = __shfl_sync(0xFFFFFFFFu, inc, j + st - 1);
          if (t <= e) j += st;
        }
        int32_t bj = __shfl_sync(0xFFFFFFFFu, b, j & 31);
        int32_t ej = __shfl_sync(0xFFFFFFFFu, inc - d, j & 31);
        if (e < tot) {
          int32_t q = bj + (e - ej);
          int32_t y = map[g.adj[q]];
          if (y != x) ht_add(K, V, cap - 1, y, lg_w(g, q));
        }
      }
    }
    __syncwarp();
    int32_t c = 0;
    for (uint32_t i0 = 0; i0 < cap; i0 += 32) {
      uint32_t i = i0 + lane;
      bool has = K[i] != HT_EMPTY;
      unsigned bal = __ballot_sync(0xFFFFFFFFu, has);
      if (has) L[c + __popc(bal & ((1u << lane) - 1u))] = ((uint64_t)(uint32_t)K[i] << 32) | (uint32_t)V[i];
      c += __popc(bal);
    }
    int32_t P = pow2_at_least(c > 1 ? c : 2);
    for (int32_t i = c + lane; i < P; i += 32) L[i] = ~0ull;
    __syncwarp();
    warp_bitonic_u64(L, P);
    for (int32_t i = lane; i < c; i += 32) {
      tadj[toff[x] + i] = (uint16_t)(L[i] >> 32);
      tw[toff[x] + i] = (int32_t)(uint32_t)L[i];
    }
    if (lane == 0) rowlen[x] = c;
    __syncwarp();
  }
  __syncthreads();
  if (threadIdx.x == 0) rowlen[nc] = 0;
  __syncthreads();
  int32_t m2 = block_scan_excl<int32_t>(rowlen, cx, nc + 1);
  for (int32_t x = w; x < nc; x += IPW)
    for (int32_t i = lane; i < cx[x + 1] - cx[x]; i += 32) {
      cadj[cx[x] + i] = tadj[toff[x] + i];
      cew[cx[x] + i] = tw[toff[x] + i];
    }
  __syncthreads();
  B.top = mark;
  out->n = nc;
  out->m = m2;
  out->xadj = cx;
  out->adj = cadj;
  out->ew = cew;
  out->vw = cvw;
  __syncthreads();
}

// ------------------------------------------------------------ warp FM
// A pass of 2-way FM is a chain of steps on one warp, each a scan for the tops
// of both sides and an update of one row's gains, so its time is the latency of
// what a step does in turn.  Its state is small enough for shared memory at
// every level that occurs in large numbers (6.1 bytes a node, 14.1 with row
// offsets and node weights): a 32-bit key a node; a bit a node for its side at
// the start of the pass (a move locks, so sides change once, at the end of the
// pass, by the kept moves); the move log in 16 bits.
//
// The key holds gain and id: ((gain + bias) << idbits | largest id - id), as
// such on side 0, negated on side 1, 0 once locked (the next pass computes a
// locked node's gain anew).  So the tops of both sides, gain descending and id
// ascending, are the largest and the smallest key; and a move changes every
// unlocked neighbour's key by the same signed amount whichever side it is on.
// Where id and the largest weighted degree do not fit 31 bits together
// (idbits < 0) the key is the plain gain, FM_LOCKED once locked, and the scan
// reads the sides.
constexpr int32_t FM_LOCKED = INT32_MIN;  // below every gain: those fit 31 bits and a sign
struct FMState {
  int32_t *key;     // fm_pad(n) words, 16-byte aligned; locked from n on
  uint32_t *bits;   // fm_pad(n) / 32 words: sides
  uint16_t *moves;  // n node ids (IP_MAX_N)
  // the level's graph; row offsets, node weights and entries in shared memory
  // where they fit
  const int32_t *xadj, *vw;
  const uint16_t *adj;
  const int32_t *ew;  // null: unit weights
  // word offsets of the state, of the row offsets (the node weights behind them)
  // and of the edge weights (neighbour ids behind them) in the CTA's dynamic
  // shared memory; -1: not there
  int32_t off, goff, eoff;
};
__host__ __device__ __forceinline__ int32_t fm_pad(int32_t n) { return (n + 127) & ~127; }
__host__ __device__ __forceinline__ int64_t fm_words(int32_t n) { return (int64_t)fm_pad(n) / 32 * 49; }
__device__ __forceinline__ FMState fm_state(int32_t *p, const LG &g) {
  const int32_t np = fm_pad(g.n);
  uint32_t *bits = reinterpret_cast<uint32_t *>(p + np);
  return FMState{p, bits, reinterpret_cast<uint16_t *>(bits + np / 32), g.xadj, g.vw, g.adj, g.ew, -1, -1, -1};
}
__device__ __forceinline__ int32_t *align16(int32_t *p) {
  return reinterpret_cast<int32_t *>((reinterpret_cast<uintptr_t>(p) + 15) & ~(uintptr_t)15);
}
__device__ __forceinline__ int32_t fm_side(const uint32_t *bits, int32_t v) { return (bits[v >> 5] >> (v & 31)) & 1; }

// bits of a node id in the key: n <= 2^idbits, and gains within +-maxwd leave
// 1 <= (gain + bias) < 2^(31 - idbits) with bias = maxwd + 1; -1 if they do not
__device__ __forceinline__ int32_t fm_idbits(int32_t n, int32_t maxwd) {
  const int32_t b = 32 - __clz(n > 1 ? n - 1 : 1);
  return 2ll * maxwd + 2 < (1ll << (31 - b)) ? b : -1;
}
__device__ __forceinline__ int32_t fm_key(int32_t gain, int32_t v, int32_t side, int32_t idbits, int32_t bias) {
  const int32_t k = ((gain + bias) << idbits) | ((1 << idbits) - 1 - v);
  return side ? -k : k;
}

__device__ __forceinline__ bool fm_less(int32_t ia, int64_t oa, int64_t ca, int32_t ib, int64_t ob,
                                        int64_t cb) {
  if (ia != ib) return ia < ib;
  if (oa != ob) return oa < ob;
  return ca < cb;
}

// A graph whose rows may hold parallel entries (Graph::multi) has a build of these
// kernels of its own (kmp_ip_multi.cu): lanes that walk a row may change one node's
// key or gain at once, so they add atomically.  With atomics everywhere 4096 items of
// 200..4000 nodes take 32.5 ms instead of 31.8; as template variants in this file the
// plain kernel took 2 % longer on small items, for its registers.
#if KMP_IP_MULTI
#define FM_ADD(x, k, d) atomicAdd(&(x), d)
#else
#define FM_ADD(x, k, d) ((x) = (k) + (d))
#endif

// The moves of one FM pass by one warp, from keys already set: repeatedly the
// better feasible top of the two sides (gain desc, id asc), until no unlocked
// node is left or fm_stop moves bring no new best (overload, then cut); then
// the pass keeps its best prefix.  Returns the kept moves (0: the pass found
// nothing better) and updates the sides, the side weights and the cut.
//
// One warp on its own issues a dependent instruction every few cycles, so a
// step costs what its instructions count: the shared arrays are addressed as
// offsets into the CTA's shared memory (32-bit addresses; GRAPH as in FMState),
// the sums are 32-bit (caps clamped to the total weight, which is below 2^31),
// the room left on each side stands for both weights, and only the better
// side's top is looked up unless it does not fit.
// Measured a step in place: 780 cycles with all of a level of up to 256 nodes in
// shared memory (about 1900 with 64-bit selection keys reduced by shuffles), 2200
// for 2048 nodes with the entries in L2 (3800).
template <int GRAPH>
__device__ __forceinline__ int32_t fm_pass_packed(int32_t fm_stop, int32_t n, const FMState F, int32_t idbits,
                                                  int32_t bias, int32_t L0, int32_t L1, int32_t &W0, int32_t &W1,
                                                  int32_t &cut) {
  extern __shared__ __align__(16) int32_t ipdyn[];
  constexpr unsigned ALL = 0xFFFFFFFFu;
  const int lane = threadIdx.x & 31;
  const int32_t np = fm_pad(n), idmask = (1 << idbits) - 1, total = W0 + W1;
  int32_t *const key = GRAPH ? ipdyn + F.off : F.key;
  uint32_t *const bits = GRAPH ? reinterpret_cast<uint32_t *>(ipdyn + F.off + np) : F.bits;
  uint16_t *const moves = GRAPH ? reinterpret_cast<uint16_t *>(ipdyn + F.off + np + np / 32) : F.moves;
  const int32_t *const xadj = GRAPH ? ipdyn + F.goff : F.xadj;
  const int32_t *const vw = GRAPH ? ipdyn + F.goff + n + 1 : F.vw;
  const bool unit = F.ew == nullptr;
  const int32_t *const ew = GRAPH == 2 ? ipdyn + F.eoff : F.ew;
  const uint16_t *const adj =
      GRAPH == 2 ? reinterpret_cast<const uint16_t *>(ipdyn + F.eoff + (unit ? 0 : xadj[n])) : F.adj;
  int32_t r0 = min(L0, total) - W0, r1 = min(L1, total) - W1;  // room left
  int32_t c = cut, br0 = r0, bcut = c, bmin = min(min(r0, r1), 0);
  int32_t best_step = 0, nsteps = 0;
  for (;;) {
    const int4 k0 = *reinterpret_cast<const int4 *>(key + 4 * lane);
    int32_t hi = max(max(max(k0.x, k0.y), max(k0.z, k0.w)), 0);
    int32_t lo = min(min(min(k0.x, k0.y), min(k0.z, k0.w)), 0);
#pragma unroll 4
    for (int32_t v = 4 * lane + 128; v < np; v += 128) {
      const int4 k = *reinterpret_cast<const int4 *>(key + v);
      hi = max(hi, max(max(k.x, k.y), max(k.z, k.w)));
      lo = min(lo, min(min(k.x, k.y), min(k.z, k.w)));
    }
    const int32_t m0 = __reduce_max_sync(ALL, hi), m1 = -__reduce_min_sync(ALL, lo);
    if ((m0 | m1) == 0) break;
    bool from0 = m0 > m1;
    int32_t m = from0 ? m0 : m1, v = idmask - (m & idmask);
    int32_t cv = vw[v], qb = xadj[v], qe = xadj[v + 1];
    if (cv > (from0 ? r1 : r0)) {  // the other side's top
      const int32_t o = from0 ? m1 : m0, u = idmask - (o & idmask);
      bool fits = false;
      if (o) {
        cv = vw[u];
        fits = cv <= (from0 ? r0 : r1);
      }
      if (!fits) {
        if (lane == 0) {
          key[v] = 0;
          if (o) key[u] = 0;
        }
        __syncwarp();
        continue;
      }
      from0 = !from0;
      m = o;
      v = u;
      qb = xadj[v];
      qe = xadj[v + 1];
    }
    const int32_t sg = from0 ? 1 << (idbits + 1) : -(1 << (idbits + 1));
    for (int32_t q = qb + lane; q < qe; q += 32) {
      const int32_t x = adj[q], d = (unit ? 1 : ew[q]) * sg, k = key[x];
      if (k) FM_ADD(key[x], k, d);
    }
    if (lane == 0) {
      key[v] = 0;
      moves[nsteps] = (uint16_t)v;
    }
    __syncwarp();
    ++nsteps;
    const int32_t d = from0 ? cv : -cv;
    r0 += d;
    r1 -= d;
    c += bias - (m >> idbits);
    const int32_t mn = min(min(r0, r1), 0);
    if (mn > bmin || (mn == bmin && c < bcut)) {
      bmin = mn;
      bcut = c;
      br0 = r0;
      best_step = nsteps;
    }
    if (nsteps - best_step >= fm_stop) break;
  }
  for (int32_t i = lane; i < best_step; i += 32) {
    const int32_t v = moves[i];
    atomicXor(&bits[v >> 5], 1u << (v & 31));
  }
  __syncwarp();
  W0 = min(L0, total) - br0;
  W1 = total - W0;
  cut = bcut;
  return best_step;
}

// the same pass from plain gains, for levels whose keys do not pack
__device__ __noinline__ int32_t fm_pass_plain(int32_t fm_stop, int32_t n, const FMState F, int64_t L0, int64_t L1,
                                              int32_t &W0, int32_t &W1, int32_t &cut) {
  constexpr unsigned ALL = 0xFFFFFFFFu;
  const int lane = threadIdx.x & 31;
  int64_t w0 = W0, w1 = W1, bw0 = w0;
  const int64_t total = w0 + w1;
  auto overload = [&]() -> int64_t { return max(max(w0 - L0, w1 - L1), (int64_t)0); };
  int64_t bov = overload();
  int32_t c = cut, bcut = c, best_step = 0, nsteps = 0;
  for (;;) {
    int32_t g0 = FM_LOCKED, g1 = FM_LOCKED;
    uint32_t i0 = ~0u, i1 = ~0u;
    for (int32_t v = lane; v < n; v += 32) {
      const int32_t x = F.key[v];
      if (!fm_side(F.bits, v)) {
        if (x > g0) {
          g0 = x;
          i0 = (uint32_t)v;
        }
      } else if (x > g1) {
        g1 = x;
        i1 = (uint32_t)v;
      }
    }
    const int32_t m0 = __reduce_max_sync(ALL, g0), m1 = __reduce_max_sync(ALL, g1);
    if (m0 == FM_LOCKED && m1 == FM_LOCKED) break;
    const int32_t v0 = (int32_t)__reduce_min_sync(ALL, g0 == m0 ? i0 : ~0u);  // -1: no unlocked node
    const int32_t v1 = (int32_t)__reduce_min_sync(ALL, g1 == m1 ? i1 : ~0u);
    const bool f0 = v0 >= 0 && w1 + F.vw[v0] <= L1;
    const bool f1 = v1 >= 0 && w0 + F.vw[v1] <= L0;
    if (!f0 && !f1) {
      if (lane == 0) {
        if (v0 >= 0) F.key[v0] = FM_LOCKED;
        if (v1 >= 0) F.key[v1] = FM_LOCKED;
      }
      __syncwarp();
      continue;
    }
    const bool from0 = f0 && (!f1 || m0 > m1 || (m0 == m1 && v0 < v1));
    const int32_t v = from0 ? v0 : v1, to = from0 ? 1 : 0;
    for (int32_t q = F.xadj[v] + lane; q < F.xadj[v + 1]; q += 32) {
      const int32_t x = F.adj[q], d = 2 * (F.ew ? F.ew[q] : 1), k = F.key[x];
      if (k != FM_LOCKED) FM_ADD(F.key[x], k, fm_side(F.bits, x) == to ? -d : d);
    }
    if (lane == 0) {
      F.key[v] = FM_LOCKED;
      F.moves[nsteps] = (uint16_t)v;
    }
    __syncwarp();
    ++nsteps;
    w0 += from0 ? -(int64_t)F.vw[v] : F.vw[v];
    w1 = total - w0;
    c -= from0 ? m0 : m1;
    const int64_t ov = overload();
    if (ov < bov || (ov == bov && c < bcut)) {
      bov = ov;
      bcut = c;
      bw0 = w0;
      best_step = nsteps;
    }
    if (nsteps - best_step >= fm_stop) break;
  }
  for (int32_t i = lane; i < best_step; i += 32) {
    const int32_t v = F.moves[i];
    atomicXor(&F.bits[v >> 5], 1u << (v & 31));
  }
  __syncwarp();
  W0 = (int32_t)bw0;
  W1 = (int32_t)(total - bw0);
  cut = bcut;
  return best_step;
}

__device__ __forceinline__ int32_t pass_moves(int32_t fm_stop, int32_t n, const FMState F, int32_t idbits,
                                              int32_t bias, int32_t L0, int32_t L1, int32_t &W0, int32_t &W1,
                                              int32_t &cut) {
  if (idbits < 0) return fm_pass_plain(fm_stop, n, F, L0, L1, W0, W1, cut);
  if (F.eoff >= 0) return fm_pass_packed<2>(fm_stop, n, F, idbits, bias, L0, L1, W0, W1, cut);
  if (F.off >= 0) return fm_pass_packed<1>(fm_stop, n, F, idbits, bias, L0, L1, W0, W1, cut);
  return fm_pass_packed<0>(fm_stop, n, F, idbits, bias, L0, L1, W0, W1, cut);
}

// 2-way FM by one warp (same decisions as the oracle) from the sides in
// F.bits, which it improves; returns the final cut, W0 and W1 the side weights
__device__ int32_t warp_fm(const IPArgs &A, int32_t n, int32_t L0, int32_t L1, const FMState F, int32_t &W0,
                           int32_t &W1) {
  const int lane = threadIdx.x & 31;
  int32_t cut = 0, idbits = 0, bias = 0;
  W0 = W1 = 0;
  for (int32_t pass = 0; pass < A.fm_passes || pass == 0; ++pass) {
    int64_t lcut = 0;
    int32_t maxwd = 0;
    for (int32_t v = lane; v < n; v += 32) {
      const int32_t sv = fm_side(F.bits, v);
      int32_t ext = 0, in = 0;
      for (int32_t q = F.xadj[v]; q < F.xadj[v + 1]; ++q) {
        const int32_t wq = F.ew ? F.ew[q] : 1;
        if (fm_side(F.bits, F.adj[q]) != sv) ext += wq;
        else in += wq;
      }
      const int32_t gs = ext - in;
      if (pass == 0) {
        lcut += ext;
        maxwd = max(maxwd, ext + in);
        if (sv == 0) W0 += F.vw[v];
        else W1 += F.vw[v];
      }
      F.key[v] = pass == 0 || idbits < 0 ? gs : fm_key(gs, v, sv, idbits, bias);
    }
    if (pass == 0) {
      cut = (int32_t)(warp_sum64(lcut) / 2);
      W0 = warp_sum32(W0);
      W1 = warp_sum32(W1);
      if (A.fm_passes == 0) break;
      maxwd = __reduce_max_sync(0xFFFFFFFFu, maxwd);
      idbits = L0 < 0 || L1 < 0 ? -1 : fm_idbits(n, maxwd);
      bias = maxwd + 1;
      for (int32_t v = lane; v < fm_pad(n); v += 32) {
        if (v >= n) F.key[v] = idbits < 0 ? FM_LOCKED : 0;
        else if (idbits >= 0) F.key[v] = fm_key(F.key[v], v, fm_side(F.bits, v), idbits, bias);
      }
    }
    __syncwarp();
    if (pass_moves(A.fm_stop, n, F, idbits, bias, L0, L1, W0, W1, cut) == 0) break;
  }
  return cut;
}

// the same FM with the whole CTA: cut, keys and weights by all warps (a
// half-warp per node and four nodes at a time, so the loads of four rows are in
// flight together), the moves by warp 0
__device__ void cta_fm(const IPArgs &A, int32_t n, int32_t L0, int32_t L1, const FMState F) {
  __shared__ int32_t s_kept;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int hl = lane & 15, h = 2 * w + (lane >> 4);
  constexpr int ROWS = 4, STEP = 2 * IPW;  // half-warps
  int64_t lcut = 0, lw0 = 0, lw1 = 0;
  int32_t cut = 0, W0 = 0, W1 = 0, idbits = 0, bias = 0;  // warp 0's from the second pass on
  for (int32_t pass = 0; pass < A.fm_passes; ++pass) {
    int32_t maxwd = 0;
    for (int32_t v0 = h; v0 - h < n; v0 += ROWS * STEP) {
      int32_t b[ROWS], e[ROWS], x[ROWS], wt[ROWS];
#pragma unroll
      for (int r = 0; r < ROWS; ++r) {
        const int32_t v = v0 + r * STEP;
        b[r] = v < n ? F.xadj[v] : 0;
        e[r] = v < n ? F.xadj[v + 1] : 0;
      }
#pragma unroll
      for (int r = 0; r < ROWS; ++r) {
        x[r] = -1;
        wt[r] = 0;
        if (b[r] + hl < e[r]) {
          x[r] = F.adj[b[r] + hl];
          wt[r] = F.ew ? F.ew[b[r] + hl] : 1;
        }
      }
#pragma unroll
      for (int r = 0; r < ROWS; ++r) {
        const int32_t v = v0 + r * STEP;
        const int32_t sv = v < n ? fm_side(F.bits, v) : 0;
        int32_t ext = 0, wd = wt[r];
        if (x[r] >= 0 && fm_side(F.bits, x[r]) != sv) ext = wt[r];
        for (int32_t q = b[r] + 16 + hl; q < e[r]; q += 16) {
          const int32_t wq = F.ew ? F.ew[q] : 1;
          wd += wq;
          if (fm_side(F.bits, F.adj[q]) != sv) ext += wq;
        }
        if (pass == 0) lcut += ext;
        int32_t gs = 2 * ext - wd;  // external less internal
#pragma unroll
        for (int m = 8; m > 0; m >>= 1) gs += __shfl_xor_sync(0xFFFFFFFFu, gs, m);  // within the half
        if (pass == 0) {
#pragma unroll
          for (int m = 8; m > 0; m >>= 1) wd += __shfl_xor_sync(0xFFFFFFFFu, wd, m);
          maxwd = max(maxwd, wd);
          if (hl == 0 && v < n) {
            if (sv == 0) lw0 += F.vw[v];
            else lw1 += F.vw[v];
          }
        }
        if (hl == 0 && v < n) F.key[v] = pass == 0 || idbits < 0 ? gs : fm_key(gs, v, sv, idbits, bias);
      }
    }
    if (pass == 0) {
      cut = (int32_t)(block_sum64(lcut) / 2);
      W0 = (int32_t)block_sum64(lw0);
      W1 = (int32_t)block_sum64(lw1);
      maxwd = block_max32(maxwd);
      idbits = L0 < 0 || L1 < 0 ? -1 : fm_idbits(n, maxwd);
      bias = maxwd + 1;
      for (int32_t v = threadIdx.x; v < fm_pad(n); v += IPT) {
        if (v >= n) F.key[v] = idbits < 0 ? FM_LOCKED : 0;
        else if (idbits >= 0) F.key[v] = fm_key(F.key[v], v, fm_side(F.bits, v), idbits, bias);
      }
    }
    __syncthreads();  // the keys are complete
    if (w == 0) {
      const int32_t kept = pass_moves(A.fm_stop, n, F, idbits, bias, L0, L1, W0, W1, cut);
      if (lane == 0) s_kept = kept;
    }
    __syncthreads();
    const int32_t kept = s_kept;
    __syncthreads();
    if (kept == 0) break;
  }
}

// sides of a level (given by side(v)) into its bits, by all threads
template <class F>
__device__ __forceinline__ void cta_set_bits(uint32_t *bits, int32_t n, F side) {
  for (int32_t v = threadIdx.x; v < fm_pad(n); v += IPT) {
    const unsigned m = __ballot_sync(0xFFFFFFFFu, v < n && side(v) != 0);
    if ((threadIdx.x & 31) == 0) bits[v >> 5] = m;
  }
}

// words of a level's row offsets and node weights, and of its entries
__device__ __forceinline__ int64_t fm_graph_words(const LG &g) { return 2ll * g.n + 1; }
__device__ __forceinline__ int64_t fm_entry_words(const LG &g) { return (g.ew ? (int64_t)g.m : 0) + (g.m + 1) / 2; }

// the level's graph at word `at` of the dynamic shared memory, its entries too
// when they end within `words`; complete after the caller's next barrier
__device__ void cta_fm_graph(const LG &g, FMState &F, int32_t *dyn, int32_t at, int32_t words) {
  int32_t *x = dyn + at, *vw = x + g.n + 1;
  for (int32_t v = threadIdx.x; v <= g.n; v += IPT) {
    x[v] = g.xadj[v];
    if (v < g.n) vw[v] = g.vw[v];
  }
  F.xadj = x;
  F.vw = vw;
  F.goff = at;
  const int32_t eo = at + (int32_t)fm_graph_words(g);
  if (eo + fm_entry_words(g) > words) return;
  int32_t *ew = dyn + eo;
  uint16_t *adj = reinterpret_cast<uint16_t *>(ew + (g.ew ? g.m : 0));
  for (int32_t q = threadIdx.x; q < g.m; q += IPT) {
    adj[q] = g.adj[q];
    if (g.ew) ew[q] = g.ew[q];
  }
  F.adj = adj;
  if (g.ew) F.ew = ew;
  F.eoff = eo;
}

// FM state of a level: in shared memory (dyn) when it fits there with the row
// offsets and node weights, and with the entries too when those fit as well;
// else in the item's scratch (glob, 16-byte aligned)
__device__ FMState cta_fm_state(const LG &g, int32_t *dyn, int32_t dyn_words, int32_t *glob) {
  const int64_t st = fm_words(g.n);
  if (st + fm_graph_words(g) > dyn_words) return fm_state(glob, g);
  FMState F = fm_state(dyn, g);
  F.off = 0;
  cta_fm_graph(g, F, dyn, (int32_t)st, dyn_words);
  return F;
}

// portfolio initial bipartition by one warp:
// algo 0 random, 1 BFS, 2 greedy graph growing, 3 learned (first fit in the
// order of `score`, like random with a learned order)
__device__ void warp_initial(int algo, const LG &g, int32_t t0, uint64_t key, int32_t *side,
                             uint64_t *oh, int32_t *ov, int32_t *gain, int32_t *vis, int32_t *queue,
                             const float *score) {
  int lane = threadIdx.x & 31;
  int32_t n = g.n;
  int32_t P = pow2_at_least(n > 1 ? n : 2);
  for (int32_t i = lane; i < P; i += 32) {
    if (i < n) {
      oh[i] = algo == 3 ? (uint64_t)mp_score_key(score[i]) : key_step(key, (uint64_t)(uint32_t)i);
      ov[i] = i;
    } else {
      oh[i] = ~0ull;
      ov[i] = INT32_MAX;
    }
  }
  for (int32_t v = lane; v < n; v += 32) side[v] = 1;
  __syncwarp();
  warp_bitonic_hv(oh, ov, P);
  if (algo == 0 || algo == 3) {
    if (lane == 0) {
      int64_t W0 = 0;
      for (int32_t i = 0; i < n; ++i) {
        int32_t v = ov[i];
        if (W0 + g.vw[v] <= t0) {
          side[v] = 0;
          W0 += g.vw[v];
        }
      }
    }
  } else if (algo == 1) {
    for (int32_t v = lane; v < n; v += 32) vis[v] = 0;
    __syncwarp();
    if (lane == 0) {
      int64_t W0 = 0;
      int32_t qh = 0, qt = 0, nr = 0;
      while (qh < n) {
        if (qh == qt) {
          while (vis[ov[nr]]) ++nr;
          vis[ov[nr]] = 1;
          queue[qt++] = ov[nr];
        }
        int32_t v = queue[qh++];
        if (W0 + g.vw[v] <= t0) {
          side[v] = 0;
          W0 += g.vw[v];
        }
        for (int32_t q = g.xadj[v]; q < g.xadj[v + 1]; ++q) {
          int32_t x = g.adj[q];
          if (!vis[x]) {
            vis[x] = 1;
            queue[qt++] = x;
          }
        }
      }
    }
  } else {
    for (int32_t v = lane; v < n; v += 32) {
      int32_t s = 0;
      for (int32_t q = g.xadj[v]; q < g.xadj[v + 1]; ++q) s -= lg_w(g, q);
      gain[v] = s;
    }
    __syncwarp();
    int64_t W0 = 0;
    int32_t v = (n > 0 && g.vw[ov[0]] <= t0) ? ov[0] : -1;
    for (;;) {
      if (v >= 0) {
        if (lane == 0) side[v] = 0;
        W0 += g.vw[v];
        for (int32_t q = g.xadj[v] + lane; q < g.xadj[v + 1]; q += 32)
          FM_ADD(gain[g.adj[q]], gain[g.adj[q]], 2 * lg_w(g, q));
        __syncwarp();
      }
      uint64_t best = 0;
      for (int32_t x = lane; x < n; x += 32) {
        if (side[x] == 0 || W0 + g.vw[x] > t0) continue;
        uint64_t k = ((uint64_t)((uint32_t)gain[x] ^ 0x80000000u) << 32) | (0xFFFFFFFFu - (uint32_t)x);
        best = k > best ? k : best;
      }
      best = group_max64<32>(best);
      if (best == 0) break;
      v = (int32_t)(0xFFFFFFFFu - (uint32_t)best);
    }
  }
  __syncwarp();
}

__device__ __forceinline__ int32_t level_cap(int32_t L, int32_t t, int32_t maxc) {
  int64_t b = (int64_t)t + maxc;
  return b > L ? (int32_t)b : L;
}

// append the coarsest graph of an item and its winning sides to the sink
// (skipped and counted as dropped when the sink is full)
__device__ void record_sample(const SampleSink &K, const LG &h, const int32_t *side, uint64_t key) {
  __shared__ unsigned long long s_nb, s_eb;
  __shared__ int32_t s_ok;
  if (threadIdx.x == 0) {
    unsigned long long gi = atomicAdd(&K.counters[0], 1ull);
    unsigned long long nb = atomicAdd(&K.counters[1], (unsigned long long)h.n);
    unsigned long long eb = atomicAdd(&K.counters[2], (unsigned long long)h.m);
    bool ok = gi < (unsigned long long)K.max_graphs && nb + h.n <= (unsigned long long)K.max_nodes &&
              eb + h.m <= (unsigned long long)K.max_entries;
    if (ok) {
      int64_t *r = K.rec + 5 * gi;
      r[0] = (int64_t)nb;
      r[1] = h.n;
      r[2] = (int64_t)eb;
      r[3] = h.m;
      r[4] = (int64_t)key;
    } else {
      atomicAdd(&K.counters[3], 1ull);
    }
    s_ok = ok;
    s_nb = nb;
    s_eb = eb;
  }
  __syncthreads();
  if (s_ok) {
    for (int32_t v = threadIdx.x; v < h.n; v += IPT) {
      K.deg[s_nb + v] = h.xadj[v + 1] - h.xadj[v];
      K.vw[s_nb + v] = h.vw[v];
      K.side[s_nb + v] = side[v];
    }
    for (int32_t e = threadIdx.x; e < h.m; e += IPT) {
      K.adj[s_eb + e] = h.adj[e];
      K.ew[s_eb + e] = lg_w(h, e);
    }
  }
  __syncthreads();
}

// Learned item mode: the network scores the item graph itself, the learned
// start (first fit in score order, warp 0) is refined by the CTA's 2-way FM on
// the item graph with the finest level's caps.  1: feasible, written to
// side_out; 0: a cap is broken (the caller runs the plain method); -1: the
// item's scratch is too small.
__device__ int item_learned(const IPArgs &A, const ItemDesc &D, const LG &g, Bump &B, int32_t *dyn) {
  const int w = threadIdx.x >> 5;
  const int32_t n = g.n;
  const int32_t P = pow2_at_least(n > 1 ? n : 2);
  float *X = reinterpret_cast<float *>(B.take((int64_t)n * MF));
  int32_t *d1 = B.take(n), *d2 = B.take(n);
  float *scr = reinterpret_cast<float *>(B.take((int64_t)n * (MF + 3 * MH)));
  float *sc = reinterpret_cast<float *>(B.take(n));
  int32_t *side = B.take(n);
  uint64_t *oh = reinterpret_cast<uint64_t *>(B.take(2ll * P));
  int32_t *ov = B.take(P);
  int32_t *fmbuf = align16(B.take(fm_words(n) + 4));
  if (B.oom) return -1;
  GView<int32_t, uint16_t> G{n, g.xadj, g.adj, 0, g.vw, g.ew};
  mp_features(G, key_step(D.key, DOM_LEARNED), X, d1, d2);
  mp_forward_cta(G, A.W, X, scr, sc);
  __syncthreads();
  if (w == 0) warp_initial(3, g, D.t0, 0, side, oh, ov, nullptr, nullptr, nullptr, sc);
  __syncthreads();
  const int32_t c0 = level_cap(D.L0, D.t0, g.maxc), c1 = level_cap(D.L1, D.t1, g.maxc);
  const FMState F = cta_fm_state(g, dyn, A.dyn_words, fmbuf);
  cta_set_bits(F.bits, n, [&](int32_t v) { return side[v]; });
  __syncthreads();
  cta_fm(A, n, c0, c1, F);
  __syncthreads();
  int64_t W0 = 0, W1 = 0;
  for (int32_t v = threadIdx.x; v < n; v += IPT) {
    if (fm_side(F.bits, v) == 0) W0 += g.vw[v];
    else W1 += g.vw[v];
  }
  W0 = block_sum64(W0);
  W1 = block_sum64(W1);
  if (W0 > c0 || W1 > c1) return 0;
  for (int32_t v = threadIdx.x; v < n; v += IPT) A.side_out[D.vbase + v] = fm_side(F.bits, v);
  __syncthreads();
  return 1;
}

__device__ void run_item(const IPArgs &A, int32_t it, int32_t *wkeys, int32_t *wvals, int32_t *dyn) {
  __shared__ LG lv[IP_MAXL + 1];
  __shared__ int32_t *maps[IP_MAXL + 1];
  __shared__ int64_t s_wk[IPW][3];
  __shared__ int32_t s_wrep[IPW];
  // adaptive portfolio: per warp and algorithm, the feasible stage-1 runs,
  // their cut sum and sum of squares; the repetitions kept for stage 2
  __shared__ int32_t s_fa[IPW][3];
  __shared__ int64_t s_s1[IPW][3];
  __shared__ unsigned __int128 s_s2[IPW][3];
  __shared__ int32_t s_rest[3];
  const ItemDesc D = A.items[it];
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (D.n == 0) return;
  Bump B{0, false};
  int32_t n0 = D.n;
  int32_t *x0 = B.take(n0 + 1);
  if (B.oom) {
    if (threadIdx.x == 0) atomicExch(A.oom, 1);
    return;
  }
  const int64_t eb = A.gx[D.vbase];
  for (int32_t v = threadIdx.x; v <= n0; v += IPT) x0[v] = (int32_t)(A.gx[D.vbase + v] - eb);
  int64_t cB = 0;
  int32_t md = 0, mc = 0;
  for (int32_t v = threadIdx.x; v < n0; v += IPT) {
    cB += A.svw[D.vbase + v];
    md = max(md, (int32_t)(A.gx[D.vbase + v + 1] - A.gx[D.vbase + v]));
    mc = max(mc, A.svw[D.vbase + v]);
  }
  cB = block_sum64(cB);
  md = block_max32(md);
  mc = block_max32(mc);
  if (threadIdx.x == 0) {
    LG g0;
    g0.n = n0;
    g0.m = D.m;
    g0.xadj = x0;
    g0.adj = const_cast<uint16_t *>(A.sadj + eb);
    g0.ew = A.sew ? const_cast<int32_t *>(A.sew + eb) : nullptr;
    g0.vw = const_cast<int32_t *>(A.svw + D.vbase);
    g0.maxdeg = md;
    g0.maxc = mc;
    lv[0] = g0;
  }
  __syncthreads();
  if (A.learned_item) {
    const int64_t mark = B.top;
    const int r = item_learned(A, D, lv[0], B, dyn);
    if (r < 0) {
      if (threadIdx.x == 0) atomicExch(A.oom, 1);
      return;
    }
    if (r == 1) return;
    B.top = mark;  // infeasible: the plain method from here, in the same scratch
  }
  // 1. coarsen
  uint64_t lpkey = key_step(D.key, DOM_IP_LP);
  int32_t nl = 1;
  while (nl < IP_MAXL) {
    LG g = lv[nl - 1];
    if (g.n <= 1) break;
    int64_t UB = cB / A.ip_C;
    if (UB < g.maxc) UB = g.maxc;
    if (UB < 1) UB = 1;
    int32_t *label = B.take(g.n);
    if (B.oom) break;
    int32_t nc = item_cluster(A, g, (int32_t)UB, key_step(lpkey, (uint64_t)(nl - 1)), label, B, wkeys, wvals,
                              dyn, A.dyn_words);
    if (B.oom) break;
    if (nc == g.n) break;
    int32_t *map = B.take(g.n);
    LG c;
    item_contract(g, label, map, &c, B, A.wtab, wkeys, wvals);
    if (B.oom) break;
    int32_t cmd = 0, cmc = 0;
    for (int32_t x = threadIdx.x; x < c.n; x += IPT) {
      cmd = max(cmd, c.xadj[x + 1] - c.xadj[x]);
      cmc = max(cmc, c.vw[x]);
    }
    cmd = block_max32(cmd);
    cmc = block_max32(cmc);
    c.maxdeg = cmd;
    c.maxc = cmc;
    if (threadIdx.x == 0) {
      lv[nl] = c;
      maps[nl - 1] = map;
    }
    __syncthreads();
    ++nl;
    if ((int64_t)A.conv_den * c.n > (int64_t)A.conv_num * g.n) break;
  }
  if (B.oom) {
    if (threadIdx.x == 0) atomicExch(A.oom, 1);
    return;
  }
  // 2. portfolio on the coarsest level, one warp per repetition
  LG h = lv[nl - 1];
  int32_t nH = h.n;
  int32_t PH = pow2_at_least(nH > 1 ? nH : 2);
  int32_t hL0 = level_cap(D.L0, D.t0, h.maxc), hL1 = level_cap(D.L1, D.t1, h.maxc);
  // per warp: FM state, the best sides, the start's side, order (64-bit key and
  // id), visited marks and queue; the coarsest graph itself once for all warps
  const int64_t per_warp = (fm_words(nH) + fm_pad(nH) / 32 + 3ll * PH + 3ll * nH + 3) & ~3ll;
  // in shared memory when it fits
  const bool pf_smem = per_warp * IPW + fm_graph_words(h) <= A.dyn_words;
  int32_t *wbuf = pf_smem ? dyn : align16(B.take(per_warp * IPW + 4));
  FMState FH{};
  FH.goff = FH.eoff = -1;
  if (pf_smem) {
    FH.adj = h.adj;
    FH.ew = h.ew;
    cta_fm_graph(h, FH, dyn, (int32_t)per_warp * IPW, A.dyn_words);
    h.xadj = const_cast<int32_t *>(FH.xadj);
    h.vw = const_cast<int32_t *>(FH.vw);
    h.adj = const_cast<uint16_t *>(FH.adj);
    h.ew = const_cast<int32_t *>(FH.ew);
    __syncthreads();
  }
  int32_t *fin = B.take(nH);
  if (B.oom) {
    if (threadIdx.x == 0) atomicExch(A.oom, 1);
    return;
  }
  // learned mode: scores of the coarsest graph's nodes (whole CTA)
  const float *score = nullptr;
  if (A.W && !A.learned_item) {
    float *X = reinterpret_cast<float *>(B.take((int64_t)nH * MF));
    int32_t *d1 = B.take(nH), *d2 = B.take(nH);
    float *scr = reinterpret_cast<float *>(B.take((int64_t)nH * (MF + 3 * MH)));
    float *sc = reinterpret_cast<float *>(B.take(nH));
    if (B.oom) {
      if (threadIdx.x == 0) atomicExch(A.oom, 1);
      return;
    }
    GView<int32_t, uint16_t> G{nH, h.xadj, h.adj, 0, h.vw, h.ew};
    mp_features(G, key_step(D.key, DOM_LEARNED), X, d1, d2);
    mp_forward_cta(G, A.W, X, scr, sc);
    score = sc;
  }
  __shared__ int32_t s_bw;
  {
    int32_t *base = wbuf + per_warp * w;
    FMState F = fm_state(base, h);
    if (pf_smem) {
      F.off = (int32_t)per_warp * w;
      F.goff = FH.goff;
      F.eoff = FH.eoff;
    }
    uint32_t *best = reinterpret_cast<uint32_t *>(base + fm_words(nH));
    uint64_t *oh = reinterpret_cast<uint64_t *>(best + fm_pad(nH) / 32);  // even offset
    int32_t *ov = reinterpret_cast<int32_t *>(oh + PH);
    int32_t *side = ov + PH, *vis = side + nH, *queue = vis + nH;
    int32_t reps[3] = {A.rep_random, A.rep_bfs, A.rep_ggg};
    uint64_t doms[3] = {DOM_RANDOM, DOM_BFS, DOM_GGG};
    // candidates in order: [learned], the first `first[a]` repetitions of each
    // algorithm, then (learned mode, best still infeasible) the rest
    int32_t nlrn = score ? 1 : 0;
    int32_t first[3] = {reps[0], reps[1], reps[2]};
    const bool adaptive = A.adaptive && !score;
    if (score) {
      first[0] = min(A.lrep_random, reps[0]);
      first[1] = min(A.lrep_bfs, reps[1]);
      first[2] = min(A.lrep_ggg, reps[2]);
    } else if (adaptive) {
      for (int a = 0; a < 3; ++a) first[a] = (reps[a] + 1) / 2;  // stage 1
    }
    int32_t rest[3] = {reps[0] - first[0], reps[1] - first[1], reps[2] - first[2]};
    int32_t R0 = nlrn + first[0] + first[1] + first[2];
    int32_t R1 = rest[0] + rest[1] + rest[2];
    bool have = false;
    int32_t binf = 0, brep = -1;
    int64_t bov = 0, bcut = 0;
    int32_t fa[3] = {0, 0, 0};
    int64_t s1[3] = {0, 0, 0};
    unsigned __int128 s2[3] = {0, 0, 0};
    for (int phase = 0; phase < 2; ++phase) {
      if (phase == 1) {
        if (adaptive) {
          // stage 2 keeps an algorithm while mean - 2 sd (population) of its
          // feasible stage-1 cuts is at most the best feasible cut, exactly:
          // s1 - f b <= 2 sqrt(f s2 - s1^2); everything stays when no run is
          // feasible yet
          if (threadIdx.x == 0) {
            const bool feas = s_wk[s_bw][0] == 0;
            const int64_t b = s_wk[s_bw][2];
            for (int a = 0; a < 3; ++a) {
              int32_t f = 0;
              int64_t t1 = 0;
              unsigned __int128 t2 = 0;
              for (int x = 0; x < IPW; ++x) {
                f += s_fa[x][a];
                t1 += s_s1[x][a];
                t2 += s_s2[x][a];
              }
              bool keep = true;
              if (feas) {
                if (f == 0) {
                  keep = false;
                } else {
                  const __int128 D = (__int128)t1 - (__int128)f * b;
                  const __int128 var = (__int128)f * (__int128)t2 - (__int128)t1 * t1;
                  keep = D <= 0 || D * D <= 4 * var;
                }
              }
              s_rest[a] = keep ? reps[a] - first[a] : 0;
            }
          }
          __syncthreads();
          rest[0] = s_rest[0];
          rest[1] = s_rest[1];
          rest[2] = s_rest[2];
          R1 = rest[0] + rest[1] + rest[2];
          if (R1 == 0) break;
        } else if (R1 == 0 || s_wk[s_bw][0] == 0) {
          break;
        }
      }
      int32_t Rp = phase == 0 ? R0 : R1;
      const int32_t *cnt = phase == 0 ? first : rest;
      for (int32_t q = w; q < Rp; q += IPW) {
        int a, r;
        if (phase == 0 && q < nlrn) {
          a = 3;
          r = 0;
        } else {
          int32_t x = phase == 0 ? q - nlrn : q;
          a = x < cnt[0] ? 0 : (x < cnt[0] + cnt[1] ? 1 : 2);
          r = a == 0 ? x : (a == 1 ? x - cnt[0] : x - cnt[0] - cnt[1]);
          if (phase == 1) r += first[a];
        }
        uint64_t key = a == 3 ? 0 : key_step(key_step(D.key, doms[a]), (uint64_t)r);
        warp_initial(a, h, D.t0, key, side, oh, ov, F.key, vis, queue, score);
        for (int32_t v = lane; v < fm_pad(nH); v += 32) {
          const unsigned m = __ballot_sync(0xFFFFFFFFu, v < nH && side[v] != 0);
          if (lane == 0) F.bits[v >> 5] = m;
        }
        __syncwarp();
        int32_t W0, W1;
        const int64_t cut = warp_fm(A, nH, hL0, hL1, F, W0, W1);
        int64_t o0 = (int64_t)W0 - hL0, o1 = (int64_t)W1 - hL1;
        int64_t o = o0 > o1 ? o0 : o1;
        int32_t inf = o > 0;
        int64_t ovv = inf ? o : 0;
        if (phase == 0 && a < 3 && !inf) {
          fa[a] += 1;
          s1[a] += cut;
          s2[a] += (unsigned __int128)((uint64_t)cut) * (uint64_t)cut;
        }
        if (!have || fm_less(inf, ovv, cut, binf, bov, bcut)) {
          have = true;
          binf = inf;
          bov = ovv;
          bcut = cut;
          brep = phase == 0 ? q : R0 + q;
          for (int32_t x = lane; x < fm_pad(nH) / 32; x += 32) best[x] = F.bits[x];
        }
        __syncwarp();
      }
      if (lane == 0) {
        s_wk[w][0] = have ? binf : 2;
        s_wk[w][1] = bov;
        s_wk[w][2] = bcut;
        s_wrep[w] = have ? brep : INT32_MAX;
        for (int a = 0; a < 3; ++a) {
          s_fa[w][a] = fa[a];
          s_s1[w][a] = s1[a];
          s_s2[w][a] = s2[a];
        }
      }
      __syncthreads();
      // the first candidate with the best (infeasible?, overload, cut) wins
      if (threadIdx.x == 0) {
        int32_t bw_ = 0;
        for (int32_t x = 1; x < IPW; ++x) {
          bool better = fm_less((int32_t)s_wk[x][0], s_wk[x][1], s_wk[x][2], (int32_t)s_wk[bw_][0],
                                s_wk[bw_][1], s_wk[bw_][2]);
          bool tie = !better && !fm_less((int32_t)s_wk[bw_][0], s_wk[bw_][1], s_wk[bw_][2],
                                         (int32_t)s_wk[x][0], s_wk[x][1], s_wk[x][2]);
          if (better || (tie && s_wrep[x] < s_wrep[bw_])) bw_ = x;
        }
        s_bw = bw_;
      }
      __syncthreads();
    }
  }
  {
    const uint32_t *bsrc = reinterpret_cast<const uint32_t *>(wbuf + per_warp * s_bw + fm_words(nH));
    for (int32_t v = threadIdx.x; v < nH; v += IPT) fin[v] = fm_side(bsrc, v);
  }
  __syncthreads();
  if (A.sink.counters && !A.sink.item_level) record_sample(A.sink, h, fin, D.key);
  // 3. uncoarsen with FM on every level (warp 0)
  int32_t *cur = fin;
  int32_t *fmbuf = align16(B.take(fm_words(n0) + 4));
  if (B.oom) {
    if (threadIdx.x == 0) atomicExch(A.oom, 1);
    return;
  }
  for (int32_t l = nl - 2; l >= 0; --l) {
    LG g = lv[l];
    int32_t *fine = B.take(g.n);
    if (B.oom) {
      if (threadIdx.x == 0) atomicExch(A.oom, 1);
      return;
    }
    const int32_t *map = maps[l];
    const FMState F = cta_fm_state(g, dyn, A.dyn_words, fmbuf);
    cta_set_bits(F.bits, g.n, [&](int32_t v) { return cur[map[v]]; });
    __syncthreads();
    cta_fm(A, g.n, level_cap(D.L0, D.t0, g.maxc), level_cap(D.L1, D.t1, g.maxc), F);
    __syncthreads();
    for (int32_t v = threadIdx.x; v < g.n; v += IPT) fine[v] = fm_side(F.bits, v);
    __syncthreads();
    cur = fine;
  }
  for (int32_t v = threadIdx.x; v < n0; v += IPT) A.side_out[D.vbase + v] = cur[v];
  __syncthreads();
  if (A.sink.counters && A.sink.item_level) record_sample(A.sink, lv[0], cur, D.key);
}

#if KMP_IP_MULTI
#define k_ip_items k_ip_items_multi
#endif
__global__ void __launch_bounds__(IPT, 3) k_ip_items(const __grid_constant__ IPArgs A) {
  __shared__ int32_t s_it;
  extern __shared__ __align__(16) int32_t ipdyn[];  // working state, then the warps' tables
  int32_t *wkeys = ipdyn + A.dyn_words, *wvals = wkeys + IPW * A.wtab;
  // item b of the order first: the CTA's region is sized for it, and later ones are smaller
  if (threadIdx.x == 0) {
    const int64_t r0 = A.region[blockIdx.x];
    region() = Region{A.scratch + r0, A.region[blockIdx.x + 1] - r0};
    s_it = blockIdx.x;
  }
  for (;;) {
    __syncthreads();
    int32_t q = s_it;
    __syncthreads();
    if (q >= A.nitems) break;
    run_item(A, A.order[q], wkeys, wvals, ipdyn);
    if (threadIdx.x == 0) s_it = gridDim.x + atomicAdd(A.queue, 1);
  }
}

static void launch_items(const IPArgs &A, int grid, size_t smem) {
  static bool attr_set = false;
  if (!attr_set) {
    KMP_CUDA(cudaFuncSetAttribute(k_ip_items, cudaFuncAttributeMaxDynamicSharedMemorySize, 4 * IP_WORDS1));
    attr_set = true;
  }
  k_ip_items<<<grid, IPT, smem, ctx().stream>>>(A);
  KMP_LAUNCHED("ip_items");
}

#if KMP_IP_MULTI
}  // namespace multi
void launch_items_multi(const IPArgs &A, int grid, size_t smem) { multi::launch_items(A, grid, smem); }
#else
void launch_items_multi(const IPArgs &A, int grid, size_t smem);  // kmp_ip_multi.cu

// ------------------------------------------------------ extraction (host side kernels)
__global__ void k_block_keys(int32_t n, const int32_t *part, int bits, uint64_t *keys) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x)
    keys[v] = ((uint64_t)(uint32_t)part[v] << bits) | (uint64_t)v;
}

// Rows above EXT_BIG entries are listed and taken by a CTA each (k_*_big): on one
// warp a hub's row of 10^5 entries outlasted the rest of the kernel (both kernels
// over all rounds of R-MAT 2^22, k = 2^12: 33.6 ms).  Shorter rows stay on a warp,
// with the gathers of EXT_U chunks in flight.
constexpr int64_t EXT_BIG = 2048;
constexpr int EXT_U = 4;
__global__ void k_block_stats(int32_t n, const int64_t *__restrict__ xadj, const int32_t *__restrict__ adj,
                              const int32_t *__restrict__ vw, const int32_t *__restrict__ part,
                              const uint64_t *__restrict__ keys, uint64_t mask, int32_t *members, int32_t *bcount,
                              unsigned long long *bweight, int32_t *ideg, unsigned long long *becount, int32_t *big,
                              int32_t *nbig) {
  // a warp takes 32 consecutive positions and walks their rows one by one
  int lane = threadIdx.x & 31;
  int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t base = gw * 32; base < n; base += nw * 32) {
    int64_t i = base + lane;
    int32_t v = -1, b = -1;
    int64_t rb = 0, re = 0;
    if (i < n) {
      v = (int32_t)(keys[i] & mask);
      members[i] = v;
      b = part[v];
      rb = xadj[v];
      re = xadj[v + 1];
      if (re - rb > EXT_BIG) {
        big[atomicAdd(nbig, 1)] = (int32_t)i;
        re = rb;
      }
    }
    int32_t myd = 0;
    int jmax = (int)(n - base < 32 ? n - base : 32);
    for (int j = 0; j < jmax; ++j) {
      const int32_t bj = __shfl_sync(0xFFFFFFFFu, b, j);
      const int64_t q0 = (int64_t)__shfl_sync(0xFFFFFFFFu, (unsigned long long)rb, j);
      const int64_t q1 = (int64_t)__shfl_sync(0xFFFFFFFFu, (unsigned long long)re, j);
      int32_t d = 0;
      for (int64_t q = q0 + lane; q < q1; q += 32 * EXT_U) {
        int32_t u[EXT_U];
#pragma unroll
        for (int r = 0; r < EXT_U; ++r) u[r] = q + 32 * r < q1 ? adj[q + 32 * r] : -1;
#pragma unroll
        for (int r = 0; r < EXT_U; ++r)
          if (u[r] >= 0) d += (part[u[r]] == bj);
      }
      d = warp_sum32(d);
      if (lane == j) myd = d;
    }
    if (i < n) {
      atomicAdd(&bcount[b], 1);
      atomicAdd(&bweight[b], (unsigned long long)(vw ? vw[v] : 1));
      ideg[i] = myd;
      if (myd) atomicAdd(&becount[b], (unsigned long long)myd);
    }
  }
}
__global__ void __launch_bounds__(256) k_block_stats_big(const int32_t *big, const int32_t *nbig, const int64_t *xadj,
                                                         const int32_t *adj, const int32_t *part, const int32_t *members,
                                                         int32_t *ideg, unsigned long long *becount) {
  __shared__ int32_t s_d;
  const int32_t nb = *nbig;
  for (int32_t x = blockIdx.x; x < nb; x += gridDim.x) {
    const int32_t i = big[x], v = members[i], b = part[v];
    if (threadIdx.x == 0) s_d = 0;
    __syncthreads();
    int32_t d = 0;
    const int64_t e = xadj[v + 1];
#pragma unroll 4
    for (int64_t q = xadj[v] + threadIdx.x; q < e; q += 256) d += (part[adj[q]] == b);
    d = warp_sum32(d);
    if ((threadIdx.x & 31) == 0 && d) atomicAdd(&s_d, d);
    __syncthreads();
    if (threadIdx.x == 0) {
      ideg[i] = s_d;
      atomicAdd(&becount[b], (unsigned long long)s_d);
    }
    __syncthreads();
  }
}

__global__ void k_local_ids(int32_t n, const int32_t *members, const int32_t *part, const int32_t *boff,
                            int32_t *loc) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    int32_t v = members[i];
    loc[v] = (int32_t)(i - boff[part[v]]);
  }
}

__global__ void k_fill_sub(int32_t n, const int64_t *__restrict__ xadj, const int32_t *__restrict__ adj,
                           const int32_t *__restrict__ vw, const int32_t *__restrict__ ew,
                           const int32_t *__restrict__ part, const int32_t *__restrict__ members,
                           const int32_t *__restrict__ loc, const int64_t *__restrict__ gx,
                           uint16_t *__restrict__ sadj, int32_t *__restrict__ sew, int32_t *__restrict__ svw) {
  // a warp per row, order-preserving compaction of the entries inside the block
  int lane = threadIdx.x & 31;
  int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t i = gw; i < n; i += nw) {
    int32_t v = members[i];
    int32_t b = part[v];
    if (lane == 0) svw[i] = vw ? vw[v] : 1;
    int64_t o = gx[i];
    const int64_t rb = xadj[v], re = xadj[v + 1];
    if (re - rb > EXT_BIG) continue;  // k_fill_sub_big
    for (int64_t q0 = rb; q0 < re; q0 += 32 * EXT_U) {
      int32_t u[EXT_U], pu[EXT_U];
#pragma unroll
      for (int r = 0; r < EXT_U; ++r) u[r] = q0 + 32 * r + lane < re ? adj[q0 + 32 * r + lane] : -1;
#pragma unroll
      for (int r = 0; r < EXT_U; ++r) pu[r] = u[r] >= 0 ? part[u[r]] : -1;
#pragma unroll
      for (int r = 0; r < EXT_U; ++r) {
        const bool keep = pu[r] == b;
        const unsigned bal = __ballot_sync(0xFFFFFFFFu, keep);
        if (keep) {
          const int64_t p = o + __popc(bal & ((1u << lane) - 1u));
          sadj[p] = (uint16_t)loc[u[r]];
          if (ew) sew[p] = ew[q0 + 32 * r + lane];
        }
        o += __popc(bal);
      }
    }
  }
}
__global__ void __launch_bounds__(256) k_fill_sub_big(const int32_t *big, const int32_t *nbig, const int64_t *xadj,
                                                      const int32_t *adj, const int32_t *ew, const int32_t *part,
                                                      const int32_t *members, const int32_t *loc, const int64_t *gx,
                                                      uint16_t *sadj, int32_t *sew) {
  __shared__ int32_t s_cnt[8];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int32_t nb = *nbig;
  for (int32_t x = blockIdx.x; x < nb; x += gridDim.x) {
    const int32_t i = big[x], v = members[i], b = part[v];
    int64_t o = gx[i];
    const int64_t re = xadj[v + 1];
    for (int64_t t0 = xadj[v]; t0 < re; t0 += 256 * EXT_U) {  // a tile: EXT_U chunks of 32 a warp, in order
      const int64_t q0 = t0 + 32 * EXT_U * w;
      int32_t u[EXT_U];
      unsigned bal[EXT_U];
      int32_t cnt = 0;
#pragma unroll
      for (int r = 0; r < EXT_U; ++r) u[r] = q0 + 32 * r + lane < re ? adj[q0 + 32 * r + lane] : -1;
#pragma unroll
      for (int r = 0; r < EXT_U; ++r) {
        bal[r] = __ballot_sync(0xFFFFFFFFu, u[r] >= 0 && part[u[r]] == b);
        cnt += __popc(bal[r]);
      }
      if (lane == 0) s_cnt[w] = cnt;
      __syncthreads();
      int64_t p = o;
      int32_t tot = 0;
      for (int y = 0; y < 8; ++y) {
        if (y < w) p += s_cnt[y];
        tot += s_cnt[y];
      }
#pragma unroll
      for (int r = 0; r < EXT_U; ++r) {
        if ((bal[r] >> lane) & 1u) {
          const int64_t at = p + __popc(bal[r] & ((1u << lane) - 1u));
          sadj[at] = (uint16_t)loc[u[r]];
          if (ew) sew[at] = ew[q0 + 32 * r + lane];
        }
        p += __popc(bal[r]);
      }
      o += tot;
      __syncthreads();  // the next tile rewrites the counts
    }
  }
}

__global__ void k_set_last(int64_t *a, int64_t idx, const int64_t *v) { a[idx] = *v; }

__global__ void k_write_parts(int32_t n, const int32_t *members, const int32_t *part_old,
                              const int32_t *newid, const int32_t *split, const int32_t *side,
                              int32_t *part) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    int32_t v = members[i];
    int32_t b = part_old[v];
    part[v] = newid[b] + (split[b] ? side[i] : 0);
  }
}

// caps4 (host, nullable): explicit (t0, t1, L0, L1) per block instead of the
// caps Algorithm 2 derives from (eps, cV, k, f)
int32_t bipartition_blocks(const Graph &g, int32_t *part, int32_t nblocks, std::vector<int32_t> &f,
                           double eps, int64_t cV, int32_t k, uint64_t roundkey, int32_t *items_out,
                           const int32_t *caps4) {
  Context &C = ctx();
  const kmp_config &cfg = C.cfg;
  cudaStream_t s = C.stream;
  int32_t n = g.n;
  // new ids, child final counts
  std::vector<int32_t> newid(nblocks), split(nblocks), nf;
  int32_t nn = 0;
  for (int32_t b = 0; b < nblocks; ++b) {
    newid[b] = nn;
    if (f[b] >= 2) {
      split[b] = 1;
      nf.push_back(f[b] / 2);
      nf.push_back(f[b] - f[b] / 2);
      nn += 2;
    } else {
      split[b] = 0;
      nf.push_back(f[b]);
      nn += 1;
    }
  }
  if (items_out) *items_out = 0;
  if (n == 0) {
    f = nf;
    return nn;
  }
  int bitsN = 1;
  while ((1ll << bitsN) < (int64_t)n) ++bitsN;
  int bitsB = 1;
  while ((1ll << bitsB) < (int64_t)nblocks) ++bitsB;
  int grid = grid_for(n, 256);
  DBuf<uint64_t> keys(n), tmp(n);
  k_block_keys<<<grid, 256, 0, s>>>(n, part, bitsN, keys);
  KMP_LAUNCHED("block_keys");
  // keys are written in ascending node order, so a stable sort by the block
  // bits alone leaves every block's members in ascending id
  radix_sort_u64(keys, tmp, n, bitsB, bitsN);
  DBuf<int32_t> members(n), bcount(nblocks + 1), ideg(n), boff(nblocks + 1), loc(n);
  DBuf<unsigned long long> bweight(nblocks), becount(nblocks);
  bcount.zero();
  bweight.zero();
  becount.zero();
  DBuf<int32_t> big, nbig(1);
  big.alloc(g.m / (EXT_BIG + 1) + 1);  // at most so many rows above EXT_BIG entries
  nbig.zero();
  const int grid_big = C.sms * 8;
  k_block_stats<<<grid, 256, 0, s>>>(n, g.xadj, g.adj, g.vw, part, keys, (1ull << bitsN) - 1ull, members,
                                     bcount, bweight, ideg, becount, big, nbig);
  KMP_LAUNCHED("block_stats");
  if (g.maxdeg > EXT_BIG) {
    k_block_stats_big<<<grid_big, 256, 0, s>>>(big, nbig, g.xadj, g.adj, part, members, ideg, becount);
    KMP_LAUNCHED("block_stats_big");
  }
  scan_excl_i32(bcount, boff, nblocks + 1, nullptr);
  k_local_ids<<<grid, 256, 0, s>>>(n, members, part, boff, loc);
  KMP_LAUNCHED("local_ids");
  DBuf<int64_t> gx(n + 1), etot(1);
  scan_excl_i32_to_i64(ideg, gx, n, etot);
  k_set_last<<<1, 1, 0, s>>>(gx, n, etot);
  KMP_LAUNCHED("set_last");
  int64_t E = read1(etot.p);
  DBuf<uint16_t> sadj(E);
  DBuf<int32_t> sew, svw(n);
  if (g.ew) sew.alloc(E);
  k_fill_sub<<<grid, 256, 0, s>>>(n, g.xadj, g.adj, g.vw, g.ew, part, members, loc, gx, sadj, sew.p, svw);
  KMP_LAUNCHED("fill_sub");
  if (g.maxdeg > EXT_BIG) {
    k_fill_sub_big<<<grid_big, 256, 0, s>>>(big, nbig, g.xadj, g.adj, g.ew, part, members, loc, gx, sadj, sew.p);
    KMP_LAUNCHED("fill_sub_big");
  }
  std::vector<int32_t> hcount(nblocks + 1), hoff(nblocks + 1);
  std::vector<unsigned long long> hw(nblocks), he(nblocks);
  to_host(hcount.data(), bcount.p, nblocks);
  to_host(hoff.data(), boff.p, nblocks + 1);
  to_host(hw.data(), bweight.p, nblocks);
  to_host(he.data(), becount.p, nblocks);
  // item descriptors
  std::vector<ItemDesc> items;
  int64_t ebase = 0;
  for (int32_t b = 0; b < nblocks; ++b) {
    int64_t eb = ebase;
    ebase += (int64_t)he[b];
    if (!split[b] || hcount[b] == 0) continue;
    if (hcount[b] > IP_MAX_N)
      fail(KMP_ERR_UNSUPPORTED, "block of " + std::to_string(hcount[b]) +
                                    " nodes exceeds the bipartitioner's item limit");
    ItemDesc d{};
    d.vbase = hoff[b];
    d.ebase = eb;
    d.n = hcount[b];
    d.m = (int32_t)he[b];
    if (caps4) {
      d.t0 = caps4[4 * b];
      d.t1 = caps4[4 * b + 1];
      d.L0 = caps4[4 * b + 2];
      d.L1 = caps4[4 * b + 3];
    } else {
      split_caps(eps, cV, k, (int64_t)hw[b], f[b], &d.t0, &d.t1, &d.L0, &d.L1);
    }
    d.key = key_step(roundkey, (uint64_t)b);
    items.push_back(d);
  }
  if (items_out) *items_out = (int32_t)items.size();
  DBuf<int32_t> side(n);
  side.zero();
  if (!items.empty()) {
    DBuf<int32_t> dorder(items.size()), q(2);
    bool learned = cfg.learned && proposer().W;
    int64_t mult = 1;
    // One wave of CTAs that take items from the queue, largest first (the order does
    // not change results); each has one scratch region and reuses it, so that what
    // the CTAs touch stays in L2 (a region per item spread 8192 items of 2048 nodes
    // over 36 GB).
    int64_t maxn = 0;
    std::vector<int64_t> words;
    for (auto &d : items) {
      maxn = std::max<int64_t>(maxn, d.n);
      words.push_back(ip_scratch_words(d.n, d.m, learned ? 2 * MF + 3 * MH + 4 : 0));
    }
    const int per_sm = std::min<int>(C.tune.ip_blocks_per_sm, 3);
    const int gridip = (int)std::min<int64_t>((int64_t)items.size(), (int64_t)C.sms * per_sm);
    for (int attempt = 0; attempt < 6; ++attempt, mult *= 4) {
      const IPRegions plan = ip_regions(words, gridip, mult);
      DBuf<ItemDesc> ditems(items.size());
      DBuf<int64_t> dregion(plan.region.size());
      DBuf<int32_t> scratch(plan.region.back());
      to_dev(dorder.p, plan.order.data(), plan.order.size());
      to_dev(dregion.p, plan.region.data(), plan.region.size());
      to_dev(ditems.p, items.data(), items.size());
      q.zero();
      IPArgs A;
      A.items = ditems;
      A.order = dorder;
      A.nitems = (int32_t)items.size();
      A.queue = q.p;
      A.oom = q.p + 1;
      A.gx = gx;
      A.sadj = sadj;
      A.sew = sew.p;
      A.svw = svw;
      A.side_out = side;
      A.scratch = scratch;
      A.region = dregion;
      A.S = cfg.subrounds;
      A.ip_C = cfg.ip_C;
      A.ip_lp_rounds = cfg.ip_lp_rounds;
      A.rep_random = cfg.rep_random;
      A.rep_bfs = cfg.rep_bfs;
      A.rep_ggg = cfg.rep_ggg;
      A.fm_passes = cfg.fm_passes;
      A.fm_stop = cfg.fm_stop;
      A.conv_num = cfg.conv_num;
      A.conv_den = cfg.conv_den;
      A.W = cfg.learned ? proposer().W : nullptr;
      A.lrep_random = cfg.lrep_random;
      A.lrep_bfs = cfg.lrep_bfs;
      A.lrep_ggg = cfg.lrep_ggg;
      A.adaptive = (cfg.adaptive && !A.W) ? 1 : 0;
      A.learned_item = (cfg.learned == 2 && A.W) ? 1 : 0;
      A.sink = sample_sink();
      // working state: the LP arrays (5.5 words a node and the sort space of a
      // sub-round's contested proposals), then FM's (3.6 words a node, the entries
      // where they fit) of the largest item, at least 16 KB (the portfolio of small
      // coarsest graphs); see IP_WORDS*
      const int64_t want = std::max<int64_t>(6 * maxn + maxn / 8 + 256, 4096);
      const int64_t words = (int64_t)items.size() <= C.sms ? IP_WORDS1 : IP_WORDS3;
      int32_t wtab = IP_WTAB_MIN;
      while (wtab < IP_WTAB_MAX && 2 * IPW * (2 * wtab) + want <= words) wtab *= 2;
      A.wtab = wtab;
      A.dyn_words = (int32_t)std::min<int64_t>((want + 3) & ~3ll, words - 2 * IPW * wtab);
      const size_t dyn_bytes = 4 * (size_t)(2 * IPW * A.wtab + A.dyn_words);
      if (g.multi) launch_items_multi(A, gridip, dyn_bytes);
      else launch_items(A, gridip, dyn_bytes);
      int32_t oom = 0;
      to_host(&oom, q.p + 1, 1);
      if (!oom) break;
      if (attempt == 5) fail(KMP_ERR_NOMEM, "bipartitioner scratch could not be sized");
    }
  }
  DBuf<int32_t> dnew(nblocks), dsplit(nblocks), old(n);
  to_dev(dnew.p, newid.data(), nblocks);
  to_dev(dsplit.p, split.data(), nblocks);
  KMP_CUDA(cudaMemcpyAsync(old.p, part, (size_t)n * sizeof(int32_t), cudaMemcpyDeviceToDevice, s));
  k_write_parts<<<grid, 256, 0, s>>>(n, members, old, dnew, dsplit, side, part);
  KMP_LAUNCHED("write_parts");
  f = nf;
  return nn;
}
#endif  // KMP_IP_MULTI

}  // namespace kmp
