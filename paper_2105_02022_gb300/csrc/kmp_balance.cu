// k-way balancing (Section 4.3, "Balancing").
//
// Deterministic reading: the starting state initialises the candidates of
// every overloaded block at once (the paper's priority-queue initialisation):
// a node v of an overloaded block B with some admissible other block gets
// d = max over admissible blocks of conn(v, b) - conn(v, B) and the relative
// gain d*c(v) (d >= 0) or d/c(v) (d < 0).  Then the overloaded blocks are
// emptied in ascending id, candidates in (relative gain desc, id asc) order,
// each moved at its turn to the admissible block of largest current
// connectivity (ties: lowest id) until the block fits.
//
// GPU mapping: candidates of all overloaded blocks in one full-GPU pass (one
// warp per node, connectivity in a per-warp hash table); grouping by block
// with a radix sort of (block, node) keys; one CTA per overloaded block sorts
// its candidates by the exact rational order; then every overloaded block
// speculates its moves at once (one warp each, as if it were emptied first),
// and one CTA commits in block order: a speculated move stands while its
// target still fits, everything else is decided again exactly, in batches
// whose members are evaluated at once and committed while they provably do
// not interact.
#include <algorithm>
#include <climits>

#include "kmp_internal.cuh"

namespace kmp {

constexpr int BAL_T = 256;
constexpr int BAL_W = BAL_T / 32;
constexpr int BAL_STAB = 512;  // per-warp shared table entries

struct BalArgs {
  int32_t n, k;
  const int64_t *xadj;
  const int32_t *adj;
  const int32_t *vw;
  const int32_t *ew;
  int32_t *part;
  int64_t *bw;
  const int32_t *cap;
  const uint8_t *over;
  const int32_t *olist;  // the overloaded blocks, ascending
  int32_t nover;
  int64_t max_room;      // the largest cap - weight over all blocks at the start
  int64_t *cand_d;       // [n] d of candidate nodes
  uint64_t *keys;        // (block << bitsN | node) of candidates
  int32_t *ncand;
  int bitsN;
  int32_t *seg_lo;       // [k] candidate segment of each block
  int32_t *seg_hi;
  uint64_t *sortbuf;     // per-block sort space (2 * ncand)
  int32_t *gtab;         // per-warp global tables when labels do not fit shared memory
  uint32_t gcap;
  unsigned long long *moved;
  // speculation: per overloaded block (index in olist) up to SPEC_MAX moves
  int32_t *spec_v, *spec_t;  // [nover][SPEC_MAX]
  int32_t *spec_n;           // moves recorded
  int32_t *spec_end;         // candidate position where the speculation stopped
  int32_t *spec_sat;         // 1: the block fits after its recorded moves
};

constexpr int SPEC_MAX = 16;

__device__ __forceinline__ int32_t bw_node(const BalArgs &A, int32_t v) { return A.vw ? A.vw[v] : 1; }

// table size for v's connectivity: a power of two >= 2 * (distinct blocks
// among its neighbours, at most min(degree, k)), at least 32
__device__ __forceinline__ uint32_t conn_cap(const BalArgs &A, int32_t v) {
  int64_t d = A.xadj[v + 1] - A.xadj[v];
  if (d > A.k) d = A.k;
  uint32_t cap = 32;
  while ((int64_t)cap < 2 * d) cap <<= 1;
  return cap;
}

// connectivity of v to the blocks of its neighbours, aggregated by one warp
__device__ int64_t conn_table(const BalArgs &A, int32_t v, int32_t *K, int32_t *V, uint32_t &mask) {
  int lane = threadIdx.x & 31;
  int64_t b = A.xadj[v], e = A.xadj[v + 1];
  uint32_t cap = conn_cap(A, v);
  mask = cap - 1;
  for (uint32_t i = lane; i < cap; i += 32) {
    K[i] = HT_EMPTY;
    V[i] = 0;
  }
  __syncwarp();
  // 128 entries per pass (four gathers in flight per lane); lanes that hit the
  // same block add their weights first, so a hub's many entries into one block
  // cost one atomic per pass instead of one per entry
  for (int64_t base = b; base < e; base += 128) {
    int32_t u[4], wt[4], blk[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      int64_t q = base + r * 32 + lane;
      bool ok = q < e;
      u[r] = ok ? A.adj[q] : -1;
      wt[r] = ok ? (A.ew ? A.ew[q] : 1) : 0;
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) blk[r] = u[r] >= 0 ? A.part[u[r]] : HT_EMPTY;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      unsigned peers = __match_any_sync(0xFFFFFFFFu, blk[r]);
      int32_t s = __reduce_add_sync(peers, wt[r]);
      if (blk[r] != HT_EMPTY && lane == __ffs(peers) - 1) ht_add(K, V, mask, blk[r], s);
    }
  }
  __syncwarp();
  return ht_get(K, V, mask, A.part[v]);
}

// some block has room for weight c (the overloaded block itself has none);
// candidates are rated from the starting state, so the starting room decides
__device__ __forceinline__ bool room_somewhere(const BalArgs &A, int64_t c) { return A.max_room >= c; }

// Candidates of the overloaded blocks, one warp per node with the warp's
// shared-memory table.  Nodes whose table would not fit it are listed in
// big[] for k_bal_cand_big.
__global__ void __launch_bounds__(BAL_T) k_bal_cand(BalArgs A, int32_t *big, int32_t *nbig) {
  __shared__ int32_t sk[BAL_W][BAL_STAB], sv[BAL_W][BAL_STAB];
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int64_t gw = (int64_t)blockIdx.x * BAL_W + w, nw = (int64_t)gridDim.x * BAL_W;
  int32_t *K = sk[w], *V = sv[w];
  for (int64_t v = gw; v < A.n; v += nw) {
    int32_t B = A.part[v];
    if (!A.over[B]) continue;
    if (conn_cap(A, (int32_t)v) > (uint32_t)BAL_STAB) {
      if (lane == 0) big[atomicAdd(nbig, 1)] = (int32_t)v;
      continue;
    }
    uint32_t mask;
    int64_t cown = conn_table(A, (int32_t)v, K, V, mask);
    int64_t c = bw_node(A, (int32_t)v);
    int64_t best = -1;
    for (uint32_t i = lane; i <= mask; i += 32) {
      int32_t b = K[i];
      if (b == HT_EMPTY || b == B) continue;
      if (A.bw[b] + c > A.cap[b]) continue;
      if (V[i] > best) best = V[i];
    }
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) {
      int64_t o = (int64_t)shfl_xor64((uint64_t)best, m);
      best = o > best ? o : best;
    }
    if (best < 0 && room_somewhere(A, c)) best = 0;  // an admissible block without neighbours
    if (lane == 0 && best >= 0) {
      A.cand_d[v] = best - cown;
      int32_t p = atomicAdd(A.ncand, 1);
      A.keys[p] = ((uint64_t)(uint32_t)B << A.bitsN) | (uint64_t)v;
    }
    __syncwarp();
  }
}

// Candidates among the listed high-degree nodes: one CTA per node, the node's
// row spread over all threads into the CTA's own global table region
// (2 * gcap words; the node uses the power of two >= 2 min(degree, k)).
__global__ void __launch_bounds__(BAL_T) k_bal_cand_big(BalArgs A, const int32_t *big, const int32_t *nbig) {
  __shared__ int64_t s_best[BAL_W];
  __shared__ int64_t s_cown;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int32_t *K = A.gtab + (int64_t)blockIdx.x * 2 * A.gcap, *V = K + A.gcap;
  const int32_t nb = *nbig;
  for (int32_t i = blockIdx.x; i < nb; i += gridDim.x) {
    const int32_t v = big[i], B = A.part[v];
    const uint32_t cap = conn_cap(A, v), mask = cap - 1;
    for (uint32_t x = threadIdx.x; x < cap; x += BAL_T) {
      K[x] = HT_EMPTY;
      V[x] = 0;
    }
    if (threadIdx.x == 0) s_cown = 0;
    __syncthreads();
    const int64_t b = A.xadj[v], e = A.xadj[v + 1];
    for (int64_t base = b + 32 * w; base < e; base += BAL_T) {
      const int64_t q = base + lane;
      const bool ok = q < e;
      const int32_t u = ok ? A.adj[q] : -1;
      const int32_t wt = ok ? (A.ew ? A.ew[q] : 1) : 0;
      const int32_t blk = ok ? A.part[u] : HT_EMPTY;
      const unsigned peers = __match_any_sync(0xFFFFFFFFu, blk);
      const int32_t sm = __reduce_add_sync(peers, wt);
      if (blk != HT_EMPTY && lane == __ffs(peers) - 1) ht_add(K, V, mask, blk, sm);
    }
    __syncthreads();
    const int64_t c = bw_node(A, v);
    int64_t best = -1;
    for (uint32_t x = threadIdx.x; x < cap; x += BAL_T) {
      const int32_t blk = K[x];
      if (blk == HT_EMPTY) continue;
      if (blk == B) {
        s_cown = V[x];
        continue;
      }
      if (A.bw[blk] + c > A.cap[blk]) continue;
      if (V[x] > best) best = V[x];
    }
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) {
      int64_t o = (int64_t)shfl_xor64((uint64_t)best, m);
      best = o > best ? o : best;
    }
    if (lane == 0) {
      s_best[w] = best;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      int64_t bb = -1;
      for (int x = 0; x < BAL_W; ++x) {
        bb = s_best[x] > bb ? s_best[x] : bb;
      }
      if (bb < 0 && room_somewhere(A, c)) bb = 0;  // an admissible block without neighbours
      if (bb >= 0) {
        A.cand_d[v] = bb - s_cown;
        int32_t p = atomicAdd(A.ncand, 1);
        A.keys[p] = ((uint64_t)(uint32_t)B << A.bitsN) | (uint64_t)v;
      }
    }
    __syncthreads();
  }
}

__global__ void k_bal_segments(BalArgs A, int32_t N) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N;
       i += (int64_t)gridDim.x * blockDim.x) {
    int32_t B = (int32_t)(A.keys[i] >> A.bitsN);
    if (i == 0 || (int32_t)(A.keys[i - 1] >> A.bitsN) != B) A.seg_lo[B] = (int32_t)i;
    if (i == N - 1 || (int32_t)(A.keys[i + 1] >> A.bitsN) != B) A.seg_hi[B] = (int32_t)i + 1;
  }
}

// "a before b" in (relative gain desc, node asc); exact with 64-bit products
__device__ __forceinline__ bool rg_before(int64_t d1, int64_t c1, int32_t v1, int64_t d2, int64_t c2,
                                          int32_t v2) {
  bool s1 = d1 >= 0, s2 = d2 >= 0;
  if (s1 != s2) return s1;
  int64_t p = s1 ? d1 * c1 : d1 * c2, q = s1 ? d2 * c2 : d2 * c1;
  if (p != q) return p > q;
  return v1 < v2;
}

// one CTA per overloaded block: bitonic sort of its candidates
__global__ void __launch_bounds__(BAL_T) k_bal_sort(BalArgs A) {
  int32_t B = A.olist[blockIdx.x];
  int32_t lo = A.seg_lo[B], hi = A.seg_hi[B];
  int32_t len = hi - lo;
  if (len <= 1) return;
  int32_t P = 1;
  while (P < len) P <<= 1;
  uint64_t mask = (1ull << A.bitsN) - 1ull;
  int32_t *vv = reinterpret_cast<int32_t *>(A.sortbuf + 2ll * lo);  // 2*len >= P slots
  for (int32_t i = threadIdx.x; i < P; i += blockDim.x)
    vv[i] = i < len ? (int32_t)(A.keys[lo + i] & mask) : -1;
  __syncthreads();
  for (int32_t kk = 2; kk <= P; kk <<= 1)
    for (int32_t j = kk >> 1; j > 0; j >>= 1) {
      for (int32_t i = threadIdx.x; i < P; i += blockDim.x) {
        int32_t l = i ^ j;
        if (l > i) {
          int32_t a = vv[i], b = vv[l];
          // padding (-1) sorts last
          bool b_first;
          if (a < 0) b_first = b >= 0;
          else if (b < 0) b_first = false;
          else b_first = rg_before(A.cand_d[b], bw_node(A, b), b, A.cand_d[a], bw_node(A, a), a);
          if (b_first == ((i & kk) == 0)) {
            vv[i] = b;
            vv[l] = a;
          }
        }
      }
      __syncthreads();
    }
  for (int32_t i = threadIdx.x; i < len; i += blockDim.x)
    A.keys[lo + i] = ((uint64_t)(uint32_t)B << A.bitsN) | (uint64_t)(uint32_t)vv[i];
}

// Moves in candidate order, evaluated in batches of up to 32.  A batch holds
// the shortest prefix of the remaining candidates whose weights cover the
// overload (it may need more moves, never fewer).  The batch's adjacency rows
// are walked at once, building one connectivity table per member and marking
// which members are neighbours of each other.  A small batch (warp 0 alone) then
// decides its members in order, each from its table and the current rooms; a
// move adds its edge weights to the tables of the later members next to it.  A
// large batch (the whole CTA) picks every member's target from the state at its
// start and commits in order: while a block is emptied, every other block only
// gains weight, so a target that is still admissible is still the best (or
// still the lowest-id admissible one), and "no admissible target" stays true;
// only a move of a neighbour changes connectivity.  There a member passes iff
// its target still fits and no earlier move of the batch was its neighbour; at
// the first one that does not, the next batch starts (its first member always
// passes).  Either way the result equals one move at a time.
constexpr int BM_T = 1024;
constexpr int BM_W = BM_T / 32;

// Speculation, one warp per overloaded block B, all blocks at once: B's moves
// in candidate order as if B were the first block emptied (every other block
// at its starting weight, plus B's own recorded moves).  A decision is only
// recorded when nothing an earlier block does can change it: blocks other
// than the overloaded ones only gain weight, so a better block that does not
// fit keeps not fitting, and the chosen block is checked again at commit; an
// earlier overloaded block, however, loses weight (it may start to fit) and
// its moved nodes change their neighbours' connectivity, so a node adjacent
// to an earlier overloaded block stops the speculation, as does a node that
// would need the lowest-id fallback.
__global__ void __launch_bounds__(BAL_T) k_bal_spec(BalArgs A) {
  __shared__ int32_t sk[BAL_W][BAL_STAB], sv[BAL_W][BAL_STAB];
  __shared__ int32_t mv_v[BAL_W][SPEC_MAX], mv_t[BAL_W][SPEC_MAX], mv_c[BAL_W][SPEC_MAX];
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int64_t gw = (int64_t)blockIdx.x * BAL_W + w, nw = (int64_t)gridDim.x * BAL_W;
  int32_t *K = sk[w], *V = sv[w];
  uint64_t vmask = (1ull << A.bitsN) - 1ull;
  for (int64_t ob = gw; ob < A.nover; ob += nw) {
    int32_t B = A.olist[ob];
    int32_t lo = A.seg_lo[B], hi = A.seg_hi[B];
    int64_t wB = A.bw[B];
    int32_t nm = 0, i = lo, sat = 0;
    for (; i < hi; ++i) {
      if (wB <= A.cap[B]) {
        sat = 1;
        break;
      }
      if (nm == SPEC_MAX) break;
      int32_t v = (int32_t)(A.keys[i] & vmask);
      // a node whose table does not fit shared memory is left to the exact commit
      if (conn_cap(A, v) > (uint32_t)BAL_STAB) break;
      int64_t c = bw_node(A, v);
      uint32_t mask;
      conn_table(A, v, K, V, mask);
      // B's own recorded moves of neighbours; neighbours in earlier overloaded blocks
      bool fragile = false;
      for (int64_t q = A.xadj[v] + lane; q < A.xadj[v + 1]; q += 32) {
        int32_t u = A.adj[q], bu = A.part[u];
        if (bu != B && bu < B && A.over[bu]) fragile = true;
        if (bu == B)
          for (int j = 0; j < nm; ++j)
            if (mv_v[w][j] == u) ht_add(K, V, mask, mv_t[w][j], A.ew ? A.ew[q] : 1);
      }
      __syncwarp();
      fragile = __any_sync(0xFFFFFFFFu, fragile);
      uint64_t bestk = 0;  // (conn, ~block): largest connectivity, then lowest id
      if (!fragile)
        for (uint32_t x = lane; x <= mask; x += 32) {
          int32_t b = K[x];
          if (b == HT_EMPTY || b == B) continue;
          int64_t wb = A.bw[b];
          for (int j = 0; j < nm; ++j)
            if (mv_t[w][j] == b) wb += mv_c[w][j];
          if (wb + c > A.cap[b]) continue;
          uint64_t key = ((uint64_t)(uint32_t)V[x] << 32) | (0xFFFFFFFFu - (uint32_t)b);
          bestk = key > bestk ? key : bestk;
        }
      bestk = group_max64<32>(bestk);
      if (fragile || bestk == 0) break;  // left to the exact commit
      int32_t t = (int32_t)(0xFFFFFFFFu - (uint32_t)bestk);
      if (lane == 0) {
        mv_v[w][nm] = v;
        mv_t[w][nm] = t;
        mv_c[w][nm] = (int32_t)c;
        A.spec_v[ob * SPEC_MAX + nm] = v;
        A.spec_t[ob * SPEC_MAX + nm] = t;
      }
      __syncwarp();
      ++nm;
      wB -= c;
    }
    if (i >= hi && wB <= A.cap[B]) sat = 1;
    if (lane == 0) {
      A.spec_n[ob] = nm;
      A.spec_end[ob] = i;
      A.spec_sat[ob] = sat;
    }
    __syncwarp();
  }
}

// ---- the commit: one CTA, driven by its warp 0, block by block
// Its time is the chain of reads that every block's decision waits for, so what
// does not change during the commit is read ahead by all warps at once: a window
// per overloaded block (32 blocks at a time, a warp each) holds the speculated
// moves and the next candidates with weights, rows and adjacency entries.  The
// state that does change is the room of every block (cap less weight), in shared
// memory while k fits, and the blocks of the neighbours, the one gather from
// global memory left per batch.  A batch with at most WS_E entries and WS_T table
// slots is evaluated by warp 0 alone, in shared-memory tables; a larger one by
// the CTA, in shared memory too while its tables fit beside the windows or over them.
// Mesh of 2^20 nodes, 8192 blocks of 128 nodes brought from 10% to 3% imbalance, the whole call: 97.0 -> 58.4 ms with the windows and rooms,
// 30.8 ms with small batches decided to their end (a batch used to stop at the
// first member next to an earlier move, and its tables were built again).
constexpr int WS_E = 256;
constexpr int WS_T = 2048;
constexpr int WS_R = 4;   // entries per lane whose gathers are issued together
constexpr int WIN_E = WS_E;
constexpr int MEMB = 64;  // slots of the batch-member table (at most 32 members)

struct BalWindow {
  int64_t beg[32];        // rows of the candidates
  int64_t epre[33];       // their entries before each
  int32_t B, lo, hi;      // block, its candidate segment
  int32_t sat, send, nm;  // speculation: fits after its moves, where it stopped, moves
  int32_t base, nc;       // candidates [base, base + nc) are held
  int32_t ne;             // entries held: the first ne of theirs
  int32_t sv[SPEC_MAX], st[SPEC_MAX], sc[SPEC_MAX];
  int32_t v[32], c[32];
  int32_t u[WIN_E], w[WIN_E];
};

// window of overloaded block o from candidate `start` on (< 0: its first), one warp
__device__ void load_window(const BalArgs &A, BalWindow &W, int32_t o, int32_t start) {
  const int lane = threadIdx.x & 31;
  const uint64_t vmask = (1ull << A.bitsN) - 1ull;
  const int32_t B = A.olist[o], lo = A.seg_lo[B], hi = A.seg_hi[B], nm = A.spec_n[o];
  const int32_t base = start < 0 ? lo : start, nc = min(32, hi - base);
  int32_t v = 0, c = 0;
  int64_t beg = 0, inc = 0;
  if (lane < nc) {
    v = (int32_t)(A.keys[base + lane] & vmask);
    c = bw_node(A, v);
    beg = A.xadj[v];
    inc = A.xadj[v + 1] - beg;
  }
  if (lane < nm) {
    const int32_t sv = A.spec_v[(int64_t)o * SPEC_MAX + lane];
    W.sv[lane] = sv;
    W.st[lane] = A.spec_t[(int64_t)o * SPEC_MAX + lane];
    W.sc[lane] = bw_node(A, sv);
  }
#pragma unroll
  for (int m = 1; m < 32; m <<= 1) {
    const int64_t x = (int64_t)__shfl_up_sync(0xFFFFFFFFu, (unsigned long long)inc, m);
    if (lane >= m) inc += x;
  }
  W.v[lane] = v;
  W.c[lane] = c;
  W.beg[lane] = beg;
  W.epre[lane + 1] = inc;
  const int64_t total = (int64_t)__shfl_sync(0xFFFFFFFFu, (unsigned long long)inc, 31);
  const int32_t ne = total < WIN_E ? (int32_t)total : WIN_E;
  if (lane == 0) {
    W.epre[0] = 0;
    W.B = B;
    W.lo = lo;
    W.hi = hi;
    W.nm = nm;
    W.sat = A.spec_sat[o];
    W.send = A.spec_end[o];
    W.base = base;
    W.nc = nc;
    W.ne = ne;
  }
  __syncwarp();
#pragma unroll 4
  for (int32_t t = lane; t < ne; t += 32) {
    int32_t j = 0;
#pragma unroll
    for (int st = 16; st > 0; st >>= 1)
      if (W.epre[j + st] <= t) j += st;
    const int64_t q = W.beg[j] + (t - W.epre[j]);
    W.u[t] = A.adj[q];
    W.w[t] = A.ew ? A.ew[q] : 1;
  }
  __syncwarp();
}

// Lowest-id block with room for a member of weight c (>= 1) that has no
// admissible neighbouring block (one warp).  *hint is the lowest block that may
// have room: every block below it has room < 1.  Blocks only gain weight during
// the commit, except the block being emptied (the commit lowers the hint to it
// when it gets room), so the scan starts there and moves the hint up past the
// full blocks it passes.  The overloaded block has no room.
constexpr int LA_U = 8;  // chunks of 32 blocks checked per round trip
__device__ int32_t lowest_admissible(const int32_t *room, int32_t k, int32_t c, int lane, int32_t *hint) {
  int32_t h1 = -1, res = -1;
  for (int32_t base = *hint & ~31; base < k && res < 0; base += 32 * LA_U) {
    int32_t rm[LA_U];
#pragma unroll
    for (int u = 0; u < LA_U; ++u) {
      const int32_t b = base + 32 * u + lane;
      rm[u] = b < k ? room[b] : INT32_MIN;
    }
#pragma unroll
    for (int u = 0; u < LA_U; ++u) {
      const unsigned m1 = __ballot_sync(0xFFFFFFFFu, rm[u] >= 1);
      const unsigned mc = __ballot_sync(0xFFFFFFFFu, rm[u] >= c);
      if (h1 < 0 && m1) h1 = base + 32 * u + __ffs(m1) - 1;
      if (res < 0 && mc) res = base + 32 * u + __ffs(mc) - 1;
    }
  }
  // blocks in [*hint, h1) were seen without room (h1 = k: none has room)
  if (lane == 0) atomicMax(hint, h1 >= 0 ? h1 : k);
  __syncwarp();
  return res;
}

// the batch's members by node id (shared memory): -1 or the member
__device__ __forceinline__ void memb_add(int32_t *mk, int32_t *mv, int32_t v, int32_t j) {
  uint32_t h = fmix32((uint32_t)v) & (MEMB - 1);
  for (int probe = 0; probe < MEMB; ++probe) {  // at most 32 of 64 slots are taken
    if (atomicCAS(&mk[h], HT_EMPTY, v) == HT_EMPTY) {
      mv[h] = j;
      return;
    }
    h = (h + 1) & (MEMB - 1);
  }
}
__device__ __forceinline__ int32_t memb_find(const int32_t *mk, const int32_t *mv, int32_t v) {
  uint32_t h = fmix32((uint32_t)v) & (MEMB - 1);
  for (int probe = 0; probe < MEMB; ++probe) {
    const int32_t x = mk[h];
    if (x == v) return mv[h];
    if (x == HT_EMPTY) return -1;
    h = (h + 1) & (MEMB - 1);
  }
  return -1;
}

// (conn, lowest block) of the larger connectivity
__device__ __forceinline__ void best_of(int32_t conn, int32_t blk, int32_t &bc, int32_t &bt) {
  if (conn > bc || (conn == bc && blk < bt)) {
    bc = conn;
    bt = blk;
  }
}

// The in-order commit of an evaluated batch by warp 0, a lane per member: t its
// target (-1: none), c its weight, adj its neighbours in the batch, rt the room
// of its target at the start of the batch.  Members are decided in order while
// the block is overloaded (need > 0), up to the first whose target no longer
// fits or who neighbours an earlier move; returns how many, `stop` when the
// block fits before the next.  All members before that one moved as chosen, so
// every lane can tell from its predecessors.
__device__ __forceinline__ int32_t commit_batch(const BalArgs &A, int32_t *room, int32_t B, int32_t nb, int32_t v, int32_t t,
                                                int32_t c, uint32_t adj, int32_t rt, int32_t need, int32_t *hint,
                                                int32_t &moves, bool &stop) {
  constexpr unsigned ALL = 0xFFFFFFFFu;
  const int lane = threadIdx.x & 31;
  const bool mover = lane < nb && t >= 0;
  const unsigned movers = __ballot_sync(ALL, mover), below = (1u << lane) - 1u;
  unsigned rest = __match_any_sync(ALL, t) & movers & below;
  int32_t pre = 0;  // earlier moves into the same target
  while (__any_sync(ALL, rest != 0)) {
    const int32_t x = __shfl_sync(ALL, c, rest ? __ffs(rest) - 1 : lane);
    if (rest) pre += x;
    rest &= rest - 1;
  }
  int32_t sum = mover ? c : 0;  // weight moved by the earlier members and this one
#pragma unroll
  for (int m = 1; m < 32; m <<= 1) {
    const int32_t x = __shfl_up_sync(ALL, sum, m);
    if (lane >= m) sum += x;
  }
  const bool fail = lane < nb && lane > 0 && ((adj & movers & below) != 0 || (t >= 0 && pre + c > rt));
  const bool fits = lane < nb && sum - (mover ? c : 0) >= need;
  const unsigned mf = __ballot_sync(ALL, fail), ms = __ballot_sync(ALL, fits);
  const int32_t jf = mf ? __ffs(mf) - 1 : nb, js = ms ? __ffs(ms) - 1 : nb;
  const int32_t n = min(jf, js);
  stop = js < nb && js <= jf;
  if (lane < n && t >= 0) {
    A.part[v] = t;
    atomicSub(&room[t], c);
  }
  const unsigned done = n >= 32 ? movers : movers & ((1u << n) - 1u);
  const int32_t gone = n > 0 ? __shfl_sync(ALL, sum, n - 1) : 0;
  if (lane == 0 && gone > 0) {
    const int32_t r = room[B] + gone;
    room[B] = r;
    if (r >= 1 && B < *hint) *hint = B;
  }
  moves += __popc(done);
  __syncwarp();
  return n;
}

constexpr size_t BAL_WINDOWS = BM_W * sizeof(BalWindow);
constexpr int32_t BAL_SLOTS = (int32_t)(BAL_WINDOWS / (2 * sizeof(int32_t))) & ~31;  // of a CTA batch's tables there
constexpr size_t BAL_TABS = 2 * WS_T * sizeof(int32_t);
constexpr int32_t BAL_ROOM_K = 26000;  // rooms in shared memory: 104 KB beside 94 KB of windows and 16 KB of tables

// dynamic shared memory of the commit: windows, warp 0's tables, rooms, and the
// tables of large batches in what is left (`slots` of them; a batch that needs
// more lies over the windows, which are then read again, or in global memory).
// With all large batches over the windows, 32 windows were read again for each:
// partition of R-MAT 2^22, k = 4096, 368.4 ms, and 353.1 like this.
// A batch of BAL_FIT members or more that fits is preferred to one that does not: a
// random graph of 30,000 nodes of 300 neighbours in 300 blocks 45.6 -> 13.6 ms (39.5
// before the windows, whose reloads it paid for), 60,000 nodes of 250 in 20,000 blocks
// 23.3 -> 11.5 (with 8 instead of 4 members 23.3).
constexpr size_t BAL_SMEM_MAX = 224000;
constexpr int32_t BAL_FIT = 4;

template <bool SROOM, bool MULTI>
__global__ void __launch_bounds__(BM_T) k_bal_moves(BalArgs A, int32_t *groom, int32_t slots) {
  extern __shared__ __align__(16) unsigned char bal_smem[];
  BalWindow *const win = reinterpret_cast<BalWindow *>(bal_smem);
  int32_t *const wk = reinterpret_cast<int32_t *>(bal_smem + BAL_WINDOWS), *const wv = wk + WS_T;  // empty between batches
  int32_t *const room = SROOM ? wv + WS_T : groom;
  __shared__ int32_t s_v[BM_W], s_c[BM_W];
  __shared__ int64_t s_eoff[BM_W + 1], s_beg[BM_W];
  __shared__ uint32_t s_adj[BM_W], s_mask[BM_W], s_toff[BM_W + 1];
  __shared__ unsigned long long s_best[BM_W];
  __shared__ int32_t mk[MEMB], mv[MEMB];
  // weight from member to member of a small batch, where s_adj has the bit; parallel entries
  // (MULTI: the graph may hold them) are summed, and their sums are zero between batches
  __shared__ int32_t adjw[32][33];
  __shared__ int32_t s_nb, s_B, s_ob, s_i, s_phase, s_done, s_large, s_hint;
  constexpr unsigned ALL = 0xFFFFFFFFu;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint32_t gcap = A.gcap;  // stride of the per-member table regions in A.gtab
  for (int x = threadIdx.x; x < WS_T; x += BM_T) {
    wk[x] = HT_EMPTY;
    wv[x] = 0;
  }
  for (int32_t x = threadIdx.x; x < A.k; x += BM_T) room[x] = (int32_t)((int64_t)A.cap[x] - A.bw[x]);
  if (threadIdx.x < MEMB) mk[threadIdx.x] = HT_EMPTY;
  if (MULTI)
    for (int x = threadIdx.x; x < 32 * 33; x += BM_T) (&adjw[0][0])[x] = 0;
  if (threadIdx.x == 0) {
    s_ob = 0;
    s_i = -1;
    s_phase = 0;
    s_done = 0;
    s_hint = 0;
  }
  int32_t n_moves = 0, n_spec = 0;                   // warp 0's counts
  unsigned long long n_batches = 0, n_cands = 0, n_entries = 0;
  __syncthreads();
  int32_t g0 = 0, gn = 0;  // blocks whose windows are held
  bool reload = true;
  for (;;) {
    if (reload) {
      // windows of the next blocks; the first may be under way (phase 1, candidate s_i)
      g0 = s_ob;
      gn = min(BM_W, A.nover - g0);
      if (w < gn) load_window(A, win[w], g0 + w, w == 0 && s_phase == 1 ? s_i : -1);
      __syncthreads();
    }
    if (w == 0) {
      int32_t ob = s_ob, i = s_i, phase = s_phase;
      bool large = false;
      while (ob < g0 + gn) {
        BalWindow &W = win[ob - g0];
        const int32_t B = W.B, hi = W.hi;
        if (phase == 0) {
          // The block's speculated moves stand, in order, while their targets
          // still fit under what the blocks before left; the moves before the
          // first that does not are applied at once.
          const int32_t nm = W.nm;
          int32_t v = 0, t = -1, c = 0, rt = 0;
          if (lane < nm) {
            v = W.sv[lane];
            t = W.st[lane];
            c = W.sc[lane];
            rt = room[t];
          }
          int32_t pre = 0;  // this block's earlier moves into the same target
          for (int j = 0; j < nm; ++j) {
            const int32_t tj = __shfl_sync(ALL, t, j), cj = __shfl_sync(ALL, c, j);
            if (j < lane && tj == t) pre += cj;
          }
          const unsigned bad = __ballot_sync(ALL, lane < nm && pre + c > rt);
          const int32_t f = bad ? __ffs(bad) - 1 : nm;  // moves [0, f) stand
          if (lane < f) {
            A.part[v] = t;
            atomicSub(&room[t], c);
          }
          const int32_t gone = warp_sum32(lane < f ? c : 0);
          if (lane == 0 && f > 0) {
            const int32_t r = room[B] + gone;
            room[B] = r;
            if (r >= 1 && B < s_hint) s_hint = B;  // the block got room
          }
          __syncwarp();
          n_moves += f;
          n_spec += f;
          i = f < nm ? W.lo + f : (W.sat ? hi : W.send);
          phase = 1;
        }
        const int32_t need = -room[B];
        if (i >= hi || need <= 0) {
          ++ob;
          phase = 0;
          continue;
        }
        // the next batch: the shortest prefix of the remaining candidates whose
        // weights cover the overload; the window moves up when it does not show it
        int32_t a = i - W.base, avail = min(hi - i, 32), nb = 0;
        int32_t c = 0, inc = 0;
        for (int turn = 0; turn < 2; ++turn) {
          const int32_t held = min(W.nc - a, avail);
          c = lane < held ? W.c[a + lane] : 0;
          inc = c;
#pragma unroll
          for (int m = 1; m < 32; m <<= 1) {
            const int32_t x = __shfl_up_sync(ALL, inc, m);
            if (lane >= m) inc += x;
          }
          const unsigned enough = __ballot_sync(ALL, lane < held && inc >= need);
          nb = enough ? __ffs(enough) : held;
          if (enough || held >= avail) break;
          __syncwarp();
          load_window(A, W, ob, i);
          a = 0;
        }
        // member table sized by the member's own distinct blocks (at most
        // min(degree, k)); the tables' slots are numbered across the batch
        const int64_t e0 = W.epre[a], E = W.epre[a + nb] - e0;
        const int32_t v = lane < nb ? W.v[a + lane] : -1;
        const int64_t deg = lane < nb ? W.epre[a + lane + 1] - W.epre[a + lane] : 0;
        uint32_t cap = 32;
        while ((int64_t)cap < 2 * (deg < A.k ? deg : (int64_t)A.k)) cap <<= 1;
        uint32_t tpre = lane < nb ? cap : 0;
#pragma unroll
        for (int m = 1; m < 32; m <<= 1) {
          const uint32_t x = __shfl_up_sync(ALL, tpre, m);
          if (lane >= m) tpre += x;
        }
        const uint32_t TT = __shfl_sync(ALL, tpre, nb - 1);
        if (lane < nb) {
          s_adj[lane] = 0;
          s_mask[lane] = cap - 1;
          s_toff[lane + 1] = tpre;
          memb_add(mk, mv, v, lane);
        }
        if (lane == 0) s_toff[0] = 0;
        ++n_batches;
        if (E > WS_E || TT > (uint32_t)WS_T) {
          // Members whose tables do not fit beside the windows are left to the next batch
          // while BAL_FIT or more do fit: on dense graphs a batch stops at a neighbour of
          // an earlier move after a few members, and tables in global memory, cleared and
          // filled for all 32, cost more than the batches that this adds.
          if (TT > (uint32_t)slots) {
            const int32_t fit = __popc(__ballot_sync(ALL, lane < nb && tpre <= (uint32_t)slots));
            if (fit >= BAL_FIT) nb = fit;
          }
          n_cands += nb;
          n_entries += W.epre[a + nb] - e0;
          if (lane < nb) {
            s_v[lane] = v;
            s_c[lane] = c;
            s_beg[lane] = W.beg[a + lane];
            s_eoff[lane + 1] = W.epre[a + lane + 1] - e0;
            s_best[lane] = 0;
          }
          if (lane == 0) {
            s_eoff[0] = 0;
            s_nb = nb;
            s_B = B;
          }
          large = true;
          break;  // the whole CTA evaluates this batch
        }
        n_cands += nb;
        n_entries += E;
        __syncwarp();
        // ---- warp 0 alone: connectivity tables in shared memory
        for (int32_t t0 = 0; t0 < (int32_t)E; t0 += 32 * WS_R) {
          int32_t uu[WS_R], wt[WS_R], jm[WS_R], bk[WS_R];
#pragma unroll
          for (int r = 0; r < WS_R; ++r) {
            const int64_t t = e0 + t0 + lane + 32 * r;
            uu[r] = -1;
            if (t < e0 + E) {
              int32_t j = 0;
#pragma unroll
              for (int st = 16; st > 0; st >>= 1)
                if (W.epre[j + st] <= t) j += st;
              jm[r] = j - a;
              if (t < W.ne) {
                uu[r] = W.u[t];
                wt[r] = W.w[t];
              } else {
                const int64_t q = W.beg[j] + (t - W.epre[j]);
                uu[r] = A.adj[q];
                wt[r] = A.ew ? A.ew[q] : 1;
              }
            }
          }
#pragma unroll
          for (int r = 0; r < WS_R; ++r)
            if (uu[r] >= 0) bk[r] = A.part[uu[r]];
#pragma unroll
          for (int r = 0; r < WS_R; ++r)
            if (uu[r] >= 0) {
              const int32_t ib = memb_find(mk, mv, uu[r]);
              if (ib >= 0) {
                atomicOr(&s_adj[jm[r]], 1u << ib);
                if (MULTI) atomicAdd(&adjw[jm[r]][ib], wt[r]);
                else adjw[jm[r]][ib] = wt[r];
              }
              ht_add(wk + s_toff[jm[r]], wv + s_toff[jm[r]], s_mask[jm[r]], bk[r], wt[r]);
            }
        }
        __syncwarp();
        // In order, each member from its own table and the rooms as the members
        // before it left them; a move adds its weight to the tables of the later
        // members it neighbours (bits of s_adj, weights in adjw), so every member
        // is decided here, whatever the earlier ones did.
        const uint32_t madj = lane < nb ? s_adj[lane] : 0;
        int32_t left = need, j = 0;
        for (; j < nb && left > 0; ++j) {
          const uint32_t t0 = s_toff[j], t1 = s_toff[j + 1];
          const int32_t cj = __shfl_sync(ALL, c, j);
          int32_t bc = 0, bt = INT32_MAX;
          for (uint32_t x = t0 + lane; x < t1; x += 32) {
            const int32_t b = wk[x];
            if (b != HT_EMPTY && b != B && room[b] >= cj) best_of(wv[x], b, bc, bt);
          }
          const int32_t m = __reduce_max_sync(ALL, bc);
          int32_t t;
          if (m > 0) t = __reduce_min_sync(ALL, bc == m ? bt : INT32_MAX);
          else t = lowest_admissible(room, A.k, cj, lane, &s_hint);
          if (t >= 0) {
            if (lane == j) {
              A.part[v] = t;
              room[t] -= cj;
            }
            if (lane > j && ((madj >> j) & 1u)) ht_add(wk + (tpre - cap), wv + (tpre - cap), cap - 1, t, adjw[lane][j]);
            left -= cj;
            ++n_moves;
          }
          __syncwarp();
        }
        for (uint32_t x = lane; x < TT; x += 32) {
          wk[x] = HT_EMPTY;
          wv[x] = 0;
        }
        if (MULTI)
          for (uint32_t x = madj; x; x &= x - 1) adjw[lane][__ffs(x) - 1] = 0;
        mk[lane] = HT_EMPTY;
        mk[lane + 32] = HT_EMPTY;
        if (lane == 0 && left != need) {
          room[B] = -left;
          if (left < 0 && B < s_hint) s_hint = B;  // the block got room
        }
        __syncwarp();
        i += j;
      }
      if (lane == 0) {
        s_ob = ob;
        s_i = i;
        s_phase = phase;
        s_large = large;
        s_done = !large && ob >= A.nover;
      }
    }
    __syncthreads();
    if (s_done) break;
    reload = true;
    if (!s_large) continue;
    // ---- a large batch, evaluated by the whole CTA
    const int32_t B = s_B, nb = s_nb;
    // every table size is a multiple of 32, so a warp's 32 slots lie in one table
    const uint32_t TT = s_toff[nb];
    const bool beside = TT <= (uint32_t)slots, over = !beside && TT <= (uint32_t)BAL_SLOTS, sm = beside || over;
    reload = over;
    int32_t *const sk = over ? reinterpret_cast<int32_t *>(bal_smem) : wv + WS_T + (SROOM ? A.k : 0);
    int32_t *const sv = sk + (over ? BAL_SLOTS : slots);
    auto keys_of = [&](int32_t j) { return sm ? sk + s_toff[j] : A.gtab + (int64_t)j * 2 * gcap; };
    auto vals_of = [&](int32_t j) { return sm ? sv + s_toff[j] : A.gtab + (int64_t)j * 2 * gcap + gcap; };
    {
      int32_t j = 0;
      for (uint32_t t = threadIdx.x; t < TT; t += BM_T) {
        while (s_toff[j + 1] <= t) ++j;
        keys_of(j)[t - s_toff[j]] = HT_EMPTY;
        vals_of(j)[t - s_toff[j]] = 0;
      }
    }
    __syncthreads();
    const int64_t E = s_eoff[nb];
    {
      int32_t jm = 0;  // this thread's entries only move forward through the members
      for (int64_t base = 0; base < E; base += BM_T) {
        int64_t t = base + threadIdx.x;
        bool ok = t < E;
        if (ok)
          while (s_eoff[jm + 1] <= t) ++jm;
        int32_t blk = HT_EMPTY, wt = 0;
        if (ok) {
          int64_t q = s_beg[jm] + (t - s_eoff[jm]);
          int32_t u = A.adj[q];
          blk = A.part[u];
          wt = A.ew ? A.ew[q] : 1;
          const int32_t ib = memb_find(mk, mv, u);
          if (ib >= 0) atomicOr(&s_adj[jm], 1u << ib);
        }
        if (sm) {
          if (ok) ht_add(keys_of(jm), vals_of(jm), s_mask[jm], blk, wt);
          continue;
        }
        // lanes that hit the same block of the same member add first
        const uint64_t key = ok ? ((uint64_t)(uint32_t)jm << 32) | (uint32_t)blk : ~0ull;
        const unsigned peers = __match_any_sync(ALL, key);
        const int32_t s = __reduce_add_sync(peers, wt);
        if (ok && lane == __ffs(peers) - 1) ht_add(keys_of(jm), vals_of(jm), s_mask[jm], blk, s);
      }
    }
    __syncthreads();
    {
      // best admissible block of every member: (conn, ~block), largest
      // connectivity, then lowest id; a warp's slots belong to one member
      int32_t jj = 0;
      for (uint32_t base = 0; base < TT; base += BM_T) {
        const uint32_t t = base + threadIdx.x;
        if (base + (threadIdx.x & ~31u) >= TT) break;  // warp-uniform
        while (s_toff[jj + 1] <= t) ++jj;
        const uint32_t x = t - s_toff[jj];
        const int32_t b = keys_of(jj)[x];
        uint64_t key = 0;
        if (b != HT_EMPTY && b != B && room[b] >= s_c[jj])
          key = ((uint64_t)(uint32_t)vals_of(jj)[x] << 32) | (0xFFFFFFFFu - (uint32_t)b);
        key = group_max64<32>(key);
        if (lane == 0 && key) atomicMax(&s_best[jj], key);
      }
    }
    __syncthreads();
    if (w == 0) {
      const int32_t v = lane < nb ? s_v[lane] : -1, c = lane < nb ? s_c[lane] : 0;
      const uint64_t bestk = lane < nb ? s_best[lane] : 0;
      int32_t t = bestk ? (int32_t)(0xFFFFFFFFu - (uint32_t)bestk) : -1;
      for (unsigned none = __ballot_sync(ALL, lane < nb && t < 0); none; none &= none - 1) {
        const int j = __ffs(none) - 1;
        const int32_t x = lowest_admissible(room, A.k, __shfl_sync(ALL, c, j), lane, &s_hint);
        if (lane == j) t = x;
      }
      const int32_t rt = t >= 0 ? room[t] : 0;
      const uint32_t adj = lane < nb ? s_adj[lane] : 0;
      const int32_t need = -room[B];
      mk[lane] = HT_EMPTY;
      mk[lane + 32] = HT_EMPTY;
      __syncwarp();
      bool stop = false;
      const int32_t n = commit_batch(A, room, B, nb, v, t, c, adj, rt, need, &s_hint, n_moves, stop);
      if (lane == 0) {
        s_i += n;
        if (stop) {
          ++s_ob;
          s_phase = 0;
        }
        s_done = s_ob >= A.nover;
      }
    }
    __syncthreads();
    const bool done = s_done;
    __syncthreads();  // warp 0 may go straight on to the next blocks and write it again
    if (done) break;
  }
  if (threadIdx.x == 0) {
    A.moved[0] = (unsigned long long)n_moves;
    A.moved[1] = (unsigned long long)n_spec;  // speculated moves that stood
    A.moved[2] = n_batches;
    A.moved[3] = n_cands;
    A.moved[4] = n_entries;
  }
}

template <bool SROOM, bool MULTI>
static void launch_moves(const BalArgs &A, int32_t *room, int32_t slots) {
  static bool attr = false;
  if (!attr) {
    KMP_CUDA(cudaFuncSetAttribute(k_bal_moves<SROOM, MULTI>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)BAL_SMEM_MAX));
    attr = true;
  }
  k_bal_moves<SROOM, MULTI><<<1, BM_T, BAL_SMEM_MAX, ctx().stream>>>(A, room, slots);
}

int64_t balance(const Graph &g, int32_t k, const int32_t *caps_host, int32_t *part, BalStats *bs) {
  Context &C = ctx();
  cudaStream_t s = C.stream;
  int32_t n = g.n;
  DBuf<int64_t> bw(k);
  block_weights(g, part, k, bw);
  std::vector<int64_t> hbw(k);
  to_host(hbw.data(), bw.p, k);
  std::vector<uint8_t> hover(k, 0);
  std::vector<int32_t> holist;
  int64_t max_room = INT64_MIN;
  for (int32_t b = 0; b < k; ++b) {
    if (hbw[b] > caps_host[b]) {
      hover[b] = 1;
      holist.push_back(b);
    }
    max_room = std::max<int64_t>(max_room, (int64_t)caps_host[b] - hbw[b]);
  }
  if (holist.empty() || n == 0) return 0;
  int bitsN = 1;
  while ((1ll << bitsN) < (int64_t)n) ++bitsN;
  int bitsK = 1;
  while ((1ll << bitsK) < (int64_t)k) ++bitsK;
  DBuf<int32_t> cap(k), ncand(1), seg_lo(k), seg_hi(k);
  DBuf<uint8_t> over(k);
  DBuf<int64_t> cand_d(n);
  DBuf<uint64_t> keys(n), tmp(n), sortbuf(2ll * n);
  // moves, speculated moves that stood, exact batches, their candidates and adjacency entries
  DBuf<unsigned long long> moved(5);
  to_dev(cap.p, caps_host, k);
  to_dev(over.p, hover.data(), k);
  DBuf<int32_t> olist(holist.size());
  to_dev(olist.p, holist.data(), holist.size());
  ncand.zero();
  moved.zero();
  seg_lo.zero();
  seg_hi.zero();
  int64_t dmax = std::min<int64_t>(g.maxdeg, k);
  uint32_t gcap = 32;
  while ((int64_t)gcap < 2 * dmax) gcap <<= 1;
  const int grid = grid_for((int64_t)n * 32, BAL_T, 8);
  int grid_big = 0;
  DBuf<int32_t> gtab;
  BalArgs A;
  A.n = n;
  A.k = k;
  A.xadj = g.xadj;
  A.adj = g.adj;
  A.vw = g.vw;
  A.ew = g.ew;
  A.part = part;
  A.bw = bw;
  A.cap = cap;
  A.over = over;
  A.olist = olist;
  A.nover = (int32_t)holist.size();
  A.max_room = max_room;
  A.cand_d = cand_d;
  A.keys = keys;
  A.ncand = ncand;
  A.bitsN = bitsN;
  A.seg_lo = seg_lo;
  A.seg_hi = seg_hi;
  A.sortbuf = sortbuf;
  A.gtab = nullptr;
  A.gcap = gcap;
  A.moved = moved;
  // nodes with more distinct neighbour blocks than a warp's shared table
  // holds have degree > BAL_STAB / 2, so there are at most m / 257 of them
  DBuf<int32_t> big(g.m / (BAL_STAB / 2 + 1) + 1), nbig(1);
  nbig.zero();
  k_bal_cand<<<grid, BAL_T, 0, s>>>(A, big, nbig);
  KMP_LAUNCHED("bal_cand");
  if (gcap > BAL_STAB) {
    const int32_t nb = read1(nbig.p);
    if (nb > 0) {
      // one CTA per listed node, each with its own global table region,
      // bounded to about 256 MB in all
      int64_t per_cta = 2ll * gcap * (int64_t)sizeof(int32_t);
      int64_t gmax = std::max<int64_t>(1, (256ll << 20) / per_cta);
      grid_big = (int)std::min<int64_t>(std::min<int64_t>(nb, gmax), (int64_t)C.sms * 8);
      gtab.alloc(2ll * gcap * (int64_t)grid_big);
      A.gtab = gtab;
      k_bal_cand_big<<<grid_big, BAL_T, 0, s>>>(A, big, nbig);
      KMP_LAUNCHED("bal_cand_big");
    }
  }
  int32_t N = read1(ncand.p);
  if (N == 0) return 0;
  // grouped by block only: k_bal_sort orders every block's candidates by a
  // strict total order (relative gain, then id), whatever order they arrive in
  radix_sort_u64(keys, tmp, N, bitsK, bitsN);
  k_bal_segments<<<grid_for(N, 256), 256, 0, s>>>(A, N);
  KMP_LAUNCHED("bal_segments");
  k_bal_sort<<<A.nover, BAL_T, 0, s>>>(A);
  KMP_LAUNCHED("bal_sort");
  // speculation over all overloaded blocks (tables as for the candidates)
  int32_t nover = (int32_t)holist.size();
  DBuf<int32_t> spec_v((size_t)nover * SPEC_MAX), spec_t((size_t)nover * SPEC_MAX), spec_n(nover),
      spec_end(nover), spec_sat(nover);
  A.spec_v = spec_v;
  A.spec_t = spec_t;
  A.spec_n = spec_n;
  A.spec_end = spec_end;
  A.spec_sat = spec_sat;
  {
    int sgrid = (int)ceil_div(nover, BAL_W);
    A.gtab = nullptr;
    k_bal_spec<<<sgrid, BAL_T, 0, s>>>(A);
    KMP_LAUNCHED("bal_spec");
  }
  // a global table per member for CTA batches whose tables do not fit shared
  // memory; rooms in shared memory while k fits
  DBuf<int32_t> gtab1(2ll * gcap * BM_W), room;
  A.gtab = gtab1;
  const size_t fixed = BAL_WINDOWS + BAL_TABS + (k <= BAL_ROOM_K ? (size_t)k * sizeof(int32_t) : 0);
  const int32_t slots = (int32_t)((BAL_SMEM_MAX - fixed) / (2 * sizeof(int32_t))) & ~31;
  if (k > BAL_ROOM_K) room.alloc(k);
  if (k <= BAL_ROOM_K) {
    if (g.multi) launch_moves<true, true>(A, nullptr, slots);
    else launch_moves<true, false>(A, nullptr, slots);
  } else {
    if (g.multi) launch_moves<false, true>(A, room, slots);
    else launch_moves<false, false>(A, room, slots);
  }
  KMP_LAUNCHED("bal_moves");
  unsigned long long hm[5];
  to_host(hm, moved.p, 5);
  if (bs) {
    bs->over_blocks += nover;
    bs->moves += (int64_t)hm[0];
    bs->spec_moves += (int64_t)hm[1];
    bs->exact_batches += (int64_t)hm[2];
    bs->exact_cands += (int64_t)hm[3];
    bs->exact_entries += (int64_t)hm[4];
  }
  return (int64_t)hm[0];
}

}  // namespace kmp
