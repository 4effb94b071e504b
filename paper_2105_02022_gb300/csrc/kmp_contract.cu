// Contraction (Section 2, "Multilevel Graph Partitioning"): each cluster
// becomes one coarse node whose weight is the sum of its members' weights;
// the coarse edge between two clusters carries the summed weight of the fine
// edges between them; edges inside a cluster vanish.
//
// GPU layout: coarse ids = exclusive scan of "label used" flags (ascending
// label); members grouped by a counting sort.  A coarse node whose members'
// total degree is <= 512 is aggregated by one warp in a shared-memory hash
// table (four bins by size: 64, 128, 256, 512), one whose total degree is
// <= 8192 by one CTA in a table sized for it (three bins: 2048, 4096, 8192);
// larger rows are aggregated by all their members' warps in parallel into
// global tables.  A row is put in order by the cheapest way that its ids allow:
// the rank in a bitmap of its id span; buckets of equal id ranges; a bitonic
// network where ids crowd into few buckets (and for the shortest rows).  The
// longest rows go through one counting sort by (row, high neighbour bits) and a
// bitmap per segment.  Rows go to temporary space at upper-bound offsets; a
// prefix sum of the row lengths then places them into the final CSR.
// R-MAT 2^24 with its level-0 clusters, whole contraction: 74.0 ms with networks
// for all rows whose ids span far (66 steps an entry at 2048 entries), 33.3 now.
// Also: projection (Algorithm 1), cut and block weights (Section 2), and the
// per-graph facts the other kernels need (max degree, isolated nodes, weights).
#include <climits>
#include <cstring>

#include "kmp_internal.cuh"
#include "kmp_plan.h"

namespace kmp {

constexpr int CW_UB = 512;            // warp path: members' total degree <= CW_UB
constexpr int CB_UB = 8192;           // block path: members' total degree <= CB_UB
constexpr int NCLASS = 8;             // four warp bins, three block bins, global path
constexpr int CLS_GLOBAL = NCLASS - 1;

// row class by members' total degree ub: warp bins 64 / 128 / 256 / 512, block
// bins 2048 / 4096 / 8192, then the global path
__host__ __device__ __forceinline__ int row_class(unsigned long long ub) {
  return ub <= 64ull    ? 0
         : ub <= 128ull  ? 1
         : ub <= 256ull  ? 2
         : ub <= (unsigned long long)CW_UB ? 3
         : ub <= 2048ull ? 4
         : ub <= 4096ull ? 5
         : ub <= 8192ull ? 6
                         : CLS_GLOBAL;
}

// labels outside [0, n) set *bad and mark nothing
__global__ void k_map_used(int32_t n, const int32_t *label, uint8_t *used, int32_t *bad) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x) {
    const int32_t l = label[v];
    if (l < 0 || l >= n) *bad = 1;
    else used[l] = 1;
  }
}

__global__ void k_map(int32_t n, const int32_t *label, const int32_t *cid, int32_t *map) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x)
    map[v] = cid[label[v]];
}

__global__ void k_contract_prep(int32_t n, const int64_t *xadj, const int32_t *vw,
                                const int32_t *map, int32_t *cvw, int32_t *csize,
                                unsigned long long *cub) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x) {
    int32_t x = map[v];
    atomicAdd(&cvw[x], vw ? vw[v] : 1);
    atomicAdd(&csize[x], 1);
    atomicAdd(&cub[x], (unsigned long long)(xadj[v + 1] - xadj[v]));
  }
}

__global__ void k_members(int32_t n, const int32_t *map, const int32_t *moff, int32_t *mcur,
                          int32_t *members) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x) {
    int32_t x = map[v];
    members[moff[x] + atomicAdd(&mcur[x], 1)] = (int32_t)v;
  }
}

// Split coarse nodes by row class: list c holds its rows at lists + c * nc (in any
// order).  A CTA counts a tile's classes in shared memory and claims each class's
// places with one atomic: one atomic a row on eight counters made this the
// longest kernel of a mesh level (1.2 M rows: 117 us, 12 now).
constexpr int SPLIT_PER = 8;
__global__ void __launch_bounds__(256) k_split_ub(int32_t nc, const unsigned long long *cub, int32_t *lists,
                                                  int32_t *counts) {
  __shared__ int32_t cnt[NCLASS], base[NCLASS];
  const int lane = threadIdx.x & 31;
  for (int64_t t0 = (int64_t)blockIdx.x * 256 * SPLIT_PER; t0 < nc; t0 += (int64_t)gridDim.x * 256 * SPLIT_PER) {
    if (threadIdx.x < NCLASS) cnt[threadIdx.x] = 0;
    __syncthreads();
    int32_t cls[SPLIT_PER], rank[SPLIT_PER];
#pragma unroll
    for (int r = 0; r < SPLIT_PER; ++r) {
      const int64_t x = t0 + r * 256 + threadIdx.x;
      cls[r] = x < nc ? row_class(cub[x]) : -1;
    }
#pragma unroll
    for (int r = 0; r < SPLIT_PER; ++r) {
      rank[r] = 0;
#pragma unroll
      for (int c = 0; c < NCLASS; ++c) {
        const unsigned m = __ballot_sync(0xFFFFFFFFu, cls[r] == c);
        if (m == 0) continue;
        int32_t at = 0;
        if (lane == 0) at = atomicAdd(&cnt[c], __popc(m));
        at = __shfl_sync(0xFFFFFFFFu, at, 0);
        if (cls[r] == c) rank[r] = at + __popc(m & ((1u << lane) - 1u));
      }
    }
    __syncthreads();
    if (threadIdx.x < NCLASS && cnt[threadIdx.x] > 0)
      base[threadIdx.x] = atomicAdd(&counts[threadIdx.x], cnt[threadIdx.x]);
    __syncthreads();
#pragma unroll
    for (int r = 0; r < SPLIT_PER; ++r)
      if (cls[r] >= 0)
        lists[(int64_t)cls[r] * nc + base[cls[r]] + rank[r]] = (int32_t)(t0 + r * 256 + threadIdx.x);
    __syncthreads();
  }
}

__global__ void k_ub_to_i64(int32_t nc, const unsigned long long *cub, int64_t *ub64) {
  for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < nc;
       x += (int64_t)gridDim.x * blockDim.x)
    ub64[x] = (int64_t)cub[x];
}

// bitonic sort (ascending) of P = power-of-two entries by `nt` cooperating
// threads with index t; sync() separates the steps
template <bool BLOCK>
__device__ __forceinline__ void bitonic(uint64_t *a, uint32_t P, uint32_t t, uint32_t nt) {
  for (uint32_t k = 2; k <= P; k <<= 1) {
    for (uint32_t j = k >> 1; j > 0; j >>= 1) {
      for (uint32_t i = t; i < P; i += nt) {
        uint32_t l = i ^ j;
        if (l > i) {
          uint64_t x = a[i], y = a[l];
          bool up = (i & k) == 0;
          if ((x > y) == up) {
            a[i] = y;
            a[l] = x;
          }
        }
      }
      if (BLOCK) __syncthreads();
      else __syncwarp();
    }
  }
}

// Order of `cnt` entries (neighbour << 32 | weight, neighbours distinct) by
// neighbour through buckets of equal id ranges, about one entry each: L is
// counted by bucket (H: nb + 1 counters), scattered to M in bucket order, and an
// entry's place is its bucket's start plus the smaller entries of its bucket.
// That is a few shared-memory steps an entry, where a bitonic network of 2^p
// takes p (p + 1) / 2.  Ids that crowd into a bucket would make the last step
// quadratic: false (nothing but H and M touched) when one holds more than
// BUCKET_MAX, and the caller sorts by the network.  All threads of the group
// (a warp, or a CTA with s_wsum / s_max) call it; out(place, entry) writes.
constexpr int32_t BUCKET_MAX = 32;
template <int NT>
__device__ __forceinline__ int32_t block_scan_excl(int32_t v, int32_t *s_wsum /* NT / 32 */);
__device__ __forceinline__ int bucket_shift(int32_t ymin, int32_t ymax, int32_t nb) {
  const int sh = (32 - __clz((ymax - ymin) | 1)) - (31 - __clz(nb));
  return sh > 0 ? sh : 0;
}
template <class F>
__device__ __forceinline__ bool bucket_order_warp(const uint64_t *L, int32_t cnt, int32_t ymin, int32_t ymax, int32_t nb,
                                                  int32_t *H, uint64_t *M, F out) {
  const int lane = threadIdx.x & 31;
  const int sh = bucket_shift(ymin, ymax, nb);
  for (int32_t j = lane; j < nb; j += 32) H[j] = 0;
  __syncwarp();
  for (int32_t j = lane; j < cnt; j += 32) atomicAdd(&H[((int32_t)(L[j] >> 32) - ymin) >> sh], 1);
  __syncwarp();
  int32_t run = 0, top = 0;
  for (int32_t j0 = 0; j0 < nb; j0 += 32) {
    const int32_t h = j0 + lane < nb ? H[j0 + lane] : 0;
    top = max(top, h);
    int32_t inc = h;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t t = __shfl_up_sync(0xFFFFFFFFu, inc, o);
      if (lane >= o) inc += t;
    }
    if (j0 + lane < nb) H[j0 + lane] = run + inc - h;
    run += __shfl_sync(0xFFFFFFFFu, inc, 31);
  }
  if (__reduce_max_sync(0xFFFFFFFFu, top) > BUCKET_MAX) return false;
  __syncwarp();
  for (int32_t j = lane; j < cnt; j += 32) {
    const uint64_t e = L[j];
    M[atomicAdd(&H[((int32_t)(e >> 32) - ymin) >> sh], 1)] = e;
  }
  __syncwarp();  // H[b] is the end of bucket b now
  for (int32_t j = lane; j < cnt; j += 32) {
    const uint64_t e = M[j];
    const int32_t b = ((int32_t)(e >> 32) - ymin) >> sh, lo = b > 0 ? H[b - 1] : 0, hi = H[b];
    int32_t r = lo;
    for (int32_t q = lo; q < hi; ++q) r += M[q] < e;
    out(r, e);
  }
  return true;
}
template <int NT, class F>
__device__ __forceinline__ bool bucket_order_cta(const uint64_t *L, int32_t cnt, int32_t ymin, int32_t ymax, int32_t nb,
                                                 int32_t *H, uint64_t *M, int32_t *s_wsum, int32_t *s_max, F out) {
  const int tid = threadIdx.x;
  const int sh = bucket_shift(ymin, ymax, nb);
  for (int32_t j = tid; j < nb; j += NT) H[j] = 0;
  if (tid == 0) *s_max = 0;
  __syncthreads();
  for (int32_t j = tid; j < cnt; j += NT) atomicAdd(&H[((int32_t)(L[j] >> 32) - ymin) >> sh], 1);
  __syncthreads();
  const int32_t seg = (nb + NT - 1) / NT, a = min(tid * seg, nb), b = min(a + seg, nb);
  int32_t loc = 0, top = 0;
  for (int32_t j = a; j < b; ++j) {
    loc += H[j];
    top = max(top, H[j]);
  }
  if (top > BUCKET_MAX) *s_max = 1;
  int32_t base = block_scan_excl<NT>(loc, s_wsum);
  for (int32_t j = a; j < b; ++j) {
    const int32_t h = H[j];
    H[j] = base;
    base += h;
  }
  __syncthreads();
  if (*s_max) return false;
  for (int32_t j = tid; j < cnt; j += NT) {
    const uint64_t e = L[j];
    M[atomicAdd(&H[((int32_t)(e >> 32) - ymin) >> sh], 1)] = e;
  }
  __syncthreads();
  for (int32_t j = tid; j < cnt; j += NT) {
    const uint64_t e = M[j];
    const int32_t k = ((int32_t)(e >> 32) - ymin) >> sh, lo = k > 0 ? H[k - 1] : 0, hi = H[k];
    int32_t r = lo;
    for (int32_t q = lo; q < hi; ++q) r += M[q] < e;
    out(r, e);
  }
  return true;
}

// warp path: one coarse node per warp for rows whose members' total degree
// ub is at most TABW / 2.  The table packs (neighbour << 32 | weight) per slot
// (key and weight updated as the two 32-bit halves), is sized to the power of
// two >= 2 ub, and is compacted in place into the sort list, since every entry
// moves to a slot at or below its own.  Up to 32 members at a time spread
// their edges over the lanes (a warp prefix sum of their degrees; each lane
// finds the member of its edge by a five-step search over the prefixes).
template <int TABW, int WARPS>
__global__ void __launch_bounds__(WARPS * 32) k_aggregate_warp(
    const int32_t *list, int32_t nrows, const unsigned long long *cub, const int64_t *xadj,
    const int32_t *adj, const int32_t *ew, const int32_t *map, const int32_t *members,
    const int32_t *moff, const int64_t *toff, int32_t *tadj, int32_t *tw, int32_t *cdeg) {
  __shared__ uint64_t tab[WARPS][TABW];
  __shared__ int32_t hist[TABW >= 256 ? WARPS : 1][TABW >= 256 ? TABW / 2 : 1];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint64_t *T = tab[w];
  int32_t *H = reinterpret_cast<int32_t *>(T);  // H[2 j] weight, H[2 j + 1] key of slot j
  const int64_t gw = (int64_t)blockIdx.x * WARPS + w, nw = (int64_t)gridDim.x * WARPS;
  for (int64_t i = gw; i < nrows; i += nw) {
    const int32_t x = list[i];
    const uint32_t ub = (uint32_t)cub[x];
    uint32_t tsz = 64;
    while (tsz < 2 * ub) tsz <<= 1;
    const uint32_t mask = tsz - 1;
    for (uint32_t j = lane; j < tsz; j += 32) T[j] = (uint64_t)(uint32_t)HT_EMPTY << 32;
    __syncwarp();
    const int32_t m1 = moff[x + 1];
    for (int32_t c0 = moff[x]; c0 < m1; c0 += 32) {
      int32_t d = 0;
      int64_t b = 0;
      if (c0 + lane < m1) {
        int32_t v = members[c0 + lane];
        b = xadj[v];
        d = (int32_t)(xadj[v + 1] - b);
      }
      int32_t inc = d;
      for (int o = 1; o < 32; o <<= 1) {
        int32_t t = __shfl_up_sync(0xFFFFFFFFu, inc, o);
        if (lane >= o) inc += t;
      }
      const int32_t tot = __shfl_sync(0xFFFFFFFFu, inc, 31);
      for (int32_t e0 = 0; e0 < tot; e0 += 32) {
        const int32_t e = e0 + lane;
        int32_t j = 0;  // members before the owner of edge e: their inclusive prefix is <= e
        for (int st = 16; st > 0; st >>= 1) {
          int32_t t = __shfl_sync(0xFFFFFFFFu, inc, j + st - 1);
          if (t <= e) j += st;
        }
        int64_t bj = __shfl_sync(0xFFFFFFFFu, b, j & 31);
        int32_t ej = __shfl_sync(0xFFFFFFFFu, inc - d, j & 31);
        if (e < tot) {
          int64_t q = bj + (e - ej);
          int32_t y = map[adj[q]];
          if (y != x) {
            int32_t wq = ew ? ew[q] : 1;
            uint32_t h = fmix32((uint32_t)y) & mask;
            for (uint32_t probe = 0; probe <= mask; ++probe) {
              int32_t old = atomicCAS(&H[2 * h + 1], HT_EMPTY, y);
              if (old == HT_EMPTY || old == y) {
                atomicAdd(&H[2 * h], wq);
                break;
              }
              h = (h + 1) & mask;
            }
          }
        }
      }
    }
    __syncwarp();
    // in-place compaction: entry j goes to slot cnt + rank <= j
    int32_t cnt = 0;
    for (uint32_t j0 = 0; j0 < tsz; j0 += 32) {
      uint64_t ent = T[j0 + lane];
      bool has = (int32_t)(ent >> 32) != HT_EMPTY;
      unsigned bal = __ballot_sync(0xFFFFFFFFu, has);
      __syncwarp();
      if (has) T[cnt + __popc(bal & ((1u << lane) - 1u))] = ent;
      cnt += __popc(bal);
      __syncwarp();
    }
    uint32_t P = 1;
    while (P < (uint32_t)cnt) P <<= 1;
    const int64_t o = toff[x];
    bool done = false;
    if (TABW >= 256 && P >= 64) {
      // the entries fill at most half of the table: the other half is the scatter space
      int32_t ymin = INT32_MAX, ymax = 0;
      for (int32_t j = lane; j < cnt; j += 32) {
        const int32_t y = (int32_t)(T[j] >> 32);
        ymin = min(ymin, y);
        ymax = max(ymax, y);
      }
      ymin = __reduce_min_sync(0xFFFFFFFFu, ymin);
      ymax = __reduce_max_sync(0xFFFFFFFFu, ymax);
      done = bucket_order_warp(T, cnt, ymin, ymax, (int32_t)P, hist[w], T + TABW / 2, [&](int32_t r, uint64_t e) {
        tadj[o + r] = (int32_t)(e >> 32);
        tw[o + r] = (int32_t)(uint32_t)e;
      });
      __syncwarp();
    }
    if (!done) {
      for (uint32_t j = cnt + lane; j < P; j += 32) T[j] = ~0ull;
      __syncwarp();
      bitonic<false>(T, P, lane, 32);
      for (int32_t j = lane; j < cnt; j += 32) {
        tadj[o + j] = (int32_t)(T[j] >> 32);
        tw[o + j] = (int32_t)(uint32_t)T[j];
      }
    }
    if (lane == 0) cdeg[x] = cnt;
    __syncwarp();
  }
}

template <int TABW, int WARPS>
void launch_aggregate_warp(const int32_t *list, int32_t nrows, const unsigned long long *cub, const Graph &g,
                           const int32_t *map, const int32_t *members, const int32_t *moff,
                           const int64_t *toff, int32_t *tadj, int32_t *tw, int32_t *cdeg) {
  constexpr size_t bytes = (size_t)TABW * WARPS * sizeof(uint64_t) + (TABW >= 256 ? TABW / 2 * WARPS * sizeof(int32_t) : 4);
  static_assert(TABW >= 64 && bytes <= 48 * 1024, "bin shape");
  constexpr int per_sm_smem = (int)((227u << 10) / (bytes + 1024));
  constexpr int per_sm = per_sm_smem < 64 / WARPS ? per_sm_smem : 64 / WARPS;
  k_aggregate_warp<TABW, WARPS><<<grid_for(nrows, WARPS, per_sm), WARPS * 32, 0, ctx().stream>>>(
      list, nrows, cub, g.xadj, g.adj, g.ew, map, members, moff, toff, tadj, tw, cdeg);
  KMP_LAUNCHED("aggregate_warp");
}

// block path: one coarse node per CTA for rows whose members' total degree ub
// is at most TAB / 2.  The row's table is the power of two >= 2 ub (load
// factor <= 1/2); its distinct entries (at most ub) are sorted by neighbour id.
// The members' edges are spread evenly over all NT threads (up to NT members
// at a time: a prefix sum of their degrees, each thread finds the member of
// its edge by binary search), so one high-degree member does not serialise
// the row on one warp.  Ordering: when the row's neighbour ids span at most
// 32 TAB values (and not far more than the entries), each entry's position is
// the number of smaller ids, read from a bitmap of the span and a prefix sum
// of its word popcounts (the freed table is the space); else the entries are
// sorted by a block bitonic network.
// exclusive prefix sum of v over the NT threads of the block (all threads call it)
template <int NT>
__device__ __forceinline__ int32_t block_scan_excl(int32_t v, int32_t *s_wsum /* NT / 32 */) {
  constexpr int NW = NT / 32;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int32_t inc = v;
  for (int o = 1; o < 32; o <<= 1) {
    int32_t t = __shfl_up_sync(0xFFFFFFFFu, inc, o);
    if (lane >= o) inc += t;
  }
  if (lane == 31) s_wsum[w] = inc;
  __syncthreads();
  if (w == 0) {
    int32_t t = lane < NW ? s_wsum[lane] : 0;
    for (int o = 1; o < 32; o <<= 1) {
      int32_t u = __shfl_up_sync(0xFFFFFFFFu, t, o);
      if (lane >= o) t += u;
    }
    if (lane < NW) s_wsum[lane] = t;
  }
  __syncthreads();
  int32_t r = inc - v + (w > 0 ? s_wsum[w - 1] : 0);
  __syncthreads();  // s_wsum may be reused
  return r;
}

template <int TAB, int NT>
constexpr size_t cta_smem_bytes() {
  return (size_t)TAB / 2 * sizeof(uint64_t) + (size_t)TAB * 2 * sizeof(int32_t);
}

template <int TAB, int NT>
__global__ void __launch_bounds__(NT) k_aggregate_cta(
    const int32_t *list, int32_t nrows, const unsigned long long *cub, const int64_t *xadj,
    const int32_t *adj, const int32_t *ew, const int32_t *map, const int32_t *members,
    const int32_t *moff, const int64_t *toff, int32_t *tadj, int32_t *tw, int32_t *cdeg) {
  extern __shared__ __align__(16) unsigned char cta_smem[];
  uint64_t *L = reinterpret_cast<uint64_t *>(cta_smem);      // TAB / 2 sort entries
  int32_t *K = reinterpret_cast<int32_t *>(L + TAB / 2);     // TAB keys
  int32_t *V = K + TAB;                                       // TAB weights
  __shared__ int32_t s_cnt, s_ymin, s_ymax, s_max;
  __shared__ int32_t s_pre[NT + 1];
  __shared__ int64_t s_b[NT];
  __shared__ int32_t s_wsum[NT / 32];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  for (int32_t i = blockIdx.x; i < nrows; i += gridDim.x) {
    int32_t x = list[i];
    uint32_t ub = (uint32_t)cub[x];
    uint32_t tsz = 64;
    while (tsz < 2 * ub) tsz <<= 1;
    for (uint32_t j = tid; j < tsz; j += NT) {
      K[j] = HT_EMPTY;
      V[j] = 0;
    }
    if (tid == 0) {
      s_cnt = 0;
      s_ymin = INT32_MAX;
      s_ymax = -1;
    }
    __syncthreads();
    const int32_t m1 = moff[x + 1];
    for (int32_t c0 = moff[x]; c0 < m1; c0 += NT) {
      const int32_t cn = m1 - c0 < NT ? m1 - c0 : NT;
      int32_t d = 0;
      int64_t b = 0;
      if (tid < cn) {
        int32_t v = members[c0 + tid];
        b = xadj[v];
        d = (int32_t)(xadj[v + 1] - b);
      }
      s_pre[tid + 1] = block_scan_excl<NT>(d, s_wsum) + d;
      s_b[tid] = b;
      if (tid == 0) s_pre[0] = 0;
      __syncthreads();
      const int32_t tot = s_pre[cn];
      for (int32_t e = tid; e < tot; e += NT) {
        int32_t lo = 0, hi = cn - 1;  // the last member whose prefix is <= e owns edge e
        while (lo < hi) {
          int32_t mid = (lo + hi + 1) >> 1;
          if (s_pre[mid] <= e) lo = mid;
          else hi = mid - 1;
        }
        int64_t q = s_b[lo] + (e - s_pre[lo]);
        int32_t y = map[adj[q]];
        if (y != x) ht_add(K, V, tsz - 1, y, ew ? ew[q] : 1);
      }
      __syncthreads();  // the next chunk rewrites the prefix
    }
    // compact into L (order arbitrary; tsz is a multiple of 32)
    for (uint32_t j0 = (uint32_t)w * 32; j0 < tsz; j0 += NT) {
      uint32_t j = j0 + lane;
      bool has = K[j] != HT_EMPTY;
      unsigned bal = __ballot_sync(0xFFFFFFFFu, has);
      int32_t p0 = 0;
      if (lane == 0 && bal) p0 = atomicAdd(&s_cnt, __popc(bal));
      p0 = __shfl_sync(0xFFFFFFFFu, p0, 0);
      if (has) L[p0 + __popc(bal & ((1u << lane) - 1u))] = ((uint64_t)(uint32_t)K[j] << 32) | (uint32_t)V[j];
      int32_t mn = __reduce_min_sync(0xFFFFFFFFu, has ? K[j] : INT32_MAX);
      int32_t mx = __reduce_max_sync(0xFFFFFFFFu, has ? K[j] : -1);
      if (lane == 0 && bal) {
        atomicMin(&s_ymin, mn);
        atomicMax(&s_ymax, mx);
      }
    }
    __syncthreads();
    const int32_t cnt = s_cnt, ymin = s_ymin;
    uint32_t P = 1;
    while (P < (uint32_t)cnt) P <<= 1;
    const int32_t W = cnt > 0 ? ((s_ymax - ymin) >> 5) + 1 : 0;
    int64_t o = toff[x];
    if (W <= TAB && (uint32_t)W <= 16 * P) {
      uint32_t *Bm = reinterpret_cast<uint32_t *>(K);  // bitmap of ids ymin.. (W words)
      int32_t *Pf = V;                                 // popcount prefix per word
      for (int32_t j = tid; j < W; j += NT) Bm[j] = 0;
      __syncthreads();
      for (int32_t j = tid; j < cnt; j += NT) {
        int32_t d = (int32_t)(L[j] >> 32) - ymin;
        atomicOr(&Bm[d >> 5], 1u << (d & 31));
      }
      __syncthreads();
      const int32_t seg = (W + NT - 1) / NT, a = tid * seg < W ? tid * seg : W, b = a + seg < W ? a + seg : W;
      int32_t loc = 0;
      for (int32_t j = a; j < b; ++j) loc += __popc(Bm[j]);
      int32_t base = block_scan_excl<NT>(loc, s_wsum);
      for (int32_t j = a; j < b; ++j) {
        Pf[j] = base;
        base += __popc(Bm[j]);
      }
      __syncthreads();
      for (int32_t j = tid; j < cnt; j += NT) {
        uint64_t ent = L[j];
        int32_t y = (int32_t)(ent >> 32), d = y - ymin;
        int32_t r = Pf[d >> 5] + __popc(Bm[d >> 5] & ((1u << (d & 31)) - 1u));
        tadj[o + r] = y;
        tw[o + r] = (int32_t)(uint32_t)ent;
      }
    } else if (!bucket_order_cta<NT>(L, cnt, ymin, s_ymax, (int32_t)P, K, reinterpret_cast<uint64_t *>(V), s_wsum, &s_max,
                                     [&](int32_t r, uint64_t e) {
                                       tadj[o + r] = (int32_t)(e >> 32);
                                       tw[o + r] = (int32_t)(uint32_t)e;
                                     })) {
      for (uint32_t j = cnt + tid; j < P; j += NT) L[j] = ~0ull;
      __syncthreads();
      bitonic<true>(L, P, tid, NT);
      for (int32_t j = tid; j < cnt; j += NT) {
        tadj[o + j] = (int32_t)(L[j] >> 32);
        tw[o + j] = (int32_t)(uint32_t)L[j];
      }
    }
    if (tid == 0) cdeg[x] = cnt;
    __syncthreads();  // the next row reuses the tables and the counter
  }
}

template <int TAB, int NT>
void launch_aggregate_cta(const int32_t *list, int32_t nrows, const unsigned long long *cub, const Graph &g,
                          const int32_t *map, const int32_t *members, const int32_t *moff,
                          const int64_t *toff, int32_t *tadj, int32_t *tw, int32_t *cdeg) {
  static_assert(TAB / 2 >= NT && TAB % NT == 0, "bin shape");
  constexpr size_t bytes = cta_smem_bytes<TAB, NT>();
  static bool attr = false;
  if (!attr) {
    KMP_CUDA(cudaFuncSetAttribute(k_aggregate_cta<TAB, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)bytes));
    attr = true;
  }
  int per_sm = (int)((227u << 10) / (bytes + 1024));
  if (per_sm < 1) per_sm = 1;
  int blocks = std::min<int64_t>(nrows, (int64_t)ctx().sms * per_sm);
  k_aggregate_cta<TAB, NT><<<blocks, NT, bytes, ctx().stream>>>(list, nrows, cub, g.xadj, g.adj, g.ew, map,
                                                                members, moff, toff, tadj, tw, cdeg);
  KMP_LAUNCHED("aggregate_cta");
}

// ---- large rows (members' total degree > CW_UB)
__global__ void k_large_sizes(int32_t nc, const unsigned long long *cub, int64_t *tsz) {
  for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < nc;
       x += (int64_t)gridDim.x * blockDim.x) {
    unsigned long long ub = cub[x];
    if (ub <= (unsigned long long)CB_UB) {
      tsz[x] = 0;
    } else {
      int64_t d = (int64_t)ub < nc ? (int64_t)ub : nc;  // distinct neighbours < nc
      int64_t c = 32;
      while (c < 2 * d) c <<= 1;
      tsz[x] = c;
    }
  }
}

// work units: chunks of LARGE_CHUNK entries of the rows of members of large
// coarse nodes (so one very high-degree member is spread over many warps)
constexpr int64_t LARGE_CHUNK = 512;

__global__ void k_large_chunks(int32_t n, const int64_t *xadj, const int32_t *map,
                               const unsigned long long *cub, int64_t *nch) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x)
    nch[v] = cub[map[v]] > (unsigned long long)CB_UB ? ceil_div(xadj[v + 1] - xadj[v], LARGE_CHUNK) : 0;
}

// the node owning every chunk
__global__ void k_large_owner(int32_t n, const int64_t *nch, const int64_t *choff, int32_t *owner) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x)
    for (int64_t c = 0; c < nch[v]; ++c) owner[choff[v] + c] = (int32_t)v;
}

__global__ void __launch_bounds__(256) k_large_insert(int64_t total, const int32_t *owner, const int64_t *choff,
                                                      const int64_t *xadj, const int32_t *adj,
                                                      const int32_t *ew, const int32_t *map,
                                                      const int64_t *ltoff, const int64_t *tsz, int32_t *lk,
                                                      int32_t *lv) {
  int lane = threadIdx.x & 31;
  int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t c = gw; c < total; c += nw) {
    int32_t v = owner[c], x = map[v];
    int32_t *K = lk + ltoff[x], *V = lv + ltoff[x];
    uint32_t mask = (uint32_t)(tsz[x] - 1);
    int64_t b = xadj[v] + (c - choff[v]) * LARGE_CHUNK;
    int64_t e = b + LARGE_CHUNK < xadj[v + 1] ? b + LARGE_CHUNK : xadj[v + 1];
    for (int64_t q = b + lane; q < e; q += 32) {
      int32_t y = map[adj[q]];
      if (y != x) ht_add(K, V, mask, y, ew ? ew[q] : 1);
    }
  }
}

// Tables are powers of two >= 32 laid out back to back, so every aligned tile
// of 32 entries belongs to one row: the row of every tile (a warp per large
// row writes its tiles)
__global__ void k_large_tiles(const int32_t *large_list, const int32_t *nlarge, const int64_t *ltoff,
                              const int64_t *tsz, int32_t *tile_row) {
  int lane = threadIdx.x & 31;
  int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t i = gw; i < *nlarge; i += nw) {
    int32_t x = large_list[i];
    for (int64_t t = ltoff[x] / 32 + lane; t < (ltoff[x] + tsz[x]) / 32; t += 32) tile_row[t] = x;
  }
}

// distinct entries of every large row into its own temporary row (positions
// within the row from its entry counter; the row is sorted afterwards)
__global__ void __launch_bounds__(256) k_large_compact(int64_t LT, const int32_t *tile_row,
                                                       const int32_t *lk, const int32_t *lv,
                                                       const int64_t *toff, int32_t *tadj, int32_t *tw,
                                                       int32_t *cdeg) {
  int lane = threadIdx.x & 31;
  int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t t = gw; t * 32 < LT; t += nw) {
    int64_t e = t * 32;
    int32_t x = tile_row[t];
    int32_t y = lk[e + lane];
    bool has = y != HT_EMPTY;
    unsigned bal = __ballot_sync(0xFFFFFFFFu, has);
    if (bal == 0) continue;
    int32_t p0 = 0;
    if (lane == 0) p0 = atomicAdd(&cdeg[x], __popc(bal));
    p0 = __shfl_sync(0xFFFFFFFFu, p0, 0);
    if (has) {
      const int64_t p = toff[x] + p0 + __popc(bal & ((1u << lane) - 1u));
      tadj[p] = y;
      tw[p] = lv[e + lane];
    }
  }
}

// large rows by their distinct entries: up to SORT_S (one CTA of 256 threads
// orders them in shared memory), up to SORT_L (1024 threads), more (segments)
constexpr int32_t SORT_S = 2048;
constexpr int32_t SORT_L = 16384;
__global__ void k_large_split(const int32_t *rows, const int32_t *nrows, const int32_t *cdeg, int32_t cap,
                              int32_t *lists, int32_t *counts) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < *nrows;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t x = rows[i], d = cdeg[x];
    const int c = d <= SORT_S ? 0 : d <= SORT_L ? 1 : 2;
    lists[(int64_t)c * cap + atomicAdd(&counts[c], 1)] = x;
  }
}

// One CTA per row: the row's entries go through buckets of equal id ranges
// (bucket_order_cta's way) straight from global memory: counted, scattered to
// shared memory in bucket order, placed by rank.  A row whose ids crowd into a
// bucket is sorted by a bitonic network.
template <int P, int NT>
__global__ void __launch_bounds__(NT) k_large_sort_smem(int32_t nc, const int32_t *rows, int32_t nrows,
                                                        const int64_t *toff, const int32_t *cdeg, int32_t *tadj,
                                                        int32_t *tw) {
  extern __shared__ uint64_t srt[];  // P entries, P / 2 counters
  __shared__ int32_t s_wsum[NT / 32], s_max;
  int32_t *H = reinterpret_cast<int32_t *>(srt + P);
  const int32_t tid = threadIdx.x;
  for (int64_t i = blockIdx.x; i < nrows; i += gridDim.x) {
    const int32_t x = rows[i];
    const int64_t o = toff[x];
    const int32_t d = cdeg[x];
    int32_t Q = 64;
    while (Q < d) Q <<= 1;
    const int32_t nb = Q / 2;
    const int sh = bucket_shift(0, nc, nb);
    for (int32_t j = tid; j < nb; j += NT) H[j] = 0;
    if (tid == 0) s_max = 0;
    __syncthreads();
#pragma unroll 4
    for (int32_t j = tid; j < d; j += NT) atomicAdd(&H[tadj[o + j] >> sh], 1);
    __syncthreads();
    const int32_t seg = (nb + NT - 1) / NT, a = min(tid * seg, nb), b = min(a + seg, nb);
    int32_t loc = 0, top = 0;
    for (int32_t j = a; j < b; ++j) {
      loc += H[j];
      top = max(top, H[j]);
    }
    if (top > BUCKET_MAX) s_max = 1;
    int32_t base = block_scan_excl<NT>(loc, s_wsum);
    for (int32_t j = a; j < b; ++j) {
      const int32_t h = H[j];
      H[j] = base;
      base += h;
    }
    __syncthreads();
    if (!s_max) {
#pragma unroll 4
      for (int32_t j = tid; j < d; j += NT) {
        const int32_t y = tadj[o + j];
        srt[atomicAdd(&H[y >> sh], 1)] = ((uint64_t)(uint32_t)y << 32) | (uint32_t)tw[o + j];
      }
      __syncthreads();
      for (int32_t j = tid; j < d; j += NT) {
        const uint64_t e = srt[j];
        const int32_t k = (int32_t)(e >> 32) >> sh, lo = k > 0 ? H[k - 1] : 0, hi = H[k];
        int32_t r = lo;
        for (int32_t q = lo; q < hi; ++q) r += srt[q] < e;
        tadj[o + r] = (int32_t)(e >> 32);
        tw[o + r] = (int32_t)(uint32_t)e;
      }
    } else {
      for (int32_t j = tid; j < Q; j += NT)
        srt[j] = j < d ? ((uint64_t)(uint32_t)tadj[o + j] << 32) | (uint32_t)tw[o + j] : ~0ull;
      __syncthreads();
      bitonic<true>(srt, Q, tid, NT);
      for (int32_t j = tid; j < d; j += NT) {
        tadj[o + j] = (int32_t)(srt[j] >> 32);
        tw[o + j] = (int32_t)(uint32_t)srt[j];
      }
    }
    __syncthreads();  // the next row reuses the arrays
  }
}

template <int P, int NT>
void launch_large_sort_smem(int32_t nc, const int32_t *rows, int32_t nrows, const int64_t *toff, const int32_t *cdeg,
                            int32_t *tadj, int32_t *tw) {
  constexpr size_t bytes = (size_t)P * sizeof(uint64_t) + (size_t)P / 2 * sizeof(int32_t);
  static bool attr = false;
  if (!attr) {
    KMP_CUDA(cudaFuncSetAttribute(k_large_sort_smem<P, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)bytes));
    attr = true;
  }
  int per_sm = (int)((227u << 10) / (bytes + 1024));
  if (per_sm < 1) per_sm = 1;
  if (per_sm > 2048 / NT) per_sm = 2048 / NT;
  int blocks = std::min<int64_t>(nrows, (int64_t)ctx().sms * per_sm);
  k_large_sort_smem<P, NT><<<blocks, NT, bytes, ctx().stream>>>(nc, rows, nrows, toff, cdeg, tadj, tw);
  KMP_LAUNCHED("large_sort_smem");
}

// The longest rows (rank r, entries [boff[r], boff[r + 1]) of all of them) are
// ordered by a counting sort on (r, neighbour >> SEG_LO): such a segment holds
// distinct neighbours within 2^SEG_LO ids, so a bitmap of the segment and its
// popcount prefix give every entry's place.  The kernels take a batch of rows
// (seg_batches; nearly always all of them), N entries from boff[0] on, and index
// what they sort from there.  Entries are taken one a thread,
// whatever the rows' lengths (a warp a row took 8.5 of the 73 ms that
// contracting R-MAT 2^24 takes), read from the temporary rows, scattered once,
// and written back in place.
constexpr int SEG_LO = 14;
__device__ __forceinline__ int32_t row_of(const int64_t *boff, int32_t nrows, int64_t i) {
  int32_t lo = 0, hi = nrows - 1;  // last row with boff[row] <= i
  while (lo < hi) {
    const int32_t mid = (lo + hi + 1) >> 1;
    if (boff[mid] <= i) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}
__global__ void k_seg_hist(int64_t N, const int32_t *rows, int32_t nrows, const int64_t *boff, const int64_t *toff,
                           const int32_t *tadj, int hb, int32_t *hist) {
  const int64_t e0 = boff[0];
  for (int64_t i = e0 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < e0 + N; i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t r = row_of(boff, nrows, i);
    atomicAdd(&hist[((int64_t)r << hb) | (tadj[toff[rows[r]] + (i - boff[r])] >> SEG_LO)], 1);
  }
}
__global__ void k_seg_scatter(int64_t N, const int32_t *rows, int32_t nrows, const int64_t *boff, const int64_t *toff,
                              const int32_t *tadj, const int32_t *tw, int hb, const int32_t *off, int32_t *cur,
                              int32_t *ek, int32_t *ev) {
  const int64_t e0 = boff[0];
  for (int64_t i = e0 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < e0 + N; i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t r = row_of(boff, nrows, i);
    const int64_t q = toff[rows[r]] + (i - boff[r]);
    const int32_t y = tadj[q];
    const int64_t x = ((int64_t)r << hb) | (y >> SEG_LO);
    const int64_t p = (int64_t)off[x] + atomicAdd(&cur[x], 1);
    ek[p] = y;
    ev[p] = tw[q];
  }
}
// one CTA per non-empty segment
__global__ void __launch_bounds__(256) k_seg_place(int64_t X, const int32_t *hist, const int32_t *off, int hb,
                                                   const int32_t *ek, const int32_t *ev, const int32_t *rows,
                                                   const int64_t *boff, const int64_t *toff, int32_t *tadj,
                                                   int32_t *tw) {
  constexpr int W = 1 << (SEG_LO - 5), PER = W / 256;
  __shared__ uint32_t bm[W];
  __shared__ int32_t pf[W];
  __shared__ int32_t s_wsum[8];
  const int tid = threadIdx.x;
  for (int64_t x = blockIdx.x; x < X; x += gridDim.x) {
    const int32_t d = hist[x];
    if (d == 0) continue;
    const int64_t o = off[x];
    const int32_t r = (int32_t)(x >> hb);
    const int64_t to = toff[rows[r]] + (boff[0] + o - boff[r]);
#pragma unroll
    for (int u = 0; u < PER; ++u) bm[tid * PER + u] = 0;
    __syncthreads();
    for (int32_t j = tid; j < d; j += 256) {
      const int32_t y = ek[o + j] & ((1 << SEG_LO) - 1);
      atomicOr(&bm[y >> 5], 1u << (y & 31));
    }
    __syncthreads();
    int32_t loc = 0;
#pragma unroll
    for (int u = 0; u < PER; ++u) loc += __popc(bm[tid * PER + u]);
    int32_t base = block_scan_excl<256>(loc, s_wsum);
#pragma unroll
    for (int u = 0; u < PER; ++u) {
      pf[tid * PER + u] = base;
      base += __popc(bm[tid * PER + u]);
    }
    __syncthreads();
    for (int32_t j = tid; j < d; j += 256) {
      const int32_t y = ek[o + j], l = y & ((1 << SEG_LO) - 1);
      const int64_t p = to + pf[l >> 5] + __popc(bm[l >> 5] & ((1u << (l & 31)) - 1u));
      tadj[p] = y;
      tw[p] = ev[o + j];
    }
    __syncthreads();  // the next segment reuses the bitmap
  }
}

__global__ void k_gather_deg(const int32_t *rows, int32_t nrows, const int32_t *cdeg, int64_t *out) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nrows;
       i += (int64_t)gridDim.x * blockDim.x)
    out[i] = cdeg[rows[i]];
}

// rows from their upper-bound offsets into the final CSR; four loads per lane
// are issued before their stores
__global__ void k_copy_rows(int32_t nc, const int64_t *__restrict__ toff, const int64_t *__restrict__ cx,
                            const int32_t *__restrict__ tadj, const int32_t *__restrict__ tw,
                            int32_t *__restrict__ adj, int32_t *__restrict__ ew) {
  int lane = threadIdx.x & 31;
  int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t x = gw; x < nc; x += nw) {
    int64_t o = toff[x], p = cx[x], d = cx[x + 1] - p;
    for (int64_t j = lane; j < d; j += 128) {
      int32_t a[4], c[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (j + 32 * u < d) {
          a[u] = tadj[o + j + 32 * u];
          c[u] = tw[o + j + 32 * u];
        }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (j + 32 * u < d) {
          adj[p + j + 32 * u] = a[u];
          ew[p + j + 32 * u] = c[u];
        }
    }
  }
}

__global__ void k_set_last_i64(int64_t *a, int64_t idx, const int64_t *v) { a[idx] = *v; }

// graph facts: max degree, isolated nodes, max and total node weight, total edge weight
__global__ void k_graph_facts(int32_t n, const int64_t *xadj, const int32_t *vw,
                              unsigned long long *out /* [maxdeg, iso, maxvw, totvw] */) {
  unsigned long long md = 0, iso = 0, mw = 0, tw = 0;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x) {
    unsigned long long d = (unsigned long long)(xadj[v + 1] - xadj[v]);
    md = d > md ? d : md;
    iso += d == 0;
    unsigned long long w = vw ? (unsigned long long)vw[v] : 1ull;
    mw = w > mw ? w : mw;
    tw += w;
  }
#pragma unroll
  for (int m = 16; m > 0; m >>= 1) {
    unsigned long long a = __shfl_xor_sync(0xFFFFFFFFu, md, m);
    md = a > md ? a : md;
    iso += __shfl_xor_sync(0xFFFFFFFFu, iso, m);
    unsigned long long b = __shfl_xor_sync(0xFFFFFFFFu, mw, m);
    mw = b > mw ? b : mw;
    tw += __shfl_xor_sync(0xFFFFFFFFu, tw, m);
  }
  if ((threadIdx.x & 31) == 0) {
    atomicMax(&out[0], md);
    atomicAdd(&out[1], iso);
    atomicMax(&out[2], mw);
    atomicAdd(&out[3], tw);
  }
}

static void set_facts(Graph &g, const int64_t *h) {
  g.maxdeg = h[0];
  g.n_isolated = h[1];
  g.max_vw = (int32_t)h[2];
  g.total_vw = h[3];
}

void compute_facts(Graph &g) {
  DBuf<int64_t> f(4);
  f.zero();
  k_graph_facts<<<grid_for(g.n, 256), 256, 0, ctx().stream>>>(g.n, g.xadj, g.vw,
                                                             reinterpret_cast<unsigned long long *>(f.p));
  KMP_LAUNCHED("graph_facts");
  int64_t h[4];
  to_host(h, f.p, 4);
  set_facts(g, h);
}

void free_graph(Graph &g) {
  if (g.owned) {
    dfree(g.xadj);
    dfree(g.adj);
    dfree(g.vw);
    dfree(g.ew);
  }
  g = Graph();
}

Graph contract_graph(const Graph &g, const int32_t *label, int32_t *map) {
  Context &C = ctx();
  cudaStream_t s = C.stream;
  int32_t n = g.n;
  int grid = grid_for(n, 256);
  DBuf<uint8_t> used(n);
  used.zero();
  DBuf<int32_t> cid(n), ncd(2);  // coarse nodes, bad labels
  ncd.zero();
  k_map_used<<<grid, 256, 0, s>>>(n, label, used, ncd.p + 1);
  KMP_LAUNCHED("map_used");
  scan_excl_u8_to_i32(used, cid, n, ncd);
  int32_t hn[2];
  to_host(hn, ncd.p, 2);
  if (hn[1]) fail(KMP_ERR_ARG, "label: value out of range");
  const int32_t nc = hn[0];
  k_map<<<grid, 256, 0, s>>>(n, label, cid, map);
  KMP_LAUNCHED("map");

  Graph out;
  out.n = nc;
  out.owned = true;
  DBuf<int32_t> cvw(nc), csize(nc + 1), moff(nc + 1), mcur(nc), members(n);
  DBuf<unsigned long long> cub(nc);
  cvw.zero();
  csize.zero();
  mcur.zero();
  cub.zero();
  k_contract_prep<<<grid, 256, 0, s>>>(n, g.xadj, g.vw, map, cvw, csize, cub);
  KMP_LAUNCHED("contract_prep");
  scan_excl_i32(csize, moff, nc + 1, nullptr);
  k_members<<<grid, 256, 0, s>>>(n, map, moff, mcur, members);
  KMP_LAUNCHED("members");
  // temporary rows at upper-bound offsets
  DBuf<int64_t> ub64(nc + 1), toff(nc + 1);
  int gridc = grid_for(nc, 256);
  k_ub_to_i64<<<gridc, 256, 0, s>>>(nc, cub, ub64);
  KMP_LAUNCHED("ub_copy");
  scan_excl_i64(ub64, toff, nc, nullptr);
  DBuf<int32_t> tadj(g.m), tw(g.m), cdeg(nc + 1);  // every entry belongs to one coarse row
  cdeg.zero();
  DBuf<int32_t> lists((int64_t)NCLASS * nc), counts(NCLASS);
  counts.zero();
  k_split_ub<<<grid_for(nc, 256 * SPLIT_PER), 256, 0, s>>>(nc, cub, lists, counts);
  KMP_LAUNCHED("split_ub");
  int32_t hc[NCLASS];
  to_host(hc, counts.p, NCLASS);
  const int32_t *large_list = lists.p + (int64_t)CLS_GLOBAL * nc;
  auto L = [&](int c) { return lists.p + (int64_t)c * nc; };
  if (hc[4] > 0) launch_aggregate_cta<4096, 256>(L(4), hc[4], cub, g, map, members, moff, toff, tadj, tw, cdeg);
  if (hc[5] > 0) launch_aggregate_cta<8192, 512>(L(5), hc[5], cub, g, map, members, moff, toff, tadj, tw, cdeg);
  if (hc[6] > 0)
    launch_aggregate_cta<16384, 1024>(L(6), hc[6], cub, g, map, members, moff, toff, tadj, tw, cdeg);
  if (hc[0] > 0) launch_aggregate_warp<128, 8>(L(0), hc[0], cub, g, map, members, moff, toff, tadj, tw, cdeg);
  if (hc[1] > 0) launch_aggregate_warp<256, 8>(L(1), hc[1], cub, g, map, members, moff, toff, tadj, tw, cdeg);
  if (hc[2] > 0) launch_aggregate_warp<512, 8>(L(2), hc[2], cub, g, map, members, moff, toff, tadj, tw, cdeg);
  if (hc[3] > 0) launch_aggregate_warp<1024, 4>(L(3), hc[3], cub, g, map, members, moff, toff, tadj, tw, cdeg);
  if (hc[CLS_GLOBAL] > 0) {
    // large rows: every member inserts in parallel into its coarse node's global
    // table; each row's distinct entries are compacted into its temporary row
    // and put in order there: in shared memory by one CTA per row when they fit,
    // the longer rows by segments
    int bits = 1;
    while ((1ll << bits) < (int64_t)nc) ++bits;
    DBuf<int64_t> tsz(nc), ltoff(nc), ltot(1);
    k_large_sizes<<<gridc, 256, 0, s>>>(nc, cub, tsz);
    KMP_LAUNCHED("large_sizes");
    scan_excl_i64(tsz, ltoff, nc, ltot);
    int64_t LT = read1(ltot.p);
    DBuf<int32_t> lk(LT), lv(LT);
    lk.fill_bytes(0xFF);
    lv.zero();
    DBuf<int64_t> nch(n), choff(n), chtot(1);
    k_large_chunks<<<grid, 256, 0, s>>>(n, g.xadj, map, cub, nch);
    KMP_LAUNCHED("large_chunks");
    scan_excl_i64(nch, choff, n, chtot);
    int64_t CT = read1(chtot.p);
    DBuf<int32_t> owner(CT + 1);
    k_large_owner<<<grid, 256, 0, s>>>(n, nch, choff, owner);
    KMP_LAUNCHED("large_owner");
    k_large_insert<<<grid_for(CT * 32, 256, 8), 256, 0, s>>>(CT, owner, choff, g.xadj, g.adj, g.ew, map,
                                                             ltoff, tsz, lk, lv);
    KMP_LAUNCHED("large_insert");
    DBuf<int32_t> tile_row(LT / 32 + 1);
    k_large_tiles<<<grid_for((int64_t)hc[CLS_GLOBAL] * 32, 256), 256, 0, s>>>(large_list, counts.p + CLS_GLOBAL, ltoff, tsz,
                                                                     tile_row);
    KMP_LAUNCHED("large_tiles");
    k_large_compact<<<grid_for(LT, 256, 8), 256, 0, s>>>(LT, tile_row, lk, lv, toff, tadj, tw, cdeg);
    KMP_LAUNCHED("large_compact");
    const int32_t nlarge = hc[CLS_GLOBAL];
    DBuf<int32_t> slists(3ll * nlarge), scounts(3);
    scounts.zero();
    k_large_split<<<grid_for(nlarge, 256), 256, 0, s>>>(large_list, counts.p + CLS_GLOBAL, cdeg, nlarge, slists,
                                                       scounts);
    KMP_LAUNCHED("large_split");
    int32_t sc[3];
    to_host(sc, scounts.p, 3);
    if (sc[0] > 0) launch_large_sort_smem<SORT_S, 256>(nc, slists.p, sc[0], toff, cdeg, tadj, tw);
    if (sc[1] > 0) launch_large_sort_smem<SORT_L, 1024>(nc, slists.p + nlarge, sc[1], toff, cdeg, tadj, tw);
    if (sc[2] > 0) {
      const int32_t nbig = sc[2];
      const int32_t *brows = slists.p + 2ll * nlarge;
      DBuf<int64_t> bdeg(nbig), boff(nbig + 1);
      k_gather_deg<<<grid_for(nbig, 256), 256, 0, s>>>(brows, nbig, cdeg, bdeg);
      KMP_LAUNCHED("gather_deg");
      scan_excl_i64(bdeg, boff, nbig, boff.p + nbig);
      std::vector<int64_t> hoff((size_t)nbig + 1);
      to_host(hoff.data(), boff.p, hoff.size());
      // (a row above SORT_L entries has more than 2^SEG_LO distinct neighbours, so
      // bits > SEG_LO here)
      const int hb = bits - SEG_LO;
      for (const auto &[r0, r1] : seg_batches(hoff.data(), nbig, hb, SEG_MAX_ENTRIES, SEG_MAX_COUNTERS)) {
        const int32_t *rows = brows + r0;
        const int64_t *off0 = boff.p + r0;
        const int64_t NE = hoff[r1] - hoff[r0], X = (int64_t)(r1 - r0) << hb;
        const int gridN = grid_for(NE, 256);
        DBuf<int32_t> ek(NE), ev(NE), hist(X), off(X), cur(X);
        hist.zero();
        cur.zero();
        k_seg_hist<<<gridN, 256, 0, s>>>(NE, rows, r1 - r0, off0, toff, tadj, hb, hist);
        KMP_LAUNCHED("seg_hist");
        scan_excl_i32(hist, off, X, nullptr);
        k_seg_scatter<<<gridN, 256, 0, s>>>(NE, rows, r1 - r0, off0, toff, tadj, tw, hb, off, cur, ek, ev);
        KMP_LAUNCHED("seg_scatter");
        k_seg_place<<<grid_for(X, 1), 256, 0, s>>>(X, hist, off, hb, ek, ev, rows, off0, toff, tadj, tw);
        KMP_LAUNCHED("seg_place");
      }
    }
  }
  // entries and facts of the coarse graph in one read
  DBuf<int64_t> sizes(5);
  sizes.zero();
  out.xadj = static_cast<int64_t *>(dmalloc((nc + 1) * sizeof(int64_t)));
  scan_excl_i32_to_i64(cdeg, out.xadj, nc, sizes.p + 4);
  k_set_last_i64<<<1, 1, 0, s>>>(out.xadj, nc, sizes.p + 4);
  KMP_LAUNCHED("set_last");
  k_graph_facts<<<gridc, 256, 0, s>>>(nc, out.xadj, cvw, reinterpret_cast<unsigned long long *>(sizes.p));
  KMP_LAUNCHED("graph_facts");
  int64_t hs[5];
  to_host(hs, sizes.p, 5);
  set_facts(out, hs);
  out.m = hs[4];
  out.adj = static_cast<int32_t *>(dmalloc((out.m > 0 ? out.m : 1) * sizeof(int32_t)));
  out.ew = static_cast<int32_t *>(dmalloc((out.m > 0 ? out.m : 1) * sizeof(int32_t)));
  if (nc > 0) {
    k_copy_rows<<<grid_for((int64_t)nc * 32, 256), 256, 0, s>>>(nc, toff, out.xadj, tadj, tw,
                                                                out.adj, out.ew);
    KMP_LAUNCHED("copy_rows");
  }
  out.vw = cvw.release();
  return out;
}

__global__ void k_project(int32_t n, const int32_t *map, const int32_t *pc, int32_t *pf) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x)
    pf[v] = pc[map[v]];
}

void project(int32_t n_fine, const int32_t *map, const int32_t *part_c, int32_t *part_f) {
  k_project<<<grid_for(n_fine, 256), 256, 0, ctx().stream>>>(n_fine, map, part_c, part_f);
  KMP_LAUNCHED("project");
}

// Block weights node by node, then the cut by equal shares of rows and entries: a warp
// takes one run of them (a row counts for one more than its entries), CUT_SHARE at
// least, finds the row they start in, and reads the ends and blocks of 32 rows at a time; an
// entry's row is the number of those that end at or before it.  So a hub's row is
// shared by many warps, and a short row costs no round trip of its own (rows one
// after the other on the warp that held their 32 nodes: R-MAT 2^22 1.48 ms, mesh of
// 2^24 nodes 1.41 ms; for the cut alone).  Shares of the entries alone let one warp
// walk all rows without entries between two of its own: 2^24 isolated nodes took
// 293 ms, every 64th of 2^20 nodes joined 2.0 ms.  One run a warp, since runs of a
// fixed length leave a last wave nearly empty on large graphs and most warps without
// any on small ones (kernel alone, runs of 2048 entries against this: mesh of 2^15
// nodes, degree 12, 44 -> 21 us; of 2^21, weighted, 209 -> 172; R-MAT 2^21 324 -> 260);
// below 512 the search for its rows costs more.  Entries before xadj[0] belong
// to no row and are not read.  Weights are summed in shared memory when k is small.
// bad (nullable) is set when a block id lies outside [0, k); such ids index nothing.
constexpr int CUT_SBW = 2048;
constexpr int CUT_SHARE = 512;
constexpr int CUT_TILE = 2048;  // entries of a window taken together
constexpr int CUT_U = 4;
// The last row v with v + xadj[v] - xadj[0] <= d (d >= 0), by a warp, 32 positions a read
__device__ __forceinline__ int64_t share_row(const int64_t *__restrict__ xadj, int32_t n, int64_t d) {
  const int lane = threadIdx.x & 31;
  int64_t st = 1, v = 0;
  while (32 * st < n) st *= 32;
  d += xadj[0];
  for (; st > 0; st /= 32) {
    const int64_t p = v + st * (lane + 1);
    v += st * __popc(__ballot_sync(0xFFFFFFFFu, p < n && p + xadj[p] <= d));  // rises with p
  }
  return v;
}
// WEIGHTED: ew is not null (with the test in the loop 60 us instead of 44 for 100,000
// entries in runs of 2304)
template <bool WEIGHTED>
__global__ void __launch_bounds__(256) k_cut_bw(int32_t n, int64_t m, int32_t k, const int64_t *__restrict__ xadj,
                                                const int32_t *__restrict__ adj, const int32_t *__restrict__ vw,
                                                const int32_t *__restrict__ ew, const int32_t *__restrict__ part,
                                                unsigned long long *bw, unsigned long long *cut,
                                                unsigned long long *bad, const int *status) {
  __shared__ unsigned long long sbw[CUT_SBW];
  const bool local = k <= CUT_SBW;
  if (local)
    for (int i = threadIdx.x; i < k; i += blockDim.x) sbw[i] = 0;
  if (status && blockIdx.x == 0 && threadIdx.x == 0) bad[1] = (unsigned long long)(long long)*status;
  __syncthreads();
  bool off = false;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    const int32_t p = part[v];
    const unsigned long long w = (unsigned long long)(vw ? vw[v] : 1);
    if (p < 0 || p >= k) off = true;
    else if (local) atomicAdd(&sbw[p], w);
    else atomicAdd(&bw[p], w);
  }
  if (off && bad) atomicOr(bad, 1ull);
  const int lane = threadIdx.x & 31;
  const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  unsigned long long c = 0;
  const int64_t m0 = xadj[0], total = n + m - m0;
  const int64_t share = max((total + nw - 1) / nw, (int64_t)CUT_SHARE), d = gw * share;
  if (d < total) {
    int64_t v0 = share_row(xadj, n, d), e = m0 + d - v0, e1 = m;
    if (d + share < total) e1 = m0 + d + share - share_row(xadj, n, d + share);
    while (e < e1) {
      const int64_t v = v0 + lane;
      const int64_t end = v < n ? xadj[v + 1] : m;
      const int32_t pv = v < n ? part[v] : -1;
      const int64_t top = (int64_t)__shfl_sync(0xFFFFFFFFu, (unsigned long long)end, 31);
      const int64_t lim = min(min(top, e1), e + CUT_TILE);
      const int32_t rel = (int32_t)(end - e < 2 * CUT_TILE ? end - e : 2 * CUT_TILE);  // row ends from e on
      const int32_t len = (int32_t)(lim - e);
      for (int32_t t0 = 0; t0 < len; t0 += 32 * CUT_U) {
        int32_t u[CUT_U], wt[CUT_U];
#pragma unroll
        for (int r = 0; r < CUT_U; ++r) {
          const int32_t t = t0 + 32 * r + lane;
          u[r] = t < len ? adj[e + t] : -1;
          wt[r] = WEIGHTED && t < len ? ew[e + t] : 1;
        }
#pragma unroll
        for (int r = 0; r < CUT_U; ++r) u[r] = u[r] >= 0 ? part[u[r]] : INT32_MIN;
#pragma unroll
        for (int r = 0; r < CUT_U; ++r) {
          const int32_t t = t0 + 32 * r + lane;
          int32_t j = 0;  // rows that end at or before entry t
#pragma unroll
          for (int st = 16; st > 0; st >>= 1) {
            const int32_t x = __shfl_sync(0xFFFFFFFFu, rel, j + st - 1);
            if (x <= t) j += st;
          }
          const int32_t own = __shfl_sync(0xFFFFFFFFu, pv, j);
          if (t < len && u[r] != own) c += (unsigned long long)wt[r];
        }
      }
      if (lim == top) v0 += 32;
      e = lim;
    }
  }
#pragma unroll
  for (int mm = 16; mm > 0; mm >>= 1) c += __shfl_xor_sync(0xFFFFFFFFu, c, mm);
  if (lane == 0 && c) atomicAdd(cut, c);
  __syncthreads();
  if (local)
    for (int i = threadIdx.x; i < k; i += blockDim.x)
      if (sbw[i]) atomicAdd(&bw[i], sbw[i]);
}

__global__ void k_half(int64_t *c) { *c /= 2; }  // every edge was counted from both ends

// block weights only (no edge traffic)
__global__ void __launch_bounds__(256) k_bw_only(int32_t n, int32_t k, const int32_t *vw,
                                                 const int32_t *part, unsigned long long *bw) {
  __shared__ unsigned long long sbw[CUT_SBW];
  bool local = k <= CUT_SBW;
  if (local)
    for (int i = threadIdx.x; i < k; i += blockDim.x) sbw[i] = 0;
  __syncthreads();
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x) {
    unsigned long long w = (unsigned long long)(vw ? vw[v] : 1);
    if (local) atomicAdd(&sbw[part[v]], w);
    else atomicAdd(&bw[part[v]], w);
  }
  __syncthreads();
  if (local)
    for (int i = threadIdx.x; i < k; i += blockDim.x)
      if (sbw[i]) atomicAdd(&bw[i], sbw[i]);
}

void block_weights(const Graph &g, const int32_t *part, int32_t k, int64_t *bw_dev) {
  cudaStream_t s = ctx().stream;
  KMP_CUDA(cudaMemsetAsync(bw_dev, 0, (size_t)k * sizeof(int64_t), s));
  if (g.n == 0) return;
  k_bw_only<<<grid_for(g.n, 256, 4), 256, 0, s>>>(g.n, k, g.vw, part,
                                                  reinterpret_cast<unsigned long long *>(bw_dev));
  KMP_LAUNCHED("bw_only");
}

// bad, status (nullable): as in k_cut_bw; the status word goes behind bad
static void launch_cut(const Graph &g, const int32_t *part, int32_t k, int64_t *bw, int64_t *cut, int64_t *bad,
                       const int *status) {
  const int64_t work = std::max<int64_t>(g.n, ceil_div(g.n + g.m, CUT_SHARE) * 32);
  const auto kernel = g.ew ? k_cut_bw<true> : k_cut_bw<false>;
  // one wave: 5 CTAs an SM with 48 registers a thread, 6 with 40 (8 asked for, a weighted
  // R-MAT graph of 2^19 nodes takes 107 us, one of 2^21 345)
  kernel<<<grid_for(work, 256, g.ew ? 5 : 6), 256, 0, ctx().stream>>>(
      g.n, g.m, k, g.xadj, g.adj, g.vw, g.ew, part, reinterpret_cast<unsigned long long *>(bw),
      reinterpret_cast<unsigned long long *>(cut), reinterpret_cast<unsigned long long *>(bad), status);
  KMP_LAUNCHED("cut_bw");
}

void cut_and_weights(const Graph &g, const int32_t *part, int32_t k, int64_t *bw_dev,
                     int64_t *cut_dev) {
  cudaStream_t s = ctx().stream;
  KMP_CUDA(cudaMemsetAsync(bw_dev, 0, (size_t)k * sizeof(int64_t), s));
  KMP_CUDA(cudaMemsetAsync(cut_dev, 0, sizeof(int64_t), s));
  launch_cut(g, part, k, bw_dev, cut_dev, nullptr, nullptr);
  k_half<<<1, 1, 0, s>>>(cut_dev);
  KMP_LAUNCHED("half");
}

// Cut, the range check of the block ids, the status word and the block weights behind
// them in one buffer: one clear, one kernel, one copy and one wait while the weights
// are few.  Many go straight to the caller's array in a copy of their own, none are
// copied when not asked for (k = 2^20 on a mesh of 2^21 nodes: 0.94 ms through a second
// host buffer, 0.32 like this; at 4097..12,000 one copy is 4..10 us faster, at 32,768
// two are 8).
constexpr int32_t CUT_ONE_COPY = 16384;
void cut_to_host(const Graph &g, const int32_t *part, int32_t k, int64_t head[3], int64_t *bw) {
  Context &C = ctx();
  DBuf<int64_t> d((size_t)k + 3);
  d.zero();
  launch_cut(g, part, k, d.p + 3, d.p, d.p + 1, C.d_status);
  const bool one = bw && k <= CUT_ONE_COPY;
  std::vector<int64_t> h(3 + (one ? (size_t)k : 0));
  to_host(h.data(), d.p, h.size());
  head[0] = h[0] / 2;
  head[1] = h[1];
  head[2] = h[2];
  if (!bw || head[1] || head[2]) return;
  if (one) memcpy(bw, h.data() + 3, (size_t)k * sizeof(int64_t));
  else to_host(bw, d.p + 3, (size_t)k);
}

}  // namespace kmp
