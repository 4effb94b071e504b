// Host-side size plans of the launches: plain C++, so that their limits can be
// checked without a GPU.
#ifndef KMP_PLAN_H
#define KMP_PLAN_H
#include <algorithm>
#include <cstdint>
#include <numeric>
#include <utility>
#include <vector>

namespace kmp {

// Batches [first, second) of the longest rows of a contraction, whose entries are
// put in order together: the counting sort of a batch indexes its entries and its
// counters (2^hb a row) in 32 bits, so a batch ends before either passes its limit.
// One row alone always fits (it has fewer entries than there are nodes).  boff:
// entries before each of the nrows rows, and all of them.
inline std::vector<std::pair<int32_t, int32_t>> seg_batches(const int64_t *boff, int32_t nrows, int hb,
                                                            int64_t max_entries, int64_t max_counters) {
  std::vector<std::pair<int32_t, int32_t>> out;
  for (int32_t a = 0; a < nrows;) {
    int32_t b = a + 1;
    while (b < nrows && boff[b + 1] - boff[a] <= max_entries && ((int64_t)(b + 1 - a) << hb) <= max_counters) ++b;
    out.emplace_back(a, b);
    a = b;
  }
  return out;
}
constexpr int64_t SEG_MAX_ENTRIES = 1ll << 30, SEG_MAX_COUNTERS = 1ll << 30;

// Scratch words of a bipartitioner item of n nodes and m entries (a first estimate; the
// launch says when it was too small), with `learned` words a node for the proposer
inline int64_t ip_scratch_words(int64_t n, int64_t m, int64_t learned) {
  const auto pow2 = [](int64_t x) { return x <= 2 ? 2ll : 1ll << (64 - __builtin_clzll((unsigned long long)x - 1)); };
  return (104 * n + 64 * pow2(n) + 16 * m + 8 * pow2(m) + 2048 + (learned > 0 ? learned * n + 64 : 0) + 3) & ~3ll;
}

// Work order of a round's items and the scratch regions of its CTAs.  Items are
// taken by falling scratch size, CTA b the b-th first and later ones from a queue.
// So CTA b's region needs what the b-th item needs, and the regions together never
// more than the items one by one.  (With every region sized for the largest item,
// one of 65,535 nodes beside 500 tiny ones took 330 GB.)  region: where each CTA's
// starts, and the total.
struct IPRegions {
  std::vector<int32_t> order;
  std::vector<int64_t> region;
};
inline IPRegions ip_regions(const std::vector<int64_t> &words, int32_t ctas, int64_t mult) {
  IPRegions r;
  r.order.resize(words.size());
  std::iota(r.order.begin(), r.order.end(), 0);
  std::stable_sort(r.order.begin(), r.order.end(), [&](int32_t a, int32_t b) { return words[a] > words[b]; });
  r.region.assign(1, 0);
  for (int32_t b = 0; b < ctas; ++b) r.region.push_back(r.region.back() + mult * words[r.order[b]]);
  return r;
}

}  // namespace kmp
#endif
