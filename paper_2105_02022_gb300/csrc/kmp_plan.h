// Host-side size plans of the launches: plain C++, so that their limits can be
// checked without a GPU.
#ifndef KMP_PLAN_H
#define KMP_PLAN_H
#include <cstdint>
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

}  // namespace kmp
#endif
