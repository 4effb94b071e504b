"""CPU checks of the launches' size plans (csrc/kmp_plan.h), at sizes that no test
graph reaches."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2105_02022_gb300", "csrc")
SHIM = """
#include "kmp_plan.h"
using namespace kmp;
extern "C" {
int32_t seg(const int64_t *boff, int32_t nrows, int hb, int64_t me, int64_t mc, int32_t *out) {
  int32_t n = 0;
  for (auto &b : seg_batches(boff, nrows, hb, me, mc)) { out[2 * n] = b.first; out[2 * n + 1] = b.second; ++n; }
  return n;
}
int64_t words(int64_t n, int64_t m, int64_t learned) { return ip_scratch_words(n, m, learned); }
void regions(const int64_t *w, int32_t n, int32_t ctas, int64_t mult, int32_t *order, int64_t *region) {
  IPRegions r = ip_regions(std::vector<int64_t>(w, w + n), ctas, mult);
  for (int32_t i = 0; i < n; ++i) order[i] = r.order[i];
  for (int32_t i = 0; i <= ctas; ++i) region[i] = r.region[i];
}
int64_t seg_max(int which) { return which ? SEG_MAX_COUNTERS : SEG_MAX_ENTRIES; }
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    src, out = d / "shim.cpp", d / "shim.so"
    src.write_text(SHIM)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-I", CSRC, "-o", str(out), str(src)])
    L = ctypes.CDLL(str(out))
    L.seg.argtypes = [ctypes.c_void_p, ctypes.c_int32, ctypes.c_int, ctypes.c_int64, ctypes.c_int64, ctypes.c_void_p]
    L.seg_max.restype = L.words.restype = ctypes.c_int64
    L.words.argtypes = [ctypes.c_int64] * 3
    L.regions.argtypes = [ctypes.c_void_p, ctypes.c_int32, ctypes.c_int32, ctypes.c_int64, ctypes.c_void_p, ctypes.c_void_p]
    return L


def _batches(plan, sizes, hb, me, mc):
    boff = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    out = np.zeros(2 * len(sizes), np.int32)
    n = plan.seg(boff.ctypes.data, len(sizes), hb, me, mc, out.ctypes.data)
    return boff, out[: 2 * n].reshape(-1, 2)


@pytest.mark.parametrize("name", ["few", "past 2^31 entries", "past 2^30 counters", "rows near 2^31", "one"])
def test_batches_of_the_longest_rows(plan, name):
    """Every row once, in order; entries and counters of a batch fit 32-bit indices."""
    rng = np.random.default_rng(1)
    sizes, hb = {"few": (rng.integers(16385, 100000, 500), 8),
                 "past 2^31 entries": (rng.integers(16385, 1 << 20, 9000), 12),
                 "past 2^30 counters": (rng.integers(16385, 30000, 20000), 17),
                 "rows near 2^31": (np.array([2**31 - 1, 2**31 - 5, 20000, 2**30, 1 << 20, 2**31 - 1]), 17),
                 "one": (np.array([17000]), 5)}[name]
    me, mc = plan.seg_max(0), plan.seg_max(1)
    boff, b = _batches(plan, sizes, hb, me, mc)
    assert b[0, 0] == 0 and b[-1, 1] == len(sizes) and np.array_equal(b[1:, 0], b[:-1, 1])
    entries, counters = boff[b[:, 1]] - boff[b[:, 0]], (b[:, 1] - b[:, 0]).astype(np.int64) << hb
    assert entries.max() < 2**31 and counters.max() < 2**31
    alone = b[:, 1] - b[:, 0] == 1
    assert np.all((entries <= me) | alone) and np.all((counters <= mc) | alone)
    if name in ("few", "one"):
        assert len(b) == 1


@pytest.mark.parametrize("learned", [0, 212])
@pytest.mark.parametrize("mult", [1, 4, 1024])
@pytest.mark.parametrize("items,ctas", [("skewed", 444), ("skewed", 456), ("equal", 456), ("few", 7), ("one", 1)])
def test_scratch_regions(plan, items, ctas, mult, learned):
    """Whichever CTA takes an item, its region holds it, whatever the queue's order after the
    first items; all regions together take no more than the items one by one."""
    rng = np.random.default_rng(2)
    n = {"skewed": np.concatenate([rng.integers(1, 40, 600), [65535, 30000]]), "equal": np.full(1000, 2048),
         "few": np.array([5, 60000, 1, 2, 3, 4, 9]), "one": np.array([1])}[items]
    m = np.where(n > 20000, 6_500_000, 8 * n)
    words = np.array([plan.words(int(a), int(b), learned) for a, b in zip(n, m)], np.int64)
    assert np.all(words % 4 == 0) and np.all(words > 104 * n + 16 * m)
    order, region = np.zeros(len(n), np.int32), np.zeros(ctas + 1, np.int64)
    plan.regions(words.ctypes.data, len(n), ctas, mult, order.ctypes.data, region.ctypes.data)
    assert np.array_equal(np.sort(order), np.arange(len(n))) and region[0] == 0
    size = np.diff(region)
    need = mult * words[order]
    assert np.array_equal(size, need[:ctas])
    if len(n) > ctas:  # any CTA may take any later item
        assert size.min() >= need[ctas:].max()
    assert region[-1] <= mult * words.sum()
    if items == "skewed" and mult == 1:
        assert 4 * region[-1] < 3 << 30
