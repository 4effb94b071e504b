"""GPU tests of the cut on rows without entries: runs of them of every length
between the others, and millions of them in one run, which cost no walk."""
import time

import numpy as np
import pytest
import torch

import oracle as O
from paper_2105_02022_gb300 import graphgen as gg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kmp():
    from paper_2105_02022_gb300 import _build
    from paper_2105_02022_gb300 import kmp as K

    _build.build_all()
    O.build()
    assert torch.cuda.is_available()
    yield K


def _matched(n, ends, degree=1):
    """Consecutive nodes of `ends` (an even number) joined in pairs by `degree` entries; the rest alone."""
    xadj = np.zeros(n + 1, np.int64)
    deg = np.zeros(n, np.int64)
    deg[ends] = degree
    np.cumsum(deg, out=xadj[1:])
    adj = np.repeat(np.asarray(ends).reshape(-1, 2)[:, ::-1].reshape(-1), degree)
    return gg.Graph(n, xadj, adj.astype(np.int32))


@pytest.mark.parametrize("gap", [1, 30, 31, 32, 33, 63, 64, 65, 1023, 1024, 1025, 1056, 1057, 33000, 40000])
@pytest.mark.parametrize("degree", [1, 40])
def test_runs_of_rows_without_entries(kmp, gap, degree):
    ends = np.concatenate([[3], np.arange(1, 40) * (gap + 1) + 3])
    for tail in (0, 1, 40, 5000):
        g = _matched(int(ends[-1]) + 1 + tail, ends, degree)
        part = (np.arange(g.n) * 7 % 5).astype(np.int32)
        part[ends[::4]] = part[ends[1::4]]  # some pairs uncut
        cut, bw = kmp.cut(kmp.DeviceGraph.from_host(g), torch.from_numpy(part).cuda(), 5)
        assert cut == O.cut(g, part)
        assert np.array_equal(bw, np.bincount(part, minlength=5))


def test_a_long_run_is_not_walked(kmp):
    """2^24 rows between two nodes: a walk takes 0.3 s, the skip microseconds."""
    n = 1 << 24
    g = _matched(n, np.array([0, n - 1]))
    dg = kmp.DeviceGraph.from_host(g)
    part = torch.zeros(n, dtype=torch.int32, device="cuda")
    part[-1] = 1
    times = []
    for _ in range(4):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        cut, bw = kmp.cut(dg, part, 2)
        times.append(time.perf_counter() - t0)
    assert cut == 1 and bw.tolist() == [n - 1, 1]
    assert min(times) < 0.05
