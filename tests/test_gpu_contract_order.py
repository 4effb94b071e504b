"""GPU tests of the contraction's row orders, bit-exact against the oracle: rows
whose neighbour ids crowd into one place of a wide range (the buckets overflow and
the sorting network takes over), rows spread evenly over it (the buckets), in
every row class from the warp tables to the longest rows."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2105_02022_gb300 import graphgen as gg

pytestmark = pytest.mark.gpu

N = 300000
DEGREES = [90, 200, 300, 500, 700, 2000, 3000, 6000, 8000, 9000, 17000]


@pytest.fixture(scope="module")
def kmp():
    from paper_2105_02022_gb300 import _build
    from paper_2105_02022_gb300 import kmp as K

    _build.build_all()
    O.build()
    assert torch.cuda.is_available()
    yield K


def _graph(spread):
    """Hubs 0, 1, ... with the given degrees: neighbours in one run of ids and the last node, or all over."""
    rng = np.random.default_rng(4)
    rows, cols = [], []
    for h, d in enumerate(DEGREES):
        nb = rng.choice(np.arange(1000, N - 1), d, replace=False) if spread else np.arange(1000 + 7 * h, 1000 + 7 * h + d)
        nb = np.append(nb, N - 1)
        rows += [np.full(len(nb), h), nb]
        cols += [nb, np.full(len(nb), h)]
    r, c = np.concatenate(rows).astype(np.int64), np.concatenate(cols).astype(np.int64)
    order = np.lexsort((c, r))
    r, c = r[order], c[order]
    xadj = np.zeros(N + 1, np.int64)
    np.cumsum(np.bincount(r, minlength=N), out=xadj[1:])
    w = (1 + (np.minimum(r, c) * 31 + np.maximum(r, c)) % 13).astype(np.int32)
    return gg.Graph(N, xadj, c.astype(np.int32), None, w, "hub rows")


@pytest.mark.parametrize("spread", [False, True])
@pytest.mark.parametrize("merge", [1, 2])
def test_rows_equal_the_oracle(kmp, spread, merge):
    g = _graph(spread)
    label = (np.arange(N) // merge * merge).astype(np.int32)
    cg, mp = kmp.contract(kmp.DeviceGraph.from_host(g), torch.from_numpy(label).cuda())
    rc, rmp = O.contract(g, label)
    h = cg.to_host()
    assert np.array_equal(mp.cpu().numpy(), rmp)
    assert np.array_equal(h.xadj, rc.xadj)
    assert np.array_equal(h.adjncy, rc.adjncy)
    assert np.array_equal(h.adjwgt, rc.adjwgt)
    assert np.array_equal(h.vwgt, rc.vwgt)
