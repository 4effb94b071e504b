"""GPU tests of graphs in which a pair of nodes is joined by several entries: their
weights count together everywhere, bit-exact against the oracle."""
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
    K.set_config(K.config())
    yield K


def _multi(g, seed, unit=False):
    """g with one to three more entries, of other weights, for half of its pairs."""
    rng = np.random.default_rng(seed)
    src = np.repeat(np.arange(g.n), np.diff(g.xadj))
    low = src < g.adjncy
    u, v, w = src[low], g.adjncy[low], g.ew()[low]
    more = np.where(rng.random(len(u)) < 0.5, rng.integers(1, 4, len(u)), 0)
    u, v = np.repeat(u, more + 1), np.repeat(v, more + 1)
    w = np.concatenate([w, rng.integers(1, 12, more.sum())])[: len(u)]
    r, c, w = np.concatenate([u, v]), np.concatenate([v, u]), np.concatenate([w, w])
    order = np.lexsort((c, r))
    xadj = np.zeros(g.n + 1, np.int64)
    np.cumsum(np.bincount(r, minlength=g.n), out=xadj[1:])
    return gg.Graph(g.n, xadj, c[order].astype(np.int32), g.vwgt, None if unit else w[order].astype(np.int32), "multi")


@pytest.mark.parametrize("unit", [False, True])
@pytest.mark.parametrize("n,deg,k", [(3000, 6, 200), (3000, 10, 60), (20000, 8, 1500)])
def test_balance(kmp, n, deg, k, unit):
    g = _multi(gg.rgg(n, deg, n + k), 3, unit)
    rng = np.random.default_rng(k)
    # neighbouring blocks overloaded, so that batches hold members next to one another
    part = (np.arange(n) * k // n).astype(np.int32)
    part = np.where(rng.random(n) < 0.5, part // 3 * 3, part).astype(np.int32)
    cap = np.full(k, int(1.1 * g.vw().sum() / k) + 2, np.int64)
    rp, rmv = O.balance(g, k, cap.astype(np.int32), part)
    pt = torch.from_numpy(part.copy()).cuda()
    mv = kmp.balance(kmp.DeviceGraph.from_host(g), k, cap, pt)
    assert mv == rmv and mv > 100
    assert np.array_equal(pt.cpu().numpy(), rp)
