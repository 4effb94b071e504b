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


def _multi(g, seed, unit=False, mixed=False):
    """g with one to three more entries, of other weights, for half of its pairs; rows by id, or
    mixed, so that the entries of a pair lie apart."""
    rng = np.random.default_rng(seed)
    src = np.repeat(np.arange(g.n), np.diff(g.xadj))
    low = src < g.adjncy
    u, v, w = src[low], g.adjncy[low], g.ew()[low]
    more = np.where(rng.random(len(u)) < 0.5, rng.integers(1, 4, len(u)), 0)
    u, v = np.repeat(u, more + 1), np.repeat(v, more + 1)
    w = np.concatenate([w, rng.integers(1, 12, more.sum())])[: len(u)]
    r, c, w = np.concatenate([u, v]), np.concatenate([v, u]), np.concatenate([w, w])
    order = np.lexsort((rng.random(len(c)) if mixed else c, r))
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


@pytest.mark.parametrize("unit,mixed", [(False, False), (True, False), (False, True)])
@pytest.mark.parametrize("n,deg", [(60, 6), (300, 8), (1500, 10), (6000, 8)])
def test_bipartition(kmp, n, deg, unit, mixed):
    """Items whose levels FM holds in shared memory or in scratch; a heavy one whose
    keys do not pack."""
    graphs = [_multi(gg.with_weights(gg.rgg(n, deg, n + i), 5, 9, i), i, unit, mixed) for i in range(6)]
    if n == 300 and not unit:
        graphs.append(_multi(gg.with_weights(gg.random_graph(400, 1200, 3), 5, 1 << 18, 2), 9, False, mixed))
    xs, at = [np.zeros(1, np.int64)], 0
    for g in graphs:
        xs.append(g.xadj[1:] + at)
        at += g.m_directed
    off = np.cumsum([0] + [g.n for g in graphs])
    u = gg.Graph(int(off[-1]), np.concatenate(xs), np.concatenate([g.adjncy + o for g, o in zip(graphs, off)]).astype(np.int32),
                 np.concatenate([g.vw() for g in graphs]).astype(np.int32),
                 None if unit else np.concatenate([g.ew() for g in graphs]).astype(np.int32))
    part = np.repeat(np.arange(len(graphs), dtype=np.int32), np.diff(off))
    caps = []
    for g in graphs:
        c = int(g.vw().sum())
        caps += [c // 2, c - c // 2, int(1.03 * ((c + 1) // 2)), int(1.03 * ((c + 1) // 2))]
    out = torch.from_numpy(part.copy()).cuda()
    kmp.bipartition_each(kmp.DeviceGraph.from_host(u), len(graphs), np.array(caps, np.int32), 31, out)
    got = out.cpu().numpy()
    for i, g in enumerate(graphs):
        t0, t1, L0, L1 = caps[4 * i: 4 * i + 4]
        side, _ = O.bipartition(g, L0, L1, t0, t1, O.step(31, i), O.config())
        assert np.array_equal(got[part == i], 2 * i + side), i


@pytest.mark.parametrize("k", [2, 16])
def test_partition(kmp, k):
    g = _multi(gg.with_weights(gg.rgg(4000, 8, 2), 3, 9, 4), 5)
    part, rc, st = kmp.partition_graph(kmp.DeviceGraph.from_host(g), k, 0.03, 3)
    rp, rrc, _ = O.partition(g, k, 0.03, 3)
    assert rc == rrc
    assert np.array_equal(part.cpu().numpy(), rp)
    assert st.cut == O.cut(g, rp)
