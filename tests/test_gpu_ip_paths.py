"""GPU tests of the bipartitioner's paths, bit-exact against the oracle: FM keys
that pack gain and id and the plain ones for weights too large to pack, FM and LP
state in shared memory and in scratch (item sizes around the bounds), entries in
shared and global memory, unit and weighted items, rows beyond the shared hash
tables, caps that no node or almost none fits."""
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
    K.set_config(K.config())


def _union(graphs):
    """Disjoint union, the graph index of every node, and per-graph totals."""
    xs, adj, vw, ew, part = [np.zeros(1, np.int64)], [], [], [], []
    nb = eb = 0
    for i, g in enumerate(graphs):
        xs.append(np.asarray(g.xadj[1:]) + eb)
        adj.append(np.asarray(g.adjncy) + nb)
        vw.append(g.vw())
        ew.append(g.ew())
        part.append(np.full(g.n, i, np.int32))
        nb, eb = nb + g.n, eb + len(g.adjncy)
    unit = all(g.adjwgt is None for g in graphs)
    u = gg.Graph(nb, np.concatenate(xs), np.concatenate(adj).astype(np.int32), np.concatenate(vw).astype(np.int32),
                 None if unit else np.concatenate(ew).astype(np.int32))
    return u, np.concatenate(part)


def _graphs(name):
    if name == "sizes":  # more items than SMs; LP state leaves shared memory above 2300 nodes, FM's above 3550
        big = [gg.with_weights(gg.rgg(n, 8, n), 3, 9, 1) for n in (2290, 2330, 3540, 3570, 5000)]
        return big + [gg.with_weights(gg.grid(3 + i % 4, 4), 2, 5, i) for i in range(160)]
    if name == "unit":  # no edge weights stored; one item per SM at most, entries in shared memory or not
        return [gg.rgg(n, d, 3) for n, d in ((1500, 8), (4000, 16), (127, 6), (128, 6), (129, 6), (2, 1), (1, 1))]
    if name == "heavy":  # weighted degrees that do not pack with the id into 31 bits, and ones that just do
        return [gg.with_weights(gg.random_graph(400, 1200, 3), 5, 1 << 19, 2),
                gg.with_weights(gg.random_graph(400, 1200, 4), 5, 1 << 16, 2)]
    if name == "hubs":  # rows above the shared tables of 256 and 512 slots
        return [gg.with_weights(gg.hubs(1800, [100, 127, 128, 129, 255, 257, 600], 4000, 4), 4, 20, 5),
                gg.hubs(900, [300, 300, 500], 1500, 5)]
    return [gg.with_weights(gg.rgg(600, 8, 5), 60, 9, 5), gg.with_weights(gg.random_graph(90, 300, 5), 200, 9, 6)]


@pytest.mark.parametrize("name,slack", [("sizes", 1.03), ("unit", 1.03), ("heavy", 1.03), ("hubs", 1.03), ("tight", 1.0),
                                        ("tight", 0.6)])
def test_items_equal_the_oracle(kmp, name, slack):
    graphs = _graphs(name)
    u, part = _union(graphs)
    caps = []
    for g in graphs:
        c = int(g.vw().sum())
        t0 = c // 2
        L = max(int(slack * ((c + 1) // 2)), 1)
        caps += [t0, c - t0, L, L]
    caps = np.array(caps, np.int32)
    out = torch.from_numpy(part.copy()).cuda()
    kmp.bipartition_each(kmp.DeviceGraph.from_host(u), len(graphs), caps, 77, out)
    got = out.cpu().numpy()
    for i, g in enumerate(graphs):
        t0, t1, L0, L1 = (int(x) for x in caps[4 * i: 4 * i + 4])
        side, _ = O.bipartition(g, L0, L1, t0, t1, O.step(77, i), O.config())
        assert np.array_equal(got[part == i], 2 * i + side), (name, i)
