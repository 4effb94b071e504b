"""GPU test of the bipartitioner's scratch: one large item beside hundreds of tiny
ones takes the memory of its parts, not the largest item's for every CTA."""
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


def test_one_large_item_beside_many_tiny_ones(kmp):
    graphs = [gg.with_weights(gg.grid(2 + i % 5, 3), 3, 9, i) for i in range(600)]
    at = 417  # not the first block
    graphs.insert(at, gg.with_weights(gg.rgg(60000, 8, 5), 3, 9, 5))
    off = np.cumsum([0] + [g.n for g in graphs])
    xs, e = [np.zeros(1, np.int64)], 0
    for g in graphs:
        xs.append(g.xadj[1:] + e)
        e += g.m_directed
    u = gg.Graph(int(off[-1]), np.concatenate(xs),
                 np.concatenate([g.adjncy + o for g, o in zip(graphs, off)]).astype(np.int32),
                 np.concatenate([g.vw() for g in graphs]).astype(np.int32),
                 np.concatenate([g.ew() for g in graphs]).astype(np.int32))
    part = np.repeat(np.arange(len(graphs), dtype=np.int32), np.diff(off))
    caps = []
    for g in graphs:
        c = int(g.vw().sum())
        caps += [c // 2, c - c // 2, int(1.03 * ((c + 1) // 2)) + 1, int(1.03 * ((c + 1) // 2)) + 1]
    dg = kmp.DeviceGraph.from_host(u)
    out = torch.from_numpy(part.copy()).cuda()
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    kmp.bipartition_each(dg, len(graphs), np.array(caps, np.int32), 5, out)
    # the regions of all items together are below 0.2 GB; the library's pool keeps what it took
    assert before - torch.cuda.mem_get_info()[0] < 1 << 30
    got = out.cpu().numpy()
    for i in [0, 1, 150, 151, 443, 444, 445, 600, at]:
        t0, t1, L0, L1 = caps[4 * i: 4 * i + 4]
        side, _ = O.bipartition(graphs[i], L0, L1, t0, t1, O.step(5, i), O.config())
        assert np.array_equal(got[part == i], 2 * i + side), i
