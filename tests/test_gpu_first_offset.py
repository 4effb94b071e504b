"""GPU tests of device graphs whose first offset is above 0: the entries before it
belong to no row, so every call answers as for the same rows from offset 0.  (They
hold node ids here, with heavy weights: counted, they would show.)"""
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


def _handles(kmp, g, shift):
    """The graph's handle, and one whose rows start `shift` entries into the arrays."""
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    lead = np.arange(shift) % g.n
    adj = np.concatenate([lead, g.adjncy]).astype(np.int32)
    ew = None if g.adjwgt is None else dev(np.concatenate([np.full(shift, 1 << 20), g.adjwgt]).astype(np.int32))
    vw = None if g.vwgt is None else dev(g.vwgt)
    return (kmp.DeviceGraph.from_host(g),
            kmp.DeviceGraph.from_device(g.n, dev(g.xadj + shift), dev(adj), vw, ew))


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("shift", [1, 31, 2047, 2048, 2049, 100003])
def test_calls_equal_those_from_offset_zero(kmp, shift, weighted):
    g = gg.rgg(5000, 8, 3)
    if weighted:
        g = gg.with_weights(g, 4, 9, 2)
    a, b = _handles(kmp, g, shift)
    k = 6
    part = (np.arange(g.n) * 5 % k).astype(np.int32)
    pt = torch.from_numpy(part).cuda()
    cut, bw = kmp.cut(b, pt, k)
    assert cut == O.cut(g, part)
    assert np.array_equal(bw, np.bincount(part, weights=g.vw(), minlength=k).astype(np.int64))
    caps = np.full(k, int(1.1 * g.vw().sum() / k) + 4, np.int64)
    pa, pb = pt.clone(), pt.clone()
    assert kmp.refine(a, k, caps, 3, 5, pa) == kmp.refine(b, k, caps, 3, 5, pb) == O.cut(g, pb.cpu().numpy())
    assert torch.equal(pa, pb)
    U = 60 * int(g.vw().max())
    la, lb = kmp.coarsen_level(a, U, 3, 5, 0), kmp.coarsen_level(b, U, 3, 5, 0)
    assert torch.equal(la, lb)
    ha, hb = kmp.contract(a, la)[0].to_host(), kmp.contract(b, lb)[0].to_host()
    for x in ("xadj", "adjncy", "vwgt", "adjwgt"):
        assert np.array_equal(getattr(ha, x), getattr(hb, x))
    (qa, ra, sa), (qb, rb, sb) = kmp.partition_graph(a, k, 0.03, 5), kmp.partition_graph(b, k, 0.03, 5)
    assert torch.equal(qa, qb) and ra == rb
    assert sa.cut == sb.cut == O.cut(g, qb.cpu().numpy())
