"""GPU tests of the LP schedule's size classes, bit-exact against the oracle: degrees
at the edges of the rating classes (a warp's table, a CTA's, a wide CTA's, hubs),
graphs at the edge of the one-CTA run, few and many labels, unit and weighted."""
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


def _stars(degrees, n, seed):
    """A sparse random background on nodes from len(degrees) on, and hub h joined to exactly degrees[h] of them."""
    rng = np.random.default_rng(seed)
    h = len(degrees)
    pairs = [np.stack([np.full(d, i), rng.choice(np.arange(h, n), d, replace=False)]) for i, d in enumerate(degrees)]
    a, b = rng.integers(h, n, (2, n))
    e = np.concatenate(pairs + [np.stack([a, b])[:, a != b]], 1)
    e = np.unique(np.sort(e, 0), axis=1)
    r, c = np.concatenate([e[0], e[1]]), np.concatenate([e[1], e[0]])
    order = np.lexsort((c, r))
    xadj = np.zeros(n + 1, np.int64)
    np.cumsum(np.bincount(r, minlength=n), out=xadj[1:])
    return gg.Graph(n, xadj, c[order].astype(np.int32), None, None, "stars")


CLASSES = [4, 5, 8, 9, 16, 17, 32, 33, 256, 257, 2048, 2049, 8191, 8192, 8193, 12000]


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("what", ["coarsen", "refine_few", "refine_many"])
def test_degree_classes(kmp, what, weighted):
    g = _stars(CLASSES, 20000, 3)
    assert list(np.diff(g.xadj)[: len(CLASSES)]) == CLASSES
    if weighted:
        g = gg.with_weights(g, 5, 40, 3)
    dg = kmp.DeviceGraph.from_host(g)
    if what == "coarsen":
        U = max(60, int(g.vw().max()))
        label = kmp.coarsen_level(dg, U, 5, 9, 0).cpu().numpy()
        assert np.array_equal(label, O.cluster(g, U, 5, 9, 0))
        return
    k = 500 if what == "refine_few" else 3000
    part = np.random.default_rng(5).integers(0, k, g.n).astype(np.int32)
    cap = np.full(k, int(1.1 * g.vw().sum() / k) + 6, np.int64)
    pt = torch.from_numpy(part.copy()).cuda()
    cut = kmp.refine(dg, k, cap, 3, 4, pt)
    rp, rcut = O.refine(g, k, cap.astype(np.int32), 3, 4, part)
    assert np.array_equal(pt.cpu().numpy(), rp)
    assert cut == rcut


@pytest.mark.parametrize("n,hub", [(4095, 256), (4096, 256), (4097, 256), (4096, 257), (300, 200), (2, 1)])
@pytest.mark.parametrize("weighted", [False, True])
def test_small_runs(kmp, n, hub, weighted):
    g = gg.path(2) if n == 2 else _stars([hub, 40, 33], n, n)
    if weighted:
        g = gg.with_weights(g, 6, 30, 2)
    dg = kmp.DeviceGraph.from_host(g)
    for U in (int(g.vw().max()), 25 * int(g.vw().max())):  # a cap that most targets exceed, and one that leaves room
        label, fav = kmp.coarsen_level(dg, U, 5, 11, 1, fav=True)
        assert np.array_equal(label.cpu().numpy(), O.cluster(g, U, 5, 11, 1))
    k = min(7, n)
    part = (np.arange(g.n) * k // g.n).astype(np.int32)
    cap = np.full(k, int(1.03 * g.vw().sum() / k) + 2, np.int64)
    pt = torch.from_numpy(part.copy()).cuda()
    cut = kmp.refine(dg, k, cap, 5, 4, pt)
    rp, rcut = O.refine(g, k, cap.astype(np.int32), 5, 4, part)
    assert np.array_equal(pt.cpu().numpy(), rp)
    assert cut == rcut
