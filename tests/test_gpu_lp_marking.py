"""GPU tests of neighbour marking after moves, bit-exact against the oracle: rows around
the lengths that a warp marks itself and that a CTA takes, in the one-launch run, below
and above the size where the longer limit holds."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2105_02022_gb300 import graphgen as gg

pytestmark = pytest.mark.gpu

ROWS = [31, 32, 33, 95, 96, 97, 128, 255, 256, 257, 300]


def _hubs(n, copies, seed, limit):
    """A sparse random background, and `copies` nodes of each row length up to `limit`."""
    rng = np.random.default_rng(seed)
    deg = np.repeat([r for r in ROWS if r <= limit], copies)
    h = len(deg)
    hub = np.repeat(np.arange(h), deg)
    other = np.concatenate([h + rng.choice(n - h, d, replace=False) for d in deg])
    a, b = rng.integers(h, n, (2, n))
    code = np.concatenate([hub * n + other, np.minimum(a, b)[a != b] * n + np.maximum(a, b)[a != b]])
    code = np.unique(code)
    u, v = code // n, code % n
    r, c = np.concatenate([u, v]), np.concatenate([v, u])
    order = np.lexsort((c, r))
    xadj = np.zeros(n + 1, np.int64)
    np.cumsum(np.bincount(r, minlength=n), out=xadj[1:])
    return gg.Graph(n, xadj, c[order].astype(np.int32), None, None, "hubs")


@pytest.mark.parametrize("n,copies,limit", [(4000, 3, 256), (4000, 40, 300), (60000, 60, 300), ((1 << 19) - 1, 30, 300),
                                            (1 << 19, 30, 300)])
def test_marking(n, copies, limit):
    from paper_2105_02022_gb300 import _build, kmp

    _build.build_all()
    O.build()
    g = _hubs(n, copies, n, limit)
    dg = kmp.DeviceGraph.from_host(g)
    U = 50
    assert np.array_equal(kmp.coarsen_level(dg, U, 5, 3, 0).cpu().numpy(), O.cluster(g, U, 5, 3, 0))
    k = 9
    part = (np.arange(n) % k).astype(np.int32)
    cap = np.full(k, int(1.1 * n / k) + 4, np.int64)
    pt = torch.from_numpy(part.copy()).cuda()
    cut = kmp.refine(dg, k, cap, 5, 4, pt)
    rp, rcut = O.refine(g, k, cap.astype(np.int32), 5, 4, part)
    assert np.array_equal(pt.cpu().numpy(), rp) and cut == rcut
