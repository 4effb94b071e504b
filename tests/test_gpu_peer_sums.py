"""GPU test of ratings of short weighted rows, bit-exact against the oracle: every row
length up to 32, with label sets from one that holds all neighbours to one of each."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2105_02022_gb300 import graphgen as gg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1, 2, 3, 5, 17, 40, 2000])
@pytest.mark.parametrize("copies", [20, 300])  # the one-launch run, and the separate kernels
def test_rows_and_label_sets(k, copies):
    from paper_2105_02022_gb300 import _build, kmp

    _build.build_all()
    O.build()
    rng = np.random.default_rng(k)
    length = np.repeat(np.arange(1, 33), copies)
    h, n = len(length), 3 * len(length)
    hub = np.repeat(np.arange(h), length)
    other = np.concatenate([h + rng.choice(n - h, d, replace=False) for d in length])
    r, c = np.concatenate([hub, other]), np.concatenate([other, hub])
    order = np.lexsort((c, r))
    xadj = np.zeros(n + 1, np.int64)
    np.cumsum(np.bincount(r, minlength=n), out=xadj[1:])
    g = gg.with_weights(gg.Graph(n, xadj, c[order].astype(np.int32), None, None, "rows"), 3, 1 << 14, 5)
    assert set(range(1, 33)) <= set(np.diff(g.xadj).tolist())
    part = rng.integers(0, k, n).astype(np.int32)
    cap = np.full(k, int(1.3 * g.vw().sum() / k) + 4, np.int64)
    pt = torch.from_numpy(part.copy()).cuda()
    dg = kmp.DeviceGraph.from_host(g)
    cut = kmp.refine(dg, k, cap, 3, 4, pt)
    rp, rcut = O.refine(g, k, cap.astype(np.int32), 3, 4, part)
    assert np.array_equal(pt.cpu().numpy(), rp) and cut == rcut
    U = 40
    assert np.array_equal(kmp.coarsen_level(dg, U, 4, 6, 0).cpu().numpy(), O.cluster(g, U, 4, 6, 0))
