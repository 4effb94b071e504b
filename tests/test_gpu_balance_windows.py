"""GPU tests of the balancer's commit, bit-exact against the oracle: block rooms in
shared and in global memory (k around the bound), blocks that need more
candidates than a window holds, batches whose entries exceed a window or whose
tables exceed shared memory, and blocks that only the lowest-id fallback helps."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2105_02022_gb300 import graphgen as gg

pytestmark = pytest.mark.gpu

ROOMS_IN_SMEM = 26000  # blocks


@pytest.fixture(scope="module")
def kmp():
    from paper_2105_02022_gb300 import _build
    from paper_2105_02022_gb300 import kmp as K

    _build.build_all()
    O.build()
    assert torch.cuda.is_available()
    yield K


def _case(name):
    rng = np.random.default_rng(9)
    if name.startswith("k"):  # random blocks of three nodes, a cap of four
        k = int(name[1:])
        g = gg.rgg(3 * k, 8, 3)
        return g, k, rng.integers(0, k, g.n).astype(np.int32), 4
    if name == "long":  # two blocks with nearly everything: hundreds of moves each, every batch past a window
        g, k = gg.with_weights(gg.rgg(6000, 12, 4), 4, 9, 4), 40
        part = np.where(np.arange(6000) % 3 == 0, 7, 21).astype(np.int32)
        return g, k, part, int(1.05 * g.vw().sum() / k) + 4
    if name == "dense":  # batches of more than 256 entries
        g, k = gg.random_graph(3000, 120000, 5), 30
        return g, k, (np.arange(3000) * k // 3000 * (rng.random(3000) < 0.8)).astype(np.int32), 110
    if name == "tables":  # tables of a batch above what shared memory holds
        g, k = gg.random_graph(12000, 1500000, 6), 3000
        return g, k, np.minimum(rng.integers(0, 3600, 12000), k - 1).astype(np.int32), 8
    # an isolated clique's nodes find no room next to them
    g, k = gg.with_weights(gg.random_graph(900, 4000, 7), 6, 5, 8), 90
    return g, k, (np.arange(900) // 100 * 10).astype(np.int32), int(g.vw().sum() / k) + 6


@pytest.mark.parametrize("name", ["k%d" % (ROOMS_IN_SMEM - 1), "k%d" % ROOMS_IN_SMEM, "k%d" % (ROOMS_IN_SMEM + 1), "long",
                                  "dense", "tables", "fallback"])
def test_balance_equals_the_oracle(kmp, name):
    g, k, part, cap = _case(name)
    caps = np.full(k, cap, np.int64)
    rp, rmv = O.balance(g, k, caps.astype(np.int32), part)
    pt = torch.from_numpy(part.copy()).cuda()
    mv = kmp.balance(kmp.DeviceGraph.from_host(g), k, caps, pt)
    assert mv == rmv and mv > 0
    assert np.array_equal(pt.cpu().numpy(), rp)
