"""GPU tests of the one-launch LP run's bounds on entries: bit-exact against the oracle on
both sides of them, and a dense graph of as few nodes takes the kernels of all SMs."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2105_02022_gb300 import graphgen as gg

pytestmark = pytest.mark.gpu

ENTRIES = [49152, 65536]  # clustering, refinement


@pytest.fixture(scope="module")
def kmp():
    from paper_2105_02022_gb300 import _build
    from paper_2105_02022_gb300 import kmp as K

    _build.build_all()
    O.build()
    assert torch.cuda.is_available()
    K.set_config(K.config())
    yield K


def _random(n, edges, seed):
    """A simple random graph of exactly `edges` edges."""
    rng = np.random.default_rng(seed)
    code = rng.choice(n * (n - 1) // 2, edges, replace=False)
    u = (np.sqrt(2 * code + 0.25) + 0.5).astype(np.int64)  # pair (u, v), v < u, at u (u - 1) / 2 + v
    v = code - u * (u - 1) // 2
    r, c = np.concatenate([u, v]), np.concatenate([v, u])
    order = np.lexsort((c, r))
    xadj = np.zeros(n + 1, np.int64)
    np.cumsum(np.bincount(r, minlength=n), out=xadj[1:])
    return gg.Graph(n, xadj, c[order].astype(np.int32), None, None, "random")


@pytest.mark.parametrize("n", [500, 1500, 4096])
@pytest.mark.parametrize("edges", [e // 2 + x for e in ENTRIES for x in (0, 1)])
@pytest.mark.parametrize("weighted", [False, True])
def test_both_sides_of_the_bound(kmp, n, edges, weighted):
    g = _random(n, edges, n)
    assert g.m_directed == 2 * edges and np.diff(g.xadj).max() <= 256
    if weighted:
        g = gg.with_weights(g, 4, 20, 3)
    dg = kmp.DeviceGraph.from_host(g)
    U = 12 * int(g.vw().max())
    assert np.array_equal(kmp.coarsen_level(dg, U, 5, 3, 0).cpu().numpy(), O.cluster(g, U, 5, 3, 0))
    k = 5
    part = (np.arange(n) * k // n).astype(np.int32)
    cap = np.full(k, int(1.05 * g.vw().sum() / k) + 4, np.int64)
    pt = torch.from_numpy(part.copy()).cuda()
    cut = kmp.refine(dg, k, cap, 5, 4, pt)
    rp, rcut = O.refine(g, k, cap.astype(np.int32), 5, 4, part)
    assert np.array_equal(pt.cpu().numpy(), rp) and cut == rcut


def test_dense_graphs_use_the_whole_gpu(kmp):
    """5 rounds of 8 sub-rounds of the separate kernels are hundreds of launches; a sparse
    graph of as many nodes has about a hundred in its whole partition."""
    sparse, dense = gg.rgg(4096, 6, 5), _random(4096, 200000, 5)
    assert np.diff(dense.xadj).max() <= 256
    launches = [kmp.partition_graph(kmp.DeviceGraph.from_host(g), 2, 0.03, 7)[2].gpu_launches for g in (sparse, dense)]
    assert launches[0] < 200 < launches[1] - 200
