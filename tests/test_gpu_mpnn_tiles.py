"""GPU tests of the proposer's tiled kernels at their edges: node totals around
a 64-node tile, graphs below, at and above the size whose hop counts stay in
shared memory, hub rows longer than the unrolled loads.  Features and scores
are bit-exact; gradients sum at most a few thousand products per partial sum,
each rounded to 2^-24 of itself, which stays below 1e-4 of the largest."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2105_02022_gb300 import graphgen as gg

pytestmark = pytest.mark.gpu

HOPS_IN_SMEM = 12288  # nodes


@pytest.fixture(scope="module")
def kmp():
    from paper_2105_02022_gb300 import _build
    from paper_2105_02022_gb300 import kmp as K

    _build.build_all()
    O.build()
    assert torch.cuda.is_available()
    yield K


def _graphs(name):
    if name == "one":
        return [gg.from_edges(1, [])]
    if name in ("63", "64", "65", "129"):
        return [gg.with_weights(gg.random_graph(int(name), 3 * int(name), 5), 9, 13, 6)]
    if name == "hub_rows":
        return [gg.with_weights(gg.hubs(500, [3, 5, 90, 400], 700, 4), 5, 30, 5), gg.grid(5, 7)]
    return [gg.with_weights(gg.rgg(n, 8, n), 7, 30, 3) for n in (HOPS_IN_SMEM - 1, HOPS_IN_SMEM, HOPS_IN_SMEM + 1)]


@pytest.mark.parametrize("name", ["one", "63", "64", "65", "129", "hub_rows", "hop_bound"])
def test_tiles_and_hops(kmp, name):
    graphs = _graphs(name)
    keys = [O.key(7, [i]) for i in range(len(graphs))]
    rng = np.random.default_rng(7)
    sides = [rng.integers(0, 2, g.n).astype(np.int32) for g in graphs]
    b = kmp.Batch.from_graphs(graphs, keys, sides)
    P = torch.from_numpy(rng.normal(0, 0.25, O.mpnn_num_params()).astype(np.float32)).bfloat16().float().numpy()
    m = kmp.Mpnn(1)
    try:
        m.set_params(P)
        S, X = m.forward(b, features=True)
        loss, grad = m.gradients(b)
    finally:
        m.free()
    gref, lref = np.zeros(O.mpnn_num_params()), 0.0
    for i, g in enumerate(graphs):
        lo, hi = b.noff[i], b.noff[i + 1]
        F = O.mpnn_features(g, keys[i])
        assert np.array_equal(X[lo:hi], F.astype(np.float32)), i
        assert np.array_equal(S[lo:hi], O.mpnn_scores_f32(g, keys[i], P)), i
        L, gS = O.mpnn_loss(O.mpnn_forward(g, F, P.astype(np.float64)), sides[i])
        lref += L / len(graphs)
        gref += O.mpnn_backward(g, F, P.astype(np.float64), gS) / len(graphs)
    assert loss == pytest.approx(lref, rel=1e-5)
    assert np.max(np.abs(grad - gref)) <= 1e-4 * np.max(np.abs(gref))
