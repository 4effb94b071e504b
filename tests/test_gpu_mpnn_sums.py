"""GPU test of the proposer's features where weights sum to a negative number:
equal to the oracle's (whole sums, as doubles)."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2105_02022_gb300 import graphgen as gg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("which", ["edges", "nodes", "both"])
def test_negative_weight_sums(which):
    from paper_2105_02022_gb300 import _build, kmp

    _build.build_all()
    O.build()
    g = gg.with_weights(gg.rgg(500, 8, 3), 6, 9, 2)
    if which != "nodes":
        g.adjwgt = (g.adjwgt - 20).astype(np.int32)
    if which != "edges":
        g.vwgt = (g.vwgt - 9).astype(np.int32)
    key = O.key(7, [1])
    b = kmp.Batch.from_graphs([g], [key], [np.zeros(g.n, np.int32)])
    m = kmp.Mpnn(1)
    try:
        X = m.forward(b, features=True)[1]
    finally:
        m.free()
    assert np.array_equal(X, O.mpnn_features(g, key).astype(np.float32))
