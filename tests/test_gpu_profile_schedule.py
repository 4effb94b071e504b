"""GPU test of the rating profile: with it on, a call launches the same kernels as
without it but for the one that saves a round's bin offsets, and every sub-round of a
small graph's one-launch run is counted."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2105_02022_gb300 import graphgen as gg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("n", [2, 300, 4096])
def test_small_runs_keep_their_schedule(n, weighted):
    from paper_2105_02022_gb300 import _build, kmp

    _build.build_all()
    O.build()
    g = gg.path(2) if n == 2 else gg.rgg(n, 6, 5)
    if weighted:
        g = gg.with_weights(g, 3, 9, 4)
    dg = kmp.DeviceGraph.from_host(g)
    k = 2
    plain, _, st0 = kmp.partition_graph(dg, k, 0.03, 7)
    rounds = st0.lp_rounds_run
    kmp.set_profiling(True)
    try:
        kmp.profile_read(reset=True)
        prof, _, st1 = kmp.partition_graph(dg, k, 0.03, 7)
        p = kmp.profile_read(reset=True)
    finally:
        kmp.set_profiling(False)
    assert torch.equal(plain, prof)
    assert st0.gpu_launches == st1.gpu_launches  # every level runs in one launch a call
    S = kmp.get_config().subrounds
    assert p.stage_spans % S == 0 and p.stage_spans >= S * rounds
    assert p.rate_launches == p.stage_spans
    assert 0 < p.rate_ms <= p.stage_ms < st1.ms_total
    entries = st1.lp_scanned + st1.refine_scanned
    per_entry = 12 if weighted else 8
    assert p.stage_bytes >= entries * per_entry  # and the nodes' share
    assert p.stage_bytes <= entries * (per_entry + 28)
