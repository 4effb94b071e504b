"""GPU tests of the cut's outputs: block weights below and above the number that comes
back in one copy, with and without them, and block ids out of range, which leave the
caller's arrays alone."""
import ctypes

import numpy as np
import pytest
import torch

import oracle as O
from paper_2105_02022_gb300 import graphgen as gg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1, 2, 4097, 16383, 16384, 16385, 1 << 20])
@pytest.mark.parametrize("weighted", [False, True])
def test_cut_and_weights(k, weighted):
    from paper_2105_02022_gb300 import _build, kmp

    _build.build_all()
    O.build()
    g = gg.rgg(9000, 8, 3)
    if weighted:
        g = gg.with_weights(g, 5, 9, 2)
    dg = kmp.DeviceGraph.from_host(g)
    part = np.random.default_rng(k).integers(0, k, g.n).astype(np.int32)
    pt = torch.from_numpy(part).cuda()
    ref = O.cut(g, part)
    cut, bw = kmp.cut(dg, pt, k)
    assert cut == ref
    assert np.array_equal(bw, np.bincount(part, weights=g.vw(), minlength=k).astype(np.int64))
    kmp_cut, c = kmp.load().kmp_cut, ctypes.c_int64(-7)
    p = ctypes.c_void_p(pt.data_ptr())
    assert kmp_cut(dg.h, p, k, ctypes.byref(c), None) == 0 and c.value == ref
    out = np.full(k, -7, np.int64)
    assert kmp_cut(dg.h, p, k, None, out.ctypes.data_as(ctypes.c_void_p)) == 0 and np.array_equal(out, bw)
    for wrong in (-1, k):
        pt[17] = wrong
        c, out = ctypes.c_int64(-7), np.full(k, -7, np.int64)
        assert kmp_cut(dg.h, p, k, ctypes.byref(c), out.ctypes.data_as(ctypes.c_void_p)) == kmp.KMP_ERR_ARG
        assert c.value == -7 and np.all(out == -7)
