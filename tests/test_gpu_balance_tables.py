"""GPU tests of where the balancer's large batches keep their tables, bit-exact against
the oracle: beside the windows with fewer members than the overload asks for, over the
windows, which are then read again with a block under way, and in global memory."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2105_02022_gb300 import graphgen as gg

pytestmark = pytest.mark.gpu

SMEM, WINDOWS, SMALL, ROOMS_K, FIT = 224000, 97792, 16384, 26000, 4  # bytes; blocks; members
OVER = WINDOWS // 8 & ~31  # slots over the windows


def _slots(k):
    return (SMEM - WINDOWS - SMALL - (4 * k if k <= ROOMS_K else 0)) // 8 & ~31


def _table(degree, k):
    t = 32
    while t < 2 * min(degree, k):
        t *= 2
    return t


def _heavy(n, k, blocks, per_block, degree, seed):
    """`blocks` blocks of `per_block` nodes of about `degree` neighbours, linked densely inside
    (batches stop early), and light nodes spread over all other blocks."""
    rng = np.random.default_rng(seed)
    h = blocks * per_block
    u = np.repeat(np.arange(h), degree)
    v = rng.integers(h, n, len(u))
    a, b = np.meshgrid(np.arange(per_block), np.arange(per_block))
    inside = [np.stack([a[a < b], b[a < b]]) + i * per_block for i in range(blocks)]
    inside = np.concatenate(inside, 1)[:, rng.random(blocks * per_block * (per_block - 1) // 2) < 0.4]
    u, v = np.concatenate([u, inside[0]]), np.concatenate([v, inside[1]])
    code = np.unique(np.minimum(u, v).astype(np.int64) * n + np.maximum(u, v))
    u, v = code // n, code % n
    r, c = np.concatenate([u, v]), np.concatenate([v, u])
    order = np.lexsort((c, r))
    xadj = np.zeros(n + 1, np.int64)
    np.cumsum(np.bincount(r, minlength=n), out=xadj[1:])
    g = gg.with_weights(gg.Graph(n, xadj, c[order].astype(np.int32), None, None, "heavy"), 0, 7, seed)
    part = np.empty(n, np.int32)
    ids = np.sort(rng.choice(k, blocks, replace=False))
    part[:h] = np.repeat(ids, per_block)
    rest = np.setdiff1d(np.arange(k), ids)
    part[h:] = rest[rng.integers(0, len(rest), n - h)]
    return g, part


@pytest.mark.parametrize("name", ["beside", "over", "global", "mixed"])
def test_tables(name):
    from paper_2105_02022_gb300 import _build, kmp

    _build.build_all()
    O.build()
    if name == "beside":  # more members than fit, at least FIT of them
        k, degree, per_block, room = 300, 280, 90, 40
        assert FIT * _table(400, k) <= _slots(k) < 32 * _table(260, k)
        g, part = _heavy(4000, k, 12, per_block, degree, 1)
    elif name == "over":  # fewer than FIT fit; two to five members over the windows
        k, degree, per_block, room = 20000, 700, 9, 5
        assert FIT * _table(520, k) > _slots(k) and _slots(k) < 2 * _table(520, k) and 5 * _table(1000, k) <= OVER
        g, part = _heavy(40000, k, 60, per_block, degree, 2)
    elif name == "global":  # one member's table alone exceeds what lies over the windows
        k, degree, per_block, room = 20000, 7000, 9, 5
        assert _table(6200, k) > OVER
        g, part = _heavy(60000, k, 40, per_block, degree, 3)
    else:  # rooms in global memory, members of all sizes
        k, degree, per_block, room = 26001, 1500, 14, 6
        g, part = _heavy(60000, k, 50, per_block, degree, 4)
    size = np.bincount(part, minlength=k)
    # the heavy blocks have to give up nodes, and every other block has room for one or two
    cap = np.where(size >= per_block, room, size + 1 + np.arange(k) % 2).astype(np.int64)
    rp, rmv = O.balance(g, k, cap.astype(np.int32), part)
    pt = torch.from_numpy(part.copy()).cuda()
    mv = kmp.balance(kmp.DeviceGraph.from_host(g), k, cap, pt)
    assert mv == rmv and mv >= 100
    assert np.array_equal(pt.cpu().numpy(), rp)
