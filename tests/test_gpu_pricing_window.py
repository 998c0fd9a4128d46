"""Candidate sets around and beyond the fixed capacity of the pricing selection: pass 2 gathers nothing
when its bound already exceeds the capacity (the host then redoes it with an exact-size buffer or, for a
flooded FP32 window, in FP64), and the selection is the oracle's on both sides of the line."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import costs, pricing
from tests import gpu_util as U

pytestmark = pytest.mark.gpu

NONE = np.zeros(0, np.int32)
TILE = 1024                      # candidates per sort tile


def capacity(kmax):
    """The fixed capacity: four times kmax in whole tiles, 8 to 128 of them."""
    return min(max(-(-4 * kmax // TILE), 8), 128) * TILE


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _one_column(m, count, seed):
    """m sources and two targets, exactly `count` pairs of negative reduced cost, all in column 0, about
    -1.9 .. -1.1 (one octave, so that they share bins), no pair near zero."""
    x, y = np.arange(m, dtype=np.int32) % 400, np.arange(m, dtype=np.int32) // 400
    tx, ty = np.array([0, 40], np.int32), np.array([0, 60], np.int32)
    rng = np.random.default_rng(seed)
    below = np.zeros(m, bool)
    below[rng.permutation(m)[:count]] = True
    u = x.astype(float) ** 2 + y.astype(float) ** 2 + np.where(below, np.round(1.1 + 0.8 * rng.random(m), 3), -2e4)
    return x, y, tx, ty, u, np.array([0.0, -1e7])


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("kmax,over", [(1000, -1), (1000, 0), (1000, 1), (5000, 0), (5000, 1), (40000, 0),
                                       (40000, 1)])
def test_selection_at_the_capacity(kmax, over, precision):
    """The gather bound is exactly the number of negative pairs (kmax is above it) or, for kmax below it, at
    most that; capacity - 1, capacity, capacity + 1."""
    from paper_2206_11009_gb300 import price_topk
    for km, count in ((kmax, capacity(kmax) + over), (capacity(kmax) // 4, capacity(kmax) + over)):
        m = count + 5000
        sx, sy, tx, ty, u, v = _one_column(m, count, kmax + over)
        c = costs.Cost.points(sx, sy, tx, ty, "sqeuclid")
        oi, oj, od = pricing.select(c, u, v, NONE.astype(np.int64), NONE.astype(np.int64), km)
        T = U.cuda_tensors(sx, sy, tx, ty, u, v, NONE, NONE)
        gi, gj, gd = price_topk(*T, kmax=km, precision=precision)
        assert np.array_equal(gi.cpu().numpy(), oi) and np.array_equal(gj.cpu().numpy(), oj)
        assert np.array_equal(gd.cpu().numpy(), od)


def test_flooded_window_is_not_gathered():
    """151M pairs inside the FP32 window, three columns of negative ones: the FP32 pass 2 of this call has
    nothing to do and the FP64 one skips all but three columns' tiles, so that together they take less than
    the two histogram passes, which evaluate every pair (pass 2 evaluates and counts every pair of the window
    when it does not look at the bound: 151M atomics on one word)."""
    import torch
    from paper_2206_11009_gb300 import kernel_timing, price_topk
    m = n = 12288
    z = np.zeros(m, np.int32)
    u, v = np.full(m, 1e5), np.full(n, -1e5)
    v[[17, 4000, 9001]] += np.array([1.0, 3.0, 2.0])
    T = U.cuda_tensors(z, z, z, z, u, v, NONE, NONE)
    price_topk(*T, kmax=50000, precision=1)
    torch.cuda.synchronize()
    kernel_timing(True)
    out = price_topk(*T, kmax=50000, precision=1)
    t = kernel_timing()
    kernel_timing(False)
    print({k: x for k, x in t.items() if k.startswith("scan")})
    assert len(out[0]) == 3 * m
    assert t["scan_gather"][0] < t["scan_hist"][0]
