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
    """151M pairs inside the FP32 window, three columns of negative ones: the FP32 pass 2 has nothing to do
    and the call is redone in FP64, so pass 2 takes what it takes in a call in FP64 from the start (less than
    half of that more; when the FP32 pass does not look at its bound it evaluates every pair and counts those
    of the window one by one, more than the FP64 pass 2 over half of the columns)."""
    import torch
    from paper_2206_11009_gb300 import kernel_timing, price_topk
    m = n = 12288
    z = np.zeros(m, np.int32)
    u, v = np.full(m, 1e5), np.full(n, -1e5)
    v[[17, 4000, 9001]] += np.array([1.0, 3.0, 2.0])
    T = U.cuda_tensors(z, z, z, z, u, v, NONE, NONE)
    ms = {}
    for precision in (0, 1):
        price_topk(*T, kmax=50000, precision=precision)
        torch.cuda.synchronize()
        kernel_timing(True)
        out = price_topk(*T, kmax=50000, precision=precision)
        ms[precision] = kernel_timing()["scan_gather"][0]
        kernel_timing(False)
        assert len(out[0]) == 3 * m
    print(ms)
    assert ms[1] <= 1.5 * ms[0]
