"""The pricing selection's tile sort and rank searches (1024 candidates per tile), its fixed candidate
capacity (four times kmax, 16384 to 262144) with the exact-size redo beyond it, the narrow scan tiles
(n <= 1024), the support's row pointers with empty rows, and the bounding box of point sets whose
size is no multiple of a block: the selected pairs, their order and their float64 reduced costs
are the oracle's, bit for bit."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import costs, pricing
from tests import gpu_util as U

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _check(sx, sy, tx, ty, u, v, si, sj, kmax, precision, kind="sqeuclid"):
    from paper_2206_11009_gb300 import price_topk
    T = U.cuda_tensors(sx, sy, tx, ty, u, v, si, sj)
    gi, gj, gd = price_topk(*T, kmax=kmax, precision=precision, cost=kind)
    c = costs.Cost.points(sx, sy, tx, ty, kind)
    oi, oj, od = pricing.select(c, u, v, si.astype(np.int64), sj.astype(np.int64), kmax)
    assert np.array_equal(gi.cpu().numpy(), oi) and np.array_equal(gj.cpu().numpy(), oj)
    assert np.array_equal(gd.cpu().numpy(), od)
    return len(oi)


NONE = np.zeros(0, np.int32)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("count", [1, 1023, 1024, 1025, 4097, 16384, 16385])
def test_candidate_counts_around_tiles_and_capacity(precision, count):
    """Exactly `count` negative reduced costs (one column takes them), kmax below, at and above it."""
    m = 20000
    x = np.arange(m, dtype=np.int32) % 150
    y = np.arange(m, dtype=np.int32) // 150
    tx, ty = np.array([0, 40], np.int32), np.array([0, 60], np.int32)
    rng = np.random.default_rng(count)
    c0 = x.astype(float) ** 2 + y.astype(float) ** 2
    below = np.zeros(m, bool)
    below[rng.permutation(m)[:count]] = True
    # d of column 0: -1 .. -0.01 for the chosen sources (ties among them), positive elsewhere
    u = c0 + np.where(below, np.round(0.01 + rng.random(m), 3), -1.0)
    v = np.array([0.0, -1e6])
    for kmax in (1, count - 1, count, m):
        assert _check(x, y, tx, ty, u, v, NONE, NONE, kmax, precision) == min(max(kmax, 0), count)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("kind", ["sqeuclid", "euclid", "l1", "linf"])
@pytest.mark.parametrize("w,h", [(1, 1), (31, 33), (32, 32), (25, 41), (57, 36)])
def test_widths_around_the_narrow_tiles(precision, kind, w, h):
    """n = 1, 1023, 1024, 1025, 2052 targets; sources of another shape, off the origin."""
    sx, sy = U.rect_coords(23, 29, -500, 900)
    tx, ty = U.rect_coords(w, h, -498, 903)
    amp = 6.0 if kind == "sqeuclid" else 0.5
    u, v = U.banded_duals(sx, sy, tx, ty, seed=w, amp=amp, noise=3.0)
    si, sj = U.random_support(len(sx), len(tx), 0.02, seed=h)
    _check(sx, sy, tx, ty, u, v, si, sj, len(sx), precision, kind)


@pytest.mark.parametrize("rows", [[], [0], [511], [3, 4, 200], [0, 1, 2, 509, 510, 511]])
def test_support_with_empty_rows(rows):
    """Membership through row pointers built from a support that leaves long runs of rows empty."""
    sx, sy = U.rect_coords(32, 16)
    u, v = U.banded_duals(sx, sy, sx, sy, seed=5, amp=5.0, noise=2.0)
    n = len(sx)
    si = np.repeat(np.array(rows, np.int32), n)
    sj = np.tile(np.arange(n, dtype=np.int32), len(rows))
    _check(sx, sy, sx, sy, u, v, si, sj, n, 1)


@pytest.mark.parametrize("precision", [0, 1])
def test_more_candidates_than_the_capacity(precision):
    """kmax = 3000 of far more ties than the 16384 the fixed buffer holds (one bin of equal reduced
    costs), so that pass 2 is redone with an exact-size buffer."""
    sx, sy = U.rect_coords(60, 60)
    n = len(sx)
    u, v = np.zeros(n), np.zeros(n)
    v[:] = 3.0          # d = c - 3: all pairs at distance 1 tie at -2, the diagonal at -3
    u[7] = 0.25
    assert _check(sx, sy, sx, sy, u, v, NONE, NONE, 3000, precision) == 3000
    v[:] = 12.0         # 60 x 60 pairs at squared distance < 12: ~130k candidates
    assert _check(sx, sy, sx, sy, u, v, NONE, NONE, 20000, precision) == 20000
