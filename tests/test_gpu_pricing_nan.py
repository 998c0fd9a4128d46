"""Pairs whose reduced cost is not a number (a NaN in the explicit matrix or in a dual, of either sign)
are never selected and hide no other pair, and those at -infinity come first: the selection is the
oracle's, bit for bit."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import costs, pricing
from tests import gpu_util as U

pytestmark = pytest.mark.gpu

NONE = np.zeros(0, np.int32)


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("m,n", [(40, 300), (64, 1025), (257, 2500)])
def test_nan_in_the_cost_matrix(m, n, sign):
    """One NaN above, below or beside the only negative reduced costs of its columns."""
    from paper_2206_11009_gb300 import price_topk
    import torch
    rng = np.random.default_rng(n)
    C = 1.0 + rng.random((m, n))
    at = rng.permutation(n)[:9]
    for q, j in enumerate(at):
        i = int(rng.integers(1, m - 1))
        C[i, j] = 0.5 - 0.03 * q                     # d = c - 1 < 0
        C[i + (-1, 1, 0)[q % 3], (j, j, (j + 256) % n)[q % 3]] = np.copysign(np.nan, sign)
    u, v = np.full(m, 0.75), np.full(n, 0.25)
    with np.errstate(invalid="ignore"):
        d = (C - u[:, None]) - v[None, :]
        wi, wj = np.nonzero(d < 0)
    o = np.lexsort((wi + wj * m, d[wi, wj]))
    T = U.cuda_tensors(u, v, NONE, NONE)
    for kmax in (1, len(wi), 100):
        gi, gj, gd = price_topk(None, None, None, None, *T, kmax=kmax, cost="dense",
                                C=torch.as_tensor(C, device=T[0].device))
        k = min(kmax, len(wi))
        assert np.array_equal(gi.cpu().numpy(), wi[o][:k]) and np.array_equal(gj.cpu().numpy(), wj[o][:k])
        assert np.array_equal(gd.cpu().numpy(), d[wi, wj][o][:k])


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("kind", ["sqeuclid", "euclid"])
def test_nan_duals(kind, sign, precision):
    from paper_2206_11009_gb300 import price_topk
    sx, sy = U.rect_coords(36, 30)
    tx, ty = U.rect_coords(41, 30)
    u, v = U.banded_duals(sx, sy, tx, ty, seed=2, amp=5.0 if kind == "sqeuclid" else 0.5, noise=3.0)
    u[[5, 77, 600]] = np.copysign(np.nan, sign)
    v[[0, 300, 1000]] = np.copysign(np.nan, sign)
    c = costs.Cost.points(sx, sy, tx, ty, kind)
    T = U.cuda_tensors(sx, sy, tx, ty, u, v, NONE, NONE)
    for kmax in (3, 200):
        with np.errstate(invalid="ignore"):
            oi, oj, od = pricing.select(c, u, v, NONE.astype(np.int64), NONE.astype(np.int64), kmax)
        assert len(oi) == kmax
        gi, gj, gd = price_topk(*T, kmax=kmax, precision=precision, cost=kind)
        assert np.array_equal(gi.cpu().numpy(), oi) and np.array_equal(gj.cpu().numpy(), oj)
        assert np.array_equal(gd.cpu().numpy(), od)


@pytest.mark.parametrize("precision", [0, 1])
def test_infinite_duals(precision):
    """d = -infinity over a row and a column among finite negative ones."""
    from paper_2206_11009_gb300 import price_topk
    sx, sy = U.rect_coords(36, 30)
    tx, ty = U.rect_coords(41, 30)
    u, v = U.banded_duals(sx, sy, tx, ty, seed=2, amp=5.0, noise=3.0)
    u[77] = np.inf
    v[[3, 1001]] = np.inf, -np.inf
    c = costs.Cost.points(sx, sy, tx, ty, "sqeuclid")
    T = U.cuda_tensors(sx, sy, tx, ty, u, v, NONE, NONE)
    for kmax in (5, 3000):
        with np.errstate(invalid="ignore"):
            oi, oj, od = pricing.select(c, u, v, NONE.astype(np.int64), NONE.astype(np.int64), kmax)
        gi, gj, gd = price_topk(*T, kmax=kmax, precision=precision)
        assert np.array_equal(gi.cpu().numpy(), oi) and np.array_equal(gj.cpu().numpy(), oj)
        assert np.array_equal(gd.cpu().numpy(), od)
