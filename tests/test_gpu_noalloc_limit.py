"""ot_price_topk_noalloc near the largest candidate set its fixed 24 MiB hold.  At m = n = 16384 the points and
tiles take 1.5 MB of it and a candidate 40 bytes (its pair, two keys, its index, and the sort's second
key and index) and a quarter: 585k; 498k were beyond it while the reduced costs were kept once more."""
from __future__ import annotations

import ctypes

import numpy as np
import pytest

from oracle import costs, pricing
from tests import gpu_util as U

pytestmark = pytest.mark.gpu


def _duals(k, count):
    """u with `count` pairs c_ij < u_i or up to eight fewer (v = 0): all points take the 29 neighbours of
    squared distance < 9.5 inside the grid, the first ones those of distance < 10.5 too."""
    off = [(dx, dy) for dx in range(-3, 4) for dy in range(-3, 4) if dx * dx + dy * dy <= 10]
    x, y = np.arange(k * k) % k, np.arange(k * k) // k
    n9, n10 = np.zeros(k * k, int), np.zeros(k * k, int)
    for dx, dy in off:
        ok = (x + dx >= 0) & (x + dx < k) & (y + dy >= 0) & (y + dy < k)
        (n9 if dx * dx + dy * dy <= 9 else n10)[ok] += 1
    total = n9.sum() + np.cumsum(n10)
    assert n9.sum() < count <= total[-1]
    return np.where(total <= count, 10.5, 9.5), int(n9.sum() + n10[total <= count].sum())


def test_candidate_set_near_the_limit():
    import __graft_entry__
    import torch
    __graft_entry__.build()
    from paper_2206_11009_gb300 import _lib
    lib = _lib.load()
    k = 128
    sx, sy = U.rect_coords(k, k)
    u, count = _duals(k, 498_000)
    v = np.zeros(k * k)
    none = np.zeros(0, np.int64)
    kmax = 600_000
    T = U.cuda_tensors(sx, sy, sx, sy, u, v)
    dev = T[0].device
    oi, oj = (torch.empty(kmax, dtype=torch.int32, device=dev) for _ in range(2))
    od = torch.empty(kmax, dtype=torch.float64, device=dev)
    cnt = torch.full((1,), -1, dtype=torch.int32, device=dev)
    stream = ctypes.c_void_p(torch.cuda.current_stream(dev).cuda_stream)
    rc = lib.ot_price_topk_noalloc(k * k, k * k, *[t.data_ptr() for t in T], None, None, 0, kmax, 1, oi.data_ptr(),
                                   oj.data_ptr(), od.data_ptr(), cnt.data_ptr(), stream)
    torch.cuda.synchronize()
    assert rc == _lib.OT_OK, lib.ot_last_error()
    wi, wj, wd = pricing.select(costs.Cost.points(sx, sy, sx, sy, "sqeuclid"), u, v, none, none, kmax)
    assert int(cnt.item()) == count == len(wi)
    assert np.array_equal(oi[:count].cpu().numpy(), wi) and np.array_equal(oj[:count].cpu().numpy(), wj)
    assert np.array_equal(od[:count].cpu().numpy(), wd)
