"""FP32 PCG inside FP64 refinement at a tight tolerance: the last corrections start from a residual whose
mean is rounding, as large as the rest of it; they must neither stall nor diverge on it.  So the number
of iterations varies little from input to input (the systems of one size are alike), stays a small multiple
of FP64 PCG's on the same system, and the direction is FP64 PCG's."""
import numpy as np
import pytest

from paper_2206_11009_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _iterate(k, seed):
    """An interior iterate on the pairs within squared distance 5 of a k x k grid, complementary products
    around one value, and slacks that follow a smooth field (Theta spans about four decades)."""
    gx, gy = np.arange(k * k) % k, np.arange(k * k) // k
    off = [(dx, dy) for dy in range(-2, 3) for dx in range(-2, 3) if dx * dx + dy * dy <= 5]
    I, J = [], []
    for dx, dy in off:
        ok = (gx + dx >= 0) & (gx + dx < k) & (gy + dy >= 0) & (gy + dy < k)
        I.append(np.nonzero(ok)[0])
        J.append((gx + dx)[ok] + (gy + dy)[ok] * k)
    I, J = np.concatenate(I), np.concatenate(J)
    o = np.lexsort((J, I))
    I, J = I[o], J[o]
    r = synth.normal(seed, 2 * len(I) + 4)
    fx, fy, a, b = r[-4:]
    s = np.exp(1.5 * np.cos(0.09 * gx[I] + a) * np.cos(0.07 * gy[J] + b) + 0.5 * r[:len(I)]) + 0.01
    p = np.exp(0.3 * r[len(I):2 * len(I)]) / s
    return I, J, p * (k * k / p.sum()), s, np.zeros(k * k), np.zeros(k * k)


@pytest.mark.parametrize("k", [40, 56, 72, 100])
def test_iterations_are_steady_at_a_tight_tolerance(k):
    from paper_2206_11009_gb300 import Solver
    its = []
    for seed in range(1, 8):
        inst = synth.image_pair(k, seed)
        with Solver(inst.a, inst.b, grid=(k, k)) as h:
            h.set_state(*_iterate(k, seed))
            out = h.newton_direction("mixed", cg_tol=1e-12)
            ref = h.newton_direction("pcg64", cg_tol=1e-12)
        its.append(out[4])
        print(k, seed, out[4], ref[4], [float(np.abs(x - y).max() / np.abs(y).max()) for x, y in zip(out[:4], ref[:4])])
        assert out[4] <= 4 * ref[4]
        for x, y in zip(out[:4], ref[:4]):
            assert np.abs(x - y).max() <= 1e-9 * np.abs(y).max()
    assert max(its) <= 2 * np.median(its), its


@pytest.mark.parametrize("cut", [(20, 17), (31, 9)])
def test_several_components(cut):
    """The same on a support of two components (no pair across a line): a mean each."""
    from paper_2206_11009_gb300 import Solver
    k = 48
    inst = synth.image_pair(k, 3)
    I, J, p, s, u, v = _iterate(k, 5)
    x = [(q % k < cut[0]) | (q // k < cut[1]) for q in (I, J)]
    keep = x[0] == x[1]
    with Solver(inst.a, inst.b, grid=(k, k)) as h:
        h.set_state(I[keep], J[keep], p[keep], s[keep], u, v)
        out = h.newton_direction("mixed", cg_tol=1e-12)
        ref = h.newton_direction("pcg64", cg_tol=1e-12)
    print(cut, out[4], ref[4], [float(np.abs(x - y).max() / np.abs(y).max()) for x, y in zip(out[:4], ref[:4])])
    assert out[4] <= 4 * ref[4]
    for a, b in zip(out[:4], ref[:4]):
        assert np.abs(a - b).max() <= 1e-9 * np.abs(b).max()
