"""Linear solvers of the Newton system used in turn on one handle: a dense factorisation assembles the
same Schur complement into the arrays that the sparse one keeps between calls, and must leave nothing
stale behind.  Directions against the oracle's exact one (sparse LU of the grounded S_M); the solves
stop at a relative residual of 1e-12 and cond(S_M) is at most 420 here: below 1e-9 of max|ref|."""
import numpy as np
import pytest

from oracle import costs, ipm
from paper_2206_11009_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _state(k, radius2, seed):
    """An interior iterate on the pairs within squared distance radius2 of a k x k grid."""
    gx, gy = np.arange(k * k) % k, np.arange(k * k) // k
    d2 = (gx[:, None] - gx[None, :]) ** 2 + (gy[:, None] - gy[None, :]) ** 2
    I, J = np.nonzero(d2 <= radius2)
    r = synth.uniform01(seed, 2 * len(I))
    return ipm.State(I, J, 0.1 + r[:len(I)], 0.1 + 2.0 * r[len(I):], np.zeros(k * k), np.zeros(k * k))


def _direction(h, st, solver):
    h.set_state(st.I, st.J, st.p, st.s, st.u, st.v)
    return h.newton_direction(solver, cg_tol=1e-12, max_cg=2000)[:4]


def _reference(prob, st):
    res = ipm.residuals(prob, st)
    d = ipm.newton_direction(prob, st, res.r1a, res.r1b, res.r2, -st.p * st.s)
    return d.du, d.dv, d.dp, d.ds


def _close(out, ref):
    for x, y in zip(out, ref):
        assert np.abs(x - y).max() <= 1e-9 * np.abs(y).max()


@pytest.mark.parametrize("between", ["dense64", "ic", "dense32"])
@pytest.mark.parametrize("k,small,large", [(8, 2, 9), (23, 1, 5)])
def test_sparse_again_after_another_solver_on_a_larger_support(k, small, large, between):
    """The larger support makes the assembled arrays grow between two sparse factorisations of one
    pattern."""
    from paper_2206_11009_gb300 import Solver
    inst = synth.image_pair(k, 1)
    prob = ipm.Problem(costs.square_grid(k), inst.a, inst.b)
    A, B = _state(k, small, 3), _state(k, large, 4)
    ra, rb = _reference(prob, A), _reference(prob, B)
    with Solver(inst.a, inst.b, grid=(k, k), tol=1e-8) as h:
        _close(_direction(h, A, "sparse"), ra)
        _close(_direction(h, B, between), rb)
        _close(_direction(h, A, "sparse"), ra)
        _close(_direction(h, B, "sparse"), rb)


def test_dense_directions_between_sparse_steps():
    """A handle whose steps factor sparsely (with dropped pairs), with dense directions (which drop none)
    taken between its steps: the same iterates as without them."""
    from paper_2206_11009_gb300 import Solver
    k = 12
    inst = synth.image_pair(k, 1)
    runs = []
    for dense in (False, True):
        with Solver(inst.a, inst.b, grid=(k, k), tol=1e-8, precision=0, linear_solver=2, dense_max_n=-1) as h:
            for _ in range(8):
                h.step()
                if dense:
                    h.newton_direction("dense64")
            runs.append(h.state())
    for x, y in zip(*runs):
        assert np.array_equal(x, y) if x.dtype.kind == "i" else np.abs(x - y).max() <= 1e-9 * np.abs(y).max()
