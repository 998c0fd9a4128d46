"""The Newton direction at the edges of the factorisations' and iterations' blocks -- one panel, a
full last panel, one column more, the larger update tiles -- against the oracle's sparse LU of the
grounded system.  The iterate is the library's own after two IPM iterations (Theta spans a few
decades).  Solves stop at a relative residual of 1e-12, so the error of the directions is bounded by
cond(S_M) 1e-12: below 1e-9 of max|ref| here."""
import numpy as np
import pytest

from oracle import costs, ipm
from paper_2206_11009_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


_states = {}


def _state(ks, kt):
    """(a, b, state, oracle direction) of a ks x ks / kt x kt pair after two iterations."""
    from paper_2206_11009_gb300 import Solver
    if (ks, kt) not in _states:
        a, b = synth.grf_image(ks, 4), synth.grf_image(kt, 5)
        with Solver(a, b, grid=(ks, kt), tol=1e-8) as s:
            s.step()
            s.step()
            I, J, P, S, u, v = s.state()
        c = costs.Cost.points(*synth.grid_coords(ks), *synth.grid_coords(kt), "sqeuclid")
        prob = ipm.Problem(c, a, b)
        st = ipm.State(I.astype(np.int64), J.astype(np.int64), P, S, u, v)
        res = ipm.residuals(prob, st)
        _states[ks, kt] = a, b, st, ipm.newton_direction(prob, st, res.r1a, res.r1b, res.r2, -P * S)
    return _states[ks, kt]


@pytest.mark.parametrize("solver", ["dense64", "dense32", "pcg64", "mixed"])
@pytest.mark.parametrize("ks,kt", [(2, 2), (5, 5), (8, 8), (9, 9), (11, 11), (9, 6), (6, 11), (16, 16), (31, 31),
                                   (47, 47)])
def test_direction_at_block_edges(solver, ks, kt):
    from paper_2206_11009_gb300 import Solver
    a, b, st, ref = _state(ks, kt)
    with Solver(a, b, grid=(ks, kt), tol=1e-8) as s:
        s.set_state(st.I, st.J, st.p, st.s, st.u, st.v)
        out = s.newton_direction(solver, cg_tol=1e-12, max_cg=20000)
    for x, y in zip(out[:4], (ref.du, ref.dv, ref.dp, ref.ds)):
        assert np.abs(x - y).max() <= 1e-9 * max(np.abs(y).max(), 1e-300)
