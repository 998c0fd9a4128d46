"""The stopping rule of the FP64 CG preconditioned by the FP32 dense factor: the direction's residual,
recomputed in extended precision, is at or below the tolerance asked for, also on late iterates, where
S_M's entries span many decades and a residual small in the preconditioner's norm is not small.

Bar on |rhs - S_M dv| / |rhs|: the tolerance, plus what FP64 arithmetic leaves: q = S_M p is rounded by
at most (row length + 3) eps per term, so each of the at most 60 steps adds that much of |S_M| |x| to the
residual; 64 eps (|S_M| |dv|) bounds it with room for the few steps that carry x."""
import numpy as np
import pytest

from oracle import costs, ipm
from paper_2206_11009_gb300 import synth

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53
LD = np.longdouble


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _sum_by(idx, w, size):
    """Sums of w per index in extended precision."""
    out = np.zeros(size, LD)
    np.add.at(out, idx, w)
    return out


def _residual(prob, st, dv):
    """(|rhs - S_M dv| / |rhs|, 64 eps ||S_M| |dv|| / |rhs|) for the predictor's right-hand side."""
    m, n = prob.m, prob.n
    I, J = st.I, st.J
    th = (st.p.astype(LD) / st.s.astype(LD))
    res = ipm.residuals(prob, st)
    g = th * (res.r2.astype(LD) + st.s.astype(LD))            # r2 - r3 / p with r3 = -p s
    b1 = res.r1a.astype(LD) + _sum_by(I, g, m)
    b2 = res.r1b.astype(LD) + _sum_by(J, g, n)
    M = _sum_by(I, th, m)
    Minv = np.where(M > 0, 1 / np.where(M > 0, M, 1), 0)
    rhs = b2 - _sum_by(J, th * (Minv * b1)[I], n)
    rhs -= rhs.mean()
    x = dv.astype(LD)
    w = Minv * _sum_by(I, th * x[J], m)
    r = rhs - _sum_by(J, th * (x[J] - w[I]), n)
    wa = Minv * _sum_by(I, th * np.abs(x)[J], m)
    ra = _sum_by(J, th * (np.abs(x)[J] + wa[I]), n)
    nrm = lambda z: float(np.sqrt((z * z).sum()))
    return nrm(r) / nrm(rhs), 64 * EPS * nrm(ra) / nrm(rhs)


@pytest.mark.parametrize("k,seed", [(16, 1), (23, 1), (23, 2)])
def test_residual_meets_the_tolerance_on_late_iterates(k, seed):
    """Right-hand sides along the weakest directions of a late iterate's S_M (the duals moved by an
    eigenvector, which adds -S_M times it): the FP32 factor is at its limit there, and its first steps leave
    residuals along the large eigenvalues."""
    from paper_2206_11009_gb300 import Solver
    inst = synth.image_pair(k, seed)
    prob = ipm.Problem(costs.square_grid(k), inst.a, inst.b)
    states = []
    with Solver(inst.a, inst.b, grid=(k, k), tol=1e-8, max_corr=1) as h:
        for _ in range(100):
            states.append(h.state())
            if h.step()["done"]:
                break
    worst = 0.0
    for z in states[-4:]:
        I, J = z[0].astype(np.int64), z[1].astype(np.int64)
        S, *_ = ipm.schur_matrix(k * k, k * k, I, J, z[2] / z[3])
        vec = np.linalg.eigh(S.toarray())[1]
        for e in (1, 2, 5):
            st = ipm.State(I, J, z[2], z[3], z[4], z[5] + 1e4 * vec[:, e])
            for tol in (1e-2, 1e-4, 1e-6):
                with Solver(inst.a, inst.b, grid=(k, k), direct_cg_tol=tol) as h:
                    h.set_state(st.I, st.J, st.p, st.s, st.u, st.v)
                    _, dv, _, _, its = h.newton_direction("dense32", cg_tol=1e-6)
                rel, floor = _residual(prob, st, dv)
                worst = max(worst, (rel - floor) / tol)
                print(f"k={k} e={e} tol={tol:.0e} its={its} rel={rel:.1e} floor={floor:.1e}")
    assert worst <= 1.0, worst


@pytest.mark.parametrize("k,seed", [(96, 1), (96, 6), (112, 2)])
def test_few_iterations_at_a_tight_tolerance(k, seed):
    """A residual that rounding leaves in the one equation implied by the others (the columns of S_M add up
    to zero) does not keep the iteration going: the factor is accurate to FP32, so a step gains three digits
    or more and five suffice for 1e-12."""
    from paper_2206_11009_gb300 import Solver
    inst = synth.image_pair(k, seed)
    with Solver(inst.a, inst.b, grid=(k, k), tol=1e-8) as h:
        h.step()
        h.step()
        *_, its = h.newton_direction("dense32", cg_tol=1e-12)
    assert its <= 5
