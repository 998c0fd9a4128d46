"""The tensor-core rest-update of the FP32 dense factor (three BF16 pieces, two panels per pass) against
the SIMT update, at the edges of its tiles and pairs of panels: no rest at all (4 blocks of 64), one
ragged block, an odd last panel, several tiles per CTA.  Both directions are refined to a relative
residual of 1e-12, so each is within cond(S_M) 1e-12 < 1e-9 of the exact one and 2e-9 of the other; and
the factor has FP32 accuracy (relative error below 1e-5 against 1e-6, either far below what one CG
iteration gains), so the refinement takes at most two iterations more -- a tile left out or applied
twice costs dozens."""
import numpy as np
import pytest

from paper_2206_11009_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [15, 16, 17, 18, 20, 23, 47, 67])
def test_tensor_core_rest_update_at_tile_edges(k):
    from paper_2206_11009_gb300 import Solver
    a, b = synth.grf_image(k, 6), synth.grf_image(k, 7)
    with Solver(a, b, grid=(k, k), tol=1e-8) as s:
        s.step()
        s.step()
        st = s.state()
    out = {}
    for tc in (-1, 1):
        with Solver(a, b, grid=(k, k), tol=1e-8, tc_update=tc) as s:
            s.set_state(*st)
            out[tc] = s.newton_direction("dense32", cg_tol=1e-12, max_cg=20000)
    for x, y in zip(out[1][:4], out[-1][:4]):
        assert np.abs(x - y).max() <= 2e-9 * max(np.abs(y).max(), 1e-300)
    assert out[1][4] <= out[-1][4] + 2
