"""Strongly nonlinear and shifted small eigenproblems, on which Newton's iteration from far away can
wander to the iteration cap: the solve starts again with a smaller reach and converges."""
import numpy as np
import pytest

from tests.test_gpu_parity import _fmg

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = {
    "shift_down_2d": dict(dim=2, coarse_cells=3, zeta=5e3, w_const=-19.0, box_len=10.0),
    "small_box_3d": dict(dim=3, coarse_cells=4, zeta=10.0, box_len=0.01),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_converges(name):
    fmg = _fmg()
    p = fmg.Problem(**CASES[name], levels=3, flags=fmg.FMG_FLAG_NO_AUTOTUNE)
    with fmg.Solver(p) as s:
        u = np.empty(p.size(3))
        lam, st, rc = s.solve(u, stats=True)
    assert rc == 0 and max(st.scf_iters[:3]) <= p.scf_max_iter
    assert abs(st.norm_defect) < 1e-12 and abs(st.identity_defect) < 1e-10 * abs(lam)


def test_the_cap_still_ends_the_iteration():
    """One step is not enough, from either start."""
    fmg = _fmg()
    p = fmg.Problem(dim=2, coarse_cells=8, levels=2, zeta=200.0, scf_max_iter=1)
    with fmg.Solver(p) as s:
        _, st, rc = s.solve(None, stats=True)
    assert rc == fmg.FMG_ENOCONV and list(st.scf_iters[:2]) == [1, 1]
