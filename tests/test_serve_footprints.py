"""Admission of served requests: a request's device bytes depend on its smoother too (Chebyshev
steps read stored couplings on the levels whose other smoothers need none)."""
import pytest

from tests.test_gpu_parity import _fmg

pytest.importorskip("torch")


def _pair():
    fmg = _fmg()
    kw = dict(dim=2, coarse_cells=8, levels=8, w_quad=(1.0, 4.0, 0.0), zeta=5.0)
    return fmg.Problem(**kw), fmg.Problem(**kw, smoother=fmg.FMG_SMOOTH_CHEBYSHEV)


def test_chebyshev_needs_more_bytes():
    fmg = _fmg()
    jacobi, cheb = (fmg.estimate_bytes([p]) for p in _pair())
    assert cheb - jacobi > 0.9 * 4 * 8 * 1025 ** 2


@pytest.mark.gpu
@pytest.mark.parametrize("order", [(0, 1), (1, 0)], ids=["jacobi_first", "chebyshev_first"])
def test_a_request_that_never_fits_is_refused_whatever_came_before(order):
    """A budget between the two footprints admits the Jacobi request and never the other one."""
    fmg = _fmg()
    probs = _pair()
    small, large = (fmg.estimate_bytes([p]) for p in probs)
    with pytest.raises(fmg.FmgError) as e:
        fmg.serve([probs[i] for i in order], [0.0, 0.0], budget_bytes=(small + large) / 2)
    assert e.value.code == fmg.FMG_EINVAL
    res, st = fmg.serve([probs[0]], [0.0], budget_bytes=(small + large) / 2)
    assert res[0]["status"] == 0 and st["peak_bytes"] <= st["budget_bytes"]
