"""The level operators in fixed point (2D n >= 512, 3D n >= 96) on values of extreme size and range.
Reference in 3D: a mixed-precision handle, whose operator is FP64 with stored couplings."""
import numpy as np
import pytest

from tests.test_gpu_parity import _fmg, dev, host

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _mixed_and_fp64(**kw):
    """A 3D handle of the fixed-point operator and one whose operator is FP64 with stored
    couplings (mixed precision)."""
    fmg = _fmg()
    return [fmg.Solver(fmg.Problem(**kw, precision=p)) for p in (fmg.FMG_FP64, fmg.FMG_MIXED_FP32)]


def test_right_hand_side_near_the_largest_number_3d():
    """|f| to 1.7e308 at n = 96: f / h leaves the range of FP64, f and omega / D f do not."""
    kw = dict(dim=3, coarse_cells=3, levels=6, w_const=0.3, w_quad=(1.0, 2.0, 1.5), omega=0.01)
    out = []
    for s in _mixed_and_fp64(**kw):
        with s:
            size = s.level_size(6)
            rng = np.random.default_rng(3200)
            x = rng.normal(size=size)
            f = rng.uniform(0.3, 1.0, size=size) * 1.7e308
            y = torch.empty(size, dtype=torch.float64, device="cuda")
            s.jacobi(6, dev(f), dev(x), y)
            out.append(host(y))
    assert np.isfinite(out[1]).all()
    assert (np.abs(out[0] / out[1] - 1.0) <= 1e-13).all()
