"""The level-1 inverse of the V-cycles where a negative potential brings A + W near singularity: w_const = -(1 - gap) lambda_1, lambda_1 the smallest eigenvalue of the level-1
pencil.  The single-precision elimination loses a digit per digit of the condition number (some 100
/ gap), up to pivots of the wrong sign: these take the FP64 LDL^T.

x = X f from an explicit inverse X leaves |L x - f| <= n eps |L| |x| times a small growth: 64 x 1.1e-16
x 10 gives 1e-13."""
import numpy as np
import pytest
from scipy.linalg import eigh

from oracle import fmg_oracle as O
from tests.test_gpu_parity import _fmg, _pair, dev, host

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MESHES = [(2, 3), (2, 8), (2, 9), (3, 3), (3, 4)]
TRAPS = {"flat": (0.0, 0.0, 0.0), "trap": (100.0, 300.0, 200.0)}


def _level1(dim, cells, trap, gap, **kw):
    base = dict(dim=dim, coarse_cells=cells, levels=2, w_quad=TRAPS[trap], **kw)
    op, _ = _pair(**base, w_const=0.0)
    lev = O.build_hierarchy(op)[0]
    lam = eigh(lev.L.toarray(), lev.M.toarray(), eigvals_only=True)[0]
    op, gp = _pair(**base, w_const=-(1.0 - gap) * lam)
    return O.build_hierarchy(op)[0], gp


@pytest.mark.parametrize("gap", [1.0, 1e-2, 1e-3, 1e-4, 1e-5, 1e-6, 1e-7, 1e-9])
@pytest.mark.parametrize("trap", sorted(TRAPS))
@pytest.mark.parametrize("dim,cells", MESHES)
def test_level1_inverse(dim, cells, trap, gap):
    lev, gp = _level1(dim, cells, trap, gap, zeta=0.0)
    rng = np.random.default_rng(3400)
    lmat = lev.L.toarray()
    norm = np.abs(lmat).sum(axis=1).max()
    with _fmg().Solver(gp) as s:
        for _ in range(3):
            f = rng.normal(size=gp.size(1))
            x = dev(np.zeros(gp.size(1)))
            s.multigrid(1, dev(f), x)
            got = host(x)
            assert np.abs(lmat @ got - f).max() <= 1e-13 * norm * np.abs(got).max()
