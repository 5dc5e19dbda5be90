"""The Galerkin coarsening of the density stencil on fields of wide range, entry by entry.  With
c = (0, .., 0, 1) the augmented G holds int u~^2 psi_i psi_j alone, sums of non-negative terms
through every level, so each entry keeps its own relative accuracy: 1e-11 here (a chain of levels
rounds each term some 10 times at 2^-53; the fixed-point sums at 2^-44 of their largest term where
u~ doubles from column to column)."""
import numpy as np
import pytest

from oracle import fmg_oracle as O
from tests.test_gpu_parity import _fmg, _pair, dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _density_matrix(kw, k, ut):
    """G at c = e_u from the handle, and int u~^2 phi_a phi_b restricted exactly by the oracle."""
    op, gp = _pair(**kw)
    lv = O.build_hierarchy(op)
    c = np.zeros(gp.size(1) + 1)
    c[-1] = 1.0
    with _fmg().Solver(gp) as s:
        _, _, g = s.augmented_system(k, dev(ut), c)
    b = O.density_matrix(lv[k - 1].mesh, ut)
    for j in range(k - 1, 0, -1):
        b = lv[j].P.T @ b @ lv[j].P
    return g[:-1, :-1], b.toarray()


def _compare(got, ref):
    assert np.array_equal(got != 0.0, ref != 0.0)
    nz = ref != 0.0
    assert np.abs(got[nz] / ref[nz] - 1.0).max() <= 1e-11


CASES = {"2d": (dict(dim=2, w_quad=(1.0, 2.0, 0.0), zeta=1.0, coarse_cells=5, levels=6), 6),
         "3d": (dict(dim=3, w_quad=(1.0, 2.0, 1.5), zeta=1.0, coarse_cells=4, levels=3), 3)}


@pytest.mark.parametrize("exponent", [-146.0, -145.0, -144.0, -143.0, -142.0, -139.0])
@pytest.mark.parametrize("name", sorted(CASES))
def test_tiny_values_beside_zeros(name, exponent):
    """u~ of about 10^exponent with zeros in the upper half of the box and in scattered patches:
    entries of 1e-301 to 1e-285 beside exact zeros."""
    kw, k = CASES[name]
    n = kw["coarse_cells"] << (k - 1)
    rng = np.random.default_rng(2700)
    u = 10.0 ** exponent * rng.uniform(0.2, 1.0, size=(n - 1,) * kw["dim"])
    u[(3 * n) // 5:] = 0.0
    u[2:5, 3:9] = 0.0
    _compare(*_density_matrix(kw, k, u.ravel()))


@pytest.mark.parametrize("axis,bits", [(0, 1.0), (1, 1.0), (0, 1.7), (1, 0.5), (1, 4.0)])
@pytest.mark.parametrize("name", sorted(CASES))
def test_smooth_decay(name, axis, bits):
    """u~ falls by `bits` bits per node along one axis (0: across the columns' rows, 1: along a
    row), so that the entries of 32 coarse nodes span up to 500 bits."""
    kw, k = CASES[name]
    n = kw["coarse_cells"] << (k - 1)
    dim = kw["dim"]
    x = np.arange(1, n, dtype=np.float64)
    shape = [1] * dim
    shape[-1 if axis else 0] = n - 1
    u = np.exp2(-bits * x).reshape(shape) * np.random.default_rng(2800).uniform(0.7, 1.0, size=(n - 1,) * dim)
    _compare(*_density_matrix(kw, k, u.ravel()))


@pytest.mark.parametrize("name", sorted(CASES))
def test_zero_patches(name):
    """Exact zeros beside values of order one stay exact zeros, entry by entry."""
    kw, k = CASES[name]
    n = kw["coarse_cells"] << (k - 1)
    rng = np.random.default_rng(2900)
    u = rng.uniform(0.2, 1.0, size=(n - 1,) * kw["dim"])
    u[..., (2 * n) // 5:(4 * n) // 5] = 0.0
    u[n // 3:n // 2] = 0.0
    _compare(*_density_matrix(kw, k, u.ravel()))


@pytest.mark.parametrize("value", [np.nan, np.inf])
@pytest.mark.parametrize("name", sorted(CASES))
def test_not_finite_entries_reach_their_nodes(name, value):
    """An infinity or NaN at any place of a coarse cell (centre, edge, corner, the column that the
    lane before reads) reaches every entry of G that integrates over its star."""
    kw, k = CASES[name]
    n = kw["coarse_cells"] << (k - 1)
    op, gp = _pair(**kw)
    lv = O.build_hierarchy(op)
    rng = np.random.default_rng(3000)
    base = rng.uniform(0.2, 1.0, size=(n - 1,) * kw["dim"])
    c = np.zeros(gp.size(1) + 1)
    c[-1] = 1.0
    for shift in range(4):
        at = tuple(n // 2 + (shift >> d & 1 if d < 2 else 0) for d in range(kw["dim"]))
        u = base.copy()
        u[at] = value
        v = base.copy()
        v[at] = 2.0
        with _fmg().Solver(gp) as s:
            _, _, g = s.augmented_system(k, dev(u.ravel()), c)
        touched = O.density_matrix(lv[k - 1].mesh, v.ravel()) - O.density_matrix(lv[k - 1].mesh, base.ravel())
        for j in range(k - 1, 0, -1):
            touched = lv[j].P.T @ touched @ lv[j].P
        assert np.array_equal(~np.isfinite(g[:-1, :-1]), abs(touched.toarray()) > 1e-12)
