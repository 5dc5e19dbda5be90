"""The 64-bit fixed-point kernels at the edges of their ranges: the level operator (2D from 512
cells per side, 3D FP64 from 96), the cubic-load and density walks (2D rows 4, 8, 16; 3D planes
4, 16), the density coarsening, the fused operator and mass apply, and the FP64 forms that take
the tiles fixed point does not (mixed signs, zeros, exponents out of range, infinities and NaN,
potentials too large for the formats).

References: the oracle in 2D; in 3D, where the oracle's assembly of such levels takes minutes,
a mixed-precision handle, whose operator (stored couplings, FP64) and loads (double-float) are
separate kernels that other tests compare with the oracle.  Tolerances as in test_gpu_parity:
1e-13 of the largest value for one stencil step (a fixed-point step rounds at 2^-56 of a tile's
maximum or below, FP64 sums of up to 30 terms at 2^-53 each), 1e-12 for the augmented matrices
(sums over chains of levels, double-float's 2^-47 on the reference's side)."""
import functools

import numpy as np
import pytest

from oracle import fmg_oracle as O
from tests.test_gpu_parity import _fmg, _pair, dev, host, rel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

KW2 = dict(dim=2, w_const=0.3, w_quad=(1.0, 2.5, 0.0), zeta=7.0)


@functools.lru_cache(maxsize=None)
def _mesh(n):
    return O.Mesh(2, n, 1.0)


def _empty(p, k):
    return torch.empty(p.size(k), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("w_const,scale", [(0.3, 1.0), (0.3, 1e-90), (0.3, 1e-120), (2e8, 1.0)],
                         ids=["", "small", "out_of_range", "large_potential"])
def test_operator_2d(w_const, scale, precision):
    """n = 640: 639 = 10 x 62 + 19 columns, 39 x 16 + 15 rows.  1e-120 leaves the exponents'
    range; h^2 W / 12 = 41 leaves the formats.  Mixed handles keep no omega / D."""
    op, gp = _pair(**{**KW2, "w_const": w_const}, coarse_cells=5, levels=8)
    gp.precision = _fmg().FMG_FP64 if precision == "fp64" else _fmg().FMG_MIXED_FP32
    coarse = O.Level(_mesh(320), None, None, None, None, None, None)
    lev = O.build_level(op, 8, coarse)
    rng = np.random.default_rng(2100)
    x, f = scale * rng.normal(size=(2, gp.size(8)))
    with _fmg().Solver(gp) as s:
        y = _empty(gp, 8)
        s.apply_operator(8, dev(x), y)
        assert rel(host(y), lev.L @ x) <= 1e-13
        s.jacobi(8, dev(f), dev(x), y)
        assert rel(host(y), O.jacobi(lev, f, x, op.omega)) <= 1e-13
        rc = _empty(gp, 7)
        s.residual_restrict(8, dev(f), dev(x), rc)
        assert rel(host(rc), lev.P.T @ (f - lev.L @ x)) <= 1e-13


@pytest.mark.parametrize("cells,levels,w_const", [(3, 6, 0.3), (3, 6, 1e8), (4, 6, 0.3)],
                         ids=["n96", "n96_large_potential", "n128"])
def test_operator_and_augmented_system_3d(cells, levels, w_const):
    """n = 96, 128: ragged last tiles in every direction (95 = 2 x 32 + 31 columns, 11 x 8 + 7
    rows and planes); 4-plane walks below 128, 16-plane ones from there on."""
    fmg = _fmg()
    kw = dict(dim=3, coarse_cells=cells, levels=levels, w_const=w_const, w_quad=(1.0, 2.0, 1.5),
              zeta=5.0)
    rng = np.random.default_rng(2200 + cells)
    k = levels
    p = fmg.Problem(**kw)
    x, f = rng.normal(size=(2, p.size(k)))
    ut = rng.uniform(0.2, 1.0, size=p.size(k))
    c = rng.normal(size=p.size(1) + 1)
    got = []
    for precision in (fmg.FMG_FP64, fmg.FMG_MIXED_FP32):
        with fmg.Solver(fmg.Problem(**kw, precision=precision)) as s:
            y, z, rc = _empty(p, k), _empty(p, k), _empty(p, k - 1)
            s.apply_operator(k, dev(x), y)
            s.jacobi(k, dev(f), dev(x), z)
            s.residual_restrict(k, dev(f), dev(x), rc)
            got.append([host(y), host(z), host(rc), *s.augmented_system(k, dev(ut), c)])
    for a, b, tol in zip(*got, (1e-13, 1e-13, 1e-13, 1e-12, 1e-12, 1e-12)):
        assert rel(a, b) <= tol


@pytest.mark.parametrize("cells,levels", [(5, 7), (9, 8)], ids=["n320", "n1152"])
def test_load_2d_all_tiles(cells, levels):
    """8- and 16-row walks on a field with a negative quarter (one sign: fixed point), a zero
    one, one of 1e-95 (out of the exponents' range) and the tiles between them."""
    op, gp = _pair(**KW2, coarse_cells=cells, levels=levels)
    n = gp.cells(levels)
    u = np.random.default_rng(2300).uniform(0.2, 1.0, size=(n - 1, n - 1))
    q = (n - 1) // 4
    u[:, :q] *= -1.0
    u[:, q:2 * q] = 0.0
    u[:, 2 * q:3 * q] *= 1e-95
    ref = O.nonlinear_load(_mesh(n), u.ravel(), 1.0).reshape(n - 1, n - 1)
    with _fmg().Solver(gp) as s:
        out = _empty(gp, levels)
        s.nonlinear_load(levels, dev(u.ravel()), out)
    out = host(out).reshape(n - 1, n - 1)
    assert rel(out, ref) <= 1e-13
    inner = np.s_[:, 2 * q + 1:3 * q - 1]  # stars within the small quarter
    assert rel(out[inner], ref[inner]) <= 1e-13


def test_load_2d_not_finite():
    """Infinities and NaN reach exactly the nodes whose star they lie in."""
    op, gp = _pair(**KW2, coarse_cells=5, levels=7)
    n = gp.cells(7)
    u = np.random.default_rng(2400).uniform(0.2, 1.0, size=(n - 1, n - 1))
    u[100, 40] = np.nan
    u[7, 311] = np.inf
    ref = O.nonlinear_load(_mesh(n), u.ravel(), 1.0)
    with _fmg().Solver(gp) as s:
        out = _empty(gp, 7)
        s.nonlinear_load(7, dev(u.ravel()), out)
    out = host(out)
    ok = np.isfinite(ref)
    assert np.array_equal(np.isfinite(out), ok) and (~ok).sum() == 14
    assert rel(out[ok], ref[ok]) <= 1e-13


def test_restriction_2d_zeros_and_not_finite():
    """r_c = P^T r_f (r = f for x = 0) with a zero quarter and an infinity, n = 640."""
    op, gp = _pair(**KW2, coarse_cells=5, levels=8)
    f = np.random.default_rng(2450).normal(size=(639, 639))
    f[:, :160] = 0.0
    f[333, 401] = np.inf
    with _fmg().Solver(gp) as s:
        rc = _empty(gp, 7)
        s.residual_restrict(8, dev(f.ravel()), dev(np.zeros(f.size)), rc)
    rc = host(rc)
    ok = np.isfinite(rc)
    f[333, 401] = 0.0
    ref = O.prolongation(_mesh(320), _mesh(640)).T @ f.ravel()
    assert 1 <= (~ok).sum() <= 4 and np.all(rc[ok & (ref == 0.0)] == 0.0)
    assert np.abs((rc - ref)[ok]).max() <= 1e-13 * np.abs(ref).max()


@pytest.mark.parametrize("sign", ["one", "mixed"])
@pytest.mark.parametrize("kw,k", [(dict(KW2, coarse_cells=5, levels=7), 7),
                                  (dict(KW2, coarse_cells=7, levels=4), 4),
                                  (dict(dim=3, w_const=0.3, w_quad=(1.0, 2.0, 1.5), zeta=6.0,
                                        coarse_cells=3, levels=4), 4)],
                         ids=["2d_n320", "2d_n56", "3d_n24"])
def test_augmented_system(kw, k, sign):
    """The density stencil through its coarsening on values of one sign (fixed point, partly
    filled warps) and of both (negative entries: summed in FP64)."""
    op, gp = _pair(**kw)
    lv = O.build_hierarchy(op)
    rng = np.random.default_rng(2500 + k)
    ut = rng.uniform(0.2, 1.0, size=gp.size(k)) if sign == "one" else rng.normal(size=gp.size(k))
    psi, k0, mm = O.augmented_blocks(lv, k, ut)
    c = rng.normal(size=psi.shape[1])
    g_ref = (psi.T @ O.density_matrix(lv[k - 1].mesh, psi @ c) @ psi).toarray()
    with _fmg().Solver(gp) as s:
        K, M, G = s.augmented_system(k, dev(ut), c)
    assert rel(K, k0) <= 1e-12
    assert rel(M, mm) <= 1e-12
    assert rel(G, g_ref) <= 1e-12


@pytest.mark.parametrize("nu", [(2, 2), (1, 0), (0, 2)], ids=lambda t: f"nu{t[0]}{t[1]}")
@pytest.mark.parametrize("cells", [3, 4])
def test_vcycle_legs_3d_bit_identical(cells, nu):
    """The one-kernel legs of the 3D V-cycle (n = 6 .. 32, ragged 8 x 8 x 4 tiles) evaluate what
    the separate kernels do: component V-cycles from a random start, and whole solves."""
    fmg = _fmg()
    res = []
    for flags in (0, fmg.FMG_FLAG_SEPARATE_VCYCLE):
        p = fmg.Problem(dim=3, coarse_cells=cells, levels=4, w_const=0.2, w_quad=(1.0, 2.0, 1.5),
                        zeta=9.0, nu_pre=nu[0], nu_post=nu[1], flags=flags)
        rng = np.random.default_rng(2600)
        with fmg.Solver(p) as s:
            out = []
            for k in (2, 3, 4):
                f, x = rng.normal(size=(2, p.size(k)))
                x = dev(x)
                s.multigrid(k, dev(f), x)
                out.append(host(x))
            u = np.empty(p.size(4))
            lam, _, rc = s.solve(u)
            assert rc == 0
            res.append(out + [u, np.array([lam])])
    for a, b in zip(*res):
        assert np.array_equal(a, b)


def test_batch_of_pinned_and_other_3d_instances():
    """Mixed 3D instances with and without a level of 128 cells per side take different dense
    solvers and moment sums; a batch of both gives each the bits it has alone."""
    fmg = _fmg()
    probs = [fmg.Problem(dim=3, coarse_cells=4, levels=lv, w_quad=(1.0, 1.0, g), zeta=z,
                         precision=fmg.FMG_MIXED_FP32)
             for lv, g, z in ((3, 2.0, 30.0), (6, 1.0, 20.0), (4, 3.0, 60.0))]
    got = fmg.solve_batch(probs)
    for p, lam, u in zip(probs, got[0], got[1]):
        v = np.empty(p.size(p.levels))
        with fmg.Solver(p) as s:
            one, _, rc = s.solve(v)
        assert rc == 0 and one == lam and np.array_equal(u, v)
