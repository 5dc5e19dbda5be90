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


def _fields(n, dim):
    """Values of one sign and of both that fall by 2^-40 across 32 nodes of one axis, a wide
    Gaussian, and such a slope beside a patch of zeros."""
    rng = np.random.default_rng(3300)
    shape = (n - 1,) * dim
    x = np.arange(1, n, dtype=np.float64)
    out = {}
    for axis in range(dim):
        line = [1] * dim
        line[dim - 1 - axis] = n - 1
        decay = np.exp2(-1.25 * x).reshape(line)
        out[f"decay{axis}"] = decay * rng.uniform(0.5, 1.0, size=shape)
        out[f"mixed{axis}"] = decay * rng.normal(size=shape)
    r2 = sum(np.meshgrid(*[(x / n - 0.4) ** 2] * dim, indexing="ij"))
    out["gauss"] = np.exp(-150.0 * r2)
    patch = out["decay0"].copy()
    patch[n // 3:n // 2] = 0.0
    out["zeros"] = patch
    return out


def _star_max(v):
    """The largest magnitude of each node's stencil (its 3^dim box: the stencil and corners)."""
    from scipy.ndimage import maximum_filter

    return maximum_filter(np.abs(v), size=3, mode="constant")


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_every_node_2d(precision):
    """n = 640.  Rounding of at most 16 units of 2^-58 of the largest of 6 x 6 nodes, which lies at
    most 2^6.25 above a node's own stencil here: 2^-47 of it; 1e-13, as for values of one size."""
    from oracle import fmg_oracle as O

    fmg = _fmg()
    op = O.Problem(dim=2, coarse_cells=5, levels=8, w_const=0.3, w_quad=(1.0, 2.5, 0.0), zeta=7.0)
    p = fmg.Problem(dim=2, coarse_cells=5, levels=8, w_const=0.3, w_quad=(1.0, 2.5, 0.0), zeta=7.0,
                    precision=fmg.FMG_FP64 if precision == "fp64" else fmg.FMG_MIXED_FP32)
    coarse = O.Level(O.Mesh(2, 320, 1.0), None, None, None, None, None, None)
    lev = O.build_level(op, 8, coarse)
    n = 640
    y = torch.empty(p.size(8), dtype=torch.float64, device="cuda")
    fields = _fields(n, 2)
    with fmg.Solver(p) as s:
        for name, x in fields.items():
            f = fields["mixed0" if name != "mixed0" else "decay1"]
            top = np.maximum(8 * _star_max(x), np.abs(f))
            s.apply_operator(8, dev(x.ravel()), y)
            assert (np.abs(host(y) - lev.L @ x.ravel()) <= 1e-13 * 8 * _star_max(x).ravel()).all(), name
            s.jacobi(8, dev(f.ravel()), dev(x.ravel()), y)
            ref = O.jacobi(lev, f.ravel(), x.ravel(), op.omega)
            assert (np.abs(host(y) - ref) <= 1e-13 * top.ravel()).all(), name


def test_every_node_3d():
    """n = 96.  Blocks whose columns hold a stencil below 2^-20 of the block's largest value are
    evaluated in FP64; in the others 12 units of 2^-57 (and 2^-50 times h^4 |W''| of the formats'
    limit) leave 2^-32 of a node's own stencil; 1e-9."""
    kw = dict(dim=3, coarse_cells=3, levels=6, w_const=0.3, w_quad=(1.0, 2.0, 1.5))
    n = 96
    fields = _fields(n, 3)
    got = []
    for s in _mixed_and_fp64(**kw):
        with s:
            y = torch.empty(s.level_size(6), dtype=torch.float64, device="cuda")
            rows = []
            for name, x in fields.items():
                f = fields["mixed0" if name != "mixed0" else "decay1"] / n
                s.apply_operator(6, dev(x.ravel()), y)
                rows.append(host(y).copy())
                s.jacobi(6, dev(f.ravel()), dev(x.ravel()), y)
                rows.append(host(y).copy())
            got.append(rows)
    for i, (name, x) in enumerate(fields.items()):
        f = fields["mixed0" if name != "mixed0" else "decay1"] / n
        star = _star_max(x).ravel()
        a, b = got[0][2 * i], got[1][2 * i]
        assert (np.abs(a - b) <= 1e-9 * 12.0 / n * star).all(), name
        # Jacobi: omega / D is below n / 9
        top = np.maximum(12.0 / n * star, np.abs(f.ravel())) * n / 9
        a, b = got[0][2 * i + 1], got[1][2 * i + 1]
        assert (np.abs(a - b) <= 1e-9 * top).all(), name


def test_right_hand_side_of_wide_range_from_zero_3d():
    """x = 0: the residual is f at every node, whatever the range of f (n = 96), to rounding in its
    restriction."""
    kw = dict(dim=3, coarse_cells=3, levels=6, w_const=0.3, w_quad=(1.0, 2.0, 1.5))
    got = []
    for s in _mixed_and_fp64(**kw):
        with s:
            rc = torch.empty(s.level_size(5), dtype=torch.float64, device="cuda")
            f = _fields(96, 3)["decay0"]
            s.residual_restrict(6, dev(f.ravel()), dev(np.zeros(f.size)), rc)
            got.append(host(rc))
    assert (np.abs(got[0] / got[1] - 1.0) <= 1e-9).all()


@pytest.mark.parametrize("box", [0.01, 5.0, 30.0])
def test_box_length_2d(box):
    """n = 640 on boxes of other lengths (0.01, 5: fixed point; 30: FP64 with stored couplings), to
    1e-13 of the largest value, as test_gpu_fixed_point has it on the unit box."""
    from oracle import fmg_oracle as O

    fmg = _fmg()
    kw = dict(dim=2, coarse_cells=5, levels=8, w_const=0.3, w_quad=(1.0, 4.0, 0.0), zeta=7.0,
              box_len=box)
    op, p = O.Problem(**kw), fmg.Problem(**kw)
    inside = fmg.Problem(**{**kw, "w_quad": (0.0, 0.0, 0.0)})
    stores = fmg.estimate_bytes([p]) > fmg.estimate_bytes([inside]) + 4 * 8 * 640 ** 2
    assert stores == (box == 30.0)
    lev = O.build_level(op, 8, O.Level(O.Mesh(2, 320, box), None, None, None, None, None, None))
    rng = np.random.default_rng(3500)
    x, f = rng.normal(size=(2, p.size(8)))
    y = torch.empty(p.size(8), dtype=torch.float64, device="cuda")
    rc = torch.empty(p.size(7), dtype=torch.float64, device="cuda")
    with fmg.Solver(p) as s:
        s.apply_operator(8, dev(x), y)
        ref = lev.L @ x
        assert np.abs(host(y) - ref).max() <= 1e-13 * np.abs(ref).max()
        s.jacobi(8, dev(f), dev(x), y)
        ref = O.jacobi(lev, f, x, op.omega)
        assert np.abs(host(y) - ref).max() <= 1e-13 * np.abs(ref).max()
        s.residual_restrict(8, dev(f), dev(x), rc)
        ref = lev.P.T @ (f - lev.L @ x)
        assert np.abs(host(rc) - ref).max() <= 1e-13 * np.abs(ref).max()


@pytest.mark.parametrize("box", [0.01, 3.0])
def test_box_length_3d(box):
    """n = 96: fixed point against FP64 with stored couplings, 1e-13 of the largest value."""
    kw = dict(dim=3, coarse_cells=3, levels=6, w_const=0.3, w_quad=(1.0, 2.0, 1.5), box_len=box)
    rng = np.random.default_rng(3600)
    x, f = rng.normal(size=(2, 95 ** 3))
    got = []
    for s in _mixed_and_fp64(**kw):
        with s:
            y, z = (torch.empty(x.size, dtype=torch.float64, device="cuda") for _ in range(2))
            s.apply_operator(6, dev(x), y)
            s.jacobi(6, dev(f * box / 96), dev(x), z)
            got.append((host(y), host(z)))
    for a, b in zip(*got):
        assert np.abs(a - b).max() <= 1e-13 * np.abs(b).max()
