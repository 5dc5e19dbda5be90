"""The cubic load and the auxiliary right-hand side node by node, on fields of one sign and wide
range, for every walk (2D: 4, 8 and 16 rows; 3D: 4 and 16 planes) and node by node below them.

N(u) at a node is a sum of positive terms, so FP64 keeps it to rounding wherever u lies in its
tile.  The fixed-point walks promise 4e-10 of every node's own value (fixed.cuh); 1e-9 here.  The
reference is the closed form |K| 6 d!/(d + 4)! [h3 + u_p h2 + u_p^2 h1 + u_p^3] per simplex in
FP64 (relative error some 1e-15)."""
import itertools
import math

import numpy as np
import pytest

from tests.test_gpu_parity import _fmg, dev, host

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZES = {  # dim, coarse cells, levels: n = 48, 80, 320, 1152 and 24, 48, 128
    "2d_n48": (2, 3, 5), "2d_n80": (2, 5, 5), "2d_n320": (2, 5, 7), "2d_n1152": (2, 9, 8),
    "3d_n24": (3, 3, 4), "3d_n48": (3, 3, 5), "3d_n128": (3, 4, 6),
}


def _references(u, h):
    """N(u) and M u of the interior values u on the box of spacing h."""
    dim = u.ndim
    p = np.pad(u, 1)
    vol = h ** dim / math.factorial(dim)
    nl, mu = np.zeros_like(p), np.zeros_like(p)
    m = p.shape[0] - 1
    at = lambda o: tuple(slice(a, a + m) for a in o)
    for perm in itertools.permutations(range(dim)):
        v = [np.zeros(dim, int)]
        for axis in perm:
            v.append(v[-1] + np.eye(dim, dtype=int)[axis])
        w = [p[at(o)] for o in v]
        h1, p2, p3 = sum(w), sum(x * x for x in w), sum(x ** 3 for x in w)
        h2 = (h1 * h1 + p2) / 2
        h3 = (h1 ** 3 + 3 * h1 * p2 + 2 * p3) / 6
        for o, x in zip(v, w):
            nl[at(o)] += vol * 6 * math.factorial(dim) / math.factorial(dim + 4) * (
                h3 + x * (h2 + x * (h1 + x)))
            mu[at(o)] += vol / ((dim + 1) * (dim + 2)) * (h1 + x)
    inner = (slice(1, -1),) * dim
    return nl[inner].ravel(), mu[inner].ravel()


def _field(kind, dim, n):
    x = np.arange(1, n) / n
    rng = np.random.default_rng(3100)
    jitter = rng.uniform(0.9, 1.0, size=(n - 1,) * dim)
    axes = np.meshgrid(*[x] * dim, indexing="ij")
    if kind == "sine":  # far below a tile's largest value next to edges and corners
        u = np.prod([np.sin(np.pi * a) for a in axes], axis=0)
    elif kind == "steep":  # a ground state in a steep trap
        u = np.prod([np.sin(np.pi * a) for a in axes], axis=0) * np.exp(
            -40.0 * sum((a - 0.3) ** 2 for a in axes))
    else:  # 2^-40 across 32 nodes of one axis
        u = np.exp2(-1.25 * n * axes[dim - 1 - int(kind[-1])])
    return u * jitter


FIELDS = ["sine", "steep", "decay0", "decay1"]


@pytest.mark.parametrize("kind", FIELDS)
@pytest.mark.parametrize("size,walks", [(s, False) for s in sorted(SIZES)] +
                         [("2d_n48", True), ("3d_n24", True)])
def test_every_node_keeps_its_digits(size, walks, kind):
    """walks: forced below the levels that take them by default (n = 64 in 2D, 32 in 3D)."""
    dim, cells, levels = SIZES[size]
    fmg = _fmg()
    zeta, lam = 50.0, 17.0
    p = fmg.Problem(dim=dim, coarse_cells=cells, levels=levels, w_quad=(1.0, 1.0, 1.0), zeta=zeta,
                    flags=fmg.FMG_FLAG_NO_AUTOTUNE | (fmg.FMG_FLAG_STAR_WALKS if walks else 0))
    n = p.cells(levels)
    u = _field(kind, dim, n)
    for sign in (1.0, -1.0):
        nl, mu = _references(sign * u, 1.0 / n)
        out = torch.empty(p.size(levels), dtype=torch.float64, device="cuda")
        with fmg.Solver(p) as s:
            s.nonlinear_load(levels, dev(sign * u.ravel()), out)
            got = host(out).copy()
            s.aux_rhs(levels, lam, dev(sign * u.ravel()), out)
            f = host(out)
        tiny = np.abs(nl) < 1e-290  # underflow of u^3
        assert np.abs(got - nl)[~tiny].max() > 0.0  # (not the same arithmetic)
        assert (np.abs(got - nl)[~tiny] <= 1e-9 * np.abs(nl[~tiny])).all()
        assert (np.abs(got[tiny]) <= 1e-289).all()
        scale = np.abs(lam * mu) + np.abs(zeta * nl)
        assert (np.abs(f - (lam * mu - zeta * nl)) <= 1e-9 * scale + 1e-300).all()
