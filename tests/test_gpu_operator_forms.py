"""The two forms of the level operators (2D from 512 cells per side, 3D FP64 from 96): fixed point
where its formats hold h^2 |W|, FP64 with stored couplings for every other potential.  An instance
takes its form whatever stands beside it in a batch or was solved before on the handle, and the
potentials of the FP64 form cost what stored couplings cost.

A box of 10 oscillator lengths leaves the formats at n = 512 (2D: h^2 W / 12 = 0.016) and n = 96
(3D: h^4 (wx + wy + wz) = 2^-10.7); the same traps in a unit box are far inside them."""
import numpy as np
import pytest

from tests.test_gpu_parity import _fmg

torch = pytest.importorskip("torch")

KINDS = {
    "2d": dict(dim=2, coarse_cells=8, levels=7, w_quad=(1.0, 4.0, 0.0), box_len=10.0),
    "2d_mixed": dict(dim=2, coarse_cells=8, levels=7, w_quad=(1.0, 4.0, 0.0), box_len=10.0,
                     precision=1),
    "2d_literal": dict(dim=2, coarse_cells=8, levels=7, w_quad=(1.0, 4.0, 0.0), box_len=10.0,
                       operator_form=1),
    "2d_chebyshev": dict(dim=2, coarse_cells=8, levels=7, w_quad=(1.0, 4.0, 0.0), box_len=10.0,
                         smoother=1),
    "3d": dict(dim=3, coarse_cells=3, levels=6, w_quad=(1.0, 1.0, 4.0), box_len=10.0),
}
WEAK = 1e-4  # factor that takes a trap into the formats


def _problem(kind, scale=1.0, zeta=20.0):
    kw = dict(KINDS[kind])
    kw["w_quad"] = tuple(scale * w for w in kw["w_quad"])
    return _fmg().Problem(**kw, zeta=zeta)


def _solve(s, p):
    u = np.empty(p.size(p.levels))
    lam, st, rc = s.solve(u, stats=True)
    assert rc == 0
    return lam, u, st


def _alone(p):
    with _fmg().Solver(p) as s:
        return _solve(s, p)


def test_couplings_are_stored_for_potentials_outside_the_formats():
    """Device bytes of a handle: four (eight) more arrays on the levels of the FP64 form."""
    fmg = _fmg()
    for kind, arrays in (("2d", 4), ("3d", 8)):
        inside, outside = _problem(kind, WEAK), _problem(kind)
        nodes = (inside.cells(inside.levels) + 1) ** inside.dim
        extra = fmg.estimate_bytes([outside]) - fmg.estimate_bytes([inside])
        assert extra > 0.9 * arrays * 8 * nodes


@pytest.mark.gpu
@pytest.mark.parametrize("kind", sorted(KINDS))
def test_batch_of_both_forms_equals_solves_alone(kind):
    probs = [_problem(kind, 1.0, 30.0), _problem(kind, WEAK, 10.0), _problem(kind, 1.0, 5.0),
             _problem(kind, WEAK, 60.0)]
    with _fmg().BatchSolver(probs) as b:
        lams, us, sts, codes = b.solve_all(with_u=True, stats=True)
    for p, lam, u, st, code in zip(probs, lams, us, sts, codes):
        one, v, st1 = _alone(p)
        assert code == 0 and lam == one and np.array_equal(u, v)
        assert st.identity_defect == st1.identity_defect


@pytest.mark.gpu
@pytest.mark.parametrize("kind", sorted(KINDS))
def test_set_params_across_the_limit(kind):
    """The handle takes the form of the new potential: bits of a fresh handle, in both directions,
    for solves and for the component calls."""
    fmg = _fmg()
    steps = [_problem(kind, WEAK), _problem(kind), _problem(kind, WEAK, 3.0), _problem(kind, 1.0, 7.0)]
    k = steps[0].levels
    x = torch.randn(steps[0].size(k), dtype=torch.float64, device="cuda",
                    generator=torch.Generator("cuda").manual_seed(5))

    def components(s):
        y, z = torch.empty_like(x), torch.empty_like(x)
        s.apply_operator(k, x, y)
        s.jacobi(k, x, y, z)
        torch.cuda.synchronize()
        return y.cpu().numpy(), z.cpu().numpy()

    with fmg.Solver(steps[0]) as s:
        for p in steps:
            s.set_params(p)
            with fmg.Solver(p) as fresh:
                for a, b in zip(components(s), components(fresh)):
                    assert np.array_equal(a, b)
                one, v, _ = _solve(fresh, p)
            lam, u, _ = _solve(s, p)
            assert lam == one and np.array_equal(u, v)


@pytest.mark.gpu
def test_set_params_out_of_memory_keeps_the_handle():
    """The couplings of the new form don't fit: refused, and the old parameters still solve."""
    fmg = _fmg()
    p, q = _problem("2d", WEAK), _problem("2d")
    with fmg.Solver(p) as s:
        lam, u, _ = _solve(s, p)
        fmg.inject_alloc_failure(1)
        try:
            with pytest.raises(fmg.FmgError) as e:
                s.set_params(q)
        finally:
            fmg.inject_alloc_failure(-1)
        assert e.value.code == fmg.FMG_ENOMEM
        lam2, u2, _ = _solve(s, p)
        assert lam2 == lam and np.array_equal(u2, u)
        s.set_params(q)
        lam3, u3, _ = _solve(s, q)
    one, v, _ = _alone(q)
    assert lam3 == one and np.array_equal(u3, v)


@pytest.mark.gpu
def test_served_requests_of_both_forms_equal_solves_alone():
    fmg = _fmg()
    probs = [_problem("2d", 1.0 if i % 2 else WEAK, 5.0 * i) for i in range(8)]
    res, st = fmg.serve(probs, [1e-3 * i for i in range(8)], max_batch=4, max_inflight=2,
                        batch_window_s=0.005, with_u=True)
    assert st["completed"] == len(probs)
    for p, r in zip(probs, res):
        lam, u, _ = _alone(p)
        assert r["status"] == 0 and r["lambda"] == lam and np.array_equal(r["u"], u)


def _multigrid_ms(p):
    with _fmg().Solver(p) as s:
        k = p.levels
        f = torch.randn(p.size(k), dtype=torch.float64, device="cuda")
        x = torch.zeros_like(f)
        st = torch.cuda.Stream()
        ts = []
        for _ in range(25):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record(st)
            s.multigrid(k, f, x, st.cuda_stream)
            b.record(st)
            st.synchronize()
            ts.append(a.elapsed_time(b))
    return sorted(ts)[len(ts) // 2]


@pytest.mark.gpu
def test_time_of_potentials_outside_the_formats():
    """3D V-cycles at n = 192: the FP64 kernels with stored couplings take 1.5 times what fixed point
    takes; couplings formed from tables at every use took 4 times as much."""
    kw = dict(dim=3, coarse_cells=3, levels=7, w_quad=(1.0, 1.0, 4.0), zeta=20.0)
    fmg = _fmg()
    inside, outside = fmg.Problem(**kw), fmg.Problem(**kw, box_len=10.0)
    assert _multigrid_ms(outside) <= 2.5 * _multigrid_ms(inside)
