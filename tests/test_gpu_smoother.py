"""GS_OP_SMOOTH and the FP64 V-cycle on the caller's vectors: the smoother against the oracle's Chebyshev iteration with
the solver's eigenvalue bound, and results that overlap an input against separate vectors, bit by bit.

Tolerance.  Per row and step, r = b - A x is off by at most tol s with s = |b| + |A|_c |x| (tol of the operator tests:
1e-12 FP64, 1e-6 FP32) plus |A|_c times the error of x; the update d = c1 d + c2 D^-1 r and x + d round a few times more.
The bound is carried through the steps below with absolute values throughout."""
import numpy as np
import pytest

from oracle.fem import System
from oracle.mesh import mesh_from_problem
from oracle.mg import chebyshev
from paper_2305_08986_gb300 import inputs
from tests.rowcheck import AbsOperators

pytestmark = pytest.mark.gpu

TOL = {64: 1e-12, 32: 1e-6}
CASES = [(2, (9, 7), 0.1, inputs.FACE_XM, 1), (2, (70, 40), 0.0, inputs.FACE_XM | inputs.FACE_YP, 4),
         (2, (33, 18), 0.05, inputs.FACE_YM, 0), (3, (5, 4, 6), 0.1, inputs.FACE_ZM, 0), (3, (9, 11, 7), 0.0, inputs.FACE_XP, 2)]


def _solver(case, prec, **opts):
    from paper_2305_08986_gb300 import gs
    dim, n, void, faces, variant = case
    p = inputs.config_random_field(dim, n, levels=1, seed=9, contrast=1e4, alpha=5.0, faces=faces, void_fraction=void)
    return p, gs.Solver.from_problem(p, mg_precision=prec, coarse_mode=1, tile_autotune=variant, restart=2, **opts)


def _reference(p, hi, b, x0, degree, tol):
    """The oracle's result and the bound on the rows of its error when every operator application is off by tol."""
    m = mesh_from_problem(p)
    sysm = System(m, p.eta, p.alpha, need_pressure=False)
    absA = AbsOperators(m, p.eta, p.alpha).A
    dinv = 1.0 / sysm.A.diagonal()
    lo = hi / 15.0
    theta, delta = 0.5 * (hi + lo), 0.5 * (hi - lo)
    sigma = theta / delta
    x = np.zeros_like(b) if x0 is None else x0.copy()
    d, ex, ed, rho = np.zeros_like(b), np.zeros_like(b), np.zeros_like(b), 1.0 / sigma
    for t in range(degree):
        rn = 1.0 / (2.0 * sigma - rho)
        c1, c2 = (0.0, 1.0 / theta) if t == 0 else (rn * rho, 2.0 * rn / delta)
        s = np.abs(b) + absA @ np.abs(x)
        r, er = b - sysm.A @ x, tol * s + absA @ ex
        d = c1 * d + c2 * dinv * r
        ed = c1 * ed + c2 * dinv * er + tol * (np.abs(d) + c2 * dinv * s)
        x = x + d
        ex = ex + ed + tol * np.abs(x)
        rho = rho if t == 0 else rn
    assert np.allclose(x, chebyshev(sysm.A, dinv, b, x0, degree, lo, hi), rtol=1e-10, atol=1e-12)
    return x, ex


@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("degree", [1, 2, 4])
@pytest.mark.parametrize("start", [False, True])
@pytest.mark.parametrize("case", CASES)
def test_smoother_against_the_oracle(case, start, degree, prec):
    import torch
    from paper_2305_08986_gb300 import gs
    p, s = _solver(case, prec, cheb_degree=degree)
    dt = torch.float64 if prec == 64 else torch.float32
    rng = np.random.default_rng(4)
    b, x0 = (torch.tensor(rng.standard_normal(p.n_u), dtype=dt, device="cuda") for _ in range(2))
    y = torch.full_like(b, float("nan"))
    kept = b.clone(), x0.clone()
    s.apply_level(0, gs.OP_SMOOTH, b, y, aux=x0 if start else None)
    assert torch.equal(b, kept[0]) and torch.equal(x0, kept[1])
    ref, bound = _reference(p, s.info().lambda_max[0], b.double().cpu().numpy(),
                            x0.double().cpu().numpy() if start else None, degree, TOL[prec])
    err = np.abs(y.double().cpu().numpy() - ref)
    assert np.all(err <= bound)


@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("steps", [1, 2])
def test_smoother_with_a_result_over_its_inputs(case, prec, steps):
    import torch
    from paper_2305_08986_gb300 import gs
    p, s = _solver(case, prec, smooth_steps=steps)
    dt = torch.float64 if prec == 64 else torch.float32
    rng = np.random.default_rng(5)
    b, x0 = (torch.tensor(rng.standard_normal(p.n_u), dtype=dt, device="cuda") for _ in range(2))
    want = torch.empty_like(b)
    s.apply_level(0, gs.OP_SMOOTH, b, want, aux=x0)
    y = b.clone()
    s.apply_level(0, gs.OP_SMOOTH, y, y, aux=x0)
    assert torch.equal(y, want)
    y = x0.clone()
    s.apply_level(0, gs.OP_SMOOTH, b, y, aux=y)
    assert torch.equal(y, want)
    for shift in (1, p.n_u // 2):  # the result begins inside, or ends inside, its right-hand side
        for lower in (False, True):
            buf = torch.zeros(p.n_u + shift, dtype=dt, device="cuda")
            x, y = (buf[shift:], buf[:p.n_u]) if lower else (buf[:p.n_u], buf[shift:])
            x.copy_(b)
            s.apply_level(0, gs.OP_SMOOTH, x, y, aux=x0)
            assert torch.equal(y, want)


@pytest.mark.parametrize("dim,n", [(2, (48, 32)), (3, (8, 12, 8))])
def test_vcycle_with_the_result_over_its_input(dim, n):
    import torch
    from paper_2305_08986_gb300 import gs
    p = inputs.config_random_field(dim, n, levels=2, seed=9, contrast=1e3, alpha=5.0, void_fraction=0.05)
    for prec in (64, 32):
        s = gs.Solver.from_problem(p, mg_precision=prec, restart=2)
        r = torch.tensor(np.random.default_rng(6).standard_normal(p.n_u), device="cuda")
        z = torch.empty_like(r)
        s.vcycle(r, z)
        y = r.clone()
        s.vcycle(y, y)
        assert torch.equal(y, z) and bool(torch.isfinite(z).all())
        buf = torch.zeros(p.n_u + 3, device="cuda", dtype=torch.float64)
        buf[3:] = r
        s.vcycle(buf[3:], buf[:p.n_u])
        assert torch.equal(buf[:p.n_u], z)
