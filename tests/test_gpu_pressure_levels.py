"""Which levels of the pressure V-cycle run as two launches (gs_q1cycle.cu) and which as one launch per step: by the
launches of a call, and the cycle against the oracle's where the two kinds meet.

A general level takes the smoother's start from zero and one step, residual, restriction, interpolation and two steps;
the start is part of the restriction of a general level above it, and the finest one first takes the masked copy of
its right-hand side.  The dense coarse solve and the masked copy of the result are one launch each.

Tolerances as in test_gpu_pressure_cycle.py."""
import numpy as np
import pytest

from oracle.mesh import mesh_from_problem
from paper_2305_08986_gb300 import inputs

pytestmark = pytest.mark.gpu


def _problem(dim, n, levels, faces=None, void=0.0):
    return inputs.config_random_field(dim, n, levels=levels, seed=3, contrast=1e3, alpha=7.0, faces=faces, void_fraction=void)


def _apply(p, prec, seed=12):
    import torch
    from paper_2305_08986_gb300 import gs
    s = gs.Solver.from_problem(p, mg_precision=prec)
    dt = torch.float64 if prec == 64 else torch.float32
    x = torch.tensor(np.random.default_rng(seed).standard_normal(p.n_pnodes), dtype=dt, device="cuda")
    y = torch.full_like(x, float("nan"))
    before = s.info().kernel_launches
    s.apply_level(p.levels - 1, gs.OP_PLAP_INV, x, y)
    return x.double().cpu().numpy(), y.double().cpu().numpy(), s.info().kernel_launches - before


@pytest.mark.parametrize("dim,n,levels,prec,general", [
    (3, (16, 16, 16), 3, 64, 2), (3, (8, 8, 8), 2, 64, 1), (3, (16, 16, 16), 3, 32, 0), (2, (64, 64), 4, 64, 0),
    (2, (64, 64), 4, 32, 0), (2, (512, 272), 5, 64, 1), (2, (512, 272), 5, 32, 0), (3, (64, 64, 64), 5, 32, 1)])
def test_launches_per_level(dim, n, levels, prec, general):
    """The finest `general` levels in seven launches each, the start being fused from the second on."""
    launches = 2 * (levels - 1 - general) + 1 + 1  # halves, coarse solve, masked copy of the result
    if general:
        launches += 1 + 7 * general - (general - 1)
    assert _apply(_problem(dim, n, levels), prec)[2] == launches


@pytest.mark.parametrize("dim,n,levels,void,faces,prec,tol", [
    (2, (512, 272), 5, 0.05, inputs.FACE_XM | inputs.FACE_YM, 64, 1e-10),
    (3, (64, 64, 64), 5, 0.0, inputs.FACE_ZM, 32, 1e-4),
    (3, (16, 12, 8), 3, 0.1, inputs.FACE_XP, 64, 1e-10)])
def test_cycle_across_the_two_kinds_of_level(dim, n, levels, void, faces, prec, tol):
    from oracle.pressure import PressureHierarchy
    p = _problem(dim, n, levels, faces, void)
    x, got, _ = _apply(p, prec)
    ref = PressureHierarchy(mesh_from_problem(p), levels, degree=2).apply_inverse(x)
    assert np.linalg.norm(got - ref) <= tol * np.linalg.norm(ref)
