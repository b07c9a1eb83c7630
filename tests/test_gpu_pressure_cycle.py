"""The pressure V-cycle with two launches per level (gs_q1cycle.cu) against the oracle's, at the edges of its
boxes: 16 x 4 (2D) and 4 x 4 x 2 (3D) coarse nodes exactly, one more, and several, with obstacle cells and outflow.

Tolerances.  FP64: that of the existing cycle test.  FP32: each level rounds about ten operator sums (6e-8
each), and the coarse inverse amplifies the error of its right-hand side by at most the condition number of
the coarse Laplacian, below 300 on these meshes: 300 * 6e-8 * a few = 1e-4.
"""
import numpy as np
import pytest

from oracle.mesh import mesh_from_problem
from paper_2305_08986_gb300 import inputs

pytestmark = pytest.mark.gpu

CASES = [
    (2, (30, 6), 2, 0.0, None),                       # one box
    (2, (32, 8), 2, 0.0, inputs.FACE_XM | inputs.FACE_YM | inputs.FACE_YP),
    (2, (68, 36), 3, 0.1, inputs.FACE_XM),
    (2, (4, 4), 2, 0.0, inputs.FACE_YP),
    (3, (6, 6, 2), 2, 0.0, None),                     # one box
    (3, (8, 8, 4), 2, 0.1, inputs.FACE_ZM | inputs.FACE_XP),
    (3, (20, 12, 8), 3, 0.0, inputs.FACE_YM),
]


@pytest.mark.parametrize("prec,tol", [(64, 1e-10), (32, 1e-4)])
@pytest.mark.parametrize("dim,n,levels,void,faces", CASES)
def test_pressure_cycle_at_box_edges(dim, n, levels, void, faces, prec, tol):
    import torch
    from oracle.pressure import PressureHierarchy
    from paper_2305_08986_gb300 import gs
    p = inputs.config_random_field(dim, n, levels=levels, seed=3, contrast=1e3, alpha=7.0, faces=faces, void_fraction=void)
    s = gs.Solver.from_problem(p, mg_precision=prec)
    m = mesh_from_problem(p)
    dt = torch.float64 if prec == 64 else torch.float32
    x = torch.tensor(np.random.default_rng(12).standard_normal(m.Np), dtype=dt, device="cuda")
    y = torch.full_like(x, float("nan"))
    s.apply_level(levels - 1, gs.OP_PLAP_INV, x, y)
    ref = PressureHierarchy(m, levels, degree=2).apply_inverse(x.double().cpu().numpy())
    got = y.double().cpu().numpy()
    assert np.linalg.norm(got - ref) <= tol * np.linalg.norm(ref)
