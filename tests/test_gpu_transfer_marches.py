"""Restriction and interpolation of the velocity on meshes of several strips of 29 coarse columns and of several rows
(3D: planes) per warp: one column more and less than a strip, the last row of a march short, obstacles and free faces.

The prolongation comes from the oracle's 1D matrices; tolerances per row as in test_gpu_transfers.py."""
import numpy as np
import pytest

from oracle.mesh import mesh_from_problem
from oracle.mg import prolongation
from paper_2305_08986_gb300 import inputs
from tests.rowcheck import row_error

pytestmark = pytest.mark.gpu

CASES = [
    (2, (28, 20), 0.0, inputs.FACE_XM), (2, (1024, 600), 0.0, inputs.FACE_YP), (2, (1000, 604), 0.05, inputs.FACE_XM),
    (3, (28, 4, 6), 0.0, None), (3, (60, 6, 4), 0.1, inputs.FACE_XP), (3, (64, 36, 32), 0.0, inputs.FACE_ZM | inputs.FACE_XM),
    (3, (4, 40, 64), 0.05, None),
]


@pytest.mark.parametrize("prec,tol", [(64, 1e-14), (32, 2e-6)])
@pytest.mark.parametrize("dim,n,void,faces", CASES)
def test_transfers_on_several_strips(dim, n, void, faces, prec, tol):
    import torch
    from paper_2305_08986_gb300 import gs
    p = inputs.config_random_field(dim, n, levels=2, seed=5, contrast=1e3, alpha=7.0, faces=faces, void_fraction=void)
    s = gs.Solver.from_problem(p, mg_precision=prec, coarse_mode=1, restart=2)
    fine = mesh_from_problem(p)
    P = prolongation(fine.coarsen(), fine)
    rng = np.random.default_rng(3)
    dt = torch.float64 if prec == 64 else torch.float32
    rf = torch.tensor(rng.standard_normal(P.shape[0]), dtype=dt, device="cuda")
    xc = torch.tensor(rng.standard_normal(P.shape[1]), dtype=dt, device="cuda")
    rc = torch.full_like(xc, float("nan"))
    s.apply_level(1, gs.OP_RESTRICT, rf, rc)
    r = rf.double().cpu().numpy()
    assert row_error(rc.double().cpu().numpy(), P.T @ r, abs(P.T).tocsr(), r) <= tol
    xf = torch.zeros_like(rf)
    s.apply_level(1, gs.OP_PROLONGATE, xc, xf)
    x = xc.double().cpu().numpy()
    assert row_error(xf.double().cpu().numpy(), P @ x, abs(P).tocsr(), x) <= tol
