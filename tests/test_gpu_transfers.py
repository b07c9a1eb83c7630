"""Velocity transfers (gs_xfer.cu) against the oracle's interpolation at the edges of their boxes: 32 x 8 (2D) and
8 x 8 x 4 (3D) coarse nodes, 64 x 16 and 16 x 16 x 8 fine nodes, with obstacle cells and free faces.

Tolerances per row, relative to the row's sum of |weight| |value|: at most 8 rounded operations per axis in
sequence, 24 u in 3D; 24 * 1.1e-16 < 1e-14 and 24 * 6e-8 = 1.4e-6 < 2e-6.
"""
import numpy as np
import pytest

from oracle.mesh import mesh_from_problem
from oracle.mg import Hierarchy
from paper_2305_08986_gb300 import inputs
from tests.rowcheck import row_error

pytestmark = pytest.mark.gpu

CASES = [
    (2, (4, 4), 0.0, inputs.FACE_XM), (2, (30, 6), 0.0, None), (2, (32, 8), 0.1, inputs.FACE_YP),
    (2, (64, 16), 0.0, inputs.FACE_XM | inputs.FACE_YM), (2, (66, 18), 0.1, None),
    (3, (4, 4, 4), 0.0, inputs.FACE_XM), (3, (8, 8, 4), 0.1, None), (3, (10, 6, 8), 0.0, inputs.FACE_ZP),
]


@pytest.mark.parametrize("prec,tol", [(64, 1e-14), (32, 2e-6)])
@pytest.mark.parametrize("dim,n,void,faces", CASES)
def test_transfers_at_box_edges(dim, n, void, faces, prec, tol):
    import torch
    from paper_2305_08986_gb300 import gs
    p = inputs.config_random_field(dim, n, levels=2, seed=5, contrast=1e3, alpha=7.0, faces=faces, void_fraction=void)
    s = gs.Solver.from_problem(p, mg_precision=prec)
    P = Hierarchy(mesh_from_problem(p), p.eta, p.alpha, 2).levels[1].P
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
