"""diag(A) of an FP32 level is rounded once: within half a unit of the diagonal in FP64, on meshes with an eta per cell
that FP32 holds exactly (2^-24 relative, and 1e-14 for the FP64 sums)."""
import numpy as np
import pytest

from oracle.fem import System
from oracle.mesh import mesh_from_problem
from paper_2305_08986_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,n,void", [(2, (37, 29), 0.0), (2, (64, 20), 0.1), (3, (7, 6, 9), 0.0), (3, (5, 8, 4), 0.1)])
def test_fp32_diagonal_is_rounded_once(dim, n, void):
    import torch
    from paper_2305_08986_gb300 import gs
    p = inputs.config_random_field(dim, n, levels=1, seed=9, contrast=1e4, alpha=5.0, void_fraction=void)
    p.eta = p.eta.astype(np.float32).astype(np.float64)
    s = gs.Solver.from_problem(p, mg_precision=32, coarse_mode=1, restart=2)
    d = torch.empty(p.n_u, dtype=torch.float32, device="cuda")
    s.apply_level(0, gs.OP_DIAG_A, None, d)
    want = System(mesh_from_problem(p), p.eta, p.alpha, need_pressure=False).A.diagonal()
    assert np.max(np.abs(d.double().cpu().numpy() / want - 1.0)) <= 2.0 ** -24 + 1e-14
