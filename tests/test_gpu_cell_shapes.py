"""The 8 x 8 tiles (2D) and the march (3D) against the oracle at the edges of their patches.

2D: a CTA owns 7 x 7 cells; sizes of a few cells one tile exactly, one more and several, each against the 32 x 16
tiles bitwise (every variant sums a node's cells in the same order) and against the oracle.  3D: meshes of a few
cells, thin along each axis, and of several patches and segments, in both precisions.  Tolerances per row as in
test_gpu_ops.py: 1e-12 (FP64), 1e-6 (FP32).
"""
import numpy as np
import pytest

from oracle.fem import System
from oracle.mesh import mesh_from_problem
from paper_2305_08986_gb300 import inputs
from tests.rowcheck import AbsOperators, row_error

pytestmark = pytest.mark.gpu


def _apply(p, **opts):
    """[(x, K x)], [(x_u, A x_u)] in FP64 and FP32, and the smoother's output (None as its input)."""
    import torch
    from paper_2305_08986_gb300 import gs
    s = gs.Solver.from_problem(p, coarse_mode=1, **opts)
    rng = np.random.default_rng(2)
    x = torch.tensor(rng.standard_normal(s.n_total), device="cuda")
    y = torch.full_like(x, float("nan"))
    s.vmult(x, y)
    out = [(x, y)]
    for dt in (torch.float64, torch.float32):
        xa = x[:s.n_u].to(dt).contiguous()
        ya = torch.full_like(xa, float("nan"))
        s.vmult_A(xa, ya)
        out.append((xa, ya))
    xa = x[:s.n_u].to(torch.float64 if opts.get("mg_precision") == 64 else torch.float32).contiguous()
    z = torch.full_like(xa, float("nan"))
    s.apply_level(0, gs.OP_SMOOTH, xa, z, aux=2.0 * xa)
    return out + [(None, z)]


def _check_rows(p, out):
    m = mesh_from_problem(p)
    sysm = System(m, p.eta, p.alpha)
    ab = AbsOperators(m, p.eta, p.alpha)
    for (x, y), ref, scale, tol in zip(out, (sysm.K, sysm.A, sysm.A), (ab.K, ab.A, ab.A), (1e-12, 1e-12, 1e-6)):
        xr = x.double().cpu().numpy()
        assert row_error(y.double().cpu().numpy(), ref @ xr, scale, xr) <= tol


@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("n,void,faces", [((3, 2), 0.0, inputs.FACE_XM), ((7, 7), 0.0, None), ((8, 15), 0.0, inputs.FACE_XM),
                                          ((9, 2), 0.0, inputs.FACE_YP), ((29, 22), 0.1, inputs.FACE_XM | inputs.FACE_YM)])
def test_small_tiles_match_large_tiles(n, void, faces, prec):
    import torch
    p = inputs.config_random_field(2, n, seed=4, contrast=1e6, alpha=3.0, faces=faces, void_fraction=void)
    large = _apply(p, tile_autotune=1, mg_precision=prec)
    small = _apply(p, tile_autotune=6, mg_precision=prec)
    for (_, a), (_, b) in zip(large, small):
        assert torch.equal(a, b) and bool(torch.isfinite(a).all())
    _check_rows(p, small)


@pytest.mark.parametrize("n,void,faces", [((2, 2, 2), 0.0, inputs.FACE_XM), ((9, 2, 2), 0.0, inputs.FACE_ZP),
                                          ((2, 7, 3), 0.0, inputs.FACE_YM), ((3, 2, 17), 0.1, None),
                                          ((13, 14, 5), 0.1, inputs.FACE_XP | inputs.FACE_YP)])
def test_march_at_mesh_edges(n, void, faces):
    p = inputs.config_random_field(3, n, seed=4, contrast=1e6, alpha=3.0, faces=faces, void_fraction=void)
    _check_rows(p, _apply(p))
