"""The 3D march on the shapes of larger meshes: patches in both directions, segments of several layers, against a cell by
cell reference, row by row, and with segments of at most four layers, bit by bit (tests/test_march_shape.py has the shapes
that these meshes get).

The reference applies the oracle's dense cell matrices to all cells at once, and their absolute values for the scale of a
row (tests/rowcheck.py); tolerances as in test_gpu_ops.py."""
import numpy as np
import pytest

from oracle.fem import CellMatrices
from oracle.mesh import mesh_from_problem
from paper_2305_08986_gb300 import inputs
from tests.rowcheck import row_error
from tests.test_march_shape import SEVERAL_PATCHES

pytestmark = pytest.mark.gpu


class Cells:
    """K x with the constraints of oracle.fem.System, matrix-free; absolute: of |A_K|, |B_K|."""

    def __init__(self, p):
        self.m = mesh_from_problem(p)
        cm = CellMatrices(3, self.m.h)
        act = self.m.active_cells()
        self.u, self.q = self.m.cell_udofs()[act], self.m.cell_pnodes()[act]
        self.eta = np.asarray(p.eta)[act][:, None]
        self.alpha, self.cm = p.alpha, cm
        self.con = self.m.dof_constrained()

    def __call__(self, x, absolute=False):
        n_u = self.m.n_u
        f = np.abs if absolute else (lambda a: a)
        z = np.where(self.con, 0.0, f(x))
        xu, xp = z[:n_u][self.u], z[n_u:][self.q]
        if absolute:  # |alpha M + eta A| <= alpha |M| + eta |A|
            yu = self.alpha * (xu @ np.abs(self.cm.mass)) + self.eta * (xu @ np.abs(self.cm.visc))
        else:
            yu = self.alpha * (xu @ self.cm.mass) + self.eta * (xu @ self.cm.visc)
        div = f(self.cm.div)
        yv, yp = yu, xu @ div.T
        a = np.bincount(self.u.ravel(), yv.ravel(), n_u)
        bt = np.bincount(self.u.ravel(), (xp @ div).ravel(), n_u)
        b = np.bincount(self.q.ravel(), yp.ravel(), self.m.Np)
        y = np.concatenate([a + bt, b])
        return np.where(self.con, f(x), y), np.where(self.con[:n_u], f(x[:n_u]), a)


class Scale:
    """The row scale in the form row_error takes: (scale @ |x|)."""

    def __init__(self, rows):
        self.rows = rows

    def __matmul__(self, _):
        return self.rows


@pytest.mark.parametrize("n", SEVERAL_PATCHES)
@pytest.mark.parametrize("void,faces", [(0.0, inputs.FACE_XM), (0.05, inputs.FACE_YP | inputs.FACE_ZM)])
def test_march_on_several_patches_and_layers(n, void, faces):
    import torch
    from paper_2305_08986_gb300 import gs
    p = inputs.config_random_field(3, n, seed=4, contrast=1e6, alpha=3.0, faces=faces, void_fraction=void)
    ref = Cells(p)
    rng = np.random.default_rng(8)
    x = rng.standard_normal(p.n_total)
    b, d0 = rng.standard_normal(p.n_u), rng.standard_normal(p.n_u)
    for variant in (1, 2):  # segments by size, of at most four layers
        outs = []
        for prec, dt, tol in ((64, torch.float64, 1e-12), (32, torch.float32, 1e-6)):
            s = gs.Solver.from_problem(p, mg_precision=prec, coarse_mode=1, tile_autotune=variant, restart=2)
            xt = torch.tensor(x[:p.n_u], device="cuda", dtype=dt)
            bt = torch.tensor(b, device="cuda", dtype=dt)
            ya, yr, yc = (torch.full_like(xt, float("nan")) for _ in range(3))
            s.vmult_A(xt, ya)
            s.apply_level(0, gs.OP_RESIDUAL_A, xt, yr, aux=bt)
            dinv = torch.empty_like(xt)
            s.apply_level(0, gs.OP_DIAG_A, xt, dinv)
            dinv.reciprocal_()
            d = torch.tensor(d0, device="cuda", dtype=dt)
            aux = torch.cat([bt, d, dinv])
            s.apply_level(0, gs.OP_CHEB_STEP, xt, yc, aux=aux)
            outs += [ya, yr, yc, aux]
            if variant == 1:
                full = np.concatenate([xt.double().cpu().numpy(), x[p.n_u:]])
                _, want = ref(full)
                _, scale = ref(full, absolute=True)
                got = [v.double().cpu().numpy() for v in (ya, yr, yc, bt, d, dinv, aux[p.n_u:2 * p.n_u])]
                assert row_error(got[0], want, Scale(scale), full) <= tol
                sr = scale + np.abs(got[3])
                assert np.max(np.abs(got[1] - (got[3] - want)) / sr) <= tol
                hi = s.info().lambda_max[0]
                theta, delta = 0.5 * (hi + hi / 15.0), 0.5 * (hi - hi / 15.0)
                rho = delta / theta
                rn = 1.0 / (2.0 * theta / delta - rho)
                c1, c2 = rn * rho, 2.0 * rn / delta
                dn = c1 * got[4] + c2 * got[5] * (got[3] - want)
                sd = c1 * np.abs(got[4]) + c2 * got[5] * sr
                assert np.max(np.abs(got[6] - dn) / sd) <= tol
                assert np.max(np.abs(got[2] - (full[:p.n_u] + dn)) / (np.abs(full[:p.n_u]) + sd)) <= tol
        s = gs.Solver.from_problem(p, coarse_mode=1, tile_autotune=variant, restart=2)
        xk = torch.tensor(x, device="cuda")
        yk = torch.full_like(xk, float("nan"))
        s.vmult(xk, yk)
        outs.append(yk)
        if variant == 1:
            want, _ = ref(x)
            scale, _ = ref(x, absolute=True)
            assert row_error(yk.cpu().numpy(), want, Scale(scale), x) <= 1e-12
            first = outs
    assert all(torch.equal(a, c) for a, c in zip(first, outs))
