"""FP32 rounding of the viscous coefficients in 2D: a field that is the highest mode (2, 2) in every cell.

Nodal values p(i) p(j) with p = 1, -1/2, 1, -1/2, ... have that mode alone in every cell, with value 9 exactly, so with
alpha = 0 the unconstrained operator at a cell's centre is 9 d_K, d_K = eta_K k with the mesh's coefficient k, and
nothing is added to it.  d_K rounded once and the product rounded once leave (1 + u)^2 - 1, u = 2^-24; a coefficient
rounded before it is multiplied by eta_K leaves up to 3 u on meshes like these."""
from fractions import Fraction as Fr

import numpy as np
import pytest

from paper_2305_08986_gb300 import inputs

pytestmark = pytest.mark.gpu

# sizes whose coefficients are about half a unit from the nearest float
CASES = [((64, 48), (1.0, 0.7)), ((120, 48), (1.0, 1.7)), ((104, 38), (1.0, 1.7))]


def coefficient(c, n, length):
    h = [Fr(float(length[a] / n[a])) for a in range(2)]
    k2, m2 = Fr(4, 3), Fr(1, 45)
    return sum((2 if b == c else 1) * k2 * m2 / h[b] ** 2 for b in range(2)) * h[0] * h[1] * 4


@pytest.mark.parametrize("n,length", CASES)
@pytest.mark.parametrize("variant", [1, 4, 6])
def test_highest_mode_is_rounded_twice(n, length, variant):
    import torch
    from paper_2305_08986_gb300 import gs
    rng = np.random.default_rng(7)
    eta = np.exp(rng.uniform(0.0, np.log(1e6), size=n[0] * n[1])).astype(np.float32).astype(np.float64)
    p = inputs.Problem("mode", 2, n, length, 1, eta, 0.0, inputs.FACE_XM)
    s = gs.Solver.from_problem(p, mg_precision=32, coarse_mode=1, tile_autotune=variant, restart=2)
    one = [np.where(np.arange(2 * k + 1) % 2 == 0, 1.0, -0.5) for k in n]
    field = np.outer(one[1], one[0]).ravel()
    for c in range(2):
        x = np.zeros(p.n_u, dtype=np.float32)
        x[c * field.size:(c + 1) * field.size] = field
        xt = torch.tensor(x, device="cuda")
        yt = torch.empty_like(xt)
        s.apply_level(0, gs.OP_A_RAW, xt, yt)
        y = yt[c * field.size:(c + 1) * field.size].double().cpu().numpy().reshape(2 * n[1] + 1, 2 * n[0] + 1)
        centre = y[1::2, 1::2].ravel()
        exact = float(9 * coefficient(c, n, length)) * eta  # in doubles: 2^-53
        u = 2.0 ** -24
        assert np.max(np.abs(centre / exact - 1.0)) <= (1.0 + u) ** 2 - 1.0 + 2.0 ** -45
