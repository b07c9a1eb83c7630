"""The work a user of the generalized Stokes solver has it do, as timed cases.

One time step of the method is one FGMRES solve with a multigrid preconditioner, so the cases are the
operators that solve is made of (A x, the Chebyshev smoother, the FP64 saddle operator, the pressure
V-cycle of the Schur step, the corrector stage's residual), each called by itself through the public
binding, and whole calls (a V-cycle, single solves, a batch of solves).  Meshes and coefficients come
from paper_2305_08986_gb300.inputs: the 2.5 x 0.41 channel with an obstacle and a stiff bar, unit boxes
with a stiff inclusion, the unit cube with stiff spheres, and the mesh-extension problem.

kind        entry point                                 output
apply       Solver.vmult_A                              y = A x, float32 or float64
saddle      Solver.vmult                                y = K x, float64
smooth      Solver.apply_level(OP_SMOOTH)               Cheb(A, diag A, 4) from a nonzero start
corrector   Solver.apply_level(OP_RESIDUAL_A)           b - A_c x after Solver.set_corrector
pvcycle     Solver.apply_level(OP_PLAP_INV)             one V-cycle of the pressure Laplacian
vcycle      Solver.vcycle                               one velocity V-cycle, all FP64
solve       Solver.solve                                x of K x = rhs from zero
batch       batch_solve                                 x of several systems solved together
"""
import math

import numpy as np
import torch

from paper_2305_08986_gb300 import gs, inputs

DT = {32: torch.float32, 64: torch.float64}
MAX_CELLS = {2: 1280 * 224, 3: 64 ** 3}


def listed():
    return [
        # a smoother call on a mesh the size of a coarse level or of a small request: launches count
        dict(name="smooth2d_32", kind="smooth", mesh="box", dim=2, nx=32, ny=32, nz=1, levels=1, prec=32),
        # the operator on the channel mesh as the paper states it (210 rows: cannot be coarsened)
        dict(name="apply2d_1280x210", kind="apply", mesh="channel", dim=2, nx=1280, ny=210, nz=1, levels=1, prec=32),
        # the Arnoldi matvec of the channel solve
        dict(name="saddle2d_1280x224", kind="saddle", mesh="channel", dim=2, nx=1280, ny=224, nz=1, levels=1, prec=64),
        # the smoother on the channel's finest level, the post-smoothing form (nonzero start)
        dict(name="smooth2d_1280x224", kind="smooth", mesh="channel", dim=2, nx=1280, ny=224, nz=1, levels=1, prec=32),
        # the Arnoldi matvec on an odd-sized 3D mesh
        dict(name="saddle3d_37x29x41", kind="saddle", mesh="box", dim=3, nx=37, ny=29, nz=41, levels=1, prec=64),
        # the smoother on the finest level of the 3D spheres problem
        dict(name="smooth3d_64", kind="smooth", mesh="spheres", dim=3, nx=64, ny=64, nz=64, levels=1, prec=32),
        # the Schur step's pressure V-cycle on the channel hierarchy: many small launches
        dict(name="pvcycle2d_1280x224", kind="pvcycle", mesh="channel", dim=2, nx=1280, ny=224, nz=1, levels=6, prec=32),
        # the preconditioner of the mesh-extension solve, FP64 as in the paper
        dict(name="vcycle2d_1280x224", kind="vcycle", mesh="extension", dim=2, nx=1280, ny=224, nz=1, levels=6, prec=64),
        # the corrector stage's velocity block (convection, streamline diffusion) on a mid-sized channel
        dict(name="corrector2d_640x112", kind="corrector", mesh="channel", dim=2, nx=640, ny=112, nz=1, levels=1, prec=32),
        # one small system, a tight tolerance: host round trips and launches
        dict(name="solve2d_disc16", kind="solve", mesh="disc", dim=2, nx=16, ny=16, nz=1, levels=3, prec=32, tol=1e-11),
        # the headline solve: 2.59 M unknowns to rel-res 1e-8
        dict(name="solve2d_1280x224", kind="solve", mesh="channel", dim=2, nx=1280, ny=224, nz=1, levels=6, prec=32, tol=1e-8),
        # independent systems of mixed size and dimension (2D 32^2 .. 96^2, 3D 8^3 .. 24^3) advanced together;
        # nx .. levels describe the second of them
        dict(name="batch_6", kind="batch", mesh="box", dim=3, nx=16, ny=16, nz=16, levels=3, prec=32, tol=1e-10, count=6),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _op_size(rng, dim, most):
    """Any sizes, odd ones among them, at most `most` cells."""
    while True:
        n = [_log_int(rng, 16, 1536) for _ in range(2)] + [1] if dim == 2 else [_log_int(rng, 6, 80) for _ in range(3)]
        if n[0] * n[1] * n[2] <= most:
            return n


def _mg_size(rng, dim, lo, hi, most):
    """Sizes that can be coarsened, c 2^k per axis, with the level count of inputs.levels_for."""
    while True:
        k = rng.randint(2, 5) if dim == 2 else rng.randint(1, 4)
        n = [rng.randint(2, 7 if dim == 2 else 4) << k for _ in range(dim)] + [1] * (3 - dim)
        if dim == 2 and rng.random() < 0.5:
            n[0] *= 1 << rng.randint(0, 3)
        if all(lo <= m <= hi for m in n[:dim]) and n[0] * n[1] * n[2] <= most:
            return n, k + 1


def draw(rng):
    kind = rng.choice(["apply", "apply", "saddle", "saddle", "smooth", "smooth", "corrector", "pvcycle", "vcycle",
                       "solve", "batch"])
    dim = rng.choice([2, 3])
    prec, levels = 32, 1
    most = MAX_CELLS[dim]
    if kind in ("corrector", "pvcycle"):
        dim = 2
        most = MAX_CELLS[2]
    if kind == "saddle":
        prec = 64
        most = most if dim == 2 else 40 ** 3
    if kind == "apply":
        prec = rng.choice([32, 64])
    mesh = rng.choice(["channel", "box"]) if dim == 2 else rng.choice(["box", "spheres"])
    if kind in ("apply", "saddle", "smooth", "corrector"):
        n = _op_size(rng, dim, most)
        if dim == 3 and mesh == "spheres":
            n = [n[0]] * 3 if n[0] ** 3 <= most else [24] * 3
    else:
        mesh = "channel" if kind == "pvcycle" else "box"
        if kind == "solve" and dim == 2:
            mesh = rng.choice(["channel", "box"])
        if kind == "vcycle":
            prec = 64
            mesh = "extension" if dim == 2 else "box"
        lo, hi = (16, 1280) if dim == 2 else (8, 48)
        if mesh in ("channel", "extension"):
            lo = 28
        n, levels = _mg_size(rng, dim, lo, hi, most)
        if kind == "batch":
            dim, n, levels = 3, [16, 16, 16], 3
    c = dict(kind=kind, mesh=mesh, dim=dim, nx=n[0], ny=n[1], nz=n[2], levels=levels, prec=prec)
    if kind == "solve":
        c["tol"] = 1e-10
    if kind == "batch":
        c.update(tol=1e-10, count=rng.randint(2, 8))
    c["pick"] = rng.randrange(1 << 16)  # which coefficients the inputs take
    return c


def _problem(case, seed):
    n = (case["nx"], case["ny"], case["nz"])[:case["dim"]]
    rng = np.random.default_rng([int(seed), int(case.get("pick", 0))])
    lv, mesh = case["levels"], case["mesh"]
    if mesh == "channel":
        return inputs.config_channel(nx=n[0], ny=n[1], levels=lv, v_in=float(rng.uniform(0.5, 2.0)))
    if mesh == "extension":
        return inputs.config_extension(nx=n[0], ny=n[1], levels=lv, tip=float(rng.uniform(0.005, 0.02)))
    if mesh == "disc":
        return inputs.config_disc(n=n[0], levels=lv)
    if mesh == "spheres":
        return inputs.config_spheres(n=n[0], levels=lv, seed=int(rng.integers(1 << 31)))
    # stiff boxes: up to the largest contrast for single operators, moderate where a solve has to converge
    top = 1e6 if case["kind"] in ("apply", "saddle", "smooth") else 1e3
    return inputs.config_box_inclusion(case["dim"], n, lv, float(math.exp(rng.uniform(0.0, math.log(top)))),
                                       float(rng.uniform(1.0, 1e3)), seed=int(rng.integers(1 << 31)),
                                       align_coarse=lv > 1)


def _load(p, seed):
    """The nodal load of a solve: a smooth field of a few sine modes, as the history term of a time step."""
    rng = np.random.default_rng([int(seed), 7])
    x = inputs.vnode_coords(p.dim, p.n, p.length) / np.asarray(p.length)
    f = np.zeros(p.n_total)
    for a in range(p.dim):
        for _ in range(4):
            k = rng.integers(1, 5, size=p.dim)
            f[a * p.n_vnodes:(a + 1) * p.n_vnodes] += rng.standard_normal() * np.prod(np.sin(np.pi * k * x), axis=1)
    return f


def _batch_problems(case, seed):
    """Mixed 2D / 3D boxes, sizes of the batched workload."""
    rng = np.random.default_rng([int(seed), int(case.get("pick", 0)), 3])
    sizes = [(2, 64, 5), (3, 16, 3), (2, 96, 5), (3, 8, 2), (2, 32, 4), (3, 24, 4), (2, 128, 5), (3, 12, 3)]
    return [inputs.config_box_inclusion(d, (s,) * d, lv, float(math.exp(rng.uniform(0.0, math.log(1e3)))),
                                        float(rng.uniform(1.0, 1e3)), seed=int(rng.integers(1 << 31)), align_coarse=True)
            for d, s, lv in sizes[:case["count"]]]


def _system(p, seed, **opts):
    s = gs.Solver.from_problem(p, **opts)
    f = torch.tensor(_load(p, seed), device="cuda")
    g = torch.tensor(p.g, device="cuda")
    rhs = torch.empty_like(f)
    s.lift_rhs(f, g, rhs)
    return s, rhs, torch.zeros_like(rhs)


def _vectors(case, seed, s):
    gen = torch.Generator(device="cuda").manual_seed(int(seed) * 2 + 1)
    n = {"saddle": s.n_total, "pvcycle": s.n_p}.get(case["kind"], s.n_u)
    return [torch.randn(n, generator=gen, device="cuda", dtype=DT[case["prec"]]) for _ in range(2)]


def _convection(p, seed):
    rng = np.random.default_rng([int(seed), 11])
    return rng.standard_normal(p.n_u) * 4.0, 20.0  # v° and rho of the tests' convected meshes


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        parts = [_system(p, seed + i) for i, p in enumerate(_batch_problems(case, seed))]
        return dict(kind=kind, solvers=[q[0] for q in parts], rhs=[q[1] for q in parts], x=[q[2] for q in parts],
                    tol=case["tol"])
    p = _problem(case, seed)
    if kind == "solve":
        s, rhs, x = _system(p, seed)
        return dict(kind=kind, solver=s, rhs=rhs, x=x, tol=case["tol"])
    opts = dict(coarse_mode=1 if case["levels"] == 1 else 0)
    if case["prec"] == 64:
        opts["mg_precision"] = 64
    if kind == "corrector":
        opts["corrector"] = 1
    s = gs.Solver.from_problem(p, **opts)
    if kind == "corrector":
        s.set_corrector(*_convection(p, seed))
    a, b = _vectors(case, seed, s)
    return dict(kind=kind, solver=s, level=case["levels"] - 1, a=a, b=b, y=torch.empty_like(a))


def run(state):
    kind = state["kind"]
    if kind == "batch":
        for x in state["x"]:
            x.zero_()
        status, _, _ = gs.batch_solve(state["solvers"], state["rhs"], state["x"], tol=state["tol"])
        if status != gs.GS_OK:
            raise RuntimeError("batch_solve: status %d" % status)
        return state["x"]
    s = state["solver"]
    if kind == "solve":
        state["x"].zero_()
        s.solve(state["rhs"], state["x"], tol=state["tol"])
        return state["x"]
    a, b, y = state["a"], state["b"], state["y"]
    if kind == "apply":
        s.vmult_A(a, y)
    elif kind == "saddle":
        s.vmult(a, y)
    elif kind == "smooth":
        s.apply_level(state["level"], gs.OP_SMOOTH, a, y, aux=b)
    elif kind == "corrector":
        s.apply_level(state["level"], gs.OP_RESIDUAL_A, a, y, aux=b)
    elif kind == "pvcycle":
        s.apply_level(state["level"], gs.OP_PLAP_INV, a, y)
    else:
        s.vcycle(a, y)
    return y


def work(case):
    """Bytes of the operands each operator application has to read and write, and the flops of its cell sums."""
    dim, kind, size = case["dim"], case["kind"], case["prec"] // 8
    if kind == "batch":
        one = [work(dict(case, kind="solve", dim=d, nx=n, ny=n, nz=n if d == 3 else 1))
               for d, n in [(2, 64), (3, 16), (2, 96), (3, 8), (2, 32), (3, 24), (2, 128), (3, 12)][:case["count"]]]
        return {k: sum(w[k] for w in one) for k in ("bytes", "flops")}
    n = (case["nx"], case["ny"], case["nz"])[:dim]
    nc, nu = math.prod(n), dim * math.prod(2 * k + 1 for k in n)
    np_ = math.prod(k + 1 for k in n)
    cell = 190.0 if dim == 2 else 1200.0  # operations per cell of one application of the velocity block
    coarse = 1.0 / (1.0 - 0.5 ** dim)     # all levels over the finest
    if kind == "apply":
        return {"bytes": (2 * nu + nc) * size, "flops": cell * nc}
    if kind == "saddle":
        return {"bytes": (2 * (nu + np_) + nc) * size, "flops": 1.2 * cell * nc}
    if kind == "smooth":
        return {"bytes": (4 * nu + nc) * size, "flops": 4 * cell * nc}
    if kind == "corrector":
        return {"bytes": (4 * nu + 2 * nc) * size, "flops": 3 * cell * nc}
    if kind == "pvcycle":
        return {"bytes": coarse * 4 * np_ * size, "flops": coarse * 5 * 20 * np_}
    cycle_b, cycle_f = coarse * (8 * nu + 2 * nc), coarse * 8 * cell * nc
    if kind == "vcycle":
        return {"bytes": cycle_b * size, "flops": cycle_f}
    its = 30  # of the order of the iterations the listed solves take; each also reads half the basis twice
    return {"bytes": its * (cycle_b * 4 + (2 * (nu + np_) + nc) * 8 + its * (nu + np_) * 8.0),
            "flops": its * (cycle_f + 1.2 * cell * nc + 3.0 * its * (nu + np_))}


# ---- the same operators in 64 bits, from the weak forms (plain torch) ------------------------------------

_PTS = [0.5 - 0.5 * math.sqrt(0.6), 0.5, 0.5 + 0.5 * math.sqrt(0.6)]
_WTS = [5.0 / 18.0, 8.0 / 18.0, 5.0 / 18.0]


def _basis(dim, h, order):
    """Values [q, i], gradients [q, i, a] and weights [q] of the tensor Lagrange basis on one cell."""
    t = np.array(_PTS)
    if order == 2:
        v = np.stack([(1 - t) * (1 - 2 * t), 4 * t * (1 - t), t * (2 * t - 1)], 1)
        d = np.stack([4 * t - 3, 4 - 8 * t, 4 * t - 1], 1)
    else:
        v, d = np.stack([1 - t, t], 1), np.stack([-np.ones(3), np.ones(3)], 1)
    k = order + 1
    val, w = np.ones((1, 1)), np.ones(1)
    grad = [np.ones((1, 1)) for _ in range(dim)]
    for a in reversed(range(dim)):  # x fastest
        val = np.kron(val, v)
        w = np.kron(w, np.array(_WTS) * h[a])
        grad = [np.kron(g, d / h[a] if a == b else v) for b, g in enumerate(grad)]
    return val, np.stack(grad, -1), w, k


class _Level:
    """One mesh level: masks, per-cell coefficients and the weak forms as cell matrices."""

    def __init__(self, dim, n, length, eta, alpha, void, faces):
        self.dim, self.n, self.alpha, self.faces = dim, tuple(n), alpha, faces
        self.h = [length[a] / n[a] for a in range(dim)]
        self.cells = tuple(reversed(self.n))
        dev = dict(device="cuda", dtype=torch.float64)
        self.eta = torch.as_tensor(eta).to(**dev).reshape(-1)
        self.active = (torch.ones_like(self.eta) if void is None
                       else 1.0 - torch.as_tensor(np.asarray(void, dtype=np.float64)).to(**dev).reshape(-1))
        val, grad, w, _ = _basis(dim, self.h, 2)
        pval = _basis(dim, self.h, 1)[0]
        self.val, self.grad, self.w = (torch.as_tensor(q).to(**dev) for q in (val, grad, w))
        nb = 3 ** dim
        mass = np.einsum("q,qi,qj->ij", w, val, val)
        self.mass = torch.as_tensor(np.kron(np.eye(dim), mass)).to(**dev)
        visc = np.zeros((dim, nb, dim, nb))
        for a in range(dim):
            visc[a, :, a, :] += np.einsum("q,qid,qjd->ij", w, grad, grad)
            for b in range(dim):  # (grad u)^T part of 2 eps : eps
                visc[a, :, b, :] += np.einsum("q,qi,qj->ij", w, grad[:, :, b], grad[:, :, a])
        self.visc = torch.as_tensor(visc.reshape(dim * nb, dim * nb)).to(**dev)
        div = -np.einsum("q,qp,qia->pai", w, pval, grad)
        self.div = torch.as_tensor(div.reshape(2 ** dim, dim * nb)).to(**dev)
        pgrad = _basis(dim, self.h, 1)[1]
        self.plap = torch.as_tensor(np.einsum("q,qid,qjd->ij", w, pgrad, pgrad)).to(**dev)
        self.vshape = tuple(2 * k + 1 for k in self.cells)
        self.pshape = tuple(k + 1 for k in self.cells)
        con = torch.zeros(self.vshape, **dev)
        pcon = self.scatter(self.active.expand(2 ** dim, -1), 1).reshape(-1) == 0  # touched by no active cell
        lap = pcon.reshape(self.pshape).clone()
        for a in range(dim):
            for side in (0, 1):
                at = [slice(None)] * dim
                at[dim - 1 - a] = -1 if side else 0
                if faces >> (2 * a + side) & 1:
                    con[tuple(at)] = 1
                else:
                    lap[tuple(at)] = True
        con = con + self.scatter((1.0 - self.active).expand(3 ** dim, -1), 2)[0]
        self.con = (con.reshape(-1) > 0).repeat(dim)
        self.pcon, self.lcon = pcon, lap.reshape(-1)
        self.conv = None

    def gather(self, x, order):
        """Nodal vector -> [components * local nodes, cells]."""
        v = x.reshape((-1,) + (self.vshape if order == 2 else self.pshape))
        out = []
        for comp in v:
            for loc in np.ndindex(*([order + 1] * self.dim)):
                out.append(comp[tuple(slice(l, l + order * (k - 1) + 1, order) for l, k in zip(loc, self.cells))].reshape(-1))
        return torch.stack(out)

    def scatter(self, loc, order):
        nb = (order + 1) ** self.dim
        y = torch.zeros((loc.shape[0] // nb,) + tuple(order * k + 1 for k in self.cells), device="cuda", dtype=torch.float64)
        for i in range(loc.shape[0]):
            l = np.unravel_index(i % nb, [order + 1] * self.dim)
            y[(i // nb,) + tuple(slice(q, q + order * (k - 1) + 1, order) for q, k in zip(l, self.cells))] += loc[i].reshape(self.cells)
        return y

    def local(self, loc):
        y = self.alpha * (self.mass @ loc) + self.eta * (self.visc @ loc)
        if self.conv is not None:
            v, rho, r = self.conv
            nb = 3 ** self.dim
            vq = torch.stack([self.val @ v[a * nb:(a + 1) * nb] for a in range(self.dim)])
            for a in range(self.dim):
                u = loc[a * nb:(a + 1) * nb]
                adv = sum(vq[b] * (self.grad[:, :, b] @ u) for b in range(self.dim))
                f = rho * self.w[:, None] * adv
                y[a * nb:(a + 1) * nb] += self.val.T @ f + sum(self.grad[:, :, b].T @ (r * vq[b] * f) for b in range(self.dim))
        return y * self.active

    def A(self, x):
        return torch.where(self.con, x, self.scatter(self.local(self.gather(torch.where(self.con, 0.0, x), 2)), 2).reshape(-1))

    def K(self, x):
        nu = self.con.numel()
        u, p = torch.where(self.con, 0.0, x[:nu]), torch.where(self.pcon, 0.0, x[nu:])
        lu, lp = self.gather(u, 2), self.gather(p, 1)
        yu = self.scatter(self.local(lu) + self.active * (self.div.T @ lp), 2).reshape(-1)
        yp = self.scatter(self.active * (self.div @ lu), 1).reshape(-1)
        return torch.cat([torch.where(self.con, x[:nu], yu), torch.where(self.pcon, x[nu:], yp)])

    def diag(self):
        loc = (self.alpha * self.mass.diagonal()[:, None] + self.visc.diagonal()[:, None] * self.eta) * self.active
        return torch.where(self.con, 1.0, self.scatter(loc, 2).reshape(-1))

    def L(self, x):
        y = self.scatter((self.plap @ self.gather(torch.where(self.lcon, 0.0, x), 1)) * self.active, 1).reshape(-1)
        return torch.where(self.lcon, x, y)

    def ldiag(self):
        return torch.where(self.lcon, 1.0, self.scatter(self.plap.diagonal()[:, None] * self.active, 1).reshape(-1))


def _top_eigenvalue(op, dinv, con, code):
    """1.2 times the largest Ritz value of 12 Lanczos steps from the documented SplitMix64 start vector."""
    i = np.arange(con.numel(), dtype=np.uint64) ^ np.uint64(code << 56)
    with np.errstate(over="ignore"):
        z = i + np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    v = torch.as_tensor(2.0 * ((z >> np.uint64(11)).astype(np.float64) / 2.0 ** 53) - 1.0).to("cuda")
    v = torch.where(con, 0.0, v)
    v, before, beta, al, be, s = v / v.norm(), torch.zeros_like(v), 0.0, [], [], dinv.sqrt()
    for _ in range(12):
        w = s * op(s * v) - beta * before
        a = torch.dot(w, v)
        w = w - a * v
        beta = w.norm()
        al.append(float(a))
        be.append(float(beta))
        before, v = v, w / beta
    return 1.2 * float(np.linalg.eigvalsh(np.diag(al) + np.diag(be[:-1], 1) + np.diag(be[:-1], -1))[-1])


def _cheb(op, dinv, hi, b, x, degree):
    lo = hi / 15.0
    theta, delta = 0.5 * (hi + lo), 0.5 * (hi - lo)
    sigma = theta / delta
    d = dinv * (b if x is None else b - op(x)) / theta
    x = d if x is None else x + d
    rho = 1.0 / sigma
    for _ in range(degree - 1):
        rn = 1.0 / (2.0 * sigma - rho)
        d = rn * rho * d + 2.0 * rn / delta * (dinv * (b - op(x)))
        x, rho = x + d, rn
    return x


def _interpolations(cs, order):
    """(axis, matrix) of the nested interpolation along every axis of a [components, ...] nodal array (cs: coarse
    cells, slowest first)."""
    for ax, k in enumerate(cs):
        nc = order * k + 1
        P = torch.zeros(2 * order * k + 1, nc, device="cuda", dtype=torch.float64)
        P[torch.arange(0, 2 * nc - 1, 2), torch.arange(nc)] = 1.0
        c = torch.arange(k)
        if order == 1:
            P[2 * c + 1, c] = P[2 * c + 1, c + 1] = 0.5
        else:
            for row, w in ((1, (0.375, 0.75, -0.125)), (3, (-0.125, 0.75, 0.375))):
                for j in range(3):
                    P[4 * c + row, 2 * c + j] = w[j]
        yield ax + 1, P


def _transfer(x, coarse, order, up):
    lead = (-1,) + tuple(order * k * (1 if up else 2) + 1 for k in coarse.cells)
    y = x.reshape(lead)
    for ax, P in _interpolations(coarse.cells, order):
        y = torch.movedim(torch.tensordot(P if up else P.T, y, dims=([1], [ax])), 0, ax)
    return y.reshape(-1)


def _cycle(levels, l, b, order, degree):
    lv = levels[l]
    op, con = (lv.A, lv.con) if order == 2 else (lv.L, lv.lcon)
    if l == 0:
        free = torch.nonzero(~con).reshape(-1)
        cols = []
        for j in free.tolist():
            e = torch.zeros_like(b)
            e[j] = 1.0
            cols.append(op(e)[free])
        y = torch.zeros_like(b)
        y[free] = torch.linalg.solve(torch.stack(cols, 1), b[free])
        return y
    dinv = 1.0 / (lv.diag() if order == 2 else lv.ldiag())
    hi = _top_eigenvalue(op, dinv, con, l if order == 2 else 0x80 | l)
    x = _cheb(op, dinv, hi, b, None, degree)
    low = levels[l - 1]
    lcon = low.con if order == 2 else low.lcon
    r = _transfer(torch.where(con, 0.0, b - op(x)), low, order, False)
    e = _cycle(levels, l - 1, torch.where(lcon, 0.0, r), order, degree)
    x = x + torch.where(con, 0.0, _transfer(torch.where(lcon, 0.0, e), low, order, True))
    return _cheb(op, dinv, hi, b, x, degree)


def _hierarchy(p):
    """Levels, coarsest first: coarse eta = mean of the active children, obstacle where all children are."""
    out = []
    n, eta = tuple(p.n), np.asarray(p.eta, dtype=np.float64)
    void = np.zeros(p.n_cells) if p.void is None else np.asarray(p.void, dtype=np.float64)
    for _ in range(p.levels):
        out.insert(0, _Level(p.dim, n, p.length, eta, float(p.alpha), void, p.dirichlet_faces))
        n = tuple(k // 2 for k in n)
        if len(out) == p.levels:
            break
        shape = [q for k in reversed(n) for q in (k, 2)]
        axes = tuple(range(1, 2 * p.dim, 2))
        act = (1.0 - void).reshape(shape).sum(axes)
        tot = ((1.0 - void) * eta).reshape(shape).sum(axes)
        full = eta.reshape(shape).mean(axes)
        eta = np.where(act > 0, tot / np.maximum(act, 1.0), full).reshape(-1)
        void = (act == 0).astype(np.float64).reshape(-1)
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind in ("solve", "batch"):
        if case["mesh"] != "disc":
            return None  # a direct solution of these sizes takes minutes
        p = _problem(case, seed)
        lv = _hierarchy(p)[-1]
        g, f = torch.as_tensor(p.g).to("cuda"), torch.as_tensor(_load(p, seed)).to("cuda")
        nu = lv.con.numel()
        K = torch.stack([lv.K(e) for e in torch.eye(p.n_total, device="cuda", dtype=torch.float64)], 1)
        rhs = torch.zeros_like(f)
        rhs[:nu] = torch.where(lv.con, g[:nu], lv.scatter(lv.mass @ lv.gather(f[:nu], 2) * lv.active, 2).reshape(-1))
        one = torch.zeros_like(rhs)
        one[nu:] = 1.0  # no outflow: the pressure is fixed by a zero mean
        return torch.linalg.solve(K - torch.outer(one, one) / one.sum(), rhs)
    p = _problem(case, seed)
    lv = _hierarchy(p)
    top = lv[-1]

    class size:  # the vectors _vectors makes
        n_total, n_u, n_p = p.n_total, p.n_u, p.n_pnodes
    a, b = (v.double() for v in _vectors(case, seed, size))
    if kind == "apply":
        return top.A(a)
    if kind == "saddle":
        return top.K(a)
    if kind == "corrector":
        v, rho = _convection(p, seed)
        loc = top.gather(torch.as_tensor(v).to("cuda"), 2)
        nb = 3 ** p.dim
        speed = torch.stack([loc[c * nb + nb // 2] for c in range(p.dim)]).norm(dim=0)
        size_k = math.sqrt(sum(h * h for h in top.h))
        pe = rho * speed * size_k / (4.0 * top.eta)
        r = torch.where(pe >= 1.0, size_k / (4.0 * speed) * (1.0 / torch.tanh(pe) - 1.0 / pe), 0.0)
        top.conv = (loc, rho, r)
        return b - top.A(a)
    if kind == "smooth":
        dinv = 1.0 / top.diag()
        return _cheb(top.A, dinv, _top_eigenvalue(top.A, dinv, top.con, case["levels"] - 1), a, b, 4)
    if kind == "pvcycle":
        r = torch.where(top.lcon, 0.0, a)
        return torch.where(top.lcon, 0.0, _cycle(lv, len(lv) - 1, r, 1, 2))
    return _cycle(lv, len(lv) - 1, a, 2, 4)
