"""The workloads this solver's speed is judged on, with their inputs and exact answers.

Every case is one whole call sequence of a user's program on tensors that are
already on the GPU: the coefficient of a time step is set and the equation
div(beta grad phi) = f is solved to a relative residual of 1e-10 (the time
step of a low-Mach code, paper Sec. 1), or a batch of boxes, a coupled level,
a velocity projection or the differentiable solve around it.  Inputs follow
the recipes of ``paper_1008_2801_gb300.inputs`` (smooth, stellar and inclusion
coefficients), drawn on the GPU.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1008_2801_gb300 as mg
from paper_1008_2801_gb300.inputs import BATCH_SIZES

TOL = 1e-10


def listed():
    return [
        # one small FP64 box (the 64^3 manufactured problem): launches and latency
        dict(name="fp64_64", kind="box", nx=64, ny=64, nz=64, precision="fp64", bc="DDDDDD",
             krylov=False, field="smooth"),
        # the FP64 time step on one ordinary and on the largest single box
        dict(name="fp64_256", kind="box", nx=256, ny=256, nz=256, precision="fp64", bc="DDDDDD",
             krylov=False, field="stellar"),
        dict(name="fp64_512", kind="box", nx=512, ny=512, nz=512, precision="fp64", bc="DDDDDD",
             krylov=False, field="stellar"),
        # the same largest box with FP32 V-cycles inside FP64 refinement
        dict(name="mixed_512", kind="box", nx=512, ny=512, nz=512, precision="mixed",
             bc="DDDDDD", krylov=False, field="stellar"),
        # a ragged box in mixed precision: sides 10*16, 6*16 and 14*16
        dict(name="mixed_ragged", kind="box", nx=160, ny=96, nz=224, precision="mixed",
             bc="DDDDDD", krylov=False, field="stellar"),
        # a slab of atmosphere: periodic sideways, walls below and above
        dict(name="periodic_fp64", kind="box", nx=192, ny=128, nz=96, precision="fp64",
             bc="PPPPDD", krylov=False, field="smooth"),
        # high-contrast coefficients: CG preconditioned by the V-cycle
        dict(name="krylov_fp64", kind="box", nx=128, ny=128, nz=128, precision="fp64",
             bc="DDDDDD", krylov=True, field="inclusions"),
        # the 64 uneven boxes of one refinement level's grids, solved independently
        dict(name="batch_fp64", kind="batch", nbox=64, layout=4, precision="fp64"),
        dict(name="batch_mixed", kind="batch", nbox=64, layout=4, precision="mixed"),
        # boxes of one level solved as one domain
        dict(name="level_fp64", kind="level", bx=4, by=4, bz=2, n=64, precision="fp64"),
        # the velocity projection of an inflow jet (outflow above, flux given elsewhere)
        dict(name="project_mixed", kind="project", nx=256, ny=256, nz=256, precision="mixed",
             bc="NNNNND"),
        # training through the solve: eight right-hand sides, forward and backward
        dict(name="adjoint_fp64", kind="adjoint", n=128, nrhs=8, precision="fp64"),
    ]


def _side(rng, lo, hi, step):
    """A side spread over the logarithm of lo..hi, a multiple of step."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(step, int(round(v / step)) * step)


def draw(rng):
    kind = rng.choice(["box", "box", "box", "box", "batch", "level", "project", "adjoint"])
    prec = rng.choice(["fp64", "mixed"])
    if kind == "batch":
        return dict(kind=kind, nbox=int(round(math.exp(rng.uniform(math.log(4), math.log(64))))),
                    layout=rng.randrange(1000), precision=prec)
    if kind == "level":
        return dict(kind=kind, bx=rng.randint(1, 4), by=rng.randint(2, 4), bz=rng.randint(1, 2),
                    n=rng.choice([32, 64]), precision=prec)
    if kind == "adjoint":
        return dict(kind=kind, n=rng.choice([32, 48, 64, 80, 96, 112, 128]),
                    nrhs=rng.randint(1, 8), precision=prec)
    step = rng.choice([16, 32])
    nx, ny, nz = (_side(rng, 32, 384, step) for _ in range(3))
    if kind == "project":
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, precision=prec,
                    bc=rng.choice(["DDDDDD", "NNNNND", "NNNNDD"]))
    form = rng.choice(["plain", "plain", "plain", "periodic", "krylov"])
    if form == "krylov":
        nx, ny, nz = (min(v, 160) for v in (nx, ny, nz))
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, precision=prec, bc="DDDDDD", krylov=True,
                    field=rng.choice(["stellar", "inclusions"]))
    if form == "periodic":
        # sides of few prime factors: the coarsest level has to be a small one here
        nx, ny, nz = (rng.choice([32, 48, 64, 96, 128, 192, 256]) for _ in range(3))
    bc = rng.choice(["PPDDDD", "PPPPDD"]) if form == "periodic" else rng.choice(
        ["DDDDDD", "DDDDDD", "NNNNND", "DDDDNN"])
    return dict(kind=kind, nx=nx, ny=ny, nz=nz, precision=prec, bc=bc, krylov=False,
                field=rng.choice(["smooth", "stellar"]))


# ---- inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _uniform(g, shape):
    return torch.rand(shape, generator=g, device="cuda", dtype=torch.float64) * 2.0 - 1.0


def _centres(shape, dx):
    nz, ny, nx = shape
    x, y, z = ((torch.arange(m, device="cuda", dtype=torch.float64) + 0.5) * dx
               for m in (nx, ny, nz))
    return z[:, None, None], y[None, :, None], x[None, None, :]


def _stellar_beta(g, shape, dx, centre=(0.5, 0.5, 0.5), rc=0.3):
    z, y, x = _centres(shape, dx)
    r2 = (x - centre[0]) ** 2 + (y - centre[1]) ** 2 + (z - centre[2]) ** 2
    rho = (1.0 + r2 / (rc * rc)).pow_(-1.5)
    noise = torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)
    return 1.0 / (rho * (1.0 + 0.01 * noise))


def _beta(g, shape, dx, field):
    if field == "stellar":
        return _stellar_beta(g, shape, dx)
    z, y, x = _centres(shape, dx)
    if field == "smooth":
        # periodic over each side, with phases of its own
        ph = torch.rand(3, generator=g, device="cuda", dtype=torch.float64) * (2 * math.pi)
        w = [2 * math.pi / (m * dx) for m in shape]
        return (1.0 + 0.5 * torch.sin(w[2] * x + ph[0]) * torch.sin(w[1] * y + ph[1])
                * torch.sin(w[0] * z + ph[2])).contiguous()
    ext = torch.tensor([shape[2], shape[1], shape[0]], device="cuda", dtype=torch.float64) * dx
    c = (torch.rand((24, 3), generator=g, device="cuda", dtype=torch.float64) * 0.8 + 0.1) * ext
    r = (torch.rand(24, generator=g, device="cuda", dtype=torch.float64) * 0.06 + 0.04) * ext[0]
    inside = torch.zeros(shape, dtype=torch.bool, device="cuda")
    for i in range(24):
        inside |= (x - c[i, 0]) ** 2 + (y - c[i, 1]) ** 2 + (z - c[i, 2]) ** 2 <= r[i] ** 2
    return torch.where(inside, 1e4, 1.0).to(torch.float64)


def _boxes(case):
    """Shapes (nz, ny, nx) of a batch's boxes: sides drawn from the batch recipe."""
    d = np.random.default_rng(case["layout"]).choice(np.asarray(BATCH_SIZES),
                                                     size=(case["nbox"], 3))
    return [(int(v[2]), int(v[1]), int(v[0])) for v in d]


def _level(case):
    """Lower corners (i, j, k) and shapes of a level's boxes, and the domain's shape."""
    n, bx, by, bz = case["n"], case["bx"], case["by"], case["bz"]
    los = [(i * n, j * n, k * n) for k in range(bz) for j in range(by) for i in range(bx)]
    return los, [(n, n, n)] * len(los), (bz * n, by * n, bx * n)


def _split(a, los, n):
    return torch.cat([a[k:k + n, j:j + n, i:i + n].reshape(-1) for i, j, k in los])


def _batch_inputs(case, seed):
    g, dx = _gen(seed), 1.0 / 128
    betas, fs = [], []
    for s in _boxes(case):
        u = torch.rand(4, generator=g, device="cuda", dtype=torch.float64).tolist()
        betas.append(_stellar_beta(g, s, dx, [u[0] * s[2] * dx, u[1] * s[1] * dx,
                                              u[2] * s[0] * dx], 0.1 + 0.3 * u[3]))
        f = _uniform(g, s)
        fs.append(f - f.mean())
    return betas, fs, dx


def _level_inputs(case, seed):
    g = _gen(seed)
    shape = _level(case)[2]
    dx = 1.0 / max(shape)
    beta = _stellar_beta(g, shape, dx)
    f = _uniform(g, shape)
    return beta, f - f.mean(), dx


def _adjoint_inputs(case, seed):
    g, n = _gen(seed), case["n"]
    beta = _stellar_beta(g, (n, n, n), 1.0 / n)
    lead = (case["nrhs"],) if case["nrhs"] > 1 else ()
    return beta, _uniform(g, lead + (n, n, n)), _uniform(g, lead + (n, n, n)), 1.0 / n


def _box_inputs(case, seed):
    g = _gen(seed)
    shape, dx = (case["nz"], case["ny"], case["nx"]), 1.0 / case["nx"]
    if case["kind"] == "project":
        nz, ny, nx = shape
        beta = _stellar_beta(g, shape, dx)
        return beta, (_uniform(g, (nz, ny, nx + 1)), _uniform(g, (nz, ny + 1, nx)),
                      _uniform(g, (nz + 1, ny, nx))), dx
    beta = _beta(g, shape, dx, case["field"])
    f = _uniform(g, shape)
    return beta, f - f.mean(), dx


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        betas, fs, dx = _batch_inputs(case, seed)
        s = mg.BatchSolver(_boxes(case), dx, precision=case["precision"])
        return dict(kind=kind, solver=s, beta=s.pack(betas), f=s.pack(fs))
    if kind == "level":
        los, shapes, _ = _level(case)
        beta, f, dx = _level_inputs(case, seed)
        s = mg.LevelSolver(los, shapes, dx, precision=case["precision"])
        return dict(kind=kind, solver=s, beta=_split(beta, los, case["n"]),
                    f=_split(f, los, case["n"]))
    if kind == "adjoint":
        beta, f, target, dx = _adjoint_inputs(case, seed)
        s = mg.Solver(tuple(beta.shape), dx, precision=case["precision"])
        return dict(kind=kind, solver=s, beta=beta.requires_grad_(), f=f.requires_grad_(),
                    target=target)
    beta, f, dx = _box_inputs(case, seed)
    s = mg.Solver(tuple(beta.shape), dx, precision=case["precision"], bc=case["bc"],
                  krylov=case.get("krylov", False))
    return dict(kind=kind, solver=s, beta=beta, f=f)


def run(state):
    s, beta, f = state["solver"], state["beta"], state["f"]
    if state["kind"] == "adjoint":
        phi = mg.MGSolve.apply(f, beta, s, TOL)
        loss = 0.5 * (phi - state["target"]).square().sum()
        df, dbeta = torch.autograd.grad(loss, (f, beta))
        return {"phi": phi.detach(), "df": df, "dbeta": dbeta}
    s.set_beta(beta)
    if state["kind"] == "project":
        # the provisional velocity stays with the caller for the next predictor
        u, v, w = (t.clone() for t in f)
        phi, _ = s.project(u, v, w, tol=TOL)
        return {"phi": phi, "u": u, "v": v, "w": w}
    return s.solve(f, tol=TOL)[0]


def _cells(case):
    if case["kind"] == "batch":
        return sum(a * b * c for a, b, c in _boxes(case))
    if case["kind"] == "level":
        return case["bx"] * case["by"] * case["bz"] * case["n"] ** 3
    if case["kind"] == "adjoint":
        return case["n"] ** 3
    return case["nx"] * case["ny"] * case["nz"]


def work(case):
    """beta, f read and phi written once (8 bytes each); arithmetic: one
    stencil application of 13 operations a cell for each of the ten digits."""
    cells = _cells(case)
    if case["kind"] == "adjoint":
        # beta in, dbeta out; f, target in, phi, df out per right-hand side; two solves
        r = case["nrhs"]
        return {"bytes": cells * 8.0 * (2 + 4 * r), "flops": 2.0 * r * 130.0 * cells}
    arrays = 3 + (5 if case["kind"] == "project" else 0)  # three velocities in and out, no f
    return {"bytes": 8.0 * arrays * cells, "flops": 130.0 * cells}


# ---- exact answers: conjugate gradients in 64 bits on plain torch tensors

class _Operator:
    """-A for one box: face coefficients as stated in the solver's interface
    (harmonic means, 2 beta on a Dirichlet wall, 0 on a Neumann wall)."""

    def __init__(self, beta, dx, bc):
        self.w, self.periodic = [], []
        h2 = dx * dx
        for d in range(3):                       # 0: x (last axis), 1: y, 2: z
            ax, lo, hi = 2 - d, bc[2 * d], bc[2 * d + 1]
            n = beta.shape[ax]
            a, b = beta.narrow(ax, 0, n - 1), beta.narrow(ax, 1, n - 1)
            mid = 2 * a * b / (a + b) / h2
            first, last = beta.narrow(ax, 0, 1), beta.narrow(ax, n - 1, 1)
            if lo == "P":
                wl = wh = 2 * first * last / (first + last) / h2
            else:
                wl = first * ((2.0 if lo == "D" else 0.0) / h2)
                wh = last * ((2.0 if hi == "D" else 0.0) / h2)
            self.w.append((mid, wl, wh))
            self.periodic.append(lo == "P")
        self.diag = torch.zeros_like(beta)
        for d, (mid, wl, wh) in enumerate(self.w):
            ax, n = 2 - d, beta.shape[2 - d]
            self.diag.narrow(ax, 0, n - 1).add_(mid)
            self.diag.narrow(ax, 1, n - 1).add_(mid)
            self.diag.narrow(ax, 0, 1).add_(wl)
            self.diag.narrow(ax, n - 1, 1).add_(wh)

    def __call__(self, p):
        q = self.diag * p
        for d, (mid, wl, wh) in enumerate(self.w):
            ax, n = p.dim() - 1 - d, p.shape[p.dim() - 1 - d]
            q.narrow(ax, 0, n - 1).addcmul_(mid, p.narrow(ax, 1, n - 1), value=-1)
            q.narrow(ax, 1, n - 1).addcmul_(mid, p.narrow(ax, 0, n - 1), value=-1)
            if self.periodic[d]:
                q.narrow(ax, 0, 1).addcmul_(wl, p.narrow(ax, n - 1, 1), value=-1)
                q.narrow(ax, n - 1, 1).addcmul_(wh, p.narrow(ax, 0, 1), value=-1)
        return q


def _cg(op, f, rtol=1e-13, most=30000):
    """phi with A phi = f, A = -op, by diagonally preconditioned CG."""
    x = torch.zeros_like(f)
    r = -f
    inv = 1.0 / op.diag
    z = inv * r
    p = z.clone()
    rz = torch.dot(r.reshape(-1), z.reshape(-1))
    stop = (rtol ** 2) * float(rz)
    for it in range(most):
        q = op(p)
        a = rz / torch.dot(p.reshape(-1), q.reshape(-1))
        x.addcmul_(a, p)
        r.addcmul_(a, q, value=-1)
        torch.mul(inv, r, out=z)
        new = torch.dot(r.reshape(-1), z.reshape(-1))
        if it % 50 == 49 and not float(new) > stop:
            break
        p.mul_(new / rz).add_(z)
        rz = new
    return x


def _face_grad(beta, phi, lam, dx):
    """dL/dbeta of a box with phi = 0 on its walls, summed over right-hand sides."""
    out = torch.zeros_like(beta)
    h2 = dx * dx
    for d in range(3):
        ax = 2 - d
        n = beta.shape[ax]
        pa = 1 + ax                                # phi, lam carry a leading axis
        g = ((lam.narrow(pa, 1, n - 1) - lam.narrow(pa, 0, n - 1))
             * (phi.narrow(pa, 1, n - 1) - phi.narrow(pa, 0, n - 1))).sum(0) / h2
        a, b = beta.narrow(ax, 0, n - 1), beta.narrow(ax, 1, n - 1)
        s2 = (a + b) ** 2
        out.narrow(ax, 0, n - 1).add_(g * 2 * b * b / s2)
        out.narrow(ax, 1, n - 1).add_(g * 2 * a * a / s2)
        for i in (0, n - 1):
            out.narrow(ax, i, 1).add_((lam.narrow(pa, i, 1) * phi.narrow(pa, i, 1)).sum(0)
                                      * (2.0 / h2))
    return out


def exact(case, seed):
    if case["kind"] in ("box", "project") and _cells(case) > 20_000_000:
        return None                  # plain CG takes a minute or more on such boxes
    if case["kind"] == "batch":
        betas, fs, dx = _batch_inputs(case, seed)
        return torch.cat([_cg(_Operator(b, dx, "DDDDDD"), f).reshape(-1)
                          for b, f in zip(betas, fs)])
    if case["kind"] == "level":
        beta, f, dx = _level_inputs(case, seed)
        return _split(_cg(_Operator(beta, dx, "DDDDDD"), f), _level(case)[0], case["n"])
    if case["kind"] == "adjoint":
        beta, f, target, dx = _adjoint_inputs(case, seed)
        op = _Operator(beta, dx, "DDDDDD")
        many = (-1,) + tuple(beta.shape)
        phi = torch.stack([_cg(op, v) for v in f.reshape(many)])
        lam = torch.stack([_cg(op, v) for v in phi - target.reshape(many)])
        return {"phi": phi.reshape(f.shape), "df": lam.reshape(f.shape),
                "dbeta": _face_grad(beta, phi, lam, dx)}
    beta, f, dx = _box_inputs(case, seed)
    op = _Operator(beta, dx, case["bc"])
    if case["kind"] == "box":
        return _cg(op, f)
    u, v, w = f
    div = ((u[:, :, 1:] - u[:, :, :-1]) + (v[:, 1:] - v[:, :-1]) + (w[1:] - w[:-1])) / dx
    phi = _cg(op, div)
    out = {"phi": phi}
    for d, (key, t) in enumerate(zip("uvw", f)):
        ax = 2 - d
        n = phi.shape[ax]
        mid, wl, wh = op.w[d]
        t = t.clone()
        t.narrow(ax, 1, n - 1).sub_(mid * dx * (phi.narrow(ax, 1, n - 1)
                                                - phi.narrow(ax, 0, n - 1)))
        t.narrow(ax, 0, 1).sub_(wl * dx * phi.narrow(ax, 0, 1))
        t.narrow(ax, n, 1).add_(wh * dx * phi.narrow(ax, n - 1, 1))
        out[key] = t
    return out
