"""The work that users of this library have it do, as timed cases.

Every case is one pass through the public entry points: a setup from cell
coefficients and a solve, a solve on a kept hierarchy, a solve from host
arrays, a gradient through the solve, a batch of uneven problems, a 3D setup
and solve.  The sizes are those of the library's own workloads (255^2 Poisson,
4095^2 blocks, 8191^2 log-normal, the paper's 9088 x 568 and 16383 x 1023
grids, 255^3 blocks, sides 63 to 1023 in batches) and ragged ones between
them.  Coefficients and right-hand sides are drawn on the GPU from the seed,
with the distributions of ``paper_1803_02481_gb300.inputs``.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1803_02481_gb300 as bm
from paper_1803_02481_gb300.autograd import solve as differentiable_solve

BATCH_SIDES = (63, 127, 255, 511, 1023)
BATCH_WEIGHTS = (8, 4, 2, 1, 1)


def listed():
    return [
        # the smallest call: every launch and every coarse level shows; a
        # nonlinear outer iteration assembles such a problem anew each time
        _plane("poisson_255", 255, 255, field="constant", keep=False),
        # one window of a larger block field, many right-hand sides on one operator
        _plane("window_511", 511, 511, field="blocks", block=64, decades=2.0, keep=True),
        # host arrays in and out, sides of no special form, walls of three kinds
        _plane("host_1201x733", 1201, 733, field="lognormal", solver="pcg", keep=False, host=True,
               walls="mixed"),
        # the paper's global grid: stretched cells with the compensating anisotropy
        _plane("paper_9088x568", 9088, 568, field="constant", r=16.0, stretched=True, keep=False),
        # its larger workload, conjugate gradients with FP32 cycles, many
        # right-hand sides (time steps) on one operator
        _plane("paper_16383x1023", 16383, 1023, field="constant", r=16.0, stretched=True,
               solver="pcg", precision="fp32", keep=True),
        # the 64-cell block field at its full size, plain FP64 cycles, kept operator
        _plane("blocks_4095", 4095, 4095, field="blocks", block=64, decades=1.0, keep=True),
        # the largest: FP32 cycles inside FP64 refinement, setup included
        _plane("lognormal_8191", 8191, 8191, field="lognormal", precision="fp32", keep=False),
        # adjoint gradient of a misfit with respect to the log-coefficients
        _plane("gradient_2047", 2047, 2047, field="lognormal", keep=False, gradient=True),
        # strong anisotropy on square cells: alternating line smoothing
        _plane("lines_2047", 2047, 2047, field="constant", r=100.0, smoother="lines", keep=True),
        # many uneven problems in one call
        {"name": "batch_48", "kind": "batch", "count": 48, "block": 16, "decades": 3.0},
        # 3D, the block field of the 3D workload
        _volume("blocks3d_255", 255, 255, 255, block=16),
        # 3D, ragged, conjugate gradients with FP32 cycles
        _volume("ragged3d_161x129x97", 161, 129, 97, block=16, solver="pcg", precision="fp32"),
    ]


def _plane(name, nx, ny, field, block=0, decades=0.0, r=1.0, stretched=False, solver="vcycle",
           precision="fp64", smoother="point", walls="dirichlet", keep=False, host=False, gradient=False):
    return {"name": name, "kind": "plane", "nx": nx, "ny": ny, "field": field, "block": block,
            "decades": decades, "r": r, "stretched": stretched, "solver": solver, "precision": precision,
            "smoother": smoother, "walls": walls, "keep": keep, "host": host, "gradient": gradient}


def _volume(name, nx, ny, nz, block, solver="vcycle", precision="fp64"):
    return {"name": name, "kind": "volume", "nx": nx, "ny": ny, "nz": nz, "block": block, "decades": 2.0,
            "solver": solver, "precision": precision}


def draw(rng):
    """One more case: the entry point first, then sizes spread over their
    logarithm, then the field and the options in use there."""
    def side(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["plane"] * 7 + ["lines", "gradient", "batch", "volume", "volume"])
    if kind == "batch":
        c = {"kind": "batch", "count": rng.randint(8, 48), "block": rng.choice([8, 16, 32]),
             "decades": round(rng.uniform(0.5, 3.0), 2)}
    elif kind == "volume":
        c = _volume("", side(31, 255), side(31, 255), side(31, 255), rng.choice([8, 16, 32]),
                    rng.choice(["vcycle", "pcg"]), rng.choice(["fp64", "fp32"]))
    elif kind == "lines":
        c = _plane("", side(63, 2047), side(63, 2047), "constant", r=round(rng.uniform(10.0, 100.0), 1),
                   smoother="lines", keep=rng.random() < 0.5, solver=rng.choice(["vcycle", "pcg"]))
    elif kind == "gradient":
        c = _plane("", side(63, 2047), side(63, 2047), "lognormal", gradient=True,
                   solver=rng.choice(["vcycle", "pcg"]))
    else:
        nx, aspect = side(63, 4095), rng.choice([1.0, 1.0, rng.uniform(1.0, 4.0), rng.uniform(0.25, 1.0)])
        ny = min(4095, max(63, int(nx * aspect)))
        c = _plane("", nx, ny, rng.choice(["constant", "blocks", "lognormal"]),
                   block=rng.choice([16, 64]), decades=round(rng.uniform(0.5, 2.0 if nx * ny < 1 << 20 else 1.0), 2),
                   solver=rng.choice(["vcycle", "vcycle", "pcg"]), precision=rng.choice(["fp64", "fp32"]),
                   walls=rng.choice(["dirichlet", "dirichlet", "mixed"]), keep=rng.random() < 0.5)
        if c["field"] == "constant" and rng.random() < 0.5:
            # the paper's stretched grids
            nx, ny = side(1023, 16383), side(127, 1023)
            c.update(nx=nx, ny=ny, r=round(nx / ny, 2), stretched=True, walls="dirichlet")
        elif not c["keep"] and nx * ny < 1 << 21:
            c["host"] = rng.random() < 0.4
    c.pop("name", None)
    return c


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _uniform(g, shape, lo=-1.0, hi=1.0):
    return torch.rand(shape, generator=g, device="cuda", dtype=torch.float64) * (hi - lo) + lo


def _blocks(g, shape, block, decades):
    """10^U(-decades, decades), one draw per block of cells."""
    k = 10.0 ** _uniform(g, [-(-n // block) for n in shape], -decades, decades)
    for axis, n in enumerate(shape):
        k = k.repeat_interleave(block, axis).narrow(axis, 0, n)
    return k.contiguous()


def _gaussian_field(g, ny, nx, ell=32.0):
    """Unit Gaussian field with correlation length `ell` cells: white noise
    filtered on a periodic grid of the next powers of two, cropped."""
    my, mx = (1 << (n - 1).bit_length() for n in (ny, nx))
    f = torch.fft.rfft2(torch.randn((my, mx), generator=g, device="cuda", dtype=torch.float64))
    for axis, freq in ((0, torch.fft.fftfreq(my, device="cuda", dtype=torch.float64)),
                       (1, torch.fft.rfftfreq(mx, device="cuda", dtype=torch.float64))):
        h = torch.exp(-(math.pi * ell * freq) ** 2)
        f *= h[:, None] if axis == 0 else h
    w = torch.fft.irfft2(f, s=(my, mx))[:ny, :nx]
    return ((w - w.mean()) / w.std()).contiguous()


def _walls(case):
    """Robin parameter per wall (west, east, south, north); None: u = 0."""
    return (None, 0.0, 0.5, None) if case["walls"] == "mixed" else (None,) * 4


def _aspect(case):
    return case["nx"] / case["ny"] if case["stretched"] else 1.0


def _options(case):
    kw = {"max_cycles": 500}
    if case["solver"] == "pcg":
        kw.update(nu1=1, nu2=1, solver=bm.BMG_SOLVER_PCG)
    if case["precision"] == "fp32":
        kw["precision"] = bm.BMG_FP32_REFINE
    if case["kind"] == "plane":
        kw.update(aniso_r=case["r"], cell_aspect=_aspect(case), bc_beta=_walls(case))
        if case["smoother"] == "lines":
            kw["smoother"] = bm.BMG_SMOOTH_ALTLINE
    return bm.default_options(**kw)


def _plane_inputs(case, seed):
    """Coefficients (log-coefficients for a gradient) and right-hand side."""
    g = _generator(seed)
    ny, nx = case["ny"], case["nx"]
    if case["field"] == "constant":
        k = torch.ones((ny, nx), device="cuda", dtype=torch.float64)
    elif case["field"] == "blocks":
        k = _blocks(g, (ny, nx), case["block"], case["decades"])
    else:
        theta = 2.0 * _gaussian_field(g, ny, nx)
        k = theta if case["gradient"] else torch.exp(theta)
    return k, _uniform(g, (ny, nx)), g


def _volume_inputs(case, seed):
    g = _generator(seed)
    shape = (case["nz"], case["ny"], case["nx"])
    return _blocks(g, shape, case["block"], case["decades"]), _uniform(g, shape)


def _batch_sides(case):
    """The sides of the batch, the weights' shares of `count`, largest last."""
    total, n = sum(BATCH_WEIGHTS), case["count"]
    sides = []
    for s, w in zip(BATCH_SIDES, BATCH_WEIGHTS):
        sides += [s] * max(1, n * w // total)
    return ([BATCH_SIDES[0]] * max(0, n - len(sides)) + sides)[:max(n, len(BATCH_SIDES))]


def _batch_inputs(case, seed):
    g = _generator(seed)
    ks, bs = [], []
    for n in _batch_sides(case):
        ks.append(_blocks(g, (n, n), case["block"], case["decades"]))
        bs.append(_uniform(g, (n, n)))
    return ks, bs


def _pinned(t):
    return torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t).numpy()


def prepare(case, seed):
    state = {"case": case}
    if case["kind"] == "batch":
        ks, bs = _batch_inputs(case, seed)
        # the batch is set up once and solved for many right-hand sides
        state.update(b=bs, plan=bm.Batch(ks, bm.default_options(nu1=1, nu2=1, solver=bm.BMG_SOLVER_PCG,
                                                               max_cycles=500)))
        return state
    if case["kind"] == "volume":
        k, b = _volume_inputs(case, seed)
        state.update(k=k, b=b, options=_options(case))
        return state
    k, b, g = _plane_inputs(case, seed)
    if case["gradient"]:
        state.update(theta=k, b=b, target=_gaussian_field(g, case["ny"], case["nx"]))
    elif case["host"]:
        state.update(k=_pinned(k), b=_pinned(b), x=_pinned(torch.zeros_like(b)), options=_options(case))
    elif case["keep"]:
        state.update(b=b, plan=bm.setup(k, _options(case)))
    else:
        state.update(k=k, b=b, options=_options(case))
    return state


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------

def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        xs = [torch.zeros_like(b) for b in state["b"]]
        state["plan"].solve(state["b"], xs, tol=1e-8)
        return xs
    if case["kind"] == "volume":
        h = bm.setup3(state["k"], state["options"])
        x, _ = h.solve(state["b"], tol=1e-10)
        h.destroy()
        return x
    if case["gradient"]:
        theta = state["theta"].detach().requires_grad_()
        b = state["b"].detach().requires_grad_()
        u = differentiable_solve(theta, b, tol=1e-10, adjoint_tol=1e-9, solver=case["solver"])
        (0.5 * (u - state["target"]).square().sum()).backward()
        return {"u": u.detach(), "theta": theta.grad, "b": b.grad}
    if case["host"]:
        state["x"].fill(0.0)
        bm.solve_host(state["k"], state["b"], state["x"], state["options"], tol=1e-10)
        return state["x"]
    if case["keep"]:
        return state["plan"].solve(state["b"], tol=1e-10)[0]
    h = bm.setup(state["k"], state["options"])
    x, _ = h.solve(state["b"], tol=1e-10)
    h.destroy()
    return x


def work(case):
    """Bytes: each input read once, each output written once (coefficients,
    right-hand side, solution; a kept hierarchy's planes in place of the
    coefficients).  Flops: ten cycles of three sweeps and the residual on
    every level, the fewest that reach the tolerance on smooth fields."""
    if case["kind"] == "batch":
        n = sum(s * s for s in _batch_sides(case))
        return {"bytes": 4.0 * 13 * n + 16.0 * n, "flops": 10 * 3 * 18.0 * n}
    if case["kind"] == "volume":
        n = case["nx"] * case["ny"] * case["nz"]
        return {"bytes": 24.0 * n, "flops": 10 * (4 * 13.0 + 4 * 53.0 / 7) * n}
    n = case["nx"] * case["ny"]
    word = 4.0 if case["precision"] == "fp32" else 8.0
    kept = (3 + 2) * word + (5 + 2) * word / 3 if case["keep"] else 8.0
    passes = 2 if case["gradient"] else 1
    return {"bytes": (kept + 16.0 + (24.0 if case["gradient"] else 0.0)) * n,
            "flops": passes * 10 * (4 * 9.0 + 4 * 17.0 / 3) * n}


# ---------------------------------------------------------------------------
# The same in plain torch
# ---------------------------------------------------------------------------

def _faces(k, r, aspect, betas):
    """Face coefficients of the cell-centred operator: between columns,
    between rows, and the sum over the walls of each cell."""
    kx, ky = k / r, k * r
    ax = 2.0 * kx[:, 1:] * kx[:, :-1] / (kx[:, 1:] + kx[:, :-1]) * aspect
    ay = 2.0 * ky[1:] * ky[:-1] / (ky[1:] + ky[:-1]) / aspect

    def wall(kn, scale, beta):
        return 2.0 * kn * scale * (1.0 if beta is None else beta / (2.0 * kn + beta))

    w = torch.zeros_like(k)
    w[:, 0] += wall(kx[:, 0], aspect, betas[0])
    w[:, -1] += wall(kx[:, -1], aspect, betas[1])
    w[0] += wall(ky[0], 1.0 / aspect, betas[2])
    w[-1] += wall(ky[-1], 1.0 / aspect, betas[3])
    return ax, ay, w


def _apply(ax, ay, w, x):
    y = w * x
    fx, fy = ax * (x[:, 1:] - x[:, :-1]), ay * (x[1:] - x[:-1])
    y[:, :-1] -= fx
    y[:, 1:] += fx
    y[:-1] -= fy
    y[1:] += fy
    return y


class _Direct:
    """Direct solver of the five-point operator: elimination by grid lines
    along the shorter side, with one step of refinement."""

    def __init__(self, ax, ay, w):
        self.op = (ax, ay, w)
        self.flip = w.shape[1] > w.shape[0]
        if self.flip:
            ax, ay, w = ay.T, ax.T, w.T
        self.c = ay
        d = w.clone()
        d[:, :-1] += ax
        d[:, 1:] += ax
        d[:-1] += ay
        d[1:] += ay
        self.inv = []
        for j in range(w.shape[0]):
            m = torch.diag(d[j])
            if w.shape[1] > 1:
                m -= torch.diag(ax[j], 1) + torch.diag(ax[j], -1)
            if j:
                m -= ay[j - 1][:, None] * self.inv[-1] * ay[j - 1]
            self.inv.append(torch.cholesky_inverse(torch.linalg.cholesky(m)))

    def _sweep(self, b):
        y = [b[0]]
        for j in range(1, b.shape[0]):
            y.append(b[j] + self.c[j - 1] * (self.inv[j - 1] @ y[-1]))
        x = [self.inv[-1] @ y[-1]]
        for j in range(b.shape[0] - 2, -1, -1):
            x.append(self.inv[j] @ (y[j] + self.c[j] * x[-1]))
        return torch.stack(x[::-1])

    def solve(self, b):
        x = self._once(b)
        return x + self._once(b - _apply(*self.op, x))

    def _once(self, b):
        return self._sweep(b.T).T if self.flip else self._sweep(b)


def _direct_fits(ny, nx):
    return min(nx, ny) <= 768 and max(nx, ny) <= 1536


def _volume_solve(k, b):
    """Conjugate gradients with the diagonal, restarted from the true
    residual, to the FP64 floor."""
    a = [2.0 * k.narrow(d, 1, k.shape[d] - 1) * k.narrow(d, 0, k.shape[d] - 1)
         / (k.narrow(d, 1, k.shape[d] - 1) + k.narrow(d, 0, k.shape[d] - 1)) for d in range(3)]
    w = torch.zeros_like(k)
    for d in range(3):
        for end in (0, k.shape[d] - 1):
            w.narrow(d, end, 1).add_(2.0 * k.narrow(d, end, 1))

    def apply(x):
        y = w * x
        for d in range(3):
            m = x.shape[d] - 1
            f = a[d] * (x.narrow(d, 1, m) - x.narrow(d, 0, m))
            y.narrow(d, 0, m).sub_(f)
            y.narrow(d, 1, m).add_(f)
        return y

    diag = w.clone()
    for d in range(3):
        m = k.shape[d] - 1
        diag.narrow(d, 0, m).add_(a[d])
        diag.narrow(d, 1, m).add_(a[d])
    x = torch.zeros_like(b)
    for _ in range(3):
        r = b - apply(x)
        stop = 1e-9 * r.norm()
        z = r / diag
        p, rz = z.clone(), (r * z).sum()
        for it in range(3000):
            q = apply(p)
            alpha = rz / (p * q).sum()
            x += alpha * p
            r -= alpha * q
            if it % 50 == 49 and bool(r.norm() <= stop):
                break
            z = r / diag
            new = (r * z).sum()
            p = z + (new / rz) * p
            rz = new
    return x


def exact(case, seed):
    if case["kind"] == "batch":
        ks, bs = _batch_inputs(case, seed)
        # the smaller sides only: the others would take too long here
        return [_Direct(*_faces(k, 1.0, 1.0, (None,) * 4)).solve(b) if b.shape[0] <= 127 else None
                for k, b in zip(ks, bs)]
    if case["kind"] == "volume":
        if case["nx"] * case["ny"] * case["nz"] > 3_000_000:
            return None
        return _volume_solve(*_volume_inputs(case, seed))
    if not _direct_fits(case["ny"], case["nx"]):
        return None
    k, b, g = _plane_inputs(case, seed)
    if not case["gradient"]:
        x = _Direct(*_faces(k, case["r"], _aspect(case), _walls(case))).solve(b)
        return x.cpu().numpy() if case["host"] else x
    target = _gaussian_field(g, case["ny"], case["nx"])
    theta = k.requires_grad_()
    faces = _faces(torch.exp(theta), 1.0, 1.0, (None,) * 4)
    direct = _Direct(*(f.detach() for f in faces))
    u = direct.solve(b)
    lam = direct.solve(u - target)
    # dL/dtheta = -lam . (dA/dtheta u), dL/db = lam
    grad, = torch.autograd.grad(-(lam * _apply(*faces, u)).sum(), theta)
    return {"u": u, "theta": grad, "b": lam}
