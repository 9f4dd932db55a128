"""Workloads of the pressure solve, each one call sequence of a ship-wave program.

A time step sets the density from its water fraction and solves for the pressure; a projection
step also forms the source from the face velocities and corrects them; a server keeps many grids
on the device and submits the current step of all of them together.  Every workload runs through
the C ABI (`capi`) on device arrays, with inputs made on the GPU from a seed.

The relative residual asked for is 1e-10 (the regression grid's; the benchmark line asks for 1e-9):
the pressure is then the solution of the discrete equation to ten digits or better.
"""
import math

import numpy as np
import torch

from paper_1410_1942_gb300 import capi, inputs

DEVICE = "cuda"
DT = inputs.DT
RHO_AIR, RHO_WATER = inputs.RHO_AIR, inputs.RHO_WATER
EXACT_MAX_CELLS = 24_000_000  # above this the 64-bit answer takes too long


def _case(name, call, shape, tol, **options):
    """One workload.  call: "solve" (set the density, solve from zero), "step" (a projection step
    started from the last step's pressure), "batch" (`count` grids submitted together from zero)
    or "serve" (the same, each started from its last step's pressure).  shape: the grid, or the
    largest grid of a batch (`mix` seeds its sizes)."""
    case = {"name": name, "call": call, "nx": shape[0], "ny": shape[1], "nz": shape[2],
            "tol": tol, "body": "strut", "precision": "fp32", "precond": "jacobi",
            "inner_tol": 1e-4, "walls": 0, "periodic": False, "cut": False, "count": 1, "mix": 0}
    case.update(options)
    return case


def listed():
    return [
        # the smallest production grid, plain FP64: a regression run, all launches and latency
        _case("flat32_fp64", "solve", (32, 32, 32), 1e-10, precision="fp64"),
        # a small default solve (one served request alone): latency of one persistent launch
        _case("small_jacobi", "solve", (64, 48, 32), 1e-10),
        # the strut grid of the benchmark, each preconditioner: an ordinary single solve
        _case("strut_jacobi", "solve", (256, 128, 128), 1e-10),
        _case("strut_rbssor", "solve", (256, 128, 128), 1e-10, precond="rbssor"),
        # plain FP64 on the strut at half resolution: the run that mixed precision is checked by
        _case("strut_fp64", "solve", (128, 64, 64), 1e-10, precision="fp64"),
        # a grid whose sides fit no tile: a domain cut to a measured tank
        _case("ragged_jacobi", "solve", (250, 125, 90), 1e-10),
        # BF16 densities on the wedge at half resolution
        _case("wedge_bf16", "solve", (512, 256, 128), 1e-10, body="wedge", precision="bf16"),
        # the largest single solve, with the strongest preconditioner
        _case("wedge_mg", "solve", (1024, 512, 256), 1e-10, body="wedge", precond="mg",
              inner_tol=1e-5),
        # one projection of a running simulation: periodic strut run, multigrid, warm start
        _case("step_mg", "step", (256, 128, 128), 1e-10, precond="mg", inner_tol=1e-5,
              periodic=True),
        # the strut as a free-slip cut-cell body, side walls open (p = 0), multigrid
        _case("cut_mg", "solve", (192, 96, 96), 1e-10, precond="mg", inner_tol=1e-5, cut=True,
              walls=capi.WALL_XM | capi.WALL_XP),
        # 64 uneven grids submitted together (persistent batch launches)
        _case("batch64_jacobi", "batch", (128, 64, 64), 1e-10, count=64, mix=1),
        # a server's current step of 16 requests, warm starts, multigrid on the worker streams
        _case("serve16_mg", "serve", (256, 128, 128), 1e-10, precond="mg", inner_tol=1e-5,
              count=16, mix=2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A workload of the same ranges: any size from the smallest to the largest grid of its
    preconditioner, multiples of 8 and odd sizes, every option."""
    kind = rng.choice(["jacobi", "jacobi", "rbssor", "mg", "mg", "fp64", "step", "cut", "many"])
    if kind == "many":
        precond = rng.choice(["jacobi", "mg"])
        big = rng.random() < 0.5
        return _drawn(rng, rng.choice(["batch", "serve"]), (256, 128, 128) if big else (128, 64, 64),
                      precond, count=rng.randint(4, 16 if big else 48), mix=rng.randint(3, 999))
    nx = _log_int(rng, 32, {"jacobi": 512, "rbssor": 320, "mg": 768, "fp64": 160, "step": 448,
                            "cut": 288}[kind])
    size = [nx, nx * rng.uniform(0.35, 0.75), nx * rng.uniform(0.35, 0.6)]
    mult = rng.choice([8, 16, 32]) if rng.random() < 0.6 else 1
    # no drawn solve costs more than the largest listed one
    most = {"jacobi": 16e6, "rbssor": 6e6, "mg": 40e6, "fp64": 1e6, "step": 16e6, "cut": 5e6}[kind]
    shrink = min(1.0, ((most if mult > 1 else most / 5) / math.prod(size)) ** (1 / 3))
    nx, ny, nz = (max(16, mult * round(v * shrink / mult)) for v in size)
    options = {"walls": rng.choice([0, 0, capi.WALL_XM | capi.WALL_XP, capi.WALL_ZM])}
    if options["walls"] in (0, capi.WALL_ZM) and kind != "rbssor" and rng.random() < 0.25:
        options["periodic"] = True
    precond = {"step": "mg", "cut": rng.choice(["jacobi", "mg"]), "fp64": "jacobi"}.get(kind, kind)
    if kind == "fp64":
        options["precision"] = "fp64"
    elif kind != "cut" and rng.random() < 0.25:
        options["precision"] = "bf16"
    if kind == "cut":
        options["cut"] = True
    if kind in ("jacobi", "mg") and rng.random() < 0.4:
        options["body"] = "wedge"
    return _drawn(rng, "step" if kind == "step" else "solve", (nx, ny, nz), precond, **options)


def _drawn(rng, call, shape, precond, **options):
    case = _case("", call, shape, 1e-10, precond=precond,
                 inner_tol=1e-5 if precond == "mg" else 1e-4, **options)
    del case["name"]
    return case


# ------------------------------------------------------------------ inputs
def _shapes(case):
    shape = (case["nx"], case["ny"], case["nz"])
    if case["call"] not in ("batch", "serve"):
        return [shape]
    rng = np.random.default_rng(case["mix"])
    return [inputs.draw_shape(rng, (32, 32, 32), shape) for _ in range(case["count"])]


def _fields(case, shape, seed):
    """(grid, F, velocity modes)"""
    if case["body"] == "wedge":
        grid, F, _, _ = inputs.wedge_fields_t(shape, seed=seed, device=DEVICE)
        return grid, F, inputs.fourier_modes(np.random.default_rng(seed + 1))
    grid, F, _, modes = inputs.mixed_fields_t(shape, seed, device=DEVICE)
    return grid, F, modes


def _face_velocity(grid, modes, periodic):
    """u* of the modes on the faces; no flow through the walls, the top open, the two x ends one
    face when x is periodic."""
    nx, ny, nz, h = grid.nx, grid.ny, grid.nz, grid.h
    L = grid.lengths
    at = [[(torch.arange(n + 1, dtype=torch.float64, device=DEVICE) - (0.0 if d == f else -0.5))
           [:n + 1 if d == f else n] * h for d, n in enumerate((nx, ny, nz))] for f in range(3)]
    out = []
    for f in range(3):
        x, y, z = at[f]
        v = torch.zeros(len(z), len(y), len(x), dtype=torch.float64, device=DEVICE)
        for m in modes:
            k = [2.0 * math.pi * m.k[d] / L[d] for d in range(3)]
            v += inputs.MODE_AMPLITUDE * m.a[f] * torch.sin(
                (k[2] * z)[:, None, None] + (k[1] * y)[None, :, None] + (k[0] * x + m.phase))
        out.append(v)
    u, v, w = out
    if periodic:
        u[:, :, -1] = u[:, :, 0]
    else:
        u[:, :, 0] = 0.0
        u[:, :, -1] = 0.0
    v[:, 0] = 0.0
    v[:, -1] = 0.0
    w[0] = 0.0
    return u, v, w


def _divergence(grid, u, v, w):
    return (u.diff(dim=2) + v.diff(dim=1) + w.diff(dim=0)) / (grid.h * DT)


def _cut_strut(grid):
    """Open fractions of the faces and fluid fractions of the cells around a vertical elliptic
    strut at the domain centre (4 sample points along each side)."""
    nx, ny, nz, h = grid.nx, grid.ny, grid.nz, grid.h
    sub = 4
    inside = torch.arange(sub, dtype=torch.float64, device=DEVICE).add(0.5).div(sub)
    xs = (torch.arange(nx, dtype=torch.float64, device=DEVICE)[:, None] + inside).flatten() * h
    ys = (torch.arange(ny, dtype=torch.float64, device=DEVICE)[:, None] + inside).flatten() * h
    xf = torch.arange(nx + 1, dtype=torch.float64, device=DEVICE) * h
    yf = torch.arange(ny + 1, dtype=torch.float64, device=DEVICE) * h

    def wet(x, y):
        r = (((x - 0.5 * nx * h) / 0.1) ** 2)[None, :] + (((y - 0.5 * ny * h) / 0.02) ** 2)[:, None]
        return (r > 1.0).double()

    ax = wet(xf, ys).view(ny, sub, nx + 1).mean(1)
    ay = wet(xs, yf).view(ny + 1, nx, sub).mean(2)
    vol = wet(xs, ys).view(ny, sub, nx, sub).mean((1, 3))
    full = lambda a, n: a.expand(n, *a.shape).contiguous()  # noqa: E731
    return full(ax, nz), full(ay, nz), full(vol, nz + 1), full(vol, nz)


def _wet_cells(case, grid, s):
    """The source as a program with a cut-cell body forms it: nothing where there is no fluid."""
    return s * (_cut_strut(grid)[3] > 0.0) if case["cut"] else s


def _solver(case, grid):
    return capi.Poisson(grid.nx, grid.ny, grid.nz, grid.h, precision=case["precision"],
                        precond=case["precond"], inner_tol=case["inner_tol"],
                        dirichlet_walls=case["walls"], periodic_x=case["periodic"])


def prepare(case, seed):
    state = {"call": case["call"], "tol": case["tol"], "solvers": [], "F": [], "s": [], "p0": [],
             "p": []}
    for q, shape in enumerate(_shapes(case)):
        grid, F, modes = _fields(case, shape, seed + 7919 * q)
        u, v, w = _face_velocity(grid, modes, case["periodic"])
        s = _wet_cells(case, grid, _divergence(grid, u, v, w))
        solver = _solver(case, grid)
        if case["cut"]:
            solver.set_apertures(*_cut_strut(grid))
        p0 = torch.zeros_like(F)
        if case["call"] in ("step", "serve"):
            # the last step's pressure: the source one time step earlier
            back = _face_velocity(grid, inputs.advect_modes(modes, grid, -DT), case["periodic"])
            solver.set_density(F)
            solver.solve(_divergence(grid, *back), p0, 1e-9)
        if case["call"] == "step":
            state["u0"] = (u, v, w)
            state["u"] = tuple(torch.empty_like(a) for a in (u, v, w))
        if case["call"] in ("batch", "serve"):
            solver.set_density(F)
        state["solvers"].append(solver)
        state["F"].append(F)
        state["s"].append(s)
        state["p0"].append(p0)
        state["p"].append(torch.empty_like(F))
    return state


# ------------------------------------------------------------------ one pass
def run(state):
    for p, p0 in zip(state["p"], state["p0"]):
        p.copy_(p0)
    if state["call"] in ("batch", "serve"):
        torch.cuda.synchronize()  # the batch runs on streams of its own
        pending = capi.batch_submit(state["solvers"], state["s"], state["p"], state["tol"])
        while pending:
            waiting = []
            for ticket in pending:
                status, _ = capi.poll(ticket)
                if status == capi.PENDING:
                    waiting.append(ticket)
                elif status != capi.OK:
                    raise capi.PoissonError(status, "poisson_poll")
            pending = waiting
        return state["p"]
    solver, F, p = state["solvers"][0], state["F"][0], state["p"][0]
    solver.set_density(F, RHO_AIR, RHO_WATER)
    if state["call"] == "step":
        for a, a0 in zip(state["u"], state["u0"]):
            a.copy_(a0)
        solver.projection_step(*state["u"], DT, p, state["tol"], s=state["s"][0])
        return {"u": state["u"][0], "v": state["u"][1], "w": state["u"][2], "p": p}
    solver.solve(state["s"][0], p, state["tol"])
    return p


def work(case):
    """Each input read and each output written once, and the operator applied once (the iterations
    are the method's choice)."""
    cells = sum(a * b * c for a, b, c in _shapes(case))
    arrays = {"solve": 3 + (4 if case["cut"] else 0), "step": 2 + 6 + 1, "batch": 2, "serve": 3}
    return {"bytes": 8.0 * cells * arrays[case["call"]], "flops": 30.0 * cells}


# ------------------------------------------------------------------ the answer in 64 bits
def _operator(case, grid, F):
    """Faces between cells (x, y, z; the wrap face of x or None) and the diagonal of
    A = -h^2 div((1/rho) grad), and the cells' fluid fractions (None without a body)."""
    rho = RHO_AIR + F * (RHO_WATER - RHO_AIR)
    bx = 2.0 / (rho[:, :, 1:] + rho[:, :, :-1])
    by = 2.0 / (rho[:, 1:] + rho[:, :-1])
    bz = 2.0 / (rho[1:] + rho[:-1])
    edge = 2.0 / rho
    wrap = 2.0 / (rho[:, :, 0] + rho[:, :, -1]) if case["periodic"] else None
    ax = ay = az = vol = None
    wet = torch.ones_like(F)
    if case["cut"]:
        ax, ay, az, vol = _cut_strut(grid)
        wet = (vol > 0.0).double()
        bx = bx * ax[:, :, 1:-1] * wet[:, :, 1:] * wet[:, :, :-1]
        by = by * ay[:, 1:-1] * wet[:, 1:] * wet[:, :-1]
        bz = bz * az[1:-1] * wet[1:] * wet[:-1]
        if wrap is not None:
            wrap = wrap * ax[:, :, 0] * wet[:, :, 0] * wet[:, :, -1]
    diag = torch.zeros_like(F)
    diag[:, :, 1:] += bx
    diag[:, :, :-1] += bx
    diag[:, 1:] += by
    diag[:, :-1] += by
    diag[1:] += bz
    diag[:-1] += bz
    if wrap is not None:
        diag[:, :, 0] += wrap
        diag[:, :, -1] += wrap
    one = torch.ones((), dtype=torch.float64, device=DEVICE)
    open_ = lambda a, at: one if a is None else a[at]  # noqa: E731
    every = slice(None)
    for wall, at, a, face in ((32, (-1,), az, (-1,)), (capi.WALL_ZM, (0,), az, (0,)),
                              (capi.WALL_XM, (every, every, 0), ax, (every, every, 0)),
                              (capi.WALL_XP, (every, every, -1), ax, (every, every, -1)),
                              (capi.WALL_YM, (every, 0), ay, (every, 0)),
                              (capi.WALL_YP, (every, -1), ay, (every, -1))):
        if (case["walls"] | 32) & wall:  # 32: the top, always p = 0
            diag[at] += edge[at] * open_(a, face)
    diag = torch.where(wet > 0.0, diag, torch.ones_like(diag))
    return bx, by, bz, wrap, diag, vol


def _apply(op, x):
    bx, by, bz, wrap, diag, _ = op
    y = diag * x
    y[:, :, 1:].addcmul_(bx, x[:, :, :-1], value=-1.0)
    y[:, :, :-1].addcmul_(bx, x[:, :, 1:], value=-1.0)
    y[:, 1:].addcmul_(by, x[:, :-1], value=-1.0)
    y[:, :-1].addcmul_(by, x[:, 1:], value=-1.0)
    y[1:].addcmul_(bz, x[:-1], value=-1.0)
    y[:-1].addcmul_(bz, x[1:], value=-1.0)
    if wrap is not None:
        y[:, :, 0].addcmul_(wrap, x[:, :, -1], value=-1.0)
        y[:, :, -1].addcmul_(wrap, x[:, :, 0], value=-1.0)
    return y


def _pressure(case, grid, F, s):
    """A p = -h^2 s to about 1e-14 by conjugate gradients with the diagonal, restarted from the
    recomputed residual."""
    op = _operator(case, grid, F)
    b = -(grid.h ** 2) * s
    if case["cut"]:
        b = b * op[5]
    inv = 1.0 / op[4]
    dot = lambda a, c: torch.dot(a.reshape(-1), c.reshape(-1))  # noqa: E731
    x = torch.zeros_like(b)
    for _ in range(4):
        r = b - _apply(op, x)
        now = float(r.norm() / b.norm())
        if now < 1e-13:
            break
        target = max(1e-12, 1e-14 / now)
        e, p = torch.zeros_like(b), None
        rz_old, start = None, r.norm()
        for i in range(20000):
            z = inv * r
            rz = dot(r, z)
            p = z if p is None else z.add_(p * (rz / rz_old))
            q = _apply(op, p)
            alpha = rz / dot(p, q)
            e.addcmul_(p, alpha)
            r.addcmul_(q, -alpha)
            rz_old = rz
            if i % 25 == 24 and float(r.norm() / start) < target:
                break
        x += e
    return x


def exact(case, seed):
    found = []
    shapes = _shapes(case)
    if sum(a * b * c for a, b, c in shapes) > EXACT_MAX_CELLS:
        return None
    for q, shape in enumerate(shapes):
        grid, F, modes = _fields(case, shape, seed + 7919 * q)
        u, v, w = _face_velocity(grid, modes, case["periodic"])
        s = _wet_cells(case, grid, _divergence(grid, u, v, w))
        found.append(_pressure(case, grid, F, s))
    if case["call"] != "step":
        return found if case["call"] in ("batch", "serve") else found[0]
    p, h = found[0], grid.h
    rho = RHO_AIR + F * (RHO_WATER - RHO_AIR)
    g = DT / h
    u[:, :, 1:-1] -= g * 2.0 / (rho[:, :, 1:] + rho[:, :, :-1]) * p.diff(dim=2)
    v[:, 1:-1] -= g * 2.0 / (rho[:, 1:] + rho[:, :-1]) * p.diff(dim=1)
    w[1:-1] -= g * 2.0 / (rho[1:] + rho[:-1]) * p.diff(dim=0)
    w[-1] += g * 2.0 / rho[-1] * p[-1]
    if case["periodic"]:
        wrap = g * 2.0 / (rho[:, :, 0] + rho[:, :, -1]) * (p[:, :, 0] - p[:, :, -1])
        u[:, :, 0] -= wrap
        u[:, :, -1] -= wrap
    if case["walls"] & capi.WALL_XM:
        u[:, :, 0] -= g * 2.0 / rho[:, :, 0] * p[:, :, 0]
    if case["walls"] & capi.WALL_XP:
        u[:, :, -1] += g * 2.0 / rho[:, :, -1] * p[:, :, -1]
    if case["walls"] & capi.WALL_ZM:
        w[0] -= g * 2.0 / rho[0] * p[0]
    return {"u": u, "v": v, "w": w, "p": p}
