"""The work that users of this library have it do, as cases that can be timed
and whose outputs can be compared.

Kinds of case, each through the package's public entry points:

  step     ``Context.ns_step``: time steps of the composed method, then the
           velocity, pressure and markers fetched (the state a program goes on
           with).  Planar and axisymmetric, both spreadings, the indicator
           function, Crank-Nicolson, relocation and the measure correction.
  solve    ``mg_setup`` + ``mg_solve``: a pressure solve from zero on new
           coefficients, as a program with its own discretisation makes it.
  noalloc  ``mg_solve_noalloc``: the same without device allocations, on the
           small grids that call takes.
  markers  marker geometry, conventional spreading and interpolation: the
           coupling of an immersed boundary to another flow solver.
  infer    ``Net.infer``: the learned warm start's pressure estimate.
  grad     ``Net.grad``: loss and gradients of one training batch.

Velocities start as a vortex whose speed is of the order of the drops'
capillary velocity, so that every output is a flow of its own size and not the
difference of a balanced static drop; the time step is a quarter of the
explicit limits, so that hundreds of passes stay far from the walls.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1807_10504_gb300 as ib

RHO_G, RHO_L, MU_G, MU_L, SIGMA = 1e-3, 1.0, 1e-4, 1e-2, 1.0  # the library's defaults


# ------------------------------------------------------------------ the cases
def _step(name, nx, ny, **kw):
    case = dict(kind="step", name=name, nx=nx, ny=ny, drops=1, markers=128, rmin=0.2, rmax=0.25,
                steps=10, precision=0, spread=1, kernel=0, relocate_every=10, viscous=0,
                indicator=0, mass_every=0, axisym=0, speed=1.0)
    case.update(kw)
    return case


def listed():
    return [
        # the smallest call: one step of one drop on a coarse grid with the
        # default (FP64) solver, as interactive and parameter studies run it;
        # launches and latency are all there is
        _step("step_drop64", 64, 64, steps=1, speed=0.5),
        # the conventional scheme the paper compares with: cosine delta
        # spreading and the Poisson indicator, FP64 solves, one jittered drop
        _step("step_conventional256", 256, 256, markers=512, rmin=0.19, rmax=0.21, spread=0,
              indicator=1),
        # the paper's own settings: Crank-Nicolson, relocation every step, the
        # measure correction every 20 steps
        _step("step_paper512", 512, 512, drops=16, markers=256, rmin=0.04, rmax=0.08, steps=20,
              precision=1, relocate_every=1, viscous=1, mass_every=20, speed=2.0),
        # the benchmark's workload, an ordinary production run: 64 drops,
        # density ratio 1000, FP32 cycles in FP64 defect correction
        _step("step_drops1024", 1024, 1024, drops=64, markers=256, rmin=0.01, rmax=0.03,
              precision=2, speed=4.0),
        # the largest grid of the benchmark (markers about a cell apart):
        # operands beyond the L2
        _step("step_drops2048", 2048, 2048, drops=64, markers=384, rmin=0.01, rmax=0.03,
              precision=2, speed=4.0),
        # the free-fall drop: axisymmetric, SI units, gravity, moving frame
        _step("step_freefall", 256, 1024, markers=1024, precision=2, axisym=1, speed=0.1),
        # pressure solves on new coefficients: FP64 on the benchmark's grid ...
        dict(kind="solve", name="solve_fp64_1024", nx=1024, ny=1024, drops=64, precision=0),
        # ... and mixed on a 3:2 domain, whose coarsest level is not a few cells
        dict(kind="solve", name="solve_mixed_960x640", nx=960, ny=640, drops=24, precision=1),
        # a solve inside a program that owns all device memory
        dict(kind="noalloc", name="noalloc_256x192", nx=256, ny=192, drops=4, precision=2),
        # marker coupling alone: 64 drops, 16384 markers
        dict(kind="markers", name="markers_1024", nx=1024, ny=1024, drops=64, markers=256,
             rmin=0.01, rmax=0.03, kernel=0),
        # the warm start's estimate on an unseen 512^2 system
        dict(kind="infer", name="infer_512", n=512, batch=1, coarsen=0),
        # one training batch of the benchmark's network training
        dict(kind="grad", name="grad_8x256", n=256, batch=8),
    ]


_SIDES = [64, 80, 96, 128, 160, 192, 256, 320, 384, 512, 640, 768, 1024]


def _coarsest(nx, ny):
    while nx % 2 == 0 and ny % 2 == 0 and nx * ny > 16:
        nx, ny = nx // 2, ny // 2
    return nx * ny


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _grid(rng, most):
    """A grid with sides between 64 and `most`, at most 3:1, that coarsens well
    (a multiple of 16 now and then that is none of 64 among them)."""
    while True:
        a = _log(rng, 64, most * 1.2)
        b = a * _log(rng, 1 / 3, 3)
        if rng.random() < 0.6:
            nx = min(_SIDES, key=lambda s: abs(math.log(s / a)))
            ny = min(_SIDES, key=lambda s: abs(math.log(s / b)))
        else:
            q = rng.choice((8, 16, 32))
            nx, ny = q * max(1, round(a / q)), q * max(1, round(b / q))
        if 64 <= min(nx, ny) and max(nx, ny) <= most and _coarsest(nx, ny) <= 160:
            return nx, ny


def _lattice(nx, ny, drops):
    """Columns and rows of the lattice the drops sit on."""
    cols = max(1, round(math.sqrt(drops * nx / ny)))
    return cols, -(-drops // cols)


def _drops(rng, nx, ny, most):
    """How many drops, and their radii in units of the longer side: at least
    six cells, and eight cells between neighbours and to the walls."""
    h = 1.0 / max(nx, ny)
    while True:
        drops = max(1, round(_log(rng, 1, most)))
        cols, rows = _lattice(nx, ny, drops)
        room = 0.5 * min(nx * h / cols, ny * h / rows) - 8 * h
        if room >= 8 * h:
            rmax = min(room, 0.25) * rng.uniform(0.8, 1.0)
            return drops, max(6 * h, rmax * rng.uniform(0.4, 0.9)), max(7 * h, rmax)


def draw(rng):
    kind = rng.choice(("step", "step", "step", "solve", "solve", "noalloc", "markers", "infer", "grad"))
    if kind == "step":
        if rng.random() < 0.2:
            nx = rng.choice((128, 160, 192, 256))
            return _step_case(nx, nx * rng.choice((2, 3, 4)), markers=2 * rng.randint(nx, 2 * nx),
                              precision=rng.choice((0, 1, 2)), axisym=1, speed=0.1)
        precision = rng.choice((0, 1, 2))
        nx, ny = _grid(rng, 512 if precision == 0 else 1024)
        drops, rmin, rmax = _drops(rng, nx, ny, 64)
        # at most 150 cells: the relocation takes about 1400 markers a drop
        rmin, rmax = (min(r, 150 / max(nx, ny)) for r in (rmin, rmax))
        markers = max(24, round(2 * math.pi * rmax * max(nx, ny) * rng.uniform(0.8, 2.0)))
        return _step_case(nx, ny, drops=drops, rmin=rmin, rmax=rmax, markers=min(markers, 1300),
                          precision=precision, spread=rng.choice((0, 1, 1)),
                          kernel=rng.choice((0, 0, 1)), relocate_every=rng.choice((0, 1, 10)),
                          viscous=rng.choice((0, 0, 1)), indicator=rng.choice((0, 0, 0, 1)),
                          mass_every=rng.choice((0, 0, 20)),
                          speed=rng.uniform(0.5, 2.0) * min(1.0, max(nx, ny) / 512),
                          steps=rng.choice((1, 10)))
    if kind == "solve":
        nx, ny = _grid(rng, 1024)
        return dict(kind=kind, nx=nx, ny=ny, drops=_drops(rng, nx, ny, 64)[0],
                    precision=rng.choice((0, 1, 2)))
    if kind == "noalloc":
        while True:
            nx, ny = _grid(rng, 512)
            if nx * ny <= 65536:
                break
        return dict(kind=kind, nx=nx, ny=ny, drops=_drops(rng, nx, ny, 4)[0],
                    precision=rng.choice((0, 1, 2)))
    if kind == "markers":
        nx, ny = _grid(rng, 1024)
        drops, rmin, rmax = _drops(rng, nx, ny, 64)
        return dict(kind=kind, nx=nx, ny=ny, drops=drops, rmin=rmin, rmax=rmax,
                    markers=max(24, round(2 * math.pi * rmax * max(nx, ny) * rng.uniform(0.8, 3.0))),
                    kernel=rng.choice((0, 1)))
    if kind == "infer":
        coarsen = rng.choice((0, 0, 1, 2))
        n = 4 * 2 ** coarsen * max(1, round(_log(rng, 64, 1024) / (4 * 2 ** coarsen)))
        return dict(kind=kind, n=n, batch=1 if n > 512 else rng.choice((1, 2, 4)), coarsen=coarsen)
    n = 4 * round(_log(rng, 32, 256) / 4)
    return dict(kind=kind, n=n, batch=rng.randint(1, 8))


def _step_case(nx, ny, **kw):
    case = _step("", nx, ny, **kw)
    del case["name"]
    return case


# -------------------------------------------------------------------- inputs
def _place(case, rng):
    """Drops of radii in [rmin, rmax] on a jittered lattice of the domain
    [0, nx h] x [0, ny h], h = 1 / max(nx, ny), eight cells apart at least."""
    nx, ny, drops = case["nx"], case["ny"], case["drops"]
    h = 1.0 / max(nx, ny)
    cols, rows = _lattice(nx, ny, drops)
    px, py = nx * h / cols, ny * h / rows
    rmin = case.get("rmin", 0.25 * min(px, py))
    rmax = case.get("rmax", 0.35 * min(px, py))
    out = []
    for k in range(drops):
        R = rng.uniform(rmin, rmax)
        sx, sy = (max(0.0, 0.5 * p - R - 5 * h) * 0.5 for p in (px, py))
        out.append(((k % cols + 0.5) * px + rng.uniform(-sx, sx),
                    (k // cols + 0.5) * py + rng.uniform(-sy, sy), R))
    return out, h


def _polylines(case, rng):
    """Counter-clockwise marker polylines: slightly elliptic, one of them with
    a little radial noise (what relocation and curvature meet in earnest)."""
    centres, h = _place(case, rng)
    n = case["markers"]
    X, Y = [], []
    for k, (cx, cy, R) in enumerate(centres):
        t = 2 * math.pi * (np.arange(n) + rng.uniform()) / n
        r = R * (1 + rng.uniform(0.0, 0.05) * np.cos(2 * t))
        if k == 0:
            r = r + rng.uniform(-0.02 * h, 0.02 * h, n)
        X.append(cx + r * np.cos(t))
        Y.append(cy + r * np.sin(t))
    return np.concatenate(X), np.concatenate(Y), np.arange(len(centres) + 1, dtype=np.int32) * n, h


def _vortex(nx, ny, h, speed):
    """u, v of the stream function sin(pi x / Lx) sin(pi y / Ly) on the faces."""
    Lx, Ly, f = nx * h, ny * h, dict(dtype=torch.float64, device="cuda")
    xf, xc = torch.arange(nx + 1, **f) * h, (torch.arange(nx, **f) + 0.5) * h
    yf, yc = torch.arange(ny + 1, **f) * h, (torch.arange(ny, **f) + 0.5) * h
    u = speed * torch.sin(math.pi * xf / Lx)[None] * torch.cos(math.pi * yc / Ly)[:, None]
    v = -speed * Ly / Lx * torch.cos(math.pi * xc / Lx)[None] * torch.sin(math.pi * yf / Ly)[:, None]
    return u.contiguous(), v.contiguous()


def _indicator(case, seed):
    """A smoothed characteristic function of the case's drops (cells)."""
    rng = np.random.default_rng(seed)
    centres, h = _place(case, rng)
    f = dict(dtype=torch.float64, device="cuda")
    x = (torch.arange(case["nx"], **f) + 0.5) * h
    y = (torch.arange(case["ny"], **f) + 0.5) * h
    H = torch.zeros((case["ny"], case["nx"]), **f)
    for cx, cy, R in centres:
        d = torch.sqrt((x[None] - cx) ** 2 + (y[:, None] - cy) ** 2) - R
        H = torch.maximum(H, 0.5 * (1 - torch.tanh(d / (1.5 * h))))
    return H, h, rng


def _pressure_system(case, seed):
    """Face coefficients 1 / rho and a right-hand side div(beta F) + div u* / dt
    of a multi-drop system at density ratio 1000."""
    H, h, rng = _indicator(case, seed)
    rho = RHO_G + (RHO_L - RHO_G) * H
    ny, nx = H.shape
    bx = torch.zeros((ny, nx + 1), dtype=torch.float64, device="cuda")
    by = torch.zeros((ny + 1, nx), dtype=torch.float64, device="cuda")
    bx[:, 1:-1] = 2.0 / (rho[:, 1:] + rho[:, :-1])
    by[1:-1] = 2.0 / (rho[1:] + rho[:-1])
    qx, qy = torch.zeros_like(bx), torch.zeros_like(by)
    qx[:, 1:-1] = bx[:, 1:-1] * (H[:, 1:] - H[:, :-1]) * (SIGMA * 30.0 / h)
    qy[1:-1] = by[1:-1] * (H[1:] - H[:-1]) * (SIGMA * 30.0 / h)
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    noise = 1e-3 * float(qx.abs().max())
    qx[:, 1:-1] += noise * torch.randn(qx[:, 1:-1].shape, generator=g, dtype=torch.float64, device="cuda")
    qy[1:-1] += noise * torch.randn(qy[1:-1].shape, generator=g, dtype=torch.float64, device="cuda")
    b = (qx[:, 1:] - qx[:, :-1] + qy[1:] - qy[:-1]) / h
    return bx, by, b.contiguous(), rho, h


_NET = ((2, 16), (16, 16), (16, 32), (32, 32), (32, 32), (32, 32), (64, 32), (48, 16), (16, 1))


def _net_params(seed):
    """He-normal weights and small biases, in the network's flat order."""
    rng = np.random.default_rng(seed + 7)
    out = []
    for ci, co in _NET:
        out.append((rng.standard_normal(co * 9 * ci) * math.sqrt(2.0 / (9 * ci))).astype(np.float32))
        out.append((0.05 * rng.standard_normal(co)).astype(np.float32))
    return np.concatenate(out)


def _net_inputs(case, seed):
    n, parts = case["n"], []
    for k in range(case["batch"]):
        sys = dict(nx=n, ny=n, drops=4 if n >= 96 else 1)
        _, _, b, rho, h = _pressure_system(sys, 1000 * seed + k)
        # a pressure of the right size: a capillary jump per drop, smooth outside
        x = (torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) * h
        p = 30.0 * (rho - RHO_G) + 3.0 * torch.cos(2 * math.pi * x)[None] * torch.cos(math.pi * x)[:, None]
        parts.append((b, rho, p))
    return tuple(torch.stack(t).contiguous() for t in zip(*parts))


def prepare(case, seed):
    kind = case["kind"]
    rng = np.random.default_rng(seed)
    if kind == "step":
        return _prepare_step(case, rng)
    if kind == "markers":
        X, Y, start, h = _polylines(case, rng)
        ctx = ib.Context(ib.Config(nx=case["nx"], ny=case["ny"], h=h, kernel=case["kernel"]), X, Y, start)
        u, v = _vortex(case["nx"], case["ny"], h, 1.0)
        return dict(case=case, ctx=ctx, u=u, v=v)
    if kind in ("solve", "noalloc"):
        bx, by, b, _, h = _pressure_system(case, seed)
        state = dict(case=case, bx=bx, by=by, b=b, h=h)
        if kind == "solve":
            # the context's own drop plays no part in the solve
            t = 2 * math.pi * np.arange(32) / 32
            w, g = 0.5 * case["nx"] * h, 0.5 * case["ny"] * h
            state["ctx"] = ib.Context(ib.Config(nx=case["nx"], ny=case["ny"], h=h), w + 8 * h * np.cos(t),
                                      g + 8 * h * np.sin(t), np.array([0, 32], np.int32))
        return state
    net = ib.Net(seed)
    net.set_params(_net_params(seed))
    b, rho, p = _net_inputs(case, seed)
    if kind == "infer":
        net.set_coarsen(case["coarsen"])
        return dict(case=case, net=net, b=b, rho=rho)
    return dict(case=case, net=net, b=b, rho=rho, p=p)


def _prepare_step(case, rng):
    nx, ny = case["nx"], case["ny"]
    opt = {k: case[k] for k in ("precision", "spread", "kernel", "relocate_every", "viscous",
                                "indicator", "mass_every", "axisym")}
    if case["axisym"]:
        # a 1 mm water drop in air, 4 diameters above the inflow
        D, n = 1e-3, case["markers"]
        h = 4 * D / nx
        mat = dict(rho_l=1000.0, rho_g=1.2, mu_l=1e-3, mu_g=1.8e-5, sigma=0.072)
        th = -0.5 * math.pi + 2 * math.pi * np.arange(n // 2 + 1) / n
        r = 0.5 * D * (1 + rng.uniform(0.01, 0.05) * np.cos(2 * th))
        x, y = r * np.cos(th), min(4 * D, 0.5 * ny * h) + r * np.sin(th)
        x[0] = x[-1] = 0.0
        X, Y = np.concatenate([x, -x[-2:0:-1]]), np.concatenate([y, y[-2:0:-1]])
        start = np.array([0, n], np.int32)
        opt.update(mat, frame=1, gy=-9.81)
        f = dict(dtype=torch.float64, device="cuda")
        R, L, a = nx * h, ny * h, case["speed"] * rng.uniform(0.8, 1.2)
        rf, rc = torch.arange(nx + 1, **f) * h, (torch.arange(nx, **f) + 0.5) * h
        zf, zc = torch.arange(ny + 1, **f) * h, (torch.arange(ny, **f) + 0.5) * h
        sf, sc = 1 - (rf / R) ** 2, 1 - (rc / R) ** 2
        # stream function a r^2 (1 - r^2/R^2)^2 sin^2(pi z / L)
        u = -a * (rf * sf ** 2)[None] * (math.pi / L * torch.sin(2 * math.pi * zc / L))[:, None]
        v = a * (2 * sc ** 2 - 4 * (rc / R) ** 2 * sc)[None] * (torch.sin(math.pi * zf / L) ** 2)[:, None]
    else:
        X, Y, start, h = _polylines(case, rng)
        mat = dict(rho_l=RHO_L, rho_g=RHO_G, mu_l=MU_L, mu_g=MU_G, sigma=SIGMA)
        u, v = _vortex(nx, ny, h, case["speed"] * rng.uniform(0.8, 1.2))
    # a tenth for the coarse axisymmetric drops, whose spurious currents grow
    dt = (0.1 if case["axisym"] else 0.25) * min(
        0.5 * math.sqrt((mat["rho_l"] + mat["rho_g"]) * h ** 3 / (4 * math.pi * mat["sigma"])),
        0.25 * h * h * min(mat["rho_l"] / mat["mu_l"], mat["rho_g"] / mat["mu_g"]),
        0.5 * h / float(max(u.abs().max(), v.abs().max())))
    ctx = ib.Context(ib.Config(nx=nx, ny=ny, h=h, **opt), X, Y, start)
    ctx.set("u", u.contiguous())
    ctx.set("v", v.contiguous())
    return dict(case=case, ctx=ctx, dt=dt)


# --------------------------------------------------------------------- a pass
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "step":
        ctx = state["ctx"]
        ctx.ns_step(state["dt"], case["steps"], 1)
        X, Y = ctx.markers()
        return dict(u=ctx.get("u"), v=ctx.get("v"), p=ctx.get("p"), X=X, Y=Y)
    if kind == "solve":
        ctx, p = state["ctx"], torch.zeros_like(state["b"])
        ctx.mg_setup(state["bx"], state["by"])
        ctx.mg_solve(state["b"], p, case["precision"], 1e-10, 200)
        return dict(p=p)
    if kind == "noalloc":
        p = torch.zeros_like(state["b"])
        st, _, _ = ib.mg_solve_noalloc(state["bx"], state["by"], state["b"], p, state["h"],
                                       case["precision"], 1e-10, 200)
        if st != ib.IB_OK:
            raise RuntimeError(ib.noalloc_error())
        return dict(p=p)
    if kind == "markers":
        ctx = state["ctx"]
        kappa, nx, ny, ds = ctx.geometry()
        Fx, Fy = ctx.spread(0)
        U, V = ctx.interp(state["u"], state["v"])
        return dict(kappa=kappa, nx=nx, ny=ny, ds=ds, Fx=Fx, Fy=Fy, U=U, V=V)
    if kind == "infer":
        return dict(p=state["net"].infer(state["b"], state["rho"]))
    loss, grads = state["net"].grad(state["b"], state["rho"], state["p"])
    return dict(loss=np.float32(loss), grads=grads)


def work(case):
    """What a pass cannot do without: the state or inputs read once and the
    results written once; the arithmetic of one application of each operator
    (a solve: of the cycles that a contraction of 0.2 needs for 1e-10)."""
    kind = case["kind"]
    if kind in ("step", "solve", "noalloc"):
        n = case["nx"] * case["ny"]
        if kind == "step":
            s = case["steps"]
            return dict(bytes=s * n * 8 * 2 * 5, flops=s * n * (60 + 4 * 74))
        return dict(bytes=n * 8 * 4, flops=n * 14 * 74)
    if kind == "markers":
        m, f = case["drops"] * case["markers"], 2 * case["nx"] * case["ny"]
        return dict(bytes=8 * (8 * m + f + 2 * 16 * m), flops=m * 2 * 2 * 16 * 4)
    px = case["batch"] * case["n"] ** 2
    if kind == "infer":
        px //= 4 ** case["coarsen"]
    macs = 9 * (2 * 16 + 16 * 16 + 48 * 16 + 16 + (16 * 32 + 32 * 32 + 64 * 32) / 4 + 2 * 32 * 32 / 16)
    if kind == "infer":
        return dict(bytes=case["batch"] * case["n"] ** 2 * 24, flops=2 * px * macs)
    return dict(bytes=px * 24, flops=3 * 2 * px * macs)


# ------------------------------------------------------------- 64-bit answers
def exact(case, seed):
    """Plain 64-bit answers.  None for the time steps: a second implementation
    of the whole method (spline fits, polygon clipping, every solve to
    rounding, tens of steps) in plain tensors takes minutes at their sizes."""
    kind = case["kind"]
    if kind == "step":
        return None
    if kind in ("solve", "noalloc"):
        bx, by, b, _, h = _pressure_system(case, seed)
        return dict(p=_solve64(bx, by, b, h))
    if kind == "markers":
        return _markers64(case, seed)
    b, rho, p = _net_inputs(case, seed)
    return _infer64(case, seed, b, rho) if kind == "infer" else _grad64(seed, b, rho, p)


def _solve64(bx, by, b, h):
    """div(beta grad p) = b - mean b, mean p = 0: conjugate gradients with the
    diagonal as preconditioner, restarted on the true residual."""
    d = (bx[:, 1:] + bx[:, :-1] + by[1:] + by[:-1]) / h ** 2

    def neg_a(p):
        fx, fy = torch.zeros_like(bx), torch.zeros_like(by)
        fx[:, 1:-1] = bx[:, 1:-1] * (p[:, 1:] - p[:, :-1])
        fy[1:-1] = by[1:-1] * (p[1:] - p[:-1])
        return -(fx[:, 1:] - fx[:, :-1] + fy[1:] - fy[:-1]) / h ** 2

    rhs = -(b - b.mean())
    norm = float(rhs.norm())
    x = torch.zeros_like(b)
    for _ in range(3):
        r = rhs - neg_a(x)
        r -= r.mean()
        e = torch.zeros_like(b)
        z = r / d
        s, rz = z.clone(), (r * z).sum()
        for it in range(1, 20001):
            q = neg_a(s)
            a = rz / (s * q).sum()
            e += a * s
            r -= a * q
            z = r / d
            rz, old = (r * z).sum(), rz
            s = z + (rz / old) * s
            if it % 20 == 0:
                r -= r.mean()
                if float(r.norm()) < 1e-14 * norm:
                    break
        x += e
        x -= x.mean()
    return x


def _phi64(kernel, r):
    a = r.abs()
    if kernel == 0:
        return torch.where(a < 2, 0.25 * (1 + torch.cos(0.5 * math.pi * r)), torch.zeros_like(a))
    one = (3 - 2 * a + torch.sqrt((1 + 4 * a - 4 * a * a).clamp(min=0))) / 8
    two = (5 - 2 * a - torch.sqrt((-7 + 12 * a - 4 * a * a).clamp(min=0))) / 8
    return torch.where(a <= 1, one, torch.where(a < 2, two, torch.zeros_like(a)))


def _markers64(case, seed):
    X, Y, start, h = _polylines(case, np.random.default_rng(seed))
    nx, ny, k = case["nx"], case["ny"], case["kernel"]
    X, Y = (torch.from_numpy(a).cuda().view(len(start) - 1, -1) for a in (X, Y))
    ax, ay = X - X.roll(1, 1), Y - Y.roll(1, 1)
    bx, by = X.roll(-1, 1) - X, Y.roll(-1, 1) - Y
    la, lb = torch.hypot(ax, ay), torch.hypot(bx, by)
    tax, tay, tbx, tby = ax / la, ay / la, bx / lb, by / lb
    ds = 0.5 * (la + lb)
    kappa = torch.hypot(tbx - tax, tby - tay) / ds
    kappa = torch.where(tax * tby - tay * tbx >= 0, kappa, -kappa)
    nrx, nry = -tay - tby, tax + tbx
    ln = torch.hypot(nrx, nry)
    nrx, nry = nrx / ln, nry / ln
    kappa, nrx, nry, ds, X, Y = (t.reshape(-1) for t in (kappa, nrx, nry, ds, X, Y))
    u, v = _vortex(nx, ny, h, 1.0)
    out = dict(kappa=kappa, nx=nrx, ny=nry, ds=ds)
    for name, vel, field, c, ox, oy in (("Fx", "U", u, nrx, 0.0, 0.5), ("Fy", "V", v, nry, 0.5, 0.0)):
        F, W = torch.zeros_like(field), torch.zeros_like(X)
        sx, sy = X / h - ox, Y / h - oy
        i0, j0 = sx.floor().long() - 1, sy.floor().long() - 1
        for b in range(4):
            for a in range(4):
                i, j = i0 + a, j0 + b
                w = _phi64(k, i - sx) * _phi64(k, j - sy)
                F.index_put_((j, i), SIGMA * kappa * c * ds * w / h ** 2, accumulate=True)
                W += field[j, i] * w
        out[name], out[vel] = F, W
    return out


def _net64(params, x):
    """The network in 64 bits: params is the flat vector, x (B, 2, N, N)."""
    o, layers = 0, []
    for ci, co in _NET:
        w = params[o:o + co * 9 * ci].view(co, 3, 3, ci).permute(0, 3, 1, 2)
        o += co * 9 * ci
        layers.append((w, params[o:o + co]))
        o += co

    def conv(k, t, relu=True):
        w, b = layers[k]
        t = torch.nn.functional.pad(t, (1, 1, 1, 1))
        n, m = t.shape[2] - 2, t.shape[3] - 2
        y = sum(torch.einsum("bchw,oc->bohw", t[:, :, dy:dy + n, dx:dx + m], w[:, :, dy, dx])
                for dy in range(3) for dx in range(3)) + b[None, :, None, None]
        return y.clamp(min=0) if relu else y

    def pool(t):
        return torch.nn.functional.avg_pool2d(t, 2)

    def up(t):
        return t.repeat_interleave(2, 2).repeat_interleave(2, 3)

    s1 = conv(1, conv(0, x))
    s2 = conv(3, conv(2, pool(s1)))
    t3 = conv(5, conv(4, pool(s2)))
    t4 = conv(6, torch.cat([up(t3), s2], 1))
    return conv(8, conv(7, torch.cat([up(t4), s1], 1)), False)[:, 0]


def _features64(b, rho):
    b0 = b - b.mean((1, 2), keepdim=True)
    s = (b0 * b0).mean((1, 2), keepdim=True).sqrt()
    return torch.stack([b0 / s, rho.amin((1, 2), keepdim=True) / rho], 1), s


def _infer64(case, seed, b, rho):
    n, k = case["n"], case["coarsen"]
    for _ in range(k):
        b, rho = (torch.nn.functional.avg_pool2d(t[:, None], 2)[:, 0] for t in (b, rho))
    x, s = _features64(b, rho)
    with torch.no_grad():
        y = _net64(torch.from_numpy(_net_params(seed)).double().cuda(), x)
    p = s * (2.0 ** k / n) ** 2 * (y - y.mean((1, 2), keepdim=True))
    for _ in range(k):
        p = torch.nn.functional.interpolate(p[:, None], scale_factor=2, mode="bilinear",
                                            align_corners=False)[:, 0]
    return dict(p=p)


def _grad64(seed, b, rho, p):
    x, s = _features64(b, rho)
    t = p / (s / b.shape[-1] ** 2)
    w = torch.from_numpy(_net_params(seed)).double().cuda().requires_grad_(True)
    # one sample at a time: the 64-bit activations of a batch are many
    total, B = 0.0, b.shape[0]
    for k in range(B):
        y = _net64(w, x[k:k + 1])
        d = (y - y.mean()) - (t[k:k + 1] - t[k:k + 1].mean())
        loss = (d * d).mean() / B
        loss.backward()
        total += float(loss.detach())
    return dict(loss=np.float64(total), grads=w.grad)
