"""GPU parity of the kernels' separate paths at the sizes where they change or
end: strips and tiles that do not divide the grid, chains and rings of a few
spans, coarsest levels on either side of the one-block inverse, lists that
overflow, drops larger than a register-held share."""
import numpy as np
import pytest

import workloads as W
from oracle import cnn as OC
from test_gpu_cnn import batch, bf16, dict_of, flat_of, oracle_inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    return torch


@pytest.fixture(scope="module")
def ib():
    import paper_1807_10504_gb300 as ib
    ib.lib()
    return ib


# One column and one row short of, at and past a strip of 30 columns and a
# march of 16 rows; the smallest grid.  About fifty operations a face on
# operands whose magnitudes sum to at most a few hundred times the result's
# largest: 1e-12 of it.
@pytest.mark.parametrize("axisym", [0, 1])
@pytest.mark.parametrize("nx,ny", [(2, 2), (29, 17), (30, 16), (31, 33), (61, 1100)])
def test_predictor_strips(T, ib, O, nx, ny, axisym):
    h, dt = 1.0 / 32, 2e-4
    rho, mu, bx, by = O.coeffs(W.random_H(nx, ny, 3), 1e-3, 1.0, 1e-4, 1e-2)
    u, v = W.random_faces(nx, ny, 4)
    aup, avp = W.random_faces(nx, ny, 5)
    d = lambda a: T.from_numpy(np.ascontiguousarray(a)).cuda()
    if axisym:
        got = ib.ib_op_predictor_axi(d(rho), d(mu), d(u), d(v), h, dt, d(aup), d(avp), gy=-9.81,
                                     S=0.37, wb=0.21)
        ref = O.predictor_axi(rho, mu, u, v, h, dt, aup, avp, (0.0, -9.81 + 0.37), 0.21)
    else:
        got = ib.ib_op_predictor(d(rho), d(mu), d(u), d(v), h, dt, d(aup), d(avp), g=(0.1, -9.8))
        ref = O.predictor(rho, mu, u, v, h, dt, aup, avp, g=(0.1, -9.8))
    for a, b in zip(got, ref):
        assert np.abs(a.cpu().numpy() - b).max() <= 1e-12 * max(np.abs(b).max(), 1.0)


# Rings of 4 .. 20 spans (border of 3, 4 and 5 rows, chains of none to five
# blocks, last rows shorter and longer than the others), and a marker count
# that takes four lanes a marker.  The spline's matrix has a condition number
# below 1e3, so rounding moves a marker by less than 1e-12.
@pytest.mark.parametrize("case", ["rings", "four_lanes", "axisym_small", "axisym"])
def test_relocation_sizes(T, ib, O, case):
    axisym = case.startswith("axisym")
    if case == "rings":
        n, h = 96, 1.0 / 96
        mk = W.join([W.circle((12 + 18 * (k % 5)) * h, (12 + 24 * (k // 5)) * h, g * 1.5 * h / (2 * np.pi),
                              24 + k, theta0=0.1 * k)
                     for k, g in enumerate((4, 5, 6, 7, 8, 9, 10, 11, 12, 13, 16, 20))])
        shape = (n, n)
    elif case == "four_lanes":
        n, h = 256, 1.0 / 256
        mk = W.multidrop(n, ndrops=20, rmin=0.03, rmax=0.06, n_per_drop=256, seed=5, gap_cells=8)
        assert 4096 <= mk.X.size < 8192
        shape = (n, n)
    elif case == "axisym_small":
        h, shape = 1.0 / 32, (32, 64)
        mk = W.axi_elliptic_drop(1.0, 0.06, 1.2, 16)
    else:
        h, shape = 1.0 / 64, (64, 128)
        mk = W.axi_elliptic_drop(1.0, 0.4, 1.1, 300)
    ctx = ib.Context(ib.Config(nx=shape[0], ny=shape[1], h=h, axisym=int(axisym)), mk.X, mk.Y, mk.drop_start)
    ctx.relocate()
    X, Y = (a.cpu().numpy() for a in ctx.markers())
    oX, oY = O.bspline_relocate(mk.X, mk.Y, mk.drop_start, h)
    if axisym:
        oX, oY = O.symmetrise(oX, oY, mk.drop_start)
    assert np.abs(X - oX).max() <= 1e-12 and np.abs(Y - oY).max() <= 1e-12


# Coarsest levels of 65, 80, 143 and 1023 cells: past the one-block inverse,
# whole blocks of 16, a remainder, the largest; rows and columns that do not
# divide the residual norm's strips of 31 x 4.  The residual is reduced by
# 1e12 (1e11 in mixed precision) on systems whose solution is at most about
# 1e2 times the scaled right-hand side.
@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("nx,ny", [(26, 10), (32, 10), (26, 22), (62, 66), (124, 132)])
def test_coarsest_sizes(T, ib, O, nx, ny, precision):
    n = min(nx, ny)
    h = 1.0 / n
    X, Y = W.circle(0.5 * nx / n, 0.5 * ny / n, min(0.2, 0.45 - 3.0 / n), 16)
    ctx = ib.Context(ib.Config(nx=nx, ny=ny, h=h), X, Y, [0, 16])
    rho, mu, bx, by = O.coeffs(W.random_H(nx, ny, 3), 1e-3, 1.0, 1e-4, 1e-2)
    b = W.random_cells(nx, ny, 4)
    d = lambda a: T.from_numpy(np.ascontiguousarray(a)).cuda()
    ctx.mg_setup(d(bx), d(by))
    p = T.zeros((ny, nx), dtype=T.float64, device="cuda")
    tol = 1e-12 if precision == 0 else 1e-11
    st, cyc, rr = ctx.mg_solve(d(b), p, precision, tol, 200)
    o = O.mg_solve(bx, by, b, h, precision=0, tol=1e-12, max_cycles=200)
    assert st == 0 and rr <= tol
    assert np.abs(p.cpu().numpy() - o.p).max() <= 100 * tol * np.abs(o.p).max()


# The coefficient tables' sweeps, two a launch: one launch, whole launches, an
# odd sweep left, and an odd number of launches (the buffers then end swapped).
# As the steps of twenty sweeps: p within 1e-10 of its largest value, u and v
# within 1e-10 of the inertial-capillary velocity.
@pytest.mark.parametrize("axisym", [0, 1])
@pytest.mark.parametrize("sweeps", [1, 2, 3, 6])
def test_cn_sweep_counts(T, ib, O, sweeps, axisym):
    if axisym:
        nx, ny, h = 24, 72, 1 / 24
        mk = W.axi_elliptic_drop(1.5, 0.25, 1.1, 64)
        kw = dict(axisym=1, frame=1, gy=-1.0)
    else:
        nx, ny, h = 40, 56, 1 / 40
        mk = W.elliptic_drop(0.5, 0.7, 0.22, 1.15, 96)
        kw = {}
    kw.update(spread=1, relocate_every=0, viscous=1, cn_sweeps=sweeps, tol=1e-11)
    ctx = ib.Context(ib.Config(nx=nx, ny=ny, h=h, **kw), mk.X, mk.Y, mk.drop_start)
    ocfg = O.Config(nx=nx, ny=ny, h=h, **kw)
    st = O.init_state(ocfg, mk.X, mk.Y, mk.drop_start)
    dt = W.capillary_dt(h, 1.0, 1e-3, 1.0, 1e-2, 1e-4)
    for _ in range(2):
        ctx.ns_step(dt, 1, 1)
        O.ns_step(ocfg, st, dt)
    assert np.abs(ctx.get("p").cpu().numpy() - st.p).max() <= 1e-10 * np.abs(st.p).max()
    for name, ref in (("u", st.u), ("v", st.v)):
        assert np.abs(ctx.get(name).cpu().numpy() - ref).max() <= 1e-10 * 2.0, name


# The coefficients formed several rows a thread, from 90,000 cells up: a last strip
# of one row, and rows that repeat above and below those of the drop.  Pressure
# within 100 of the solver's tolerances, u and v within 1e-10 of the
# inertial-capillary velocity.
@pytest.mark.parametrize("axisym", [0, 1])
def test_cn_rows_in_strips(T, ib, O, axisym):
    if axisym:
        nx, ny, h = 224, 672, 1 / 224
        mk = W.axi_elliptic_drop(1.5, 0.25, 1.1, 512)
        kw = dict(axisym=1, gy=-1.0)
    else:
        nx, ny, h = 320, 416, 1 / 320
        mk = W.elliptic_drop(0.5, 0.65, 0.22, 1.15, 512)
        kw = {}
    kw.update(spread=1, relocate_every=0, viscous=1, cn_sweeps=2, tol=1e-12)
    ctx = ib.Context(ib.Config(nx=nx, ny=ny, h=h, **kw), mk.X, mk.Y, mk.drop_start)
    ocfg = O.Config(nx=nx, ny=ny, h=h, **kw)
    st = O.init_state(ocfg, mk.X, mk.Y, mk.drop_start)
    dt = W.capillary_dt(h, 1.0, 1e-3, 1.0, 1e-2, 1e-4)
    for _ in range(2):
        ctx.ns_step(dt, 1, 1)
        O.ns_step(ocfg, st, dt)
    assert np.abs(ctx.get("p").cpu().numpy() - st.p).max() <= 1e-10 * np.abs(st.p).max()
    for name, ref in (("u", st.u), ("v", st.v)):
        assert np.abs(ctx.get(name).cpu().numpy() - ref).max() <= 1e-10 * 2.0, name


# A drop of more markers than the block's threads hold in registers: the same
# bisection decisions as the oracle's, so eps to 1e-13 h.
def test_measure_correction_large_drop(T, ib, O):
    n, h = 256, 1.0 / 256
    X, Y = W.circle(0.5, 0.5, 0.3, 2500)
    start = np.array([0, 2500], np.int32)
    ctx = ib.Context(ib.Config(nx=n, ny=n, h=h), X, Y, start)
    A0 = O.drop_measures(X, Y, start, 0)
    k, nxm, nym, ds = O.curvature(X, Y, start)
    Xs, Ys = X + 0.31 * h * nxm, Y + 0.31 * h * nym
    ctx.set_markers_host(Xs, Ys)
    eps = ctx.mass_correct()
    Xo, Yo, eo = O.mass_correct(Xs, Ys, start, A0, h, 0)
    Xg, Yg = (a.cpu().numpy() for a in ctx.markers())
    assert np.abs(eps - eo).max() <= 1e-13 * h
    assert np.abs(Xg - Xo).max() <= 1e-14 and np.abs(Yg - Yo).max() <= 1e-14


def tilted_box(cx, cy, a, tilt, m):
    """A square of half-edge a, turned by tilt, m markers an edge."""
    t = np.linspace(-1.0, 1.0, m, endpoint=False)
    o = np.ones_like(t)
    x = a * np.concatenate([t, o, -t, -o])
    y = a * np.concatenate([-o, t, o, -t])
    c, s = np.cos(tilt), np.sin(tilt)
    return cx + c * x - s * y, cy + s * x + c * y


# Squares turned by less than 0.001 rad: every segment takes the edge
# integrals.  One small square (a few listed pairs) and four large ones, whose
# pairs overflow the list (the rest is integrated in place).  A cell sums a
# handful of integrals of coordinates up to n cells, each with a few roundings.
@pytest.mark.parametrize("n,ndrops", [(32, 1), (320, 4)])
def test_heaviside_along_the_axes(T, ib, O, n, ndrops):
    h = 1.0 / n
    if ndrops == 1:
        mk = W.join([tilted_box(0.5, 0.5, 0.2, 5e-4, 10)])
    else:
        mk = W.join([tilted_box(0.27 + 0.46 * (k % 2), 0.27 + 0.46 * (k // 2), 0.19, 4e-4 + 1e-4 * k, 150)
                     for k in range(4)])
    ctx = ib.Context(ib.Config(nx=n, ny=n, h=h), mk.X, mk.Y, mk.drop_start)
    H = ctx.heaviside().cpu().numpy()
    oH = O.heaviside(mk.X, mk.Y, mk.drop_start, n, n, h)
    assert np.abs(H - oH).max() <= 1e-13 + 8 * n * 2.0 ** -53


# Images that are not whole tiles at any of the three resolutions, down to one
# pixel at the coarsest; the weight gradients' streams give the same bits on
# every call and on another stream.  Bounds as for whole tiles: the loss within
# 1e-2, gradients within 5e-3 of the layer's largest.
@pytest.mark.parametrize("B,N", [(3, 20), (1, 44), (2, 4)])
def test_gradient_ragged_tiles(T, B, N):
    import paper_1807_10504_gb300 as ib
    P = OC.init_params(seed=4)
    Pq = {k: (bf16(v) if k.endswith(".w") else v) for k, v in P.items()}
    net = ib.Net(seed=0)
    net.set_params(flat_of(P))
    rhs, rho, p = batch(B, N, 8)
    d = lambda a: T.from_numpy(np.ascontiguousarray(a)).cuda()
    c = net.fit_scale(d(rhs), d(p))
    loss, g = net.grad(d(rhs), d(rho), d(p))
    x, s, t = oracle_inputs(rhs, rho, p, c)
    y, cache = OC.forward(Pq, x, keep=True, bf16=True)
    L, gy = OC.loss(y, t)
    G, _ = OC.backward(Pq, cache, gy, bf16=True)
    assert abs(loss - L) <= 1e-2 * L, (loss, L)
    Gg = dict_of(g, P)
    for n, _, _, _ in OC.LAYERS:
        for k in (".w", ".b"):
            if n + k != "c6.b":
                a, ref = Gg[n + k].ravel(), G[n + k].ravel()
                assert np.abs(a - ref).max() <= 5e-3 * np.abs(ref).max(), n + k
    side = T.cuda.Stream()
    side.wait_stream(T.cuda.current_stream())
    with T.cuda.stream(side):
        loss2, g2 = net.grad(d(rhs), d(rho), d(p))
    assert loss2 == loss and np.array_equal(g, g2)


def layered_H(nx, ny, seed):
    """Rows that repeat the row below, rows that differ in one column only and
    a band of distinct rows, at odd places."""
    rng = np.random.default_rng(seed)
    H = np.zeros((ny, nx))
    H[ny // 3:ny // 3 + 37] = rng.uniform(0.0, 1.0, (37, nx))
    H[ny // 3 + 37:] = 1.0
    H[5:11] = rng.uniform(0.0, 1.0, nx)
    H[11, nx - 1] = H[14, 0] = H[17, nx // 2] = 0.5
    return H


# The coefficients' kernel that passes on a row equal to the one below, from
# 2^18 cells up, with a ragged last strip and last rows: the oracle's formulas
# to a rounding or two.
def test_coefficients_of_repeated_rows(T, ib, O):
    nx, ny = 523, 517
    H = layered_H(nx, ny, 6)
    got = ib.ib_op_coeffs(T.from_numpy(H).cuda(), 1e-3, 1.0, 1e-4, 1e-2)
    for a, b in zip(got, O.coeffs(H, 1e-3, 1.0, 1e-4, 1e-2)):
        assert np.abs(a.cpu().numpy() - b).max() <= 1e-15 * np.abs(b).max()


# The hierarchy's kernel does the same from 2^20 cells up: the solve on such
# coefficients reaches the tolerance by the oracle's residual.
@pytest.mark.parametrize("precision", [0, 2])
def test_solve_on_repeated_rows(T, ib, O, precision):
    nx, ny = 1088, 1024
    h = 1.0 / ny
    H = layered_H(nx, ny, 7)
    rho, mu, bx, by = ib.ib_op_coeffs(T.from_numpy(H).cuda(), 1e-1, 1.0, 1e-4, 1e-2)
    X, Y = W.circle(0.5, 0.5, 0.1, 32)
    ctx = ib.Context(ib.Config(nx=nx, ny=ny, h=h), X, Y, [0, 32])
    ctx.mg_setup(bx, by)
    b = W.random_cells(nx, ny, 8)
    b -= b.mean()
    p = T.zeros((ny, nx), dtype=T.float64, device="cuda")
    st, cyc, rr = ctx.mg_solve(T.from_numpy(b).cuda(), p, precision, 1e-10, 200)
    r = O.residual(bx.cpu().numpy(), by.cpu().numpy(), b, p.cpu().numpy(), h)
    assert st == 0 and np.linalg.norm(r) <= 1.001e-10 * np.linalg.norm(b)


# One graph for the whole step (from the third step of a shape on), separate
# graphs before that, and direct launches run the same kernels on the same
# data: the same bits, also after a step of another size in between.
@pytest.mark.parametrize("kw", [dict(precision=2, spread=1, relocate_every=2),
                                dict(precision=0, spread=0, relocate_every=0),
                                dict(precision=1, viscous=1, mass_every=2),
                                dict(precision=2, axisym=1, frame=1, gy=-1.0, relocate_every=3)])
def test_step_graphs_match_direct_launches(T, ib, kw):
    if kw.get("axisym"):
        nx, ny, h = 32, 96, 1 / 32
        mk = W.axi_elliptic_drop(1.5, 0.25, 1.1, 96)
    else:
        nx, ny, h = 64, 48, 1 / 64
        mk = W.elliptic_drop(0.5, 0.375, 0.2, 1.15, 128)
    dt = W.capillary_dt(h, 1.0, 1e-3, 1.0, 1e-2, 1e-4)
    got = []
    for graphs in (True, False):
        ctx = ib.Context(ib.Config(nx=nx, ny=ny, h=h, tol=1e-10, **kw), mk.X, mk.Y, mk.drop_start)
        ctx.use_graphs(graphs)
        for step in [dt] * 5 + [0.5 * dt] + [dt] * 2:
            ctx.ns_step(step, 1, 1)
        got.append([ctx.get(f).cpu().numpy() for f in ("u", "v", "p")] +
                   [a.cpu().numpy() for a in ctx.markers()])
        ctx.close()
    for a, b in zip(*got):
        assert np.array_equal(a, b)


# The correction takes one row a block up to the most rows of a launch, and
# further ones in turn above that.  Two fused multiply-adds a face: within a few
# ulps of the operands' sizes.
@pytest.mark.parametrize("ny", [65533, 65534, 65535, 131075])
def test_correct_tall_grids(T, ib, O, ny):
    nx, h, dt = 3, 0.01, 1e-3
    rng = np.random.default_rng(ny)
    f = lambda *n: rng.standard_normal(n)
    us, vs, p = f(ny, nx + 1), f(ny + 1, nx), f(ny, nx)
    Fx, Fy = f(ny, nx + 1), f(ny + 1, nx)
    bx, by = np.abs(f(ny, nx + 1)), np.abs(f(ny + 1, nx))
    d = lambda a: T.from_numpy(a).cuda()
    gu, gv = ib.ib_op_correct(d(us), d(vs), d(p), d(Fx), d(Fy), d(bx), d(by), h, dt)
    ou, ov = O.correct(us, vs, p, Fx, Fy, bx, by, h, dt)
    for g, o in ((gu, ou), (gv, ov)):
        assert np.abs(g.cpu().numpy() - o).max() <= 1e-14 * max(np.abs(o).max(), 1.0)


# Four squares whose pairs overflow the list of edge-integral pairs, and each of
# them alone, which fits it: which pairs are listed must not show, so that every
# square's cells carry the same bits in both, and in every run.
def test_heaviside_does_not_depend_on_the_list(T, ib):
    n, h = 320, 1.0 / 320
    boxes = [tilted_box(0.27 + 0.46 * (k % 2), 0.27 + 0.46 * (k // 2), 0.19, 4e-4 + 1e-4 * k, 150)
             for k in range(4)]

    def heaviside(drops):
        mk = W.join(drops)
        ctx = ib.Context(ib.Config(nx=n, ny=n, h=h), mk.X, mk.Y, mk.drop_start)
        out = [ctx.heaviside().cpu().numpy() for _ in range(5)]
        ctx.close()
        return out

    runs = heaviside(boxes)
    assert all(np.array_equal(H, runs[0]) for H in runs[1:])
    for k, box in enumerate(boxes):
        part = np.s_[160 * (k // 2):160 * (k // 2 + 1), 160 * (k % 2):160 * (k % 2 + 1)]
        assert np.array_equal(heaviside([box])[0][part], runs[0][part])


# Four time steps, each of three shapes (relocation every second step, the
# measure correction every fourth), in turn: their graphs fit the slots, so that
# no step records one once all have been seen, and they take the time of steps of
# one size (253 us a step; 1.66 times that where they did not fit).
def test_step_graphs_of_several_time_steps(T, ib):
    import time

    nx, ny, h = 64, 48, 1 / 64
    mk = W.elliptic_drop(0.5, 0.375, 0.2, 1.15, 128)
    dt = 0.01 * W.capillary_dt(h, 1.0, 1e-3, 1.0, 1e-2, 1e-4)

    def cycle_time(sizes):
        ctx = ib.Context(ib.Config(nx=nx, ny=ny, h=h, precision=2, relocate_every=2, mass_every=4),
                         mk.X, mk.Y, mk.drop_start)
        times = []
        for _ in range(6):
            t = time.perf_counter()
            for k in range(32):
                ctx.ns_step(dt * sizes[k // 8], 1, 1)
            times.append(time.perf_counter() - t)
        ctx.close()
        return min(times[2:])

    same = cycle_time([1.0] * 4)
    assert cycle_time([1.0, 0.9, 0.8, 0.7]) <= 1.3 * same


# The lower cycle is timed also where it is the coarsest level alone (25 x 25,
# under 50 x 50, which is launched for itself).
def test_timing_of_a_coarsest_level_alone(T, ib):
    n = 200
    X, Y = W.circle(0.5, 0.5, 0.2, 16)
    ctx = ib.Context(ib.Config(nx=n, ny=n, h=1.0 / n), X, Y, [0, 16])
    one = T.ones((n, n + 1), dtype=T.float64, device="cuda")
    ctx.mg_setup(one, T.ones((n + 1, n), dtype=T.float64, device="cuda"))
    p = T.zeros((n, n), dtype=T.float64, device="cuda")
    ctx.mg_solve(T.from_numpy(W.random_cells(n, n, 4)).cuda(), p, 1, 1e-8, 100)
    us, units = ctx.bench_kernel(5)
    assert us > 0.0 and units == 25 * 25


# Markers on grid lines and cell centres, and one unit in the last place to either
# side, where a factor of the delta functions vanishes or the stencil moves on:
# sums of sixteen products of factors below 1/2 and values below 1.
@pytest.mark.parametrize("kernel", [0, 1])
def test_delta_factors_on_grid_lines(T, ib, O, kernel):
    n, h = 32, 1.0 / 32
    X, Y = W.circle(0.5, 0.5, 0.3, 48)
    X, Y = np.round(X * 2 * n) / (2 * n), np.round(Y * 2 * n) / (2 * n)
    X[1::3], Y[2::3] = np.nextafter(X[1::3], 0.0), np.nextafter(Y[2::3], 1.0)
    X[2::4], Y[3::4] = np.nextafter(X[2::4], 1.0), np.nextafter(Y[3::4], 0.0)
    start = np.array([0, 48], np.int32)
    ctx = ib.Context(ib.Config(nx=n, ny=n, h=h, kernel=kernel), X, Y, start)
    u, v = W.random_faces(n, n, 9)
    d = lambda a: T.from_numpy(np.ascontiguousarray(a)).cuda()
    U, V = (a.cpu().numpy() for a in ctx.interp(d(u), d(v)))
    oU, oV = O.interp(u, v, X, Y, h, kernel=kernel)
    assert np.abs(U - oU).max() <= 1e-14 and np.abs(V - oV).max() <= 1e-14


# Marches of as many rows as an uneven share of blocks makes them take: 17 rows
# (960 x 640, the last of 11), 11 (768^2, the last of 9) and 14 (700 x 701, the
# last of one); and columns left over by whole strips, marched by 8 lanes (up to
# 6), 16 (up to 14) or 32, with ranges beyond the grid in the last warp.  By the
# bound of the other strips.
@pytest.mark.parametrize("axisym", [0, 1])
@pytest.mark.parametrize("nx,ny", [(960, 640), (768, 768), (700, 701), (6, 9), (31, 7), (36, 50), (37, 51),
                                   (44, 33), (45, 33), (64, 1001), (102, 770)])
def test_predictor_rows(T, ib, O, nx, ny, axisym):
    test_predictor_strips(T, ib, O, nx, ny, axisym)


# Four rows a warp between 2^18 and 2^20 cells and eight above, with last strips of
# one row and of all but one: as above.
@pytest.mark.parametrize("nx,ny", [(93, 2821), (520, 519), (1023, 1025), (1030, 1023)])
def test_coefficients_rows_a_warp(T, ib, O, nx, ny):
    H = layered_H(nx, ny, 6)
    got = ib.ib_op_coeffs(T.from_numpy(H).cuda(), 1e-3, 1.0, 1e-4, 1e-2)
    for a, b in zip(got, O.coeffs(H, 1e-3, 1.0, 1e-4, 1e-2)):
        assert np.abs(a.cpu().numpy() - b).max() <= 1e-15 * np.abs(b).max()


# Cycles of other sweep counts, whose single-block tail takes more levels: 32^2 and
# (FP32) 64^2, and a coarsest level of 33 x 17 alone.  The solution to a hundred
# times the tolerance, as on the coarsest sizes.
@pytest.mark.parametrize("nu", [(1, 1), (2, 1), (3, 3), (4, 2)])
@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("nx,ny", [(64, 64), (128, 128), (132, 68)])
def test_tails_of_other_sweep_counts(T, ib, O, nx, ny, precision, nu):
    h = 1.0 / ny
    X, Y = W.circle(0.5 * nx / ny, 0.5, 0.2, 16)
    ctx = ib.Context(ib.Config(nx=nx, ny=ny, h=h, nu1=nu[0], nu2=nu[1]), X, Y, [0, 16])
    rho, mu, bx, by = O.coeffs(W.random_H(nx, ny, 3), 1e-3, 1.0, 1e-4, 1e-2)
    b = W.random_cells(nx, ny, 4)
    d = lambda a: T.from_numpy(np.ascontiguousarray(a)).cuda()
    ctx.mg_setup(d(bx), d(by))
    p = T.zeros((ny, nx), dtype=T.float64, device="cuda")
    tol = 1e-12 if precision == 0 else 1e-11
    st, cyc, rr = ctx.mg_solve(d(b), p, precision, tol, 300)
    o = O.mg_solve(bx, by, b, h, precision=0, tol=1e-12, max_cycles=300)
    assert st == 0 and rr <= tol
    assert np.abs(p.cpu().numpy() - o.p).max() <= 100 * tol * np.abs(o.p).max()
