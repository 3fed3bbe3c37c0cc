"""Infinities, NaN and zeros at the grid kernels: a value that is not finite
reaches every result that depends on it, and a solve on it says so."""
import numpy as np
import pytest

import workloads as W

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


def context(ib, n):
    X, Y = W.circle(0.5, 0.5, 0.2, 16)
    return ib.Context(ib.Config(nx=n, ny=n, h=1.0 / n), X, Y, [0, 16])


# Both forms of the coefficients' kernel (one row a warp, eight from 2^18 cells
# up), the bad cell inside, next to a row boundary and at a wall, off the
# interface (where rows repeat) and on it.
@pytest.mark.parametrize("bad", [np.nan, -np.nan, np.inf])
@pytest.mark.parametrize("nx,ny", [(64, 48), (523, 517)])
def test_coefficients_of_a_bad_cell(T, ib, O, nx, ny, bad):
    H = W.random_H(nx, ny, 3)
    cells = [(0, 0), (ny // 2, nx // 2), (ny // 2 + 5, 7), (ny - 1, nx - 1), (15, nx - 2), (16, 30)]
    for j, i in cells:
        H[j, i] = bad
    ref = O.coeffs(H, 1e-3, 1.0, 1e-4, 1e-2)
    got = [a.cpu().numpy() for a in ib.ib_op_coeffs(T.from_numpy(H).cuda(), 1e-3, 1.0, 1e-4, 1e-2)]
    rho, _, bx, by = got
    hit = np.zeros((ny + 2, nx + 2), bool)
    hit[1:-1, 1:-1] = ~np.isfinite(H)
    fx, fy = hit[1:-1, :-1] | hit[1:-1, 1:], hit[:-1, 1:-1] | hit[1:, 1:-1]
    fx[:, [0, -1]] = False  # the walls carry no coefficient
    fy[[0, -1], :] = False
    assert np.array_equal(~np.isfinite(rho), ~np.isfinite(H))
    assert np.array_equal(~np.isfinite(bx), fx) and np.array_equal(~np.isfinite(by), fy)
    for a, b, f in ((bx, ref[2], fx), (by, ref[3], fy)):
        assert np.abs(a[~f] - b[~f]).max() <= 1e-15 * np.abs(b[~f]).max()


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("n", [64, 512])
def test_solve_on_coefficients_of_a_bad_cell(T, ib, n, precision):
    H = W.random_H(n, n, 3)
    H[n // 2 + 3, n // 4] = np.nan
    _, _, bx, by = ib.ib_op_coeffs(T.from_numpy(H).cuda(), 1e-1, 1.0, 1e-4, 1e-2)
    ctx = context(ib, n)
    ctx.mg_setup(bx, by)
    b = W.random_cells(n, n, 4)
    b[n // 2 + 3, n // 4] = 0.0
    p = T.zeros((n, n), dtype=T.float64, device="cuda")
    st, _, _ = ctx.mg_solve(T.from_numpy(b - b.mean()).cuda(), p, precision, 1e-8, 50, check=False)
    assert st == ib.IB_ENAN


# Without any coefficient there is no solution: the coarsest level's inverse does
# not exist, and the solve says so (one block's inverse at 64^2, blocks of 16 at
# 104^2, whose coarsest level has 169 cells).
@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("n", [64, 104])
def test_solve_without_coefficients(T, ib, n, precision):
    ctx = context(ib, n)
    ctx.mg_setup(T.zeros((n, n + 1), dtype=T.float64, device="cuda"),
                 T.zeros((n + 1, n), dtype=T.float64, device="cuda"))
    b = W.random_cells(n, n, 4)
    p = T.zeros((n, n), dtype=T.float64, device="cuda")
    st, _, _ = ctx.mg_solve(T.from_numpy(b - b.mean()).cuda(), p, precision, 1e-8, 20, check=False)
    assert st == ib.IB_ENAN


# Two massless cells next to each other: their face has no finite acceleration
# (axisymmetric predictor: as by the division).
def test_predictor_of_massless_cells(T, ib):
    nx, ny, h, dt = 40, 24, 1.0 / 32, 1e-3
    u, v = W.random_faces(nx, ny, 5)
    rho = np.full((ny, nx), 0.7)
    rho[9, 12:14] = 0.0
    d = lambda a: T.from_numpy(np.ascontiguousarray(a)).cuda()
    us, vs, _, _ = ib.ib_op_predictor_axi(d(rho), d(np.full_like(rho, 0.1)), d(u), d(v), h, dt)
    bad = ~np.isfinite(us.cpu().numpy())
    assert bad[9, 13] and bad.sum() == 1 and np.isfinite(vs.cpu().numpy()).all()


# A coefficient that is not finite, at a face without force: b of the cells on
# either side of it.
@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("axisym", [0, 1])
def test_rhs_of_a_bad_coefficient(T, ib, bad, axisym):
    nx, ny, h, dt = 70, 33, 1.0 / 64, 1e-3
    us, vs = W.random_faces(nx, ny, 5)
    bx, by = (np.abs(a) + 0.5 for a in W.random_faces(nx, ny, 6))
    bx[7, 30] = by[20, 41] = bad
    d = lambda a: T.from_numpy(np.ascontiguousarray(a)).cuda()
    rhs = ib.ib_op_rhs_axi if axisym else ib.ib_op_rhs
    zx, zy = np.zeros_like(us), np.zeros_like(vs)
    b = rhs(d(us), d(vs), d(zx), d(zy), d(bx), d(by), h, dt).cpu().numpy()
    hit = np.zeros((ny, nx), bool)
    hit[7, 29:31] = hit[19:21, 41] = True
    assert np.array_equal(np.isnan(b), hit)
