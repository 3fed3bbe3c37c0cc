"""Which grids the no-allocation solve takes: those whose hierarchy fits its
scratch array, up to the last few hundred bytes, and none beyond."""
import ctypes as C

import numpy as np
import pytest

import workloads as W

# At the array's edge, from the layout's sizes: those that fit leave 3 to 13 KB of
# it, the others need 3 to 6 KB more than there is.
FIT = [(10, 402), (402, 10), (670, 6), (30, 134), (134, 30), (152, 320), (320, 152), (760, 64),
       (2008, 2), (2024, 24)]
BEYOND = [(76, 200), (200, 76), (100, 152), (380, 40), (1216, 40), (12, 85), (255, 4)]


# Without a device the call ends at the first step that needs one (IB_ECUDA),
# after the sizes have been looked at (IB_EINVAL).
@pytest.mark.parametrize("nx,ny", FIT + BEYOND)
def test_sizes_without_a_device(nx, ny):
    import torch

    import paper_1807_10504_gb300 as ib
    if torch.cuda.is_available():
        pytest.skip("GPU present")
    ib.build()
    some = C.c_void_p(256)  # never reached
    st = ib.lib().mg_solve_noalloc(nx, ny, 0.01, some, some, some, some, 0, 1e-8, 10, 2, 2, None, None, None)
    assert st == (ib.IB_ECUDA if (nx, ny) in FIT else ib.IB_EINVAL), ib.noalloc_error()


# The residual of the result, by the residual operator.
@pytest.mark.gpu
@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("nx,ny", [(10, 402), (670, 6), (152, 320), (2024, 24)])
def test_solves_at_the_edge(O, nx, ny, precision):
    import torch as T

    import paper_1807_10504_gb300 as ib
    if not T.cuda.is_available():
        pytest.skip("needs a GPU")
    h = 1.0 / max(nx, ny)
    _, _, bx, by = O.coeffs(W.random_H(nx, ny, 5), 1e-1, 1.0, 1e-4, 1e-2)
    d = lambda a: T.from_numpy(np.ascontiguousarray(a)).cuda()
    bx, by, b = d(bx), d(by), W.random_cells(nx, ny, 6)
    p = T.zeros((ny, nx), dtype=T.float64, device="cuda")
    st, _, rr = ib.mg_solve_noalloc(bx, by, d(b), p, h, precision, 1e-10, 400)
    assert st == ib.IB_OK and rr <= 1e-10, ib.noalloc_error()
    r = ib.ib_op_residual(bx, by, d(b - b.mean()), p, h)
    assert float(r.norm()) <= 1.01e-10 * np.linalg.norm(b - b.mean())
