"""The finest level's sweeps taken two at a time (float, 2^23 cells and more) and the
restriction of pairs of cells (float, every axis coarsened by two): the V-cycles
of one refinement from p = 0 against the oracle's in double.  Tolerance: a sweep
rounds a value in about 8 float operations, 5e-7 of it; two or three cycles of at
most 8 levels and 8 sweeps make about 128 of them in a row, 6e-5 if they all added
up.  A neighbour missed along one edge of the 24-cell tiles in one sweep changes
the result by percents there, above 1e-3 in the norm.  The coarsest solve takes
few iterations, the same number in both.
"""
import numpy as np
import pytest
import torch

import cases
from oracle import fvm_oracle as O
from tests.gpu_util import need_gpu, rel_l2

pytestmark = pytest.mark.gpu

W, P_ = cases.WALL, cases.PERIODIC


@pytest.mark.parametrize("nx,ny,nz,bc,kw", [
    (272, 176, 176, (W, P_, W), {}),                              # an even number of swaps
    (320, 168, 160, (P_, W, W), {"mx_inner_cycles": 3}),          # an odd one
    # odd rows or planes, which are not coarsened: few levels
    (256, 256, 129, (P_, W, W), {"mg_levels": 3, "coarse_maxit": 4, "mg_pre": 1}),
    (260, 255, 130, (W, W, P_), {"mg_levels": 3, "coarse_maxit": 4, "mg_pre": 3, "mg_post": 1}),
    (272, 176, 176, (W, W, P_), {"mg_post": 0}),
    # sweeps one by one; the restriction's pairs at the edges of small levels
    (36, 20, 12, (W, P_, W), {}),
    (72, 44, 36, (P_, W, P_), {}),
])
def test_cycles_equal_oracle(nx, ny, nz, bc, kw):
    P = need_gpu()
    p = cases.Params(nx=nx, ny=ny, nz=nz, h=1.0 / nx, bc=bc, rho=(1.0, 4.0),
                     precision=cases.MIXED, mg_fixed_cycles=1, **{"coarse_maxit": 8, **kw})
    x, y, z = cases.cell_centres(p)
    alpha = (np.sin(9 * x + 4 * y) * np.cos(7 * z) > 0.2).astype(np.float32)
    alpha = np.ascontiguousarray(np.broadcast_to(alpha, p.shape))
    rhs = cases.uniform(31, p.shape, -1, 1) + np.cos(5 * x) * np.cos(3 * y + z)
    s = P.Solver(p)
    dp = torch.zeros(p.shape, dtype=torch.float64, device="cuda")
    info = s.fvm_poisson_solve(torch.tensor(alpha, device="cuda"), torch.tensor(rhs, device="cuda"), dp)
    s.close()
    assert info["status"] == 0
    ref, _, _ = O.poisson_solve(alpha.astype(np.float64), rhs, np.zeros(p.shape),
                                p.replace(precision=cases.F64, mg_fixed_cycles=p.mx_inner_cycles))
    assert rel_l2(dp.cpu().numpy(), np.asarray(ref)) <= 6e-5
