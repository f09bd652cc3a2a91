"""The mixed solve on grids whose residual is updated with the float correction
between refinements (2^19 cells and more): the residual it reports is that of
the pressure it returns, formed here in double from the oracle's operator, and
the device-side loop gives the same bits as the host loop."""
import numpy as np
import pytest
import torch

import cases
from oracle import fvm_oracle as O
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu

W, P_ = cases.WALL, cases.PERIODIC


def _solve(P, p, alpha, rhs, host_loop=False):
    s = P.Solver(p)
    if host_loop:
        s.fvm_profile(True)
    dp = torch.zeros(p.shape, dtype=torch.float64, device="cuda")
    info = s.fvm_poisson_solve(torch.as_tensor(alpha, device="cuda"), torch.tensor(rhs, device="cuda"), dp)
    s.close()
    return dp.cpu(), info


@pytest.mark.parametrize("nx,ny,nz,bc,kw", [
    (128, 64, 64, (W, W, W), {}),                       # the smallest such grid
    (100, 76, 72, (W, P_, W), {}),                      # tiles and plane runs with remainders
    (1024, 512, 1, (P_, W, P_), {}),                    # one plane
    (128, 64, 64, (P_, P_, W), {"mg_pre": 1}),          # no second sweep to read the first one's values
    (128, 64, 64, (W, W, P_), {"mg_pre": 0}),           # no sweep before the correction
    (128, 64, 64, (W, W, W), {"mg_post": 0}),           # the correction added in a pass of its own
    (128, 64, 64, (W, W, W), {"mg_fixed_cycles": 4}),
])
def test_reported_residual_is_that_of_the_pressure(nx, ny, nz, bc, kw):
    P = need_gpu()
    p = cases.Params(nx=nx, ny=ny, nz=nz, h=1.0 / max(nx, ny, nz), bc=bc, rho=(1.0, 20.0),
                     precision=cases.MIXED, **kw)
    x, y, z = cases.cell_centres(p)
    L = np.array([nx, ny, nz]) * p.h
    d = np.sqrt((x - 0.4 * L[0]) ** 2 + (y - 0.55 * L[1]) ** 2 + (z - 0.5 * L[2]) ** 2)
    # a sharp drop: the mixtures and the face coefficients are then one rounding
    # of exact numbers, the same here and in the library
    alpha = np.broadcast_to(d < 0.3 * L.max(), p.shape).astype(np.float32)
    rhs = cases.uniform(31, p.shape, -1, 1)
    got, info = _solve(P, p, alpha, rhs)
    assert info["status"] == 0
    # the library's operator: beta in float from the float phase fraction
    grid = O.Grid(p)
    rho = alpha * np.float32(p.rho[1]) + (np.float32(1) - alpha) * np.float32(p.rho[0])
    rho = torch.tensor(rho)
    beta = []
    for q in range(3):
        b = torch.tensor(1.0, dtype=torch.float32) / (0.5 * (rho + rho.roll(1, 2 - q)))
        b = b.double()
        beta.append(O._zero_wall_face(b, q) if bc[q] == W else b)
    lev = O.Level(grid.n, (grid.h,) * 3, grid.bc, beta)
    b = torch.tensor(rhs - rhs.mean())
    rel = float((b - O.apply_L(got, lev)).norm() / b.norm())
    if not kw.get("mg_fixed_cycles"):
        assert info["rel_residual"][0] <= 1e-10
    # both are double residuals of the same p: they differ by rounding, 2^-53 of
    # the 12 fluxes of a cell, for a white-noise rhs at most ~400 |b| (2D)
    assert abs(rel - info["rel_residual"][0]) <= 1e-3 * info["rel_residual"][0] + 1e-12
    host, hinfo = _solve(P, p, alpha, rhs, host_loop=True)
    assert hinfo["vcycles"][0] == info["vcycles"][0]
    assert torch.equal(host, got)


def test_a_failed_solve_leaves_nothing_behind():
    """A solve whose residual overflows float, then one on the same context: the
    bits of a fresh context, also where an axis has walls and an odd number of
    cells (a wall cell's wrapped neighbour then has the cell's own colour)."""
    P = need_gpu()
    p = cases.Params(nx=100, ny=76, nz=71, h=0.01, bc=(W, W, W), rho=(1.0, 2.0),
                     precision=cases.MIXED, mg_max_cycles=30)
    alpha = torch.tensor((cases.uniform(5, p.shape, 0, 1) > 0.5).astype(np.float32), device="cuda")
    rhs = cases.uniform(31, p.shape, -1, 1)
    fresh, info = _solve(P, p, alpha, rhs)
    assert info["status"] == 0
    s = P.Solver(p)
    dp = torch.zeros(p.shape, dtype=torch.float64, device="cuda")
    bad = s.fvm_poisson_solve(alpha, torch.tensor(rhs * 1e60, device="cuda"), dp, raise_on_error=False)
    assert bad["status"] != 0
    dp.zero_()
    s.fvm_poisson_solve(alpha, torch.tensor(rhs, device="cuda"), dp)
    s.close()
    assert torch.equal(dp.cpu(), fresh)
