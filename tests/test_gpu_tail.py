"""The multigrid levels that run in one cluster launch, on hierarchies that
take each of its forms: a level on one CTA or spread over the cluster, rows of
odd length, axes of one cell, periodic wrap, the coarsest level by its inverse
(at most 32 cells), by a float inverse in defect correction or by conjugate
gradients, on one CTA or on the cluster, a tail
of the coarsest level alone, and the scratch-limited solve whose coefficients
are formed in every cycle.  FP64 with a fixed cycle count against the oracle's
V-cycles at the FP64 parity bound; mixed to 1e-12 against the FP64 solution."""
import numpy as np
import pytest
import torch

import cases
from oracle import fvm_oracle as O
from tests.gpu_util import need_gpu, rel_l2

pytestmark = pytest.mark.gpu

W, P_ = cases.WALL, cases.PERIODIC
GRIDS = [
    (8, 8, 8, (W, W, W)),         # every level on one CTA, 8 coarsest cells
    (32, 24, 16, (P_, W, W)),     # spread levels
    (64, 64, 1, (W, W, P_)),      # 2D
    (64, 1, 1, (W, P_, P_)),      # one row
    (1, 48, 1, (P_, W, P_)),      # one column
    (28, 20, 12, (W, W, W)),      # odd rows at the coarsest level
    (12, 12, 12, (P_, P_, P_)),   # coarsening stopped by the periodic colouring
    (66, 50, 1, (W, W, P_)),      # 825 coarsest cells
    (44, 20, 20, (W, P_, W)),     # coarsest level with wrap
]


def _problem(nx, ny, nz, bc, **kw):
    p = cases.Params(nx=nx, ny=ny, nz=nz, h=1.0 / max(nx, ny, nz), bc=bc, rho=(1.0, 10.0), **kw)
    x, y, z = cases.cell_centres(p)
    L = np.array([nx, ny, nz]) * p.h
    d = np.sqrt((x - 0.4 * L[0]) ** 2 + (y - 0.55 * L[1]) ** 2 + (z - 0.5 * L[2]) ** 2)
    a = np.clip(0.5 - (d - 0.3 * L.max()) / (2.0 * p.h), 0.0, 1.0)
    return p, np.broadcast_to(a, p.shape).copy(), cases.uniform(23, p.shape, -1, 1)


def _solve(P, p, alpha, rhs):
    s = P.Solver(p)
    dt = torch.float32 if p.precision == cases.MIXED else torch.float64
    dp = torch.zeros(p.shape, dtype=torch.float64, device="cuda")
    info = s.fvm_poisson_solve(torch.tensor(alpha, dtype=dt, device="cuda"),
                               torch.tensor(rhs, device="cuda"), dp)
    s.close()
    return dp.cpu().numpy(), info


@pytest.mark.parametrize("nx,ny,nz,bc", GRIDS)
def test_f64_cycles_equal_oracle(nx, ny, nz, bc):
    P = need_gpu()
    p, alpha, rhs = _problem(nx, ny, nz, bc, mg_fixed_cycles=4)
    ref, _, _ = O.poisson_solve(alpha, rhs, np.zeros(p.shape), p)
    got, _ = _solve(P, p, alpha, rhs)
    assert rel_l2(got, ref.numpy()) <= 1e-11


@pytest.mark.parametrize("nx,ny,nz,bc,maxit", [(28, 20, 12, (W, W, W), 104), (66, 50, 1, (W, W, P_), 800),
                                               (130, 34, 1, (W, P_, P_), 1000)])
def test_f64_cycles_with_conjugate_gradients(nx, ny, nz, bc, maxit):
    """An iteration cap below the cell count (or more than 1000 coarsest cells)
    keeps the coarsest level on conjugate gradients, which end before it."""
    P = need_gpu()
    p, alpha, rhs = _problem(nx, ny, nz, bc, mg_fixed_cycles=4, coarse_maxit=maxit)
    ref, _, _ = O.poisson_solve(alpha, rhs, np.zeros(p.shape), p)
    got, _ = _solve(P, p, alpha, rhs)
    assert rel_l2(got, ref.numpy()) <= 1e-11


@pytest.mark.parametrize("nx,ny,nz,bc", GRIDS)
def test_mixed_solve_reaches_double_tolerance(nx, ny, nz, bc):
    P = need_gpu()
    p, alpha, rhs = _problem(nx, ny, nz, bc, mg_rtol=1e-12)
    ref, _, _ = O.poisson_solve(alpha, rhs, np.zeros(p.shape), p)
    got, info = _solve(P, p.replace(precision=cases.MIXED), alpha, rhs)
    assert info["rel_residual"][0] <= 1e-12
    # the float phase fraction perturbs the operator by a few units of 1e-7
    assert rel_l2(got, ref.numpy()) <= 1e-6


def test_coarsest_level_alone():
    """mg_levels = 1: the whole grid by conjugate gradients on the cluster.
    Both sides stop at 1e-12 ||b||; with cond(L) of a few 10^3 their
    solutions agree to 1e-8."""
    P = need_gpu()
    p, alpha, rhs = _problem(21, 16, 12, (W, P_, W), mg_levels=1, mg_fixed_cycles=1)
    ref, _, _ = O.poisson_solve(alpha, rhs, np.zeros(p.shape), p)
    got, _ = _solve(P, p, alpha, rhs)
    assert rel_l2(got, ref.numpy()) <= 1e-8


def test_noalloc_without_room_for_the_coefficients():
    """435 456 cells leave less scratch than the packed coefficients need: the
    solve forms them in every cycle and stops at the same tolerance.  Two
    solutions at 1e-10 differ by at most cond(L) times that."""
    P = need_gpu()
    from paper_2209_09671_gb300 import fvm
    p, alpha, rhs = _problem(72, 72, 84, (W, W, W))
    ref, info = _solve(P, p, alpha, rhs)
    dp = torch.zeros(p.shape, dtype=torch.float64, device="cuda")
    got = fvm.fvm_poisson_solve_noalloc(p, torch.tensor(alpha, device="cuda"),
                                        torch.tensor(rhs, device="cuda"), dp)
    assert got["status"] == 0
    assert got["vcycles"][0] == info["vcycles"][0]
    assert got["rel_residual"][0] <= 1e-10
    assert rel_l2(dp.cpu().numpy(), ref) <= 1e-6


@pytest.mark.parametrize("nx", [128, 132])
def test_largest_grid_solved_in_one_launch_and_the_next(nx):
    """16384 double cells are solved by one launch, 16896 level by level."""
    P = need_gpu()
    p, alpha, rhs = _problem(nx, 128, 1, (W, W, P_), mg_fixed_cycles=3)
    ref, _, rel = O.poisson_solve(alpha, rhs, np.zeros(p.shape), p)
    got, info = _solve(P, p, alpha, rhs)
    assert info["vcycles"][0] == 3
    assert info["rel_residual"][0] == pytest.approx(rel, rel=1e-6)
    assert rel_l2(got, ref.numpy()) <= 1e-11


def test_one_launch_solve_of_zero_and_of_non_finite_right_hand_sides():
    P = need_gpu()
    p, alpha, rhs = _problem(16, 16, 8, (W, P_, W))
    got, info = _solve(P, p, alpha, 0.0 * rhs)
    assert info["status"] == 0 and info["vcycles"][0] == 0 and not got.any()
    s = P.Solver(p)
    rhs[1, 2, 3] = np.inf
    dp = torch.zeros(p.shape, dtype=torch.float64, device="cuda")
    info = s.fvm_poisson_solve(torch.tensor(alpha, device="cuda"), torch.tensor(rhs, device="cuda"),
                               dp, raise_on_error=False)
    assert info["status"] == 5
    s.close()
