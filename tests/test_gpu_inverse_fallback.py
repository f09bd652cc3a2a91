"""Coarsest levels whose float inverse is of no use: with a density ratio of 10^9
the operator's condition is beyond float, a step of the defect correction gains
less than a factor of two, and the level goes on by conjugate gradients in the
layout and the buffers that the correction used.

The oracle's V-cycles supply the operator and the right-hand sides of the
coarsest level; the float inverse is formed and tried on them here, to show
that the grid is one that falls back.  Tolerances: the two sides' conjugate
gradients stop at 10^-12 of the right-hand side, so what is left is rounding, u =
2^-53 times the coarsest operator's condition in the solution and times the
density ratio in the residual (the light phase's level is as large as that
ratio), each with 64 for the operations of two cycles.  A wrong coarse correction
changes both in the first digit."""
import numpy as np
import pytest
import torch

import cases
from oracle import fvm_oracle as O
from tests.gpu_util import need_gpu, rel_l2

pytestmark = pytest.mark.gpu

W, P_ = cases.WALL, cases.PERIODIC
U = 2.0 ** -53


def _float_inverse(M):
    """Gauss-Jordan without pivoting, float."""
    G = M.astype(np.float32)
    with np.errstate(all="ignore"):
        for k in range(len(G)):
            row, col = G[k] / G[k, k], G[:, k].copy()
            row[k] = np.float32(1) / G[k, k]
            G = G - np.outer(col, row)
            G[:, k] = -col * row[k]
            G[k] = row
    return G


@pytest.mark.parametrize("nx,ny,nz,bc,ratio", [
    (14, 14, 1, (W, W, P_), 1e9),      # 49 coarsest cells on one CTA
    (28, 20, 12, (W, W, W), 1e9),      # 105 on four
])
def test_f64_cycles_equal_oracle(monkeypatch, nx, ny, nz, bc, ratio):
    P = need_gpu()
    p = cases.Params(nx=nx, ny=ny, nz=nz, h=1.0 / nx, bc=bc, rho=(1.0, ratio), mg_fixed_cycles=2)
    x, y, z = cases.cell_centres(p)
    L = np.array([nx, ny, nz]) * p.h
    d = np.sqrt((x - 0.4 * L[0]) ** 2 + (y - 0.55 * L[1]) ** 2 + (z - 0.5 * L[2]) ** 2)
    alpha = np.broadcast_to(np.clip(0.5 + (d - 0.3) / (2.0 * p.h), 0.0, 1.0), p.shape).copy()
    rhs = cases.uniform(23, p.shape, -1, 1)

    seen = []
    cg = O.coarse_cg
    monkeypatch.setattr(O, "coarse_cg", lambda b, lev, *a: seen.append((b, lev)) or cg(b, lev, *a))
    ref, _, rel = O.poisson_solve(alpha, rhs, np.zeros(p.shape), p)
    b, lev = seen[0]
    n = b.numel()
    assert 32 < n <= 1000 and p.coarse_maxit >= n
    eye = torch.eye(n, dtype=torch.float64).reshape((n,) + tuple(b.shape))
    M = np.stack([O.apply_L(e, lev).numpy().ravel() for e in eye])
    ev = np.linalg.eigvalsh(M)
    s = np.trace(M) / n
    G = _float_inverse(M / s + 1.0 / n)
    for b, _ in seen:
        r = b.numpy().ravel() - b.numpy().mean()
        scale = np.linalg.norm(r)
        with np.errstate(all="ignore"):
            dx = (G @ (r / scale).astype(np.float32)).astype(np.float64) * scale / s
            assert not np.linalg.norm(r - M @ dx) <= 0.5 * scale

    solver = P.Solver(p)
    dp = torch.zeros(p.shape, dtype=torch.float64, device="cuda")
    info = solver.fvm_poisson_solve(torch.tensor(alpha, device="cuda"), torch.tensor(rhs, device="cuda"),
                                    dp)
    solver.close()
    assert info["status"] == 0 and info["vcycles"][0] == 2
    assert abs(info["rel_residual"][0] - rel) <= 64 * ratio * U
    assert rel_l2(dp.cpu().numpy(), ref.numpy()) <= 64 * ev[-1] / ev[1] * U


@pytest.mark.parametrize("nx,ny,nz,bc", [(14, 14, 1, (W, W, P_)), (28, 20, 12, (W, P_, W))])
def test_coefficients_beyond_float(nx, ny, nz, bc):
    """beta / h^2 above 10^39: the float inverse is not a number.  In double the
    problem is that of densities 1 and 10, scaled; the FP64 parity bound."""
    P = need_gpu()
    p = cases.Params(nx=nx, ny=ny, nz=nz, h=1.0 / nx, bc=bc, rho=(1e-37, 1e-36), mg_fixed_cycles=3)
    x, y, z = cases.cell_centres(p)
    alpha = np.broadcast_to((np.sin(9 * x + 4 * y) * np.cos(7 * z) > 0.2).astype(float), p.shape).copy()
    rhs = cases.uniform(37, p.shape, -1, 1)
    ref, _, _ = O.poisson_solve(alpha, rhs, np.zeros(p.shape), p)
    solver = P.Solver(p)
    dp = torch.zeros(p.shape, dtype=torch.float64, device="cuda")
    info = solver.fvm_poisson_solve(torch.tensor(alpha, device="cuda"), torch.tensor(rhs, device="cuda"),
                                    dp)
    solver.close()
    assert info["status"] == 0
    assert rel_l2(dp.cpu().numpy(), ref.numpy()) <= 1e-11
