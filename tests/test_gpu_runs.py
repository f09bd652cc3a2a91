"""The predictor on grids whose z-marching kernels take runs of different
lengths, with a shorter last run: against the oracle at the parity bounds (FP64
1e-11; mixed 1e-5 for the velocities, 1e-6 for alpha and T)."""
import numpy as np
import pytest
import torch

import cases
from oracle import fvm_oracle as O
from tests.gpu_util import need_gpu, rel_l2
from tests.test_gpu_parity import _physics_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz", [(40, 20, 7), (160, 96, 43)])
@pytest.mark.parametrize("precision", [cases.F64, cases.MIXED])
def test_predictor_equals_oracle(nx, ny, nz, precision):
    P = need_gpu()
    p = _physics_case(nx, ny, nz, (1, 0, 1), 2).replace(precision=precision)
    s = cases.random_smooth_state(p, amp_u=0.5)
    if precision == cases.MIXED:
        s = {k: v.astype(np.float64) for k, v in cases.as_float32_state(s).items()}
    dt = 0.01
    ref = O.predictor({k: torch.tensor(v) for k, v in s.items()}, p, O.Grid(p), dt, 3, 0.0)
    solver = P.Solver(p)
    got = solver.fvm_stage_predict(P.to_device(s, precision == cases.MIXED), 3, dt)
    torch.cuda.synchronize()
    tol = {"u": 1e-11, "alpha": 1e-11} if precision == cases.F64 else {"u": 1e-5, "alpha": 1e-6}
    for k, r in zip(("u", "v", "w"), ref["ustar"]):
        assert rel_l2(got[k].double().cpu().numpy(), r.numpy()) <= tol["u"], k
    for k in ("alpha", "T"):
        assert rel_l2(got[k].double().cpu().numpy(), ref[k].numpy()) <= tol["alpha"], k
    solver.close()


@pytest.mark.parametrize("nx,ny,nz", [(40, 20, 7), (160, 96, 44), (200, 120, 107)])
@pytest.mark.parametrize("precision", [cases.F64, cases.MIXED])
def test_projected_velocity_is_divergence_free(nx, ny, nz, precision):
    """From rest each stage's divergence is -dt times its solve's residual, at
    most the solve's tolerance times |D u*|, plus roundings of the velocities; a
    right-hand side wrong in one plane or column leaves |D u*| there.  Factors: 2
    for the stages after the first, 6 faces a cell and 4 roundings a face."""
    P = need_gpu()
    p = _physics_case(nx, ny, nz, (1, 0, 1), 2).replace(precision=precision, mg_fixed_cycles=0)
    s = cases.random_smooth_state(p, amp_u=0.0)
    dt = 1e-3
    solver = P.Solver(p)
    d = P.to_device(s, precision == cases.MIXED)
    star = solver.fvm_stage_predict(d, 3, dt)

    def div(f):
        u, v, w = (f[k].double().cpu() for k in ("u", "v", "w"))
        return sum((a.roll(-1, 2 - q) - a) / p.h for q, a in enumerate((u, v, w)))

    before = div(star)
    solver.fvm_step(d, 3, dt)
    torch.cuda.synchronize()
    umax = max(float(star[k].abs().max()) for k in ("u", "v", "w"))
    eps = 2.0 ** (-53 if precision == cases.F64 else -24)
    bound = 2 * p.mg_rtol * float(before.norm()) + 24 * eps * umax / p.h * before.numel() ** 0.5
    assert float(div(d).norm()) <= bound
    assert bound < 1e-2 * float(before.norm())
    solver.close()
