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
