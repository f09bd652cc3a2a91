"""Launches that the CUDA runtime refuses: two contexts driven from two host
threads must not make each other's launches fail, and a solve that lost a
launch must say so every time, not only while its graph is built."""
import threading

import numpy as np
import pytest
import torch

import cases
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu

W, P_ = cases.WALL, cases.PERIODIC


def _problem(nx, ny, nz, bc, precision):
    p = cases.Params(nx=nx, ny=ny, nz=nz, h=1.0 / max(nx, ny, nz), bc=bc, rho=(1.0, 10.0),
                     precision=precision, mg_fixed_cycles=2)
    x, _, _ = cases.cell_centres(p)
    alpha = np.broadcast_to(np.clip(x / p.h / 4.0 - 1.0, 0.0, 1.0), p.shape).copy()
    dt = torch.float32 if precision == cases.MIXED else torch.float64
    return p, torch.tensor(alpha, dtype=dt, device="cuda"), \
        torch.tensor(cases.uniform(3, p.shape, -1, 1), device="cuda")


@pytest.mark.parametrize("precision", [cases.F64, cases.MIXED])
def test_two_threads_with_coarse_levels_of_different_size(precision):
    """Solves with the per-launch host loop (fvm_profile on), whose every cycle
    launches the coarse levels with that grid's own shared memory, from two
    threads: each returns bit for bit what it returns alone."""
    P = need_gpu()
    grids = [(64, 64, 32, (W, W, W)), (16, 16, 16, (P_, W, W))]
    jobs = []
    for g in grids:
        prm, alpha, rhs = _problem(*g, precision)
        st = torch.cuda.Stream()
        torch.cuda.synchronize()
        s = P.Solver(prm, stream=st)
        s.fvm_profile(True)
        x = torch.zeros(prm.shape, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        s.fvm_poisson_solve(alpha, rhs, x)
        torch.cuda.synchronize()
        jobs.append((s, st, alpha, rhs, x.clone()))
    bad = []

    def work(job, n):
        s, st, alpha, rhs, ref = job
        with torch.cuda.stream(st):
            for _ in range(n):
                x = torch.zeros_like(ref)
                info = s.fvm_poisson_solve(alpha, rhs, x, raise_on_error=False)
                if info["status"] != 0 or not torch.equal(x, ref):
                    bad.append(info)
                    return

    threads = [threading.Thread(target=work, args=(jobs[0], 300)),
               threading.Thread(target=work, args=(jobs[1], 600))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    for s, *_ in jobs:
        s.close()
    assert not bad, bad[0]


@pytest.mark.parametrize("precision", [cases.F64, cases.MIXED])
def test_refused_launch_is_reported_by_every_solve(precision):
    """300 000 rows exceed the sweeps' launch grid (65535 blocks of 4 rows):
    the launch is refused on the host, and every solve on that pressure field
    returns FVM_ECUDA, the later ones as well."""
    P = need_gpu()
    prm, alpha, rhs = _problem(4, 300000, 1, (W, W, P_), precision)
    prm = prm.replace(coarse_maxit=10)
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(st):
        s = P.Solver(prm, stream=st)
        x = torch.zeros(prm.shape, dtype=torch.float64, device="cuda")
        got = [s.fvm_poisson_solve(alpha, rhs, x, raise_on_error=False)["status"] for _ in range(3)]
    torch.cuda.synchronize()
    s.close()
    assert got == [3, 3, 3]
