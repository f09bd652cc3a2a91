"""V-cycle levels between the finest and the coarse ones of the cluster launch.

A level of more than 32768 cells sweeps, restricts and prolongs in launches of
its own: in double with stored reciprocal diagonals, with the residuals of one
colour restricted, and with the next level's first sweep taken by the
restriction.  96 x 64 x 64 has such a level (48 x 32 x 32 = 49152 cells) under its
finest one, 192 x 128 x 128 two.  Every cycle shape runs them: no pre- or
post-smoothing, an odd number of sweeps, other counts below the finest level.
FP64 with a fixed cycle count against the oracle's V-cycle of the same shape at
the FP64 parity bound, mixed to 1e-12 against the oracle's FP64 solution.  The launch
classes say that the level did run on its own."""
import numpy as np
import pytest
import torch

import cases
from oracle import fvm_oracle as O
from tests.gpu_util import need_gpu, rel_l2

pytestmark = pytest.mark.gpu

TOL64 = 1e-11
W, P_ = cases.WALL, cases.PERIODIC
SHAPES = [(2, 2, 3), (0, 2, 3), (2, 0, 3), (1, 1, 0), (3, 1, 2), (1, 2, 1), (2, 2, 0)]


def _params(pre, post, coarse, precision, n=(96, 64, 64), **kw):
    return cases.Params(nx=n[0], ny=n[1], nz=n[2], h=1.0 / n[0], bc=(W, P_, W), rho=(1.0, 100.0),
                        mg_pre=pre, mg_post=post, mg_coarse_sweeps=coarse, precision=precision, **kw)


def _alpha(p):
    x, y, z = cases.cell_centres(p)
    L = np.array([p.nx, p.ny, p.nz]) * p.h
    d = np.sqrt((x - 0.4 * L[0]) ** 2 + (y - 0.55 * L[1]) ** 2 + (z - 0.5 * L[2]) ** 2)
    return np.broadcast_to(np.clip(0.5 - (d - 0.3 * min(L)) / (2.0 * p.h), 0.0, 1.0), p.shape).copy()


def _solve(P, p, alpha, rhs):
    """The solution by launches (profiled, so that they are counted) and by the
    solve graph, which have to agree bit for bit."""
    dt = torch.float32 if p.precision == cases.MIXED else torch.float64
    da, dr = torch.tensor(alpha, dtype=dt, device="cuda"), torch.tensor(rhs, device="cuda")
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(st):
        s = P.Solver(p, stream=st)
        s.fvm_profile(True)
        x = torch.zeros(p.shape, dtype=torch.float64, device="cuda")
        info = s.fvm_poisson_solve(da, dr, x)
        classes = s.fvm_profile_read()
        s.fvm_profile(False)
        y = torch.zeros_like(x)
        again = s.fvm_poisson_solve(da, dr, y)
    torch.cuda.synchronize()
    s.close()
    assert torch.equal(x, y) and again["vcycles"] == info["vcycles"]
    return x.cpu().numpy(), info, classes


def _own_levels(classes, pre, post, coarse):
    # restrictions from a level below the finest are launches of their own only
    # when that level is not in the cluster launch
    assert classes["restrict_coarse"][0] > 0 and classes["coarse_tail"][0] > 0
    if coarse > 0 or pre + post > 0:
        assert classes["gs_coarse"][0] > 0


@pytest.mark.parametrize("pre,post,coarse", SHAPES)
def test_f64_shapes_equal_oracle(pre, post, coarse):
    P = need_gpu()
    p = _params(pre, post, coarse, cases.F64, mg_fixed_cycles=3)
    alpha, rhs = _alpha(p), cases.uniform(13, p.shape, -1, 1)
    ref, cyc, _ = O.poisson_solve(alpha, rhs, np.zeros(p.shape), p)
    got, info, classes = _solve(P, p, alpha, rhs)
    assert info["vcycles"][0] == cyc == 3
    assert rel_l2(got, ref.numpy()) <= TOL64
    _own_levels(classes, pre, post, coarse)


@pytest.mark.parametrize("pre,post,coarse,inner", [s + (2,) for s in SHAPES] + [(2, 2, 3, 1), (1, 2, 3, 3)])
def test_mixed_shapes_reach_double_tolerance(pre, post, coarse, inner):
    P = need_gpu()
    p = _params(pre, post, coarse, cases.MIXED, mg_rtol=1e-12, mx_inner_cycles=inner,
                mg_max_cycles=200)
    alpha, rhs = _alpha(p), cases.uniform(17, p.shape, -1, 1)
    ref, _, _ = O.poisson_solve(alpha, rhs, np.zeros(p.shape), p.replace(precision=cases.F64))
    got, info, classes = _solve(P, p, alpha, rhs)
    assert info["rel_residual"][0] <= 1e-12
    assert rel_l2(got, ref.numpy()) <= 1e-6
    _own_levels(classes, pre, post, coarse)


@pytest.mark.parametrize("n,levels", [((96, 128, 128), 1), ((192, 128, 128), 2)])
@pytest.mark.parametrize("pre,post,coarse", [(2, 2, 3), (1, 1, 1)])
def test_f64_larger_own_levels_equal_oracle(pre, post, coarse, n, levels):
    P = need_gpu()
    p = _params(pre, post, coarse, cases.F64, n=n, mg_fixed_cycles=2)
    alpha, rhs = _alpha(p), cases.uniform(19, p.shape, -1, 1)
    ref, _, _ = O.poisson_solve(alpha, rhs, np.zeros(p.shape), p)
    got, _, classes = _solve(P, p, alpha, rhs)
    assert rel_l2(got, ref.numpy()) <= TOL64
    # each level below the finest that has launches of its own restricts once a cycle
    assert classes["restrict_coarse"][0] == 2 * levels


@pytest.mark.parametrize("precision", [cases.F64, cases.MIXED])
def test_no_cluster_launch(precision):
    """mg_levels = 2: the coarsest level of 49152 cells fits no cluster and takes
    conjugate gradients on one CTA, 10 iterations on both sides.  (Mixed: a few
    refinements, whose residual the solve itself measures in double.)"""
    P = need_gpu()
    p = _params(2, 2, 3, precision, mg_levels=2, coarse_maxit=10, mg_fixed_cycles=2)
    alpha, rhs = _alpha(p), cases.uniform(29, p.shape, -1, 1)
    got, info, classes = _solve(P, p, alpha, rhs)
    assert classes["coarse_tail"][0] == 0 and classes["coarse_cg"][0] > 0
    ref, _, rel = O.poisson_solve(alpha, rhs, np.zeros(p.shape), p.replace(precision=cases.F64))
    if precision == cases.F64:
        assert rel_l2(got, ref.numpy()) <= TOL64
    else:
        assert info["rel_residual"][0] < rel
