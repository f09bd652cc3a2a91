"""FP64 predictor with the phases in either order.

Which phase is number 0 is a choice of the caller: exchanging the two values
of every property pair and replacing alpha by 1 - alpha describes the same
fluids.  alpha is a multiple of 2^-20, so that 1 - alpha and the sums of a few of
them are exact; h and dt are powers of two and the smoothing is off, so that
both orders compute the same curvature, Marangoni vector and differences, up to
sign.  What is left is the rounding of the mixtures and of what follows from
them, counted for each test in units u = 2^-53 per order.  The properties differ
by a factor of 6600 between the phases; a mixture formed from the larger value
loses that factor in the light phase."""
import numpy as np
import pytest
import torch

import cases
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu

U = 2.0 ** -53
SHAPE = (12, 16, 40)
H = 2.0 ** -5
RATIO = (1.2, 7900.0)


def _alpha(seed):
    a = np.round(cases.uniform(seed, SHAPE, -1.0, 2.0).clip(0.0, 1.0) * 2.0 ** 20) / 2.0 ** 20
    near = cases.uniform(seed + 1, SHAPE, 0.0, 1.0)
    return np.where(near < 0.2, 1.0 - 2.0 ** -20, np.where(near < 0.3, 2.0 ** -20, a))


def _predict(P, p, state, dt):
    s = P.Solver(p)
    out = s.fvm_stage_predict(P.to_device(state, False), 0, dt)
    torch.cuda.synchronize()
    s.close()
    return {k: v.cpu().numpy() for k, v in out.items()}


def _both(P, p, state, dt):
    q = p.replace(rho=p.rho[::-1], mu=p.mu[::-1], cp=p.cp[::-1], lam=p.lam[::-1])
    other = dict(state, alpha=1.0 - state["alpha"])
    return _predict(P, p, state, dt), _predict(P, q, other, dt)


def _state(seed):
    z = np.zeros(SHAPE)
    return {"u": z.copy(), "v": z.copy(), "w": z.copy(), "alpha": _alpha(seed), "T": z.copy(),
            "p": z.copy()}


def _params(**kw):
    nz, ny, nx = SHAPE
    return cases.Params(nx=nx, ny=ny, nz=nz, h=H, smooth_passes=0, **kw)


@pytest.mark.parametrize("mu", [(1.0, 1.0), (0.001, 0.005), (0.005, 0.001)])
def test_density(mu):
    """Fluid at rest: u* = dt Phi / rho_f with the same force sum Phi in both
    orders.  rho_f: 2 u (the difference of the pair and one fused operation), the
    quotient at most 2.1 u, the product with dt exact.  Both orders together
    8.2 u, bounded by 10 u of the value."""
    P = need_gpu()
    p = _params(rho=RATIO, mu=mu, sigma0=1.0, dsigma_dT=-0.25)
    s = _state(1)
    s["T"] = cases.uniform(5, SHAPE, -1.0, 1.0)
    a, b = _both(P, p, s, 0.25)
    for k in ("u", "v", "w"):
        assert np.abs(a[k]).max() > 0.0
        assert (np.abs(a[k] - b[k]) <= 10 * U * np.abs(a[k])).all()


def test_viscosity():
    """u(y) alone, alpha(y) alone, no surface tension, equal densities: u* =
    u + dt (F_hi - F_lo) / h with F = mu_e du / h.  mu_e: 2 u, the product 1 u; the
    difference and the two last sums 1 u each, dt large enough to drown u.  With
    |F_hi| + |F_lo| as the measure that is 6 u per order, 12 u for both."""
    P = need_gpu()
    p = _params(mu=RATIO)
    s = _state(2)
    s["alpha"] = np.broadcast_to(s["alpha"][:1, :, :1], SHAPE).copy()
    s["u"] = np.broadcast_to(cases.uniform(7, SHAPE, -1.0, 1.0)[:1, :, :1], SHAPE).copy()
    dt = 2.0 ** 40
    a, b = _both(P, p, s, dt)
    al, u = s["alpha"], s["u"]
    mu = al * p.mu[1] + (1.0 - al) * p.mu[0]
    f = np.abs(0.5 * (mu + np.roll(mu, 1, 1)) * (u - np.roll(u, 1, 1)) / H)   # low y-edge
    scale = dt * (f + np.roll(f, -1, 1)) / H
    assert (np.abs(a["u"] - b["u"]) <= 12 * U * scale).all()


def test_conduction():
    """Fluid at rest: T + dt q / (rho c_p), q the sum over the six faces of D / h, D
    the harmonic mean conductivity times dT / h.  D: mixtures 2 u each, their
    product 1 u and sum 1 u (with the mixtures' 2 u), the product with dT 1 u, the
    quotient 2.1 u: 11 u; five sums 5 u of sum |D|; rho c_p: 3 u, its quotient 2.1 u,
    the product with dt exact and the last sum 1 u: at most 23 u of
    dt sum |D| / (h rho c_p) per order, 46 u for both."""
    P = need_gpu()
    p = _params(lam=RATIO, cp=(900.0, 0.5))
    s = _state(3)
    s["T"] = cases.uniform(11, SHAPE, -1.0, 1.0)
    dt = 2.0 ** 20
    a, b = _both(P, p, s, dt)
    al, T = s["alpha"], s["T"]
    lam = al * p.lam[1] + (1.0 - al) * p.lam[0]
    rcp = al * p.cp[1] + (1.0 - al) * p.cp[0]
    total = np.zeros(SHAPE)
    for ax in range(3):
        l2, T2 = np.roll(lam, 1, ax), np.roll(T, 1, ax)
        d = 2.0 * lam * l2 / (lam + l2) * np.abs(T - T2) / H
        total += d + np.roll(d, -1, ax)
    scale = dt * total / (H * rcp) + np.abs(a["T"])
    assert (np.abs(a["T"] - b["T"]) <= 46 * U * scale).all()
    # with U = 0 the phase fraction does not move
    assert np.array_equal(a["alpha"], al) and np.array_equal(b["alpha"], 1.0 - al)
