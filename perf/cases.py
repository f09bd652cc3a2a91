"""The work a user of this library has it do, as measurable cases.

A case names an entry point of the Python binding (``Solver.fvm_step``,
``fvm_poisson_solve``, ``fvm_stage_predict``, ``fvm_step_adjoint`` or the
allocation-free solve), a workload, a grid and a precision form.  Inputs are
drawn from a seed: smooth discretely divergence-free velocities, a blurred or
area-fraction interface and a smooth temperature, with the material data of the
workload.  ``exact`` restates the method in plain float64 PyTorch, written
independently of the library and of its oracle, with the pressure solved by
preconditioned conjugate gradients to rounding.

``fvm_step`` works in place, so a pass first copies the state it starts from
into the working fields, as a program that can reject a step does.
"""
from __future__ import annotations

import math
import random

import torch

from cases import MIXED, F64, PERIODIC, WALL, Params
from paper_2209_09671_gb300 import fvm

DEVICE = "cuda" if torch.cuda.is_available() else "cpu"
FIELDS = ("u", "v", "w", "alpha", "T")


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------
def _case(kind, nx, ny, nz, form, **more):
    return dict(kind=kind, nx=nx, ny=ny, nz=nz, form=form, **more)


def listed():
    return [
        # the 2D static drop: the smallest everyday run (verification, teaching,
        # parameter scans), its diagnostics read after every step
        dict(name="drop 64x64 f64", **_case("drop", 64, 64, 1, "f64")),
        # the paper's migrating droplet (Sec. V-A): tens of thousands of such
        # steps make one run; 100 = 4 * 25 leaves a 25 x 25 coarsest level
        dict(name="droplet 100x100 f64", **_case("droplet", 100, 100, 1, "f64")),
        # the two-layer thermocapillary channel in both precision forms
        dict(name="channel 128x128x64 mixed", **_case("channel", 128, 128, 64, "mixed")),
        dict(name="channel 128x128x64 f64", **_case("channel", 128, 128, 64, "f64")),
        # the melt pool: the headline size, the largest one, and a double run of
        # the size on which a mixed run would be verified
        dict(name="melt 256x256x256 mixed", **_case("melt", 256, 256, 256, "mixed")),
        dict(name="melt 512x512x256 mixed", **_case("melt", 512, 512, 256, "mixed")),
        dict(name="melt 128x128x128 f64", **_case("melt", 128, 128, 128, "f64")),
        # alloying: a transported concentration and the bounded phase fraction,
        # walls on x and z, sizes that fill no tile
        dict(name="alloy 88x72x40 mixed", **_case("alloy", 88, 72, 40, "mixed")),
        # the pressure solve alone with the residual read back: a ragged box
        # between walls whose coarsening stops early
        dict(name="poisson 144x112x80 mixed", **_case("poisson", 144, 112, 80, "mixed", density=100.0)),
        # the allocation-free solve at its largest cubic grid
        dict(name="noalloc 64x64x64 f64", **_case("noalloc", 64, 64, 64, "f64", density=10.0)),
        # the predictor alone (explicit operators), odd sizes between walls
        dict(name="predict 149x90x75 f64", **_case("predict", 149, 90, 75, "f64")),
        # one reverse step of a calibration gradient, unequal densities
        dict(name="adjoint 96x96x48 f64", **_case("adjoint", 96, 96, 48, "f64", density=10.0)),
    ]


def _log_int(rng, lo, hi, step=1):
    return step * max(1, round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / step))


def draw(rng: random.Random):
    # sizes in use on periodic axes: 2^k times 1, 3, 5 or 7 (the hierarchy then
    # coarsens far); wall axes take other multiples as well
    per = [32, 40, 48, 64, 80, 96, 112, 128, 160, 192, 224, 256]
    form = rng.choice(["mixed", "f64"])
    kind = rng.choice(["drop", "droplet", "channel", "channel", "melt", "melt", "alloy", "poisson",
                       "noalloc", "predict", "adjoint"])
    if kind == "drop":
        n = _log_int(rng, 32, 256, 8)
        return _case(kind, n, n, 1, form)
    if kind == "droplet":
        n = _log_int(rng, 40, 136, 4)
        return _case(kind, n, n, 1, "f64")
    if kind == "channel":
        return _case(kind, rng.choice(per[:9]), rng.choice(per[:9]), _log_int(rng, 16, 96, 8), form)
    if kind == "melt":
        m = per if form == "mixed" else per[:8]
        return _case(kind, rng.choice(m), rng.choice(m), _log_int(rng, 48, 256 if form == "mixed" else 128, 16), form)
    if kind == "alloy":
        return _case(kind, _log_int(rng, 24, 120, 4), rng.choice(per[:7]), _log_int(rng, 16, 80, 4), form)
    if kind == "poisson":
        return _case(kind, _log_int(rng, 32, 256, 16), _log_int(rng, 32, 256, 16), _log_int(rng, 16, 160, 16), form,
                     density=float(_log_int(rng, 1, 1000)))
    if kind == "noalloc":
        return _case(kind, _log_int(rng, 16, 64, 4), _log_int(rng, 16, 64, 4), _log_int(rng, 8, 64, 4), form,
                     density=float(_log_int(rng, 1, 100)))
    if kind == "predict":
        return _case(kind, _log_int(rng, 17, 250), _log_int(rng, 16, 250, 2), _log_int(rng, 13, 160), form)
    return _case("adjoint", rng.choice(per[:6]), rng.choice(per[:6]), _log_int(rng, 8, 48, 4), "f64",
                 density=rng.choice([1.0, 10.0]))


# --------------------------------------------------------------------------
# parameters and inputs
# --------------------------------------------------------------------------
def _params(case, r: random.Random) -> Params:
    nx, ny, nz, kind = case["nx"], case["ny"], case["nz"], case["kind"]
    p = Params(nx=nx, ny=ny, nz=nz, precision=MIXED if case["form"] == "mixed" else F64)
    if kind == "drop":
        return p.replace(h=1.0 / nx, bc=(WALL, WALL, PERIODIC), rho=(1.0, 10.0), mu=(0.01, 0.1),
                         lam=(1e-6, 1e-6), sigma0=1.0)
    if kind == "droplet":
        a, grad = 1.44e-3, 200.0
        # temperatures relative to 290 K
        return p.replace(h=4 * a / nx, bc=(WALL, WALL, PERIODIC), tbc=(0, 0, 1, 1, 0, 0),
                         tbc_T0=(0, 0, 0, 4 * a * grad, 0, 0), rho=(250.0, 500.0), mu=(0.012, 0.024),
                         cp=(5e-5, 1e-4), lam=(1.2e-6, 2.4e-6), sigma0=0.1, dsigma_dT=-0.02,
                         weno_scale=(1.0, 4 * a * grad, 0.01))
    if kind in ("channel", "adjoint"):
        p = p.replace(h=1.0 / nz, bc=(PERIODIC, PERIODIC, WALL), tbc=(0, 0, 0, 0, 1, 1),
                      tbc_dTamp=(0, 0, 0, 0, 1.0, 0), sigma0=1.0, dsigma_dT=-0.01)
        if kind == "adjoint":
            d = case["density"]
            p = p.replace(adjoint=1, mg_rtol=1e-12, rho=(1.0, d), cp=(1.0, 1.0 / d), q_power=0.05,
                          q_radius=8 * p.h, q_x0=0.5 * nx * p.h, q_y0=0.5 * ny * p.h)
        return p
    if kind == "melt":
        h = 2e-6
        return p.replace(h=h, bc=(PERIODIC, PERIODIC, WALL), rho=(1.0, 7900.0), mu=(5.85e-5, 5.85e-3),
                         cp=(1900.0, 790.0), lam=(0.02, 6.6), sigma0=1.908, dsigma_dT=-4.3e-4, T0=1700.0,
                         g=(0.0, 0.0, -9.81), q_power=5e-3, q_radius=8 * h, q_x0=r.uniform(0, nx) * h,
                         q_y0=r.uniform(0, ny) * h, q_speed=0.5, weno_scale=(1.0, 17.0, 1.0))
    h = 1.0 / 16
    p = p.replace(h=h, bc=(WALL, PERIODIC, WALL), tbc=(0, 0, 0, 0, 1, 1), tbc_T0=(0, 0, 0, 0, 1.3, -0.4),
                  tbc_dTamp=(0, 0, 0, 0, 0.5, 0.5), rho=(1.0, 6.0), mu=(0.02, 0.05), cp=(1.0, 2.0),
                  lam=(0.01, 0.03), sigma0=0.05, dsigma_dT=-0.02, T0=0.2, g=(0.1, -0.2, -0.5),
                  q_power=0.002, q_radius=3 * h, q_x0=5.2 * h, q_y0=4.7 * h, q_speed=0.5)
    if kind == "alloy":
        p = p.replace(concentration=1, dsigma_dc=0.03, c0=0.45, diff_c=(0.004, 0.012), alpha_scheme=1)
    if kind in ("poisson", "noalloc"):
        p = p.replace(bc=(WALL, WALL, WALL), tbc=(0,) * 6, rho=(1.0, case["density"]))
    return p


def _axes(p, node=(False, False, False)):
    """Coordinates of cell centres (or of low nodes) over the box, in [0, 1)."""
    out = []
    for d, n in enumerate((p.nx, p.ny, p.nz)):
        c = (torch.arange(n, dtype=torch.float64, device=DEVICE) + (0.0 if node[d] else 0.5)) / n
        out.append(c.reshape([n if q == 2 - d else 1 for q in range(3)]))
    return out


def _modes(p, r, count=3, top=3):
    """A smooth field of a few Fourier modes with values of order one."""
    x, y, z = _axes(p)
    out = torch.zeros(p.shape, dtype=torch.float64, device=DEVICE)
    for _ in range(count):
        f = r.uniform(0.5, 1.0)
        for c in (x, y, z):
            f = f * torch.cos(2 * math.pi * r.randint(1, top) * c + r.uniform(0, 6.28))
        out += f
    return out


def _solenoidal(p, r, amp):
    """Discretely divergence-free face velocities of largest value `amp`: the
    curl of an edge potential whose tangential parts vanish on walls."""
    pot = []
    for d in range(3):
        node = tuple(q != d for q in range(3))
        f = torch.zeros(p.shape, dtype=torch.float64, device=DEVICE)
        for _ in range(2):
            m = r.uniform(0.5, 1.0)
            for q, c in enumerate(_axes(p, node)):
                k = r.randint(1, 3)
                if p.bc[q] == WALL and node[q]:
                    m = m * torch.sin(math.pi * k * c)
                else:
                    m = m * torch.cos(2 * math.pi * k * c + r.uniform(0, 6.28))
            f += m
        pot.append(f)
    diff = lambda a, d: (a.roll(-1, 2 - d) - a) * (p.nx, p.ny, p.nz)[d]  # noqa: E731
    vel = []
    for d in range(3):
        e, f = (d + 1) % 3, (d + 2) % 3
        vel.append(diff(pot[f], e) - diff(pot[e], f))
    top = max(float(v.abs().max()) for v in vel)
    return [v * (amp / top) for v in vel]


def _fields(case, seed):
    """(params, state) of a case in float64, and the generator."""
    r = random.Random(seed)
    p = _params(case, r)
    h, kind = p.h, case["kind"]
    x, y, z = _axes(p)
    X, Y, Z = x * p.nx * h, y * p.ny * h, z * p.nz * h
    L = (p.nx * h, p.ny * h, p.nz * h)
    speed = {"drop": 0.05, "droplet": 2e-3, "channel": 0.02, "adjoint": 0.02, "melt": 0.5}.get(kind, 0.5)
    u, v, w = _solenoidal(p, r, speed)
    s = {"u": u, "v": v, "w": w, "p": torch.zeros(p.shape, dtype=torch.float64, device=DEVICE)}
    if kind in ("drop", "droplet", "alloy", "poisson", "noalloc", "predict"):
        # a drop with a slightly wavy outline; area fractions in 2D, blurred in 3D
        R = r.uniform(0.22, 0.28) * min(q for q, n in zip(L, p.shape[::-1]) if n > 1)
        d2 = (X - L[0] * r.uniform(0.45, 0.55)) ** 2 + (Y - L[1] * r.uniform(0.45, 0.55)) ** 2
        if p.nz > 1:
            d2 = d2 + (Z - L[2] * r.uniform(0.45, 0.55)) ** 2
        dist = torch.sqrt(d2) - R * (1 + 4e-3 * _modes(p, r))
        s["alpha"] = torch.clamp(0.5 - dist / h, 0, 1) if p.nz == 1 else 0.5 * (1 - torch.tanh(dist / (1.5 * h)))
    elif kind == "melt":
        # a sharp, slightly rippled free surface
        zi = L[2] / 2 + 0.6 * h * torch.cos(2 * math.pi * (x + r.random())) * torch.cos(2 * math.pi * (y + r.random()))
        s["alpha"] = torch.clamp(0.5 + (zi - Z) / h, 0, 1)
    else:
        zi = L[2] / 2 + 0.6 * h * torch.cos(2 * math.pi * (x + r.random())) * torch.cos(2 * math.pi * (y + r.random()))
        s["alpha"] = 0.5 * (1 - torch.tanh((Z - zi) / (1.2 * h)))
    noise = _modes(p, r)
    if kind == "drop":
        s["T"] = torch.zeros(p.shape, dtype=torch.float64, device=DEVICE)
    elif kind == "droplet":
        s["T"] = 200.0 * Y + 1e-3 * noise
    elif kind in ("channel", "adjoint"):
        k = 2 * math.pi / L[0]
        s["T"] = torch.cos(k * X) * torch.sinh(k * (L[2] - Z)) / math.sinh(k * L[2]) + 0.01 * noise
    elif kind == "melt":
        s["T"] = 1700.0 + 6.0 * noise
    else:
        s["T"] = noise
    if p.concentration:
        s["c"] = 0.5 + 0.1 * _modes(p, r)
    s = {k: a.expand(p.shape).contiguous() for k, a in s.items()}
    if p.precision == MIXED:
        s = {k: a if k == "p" else a.float() for k, a in s.items()}
    if kind in ("poisson", "noalloc"):
        g = torch.Generator(device=DEVICE).manual_seed(seed)
        s["rhs"] = _modes(p, r) + 0.3 * torch.randn(p.shape, generator=g, dtype=torch.float64, device=DEVICE)
    if kind == "adjoint":
        g = torch.Generator(device=DEVICE).manual_seed(seed)
        for k in FIELDS:
            s["lam_" + k] = torch.randn(p.shape, generator=g, dtype=torch.float64, device=DEVICE)
    return p, s


def _given_dt(p):
    """The step of the entry points that are handed one."""
    return 0.2 * p.h * p.h if p.adjoint else 0.16 * p.h


def prepare(case, seed):
    p, s = _fields(case, seed)
    st = {"kind": case["kind"], "params": p, "in": s}
    if case["kind"] == "noalloc":
        st["cparams"] = fvm.make_params(p)
    else:
        st["solver"] = fvm.Solver(p, device=DEVICE)
    if case["kind"] in ("poisson", "noalloc"):
        st["p"] = torch.empty_like(s["p"])
    elif case["kind"] not in ("predict", "adjoint"):
        st["work"] = {k: torch.empty_like(a) for k, a in s.items()}
    return st


def run(st):
    p, s, kind = st["params"], st["in"], st["kind"]
    if kind == "predict":
        return st["solver"].fvm_stage_predict(s, 3, _given_dt(p))
    if kind == "adjoint":
        lam, dth = st["solver"].fvm_step_adjoint(s, 2, _given_dt(p), {k: s["lam_" + k] for k in FIELDS})
        return [lam[k] for k in FIELDS], dth
    if kind in ("poisson", "noalloc"):
        st["p"].zero_()
        if kind == "poisson":
            st["solver"].fvm_poisson_solve(s["alpha"], s["rhs"], st["p"])
        else:
            fvm.fvm_poisson_solve_noalloc(st["cparams"], s["alpha"], s["rhs"], st["p"])
        return [st["p"]]
    work = st["work"]
    for k, a in s.items():
        work[k].copy_(a)
    info = st["solver"].fvm_step(work, 3, 0.0, info=kind == "drop")
    out = [work[k] for k in FIELDS] + ([work["c"]] if "c" in work else [])
    # the mixed form's pressure belongs to float velocities, and its users read
    # it as such; in double it comes as it is
    out.append(work["p"].float() if p.precision == MIXED else work["p"])
    return out + ([info["dt"], info["vol_sum"], info["mass_sum"]] if kind == "drop" else [])


def work(case):
    n, kind = case["nx"] * case["ny"] * case["nz"], case["kind"]
    rs = 4 if case["form"] == "mixed" else 8
    # operations a cell: a stage's 15 WENO5 reconstructions and forces (about
    # 1200); a V(2,2) cycle's sweeps and residual (about 100), some ten cycles a
    # solve
    if kind in ("poisson", "noalloc"):
        return {"bytes": n * (rs + 16), "flops": 1000 * n}
    if kind == "predict":
        return {"bytes": n * 10 * rs, "flops": 1200 * n}
    if kind == "adjoint":
        return {"bytes": n * 16 * 8, "flops": (3 * 2200 + 3 * 4600) * n}
    fields = 6 if kind == "alloy" else 5
    return {"bytes": n * 2 * (fields * rs + 8), "flops": 3 * 2200 * n}


# --------------------------------------------------------------------------
# the method in plain float64 PyTorch
# --------------------------------------------------------------------------
GH = 3            # ghost layers


class _Method:
    """Operators of one stage on fields [z, y, x]; every function here can be
    differentiated by autograd."""

    def __init__(self, p: Params):
        self.p, self.h = p, p.h
        self.n = (p.nx, p.ny, p.nz)
        self.eps_n = 1e-8 / p.h

    # -- ghosts: kind 'even', 'odd', 'face' per axis, or 'T' ----------------
    def _pad_axis(self, a, d, kind):
        n, dim = self.n[d], 2 - d
        i = torch.arange(-GH, n + GH + 1, device=a.device)
        sign = torch.ones(i.numel(), dtype=a.dtype, device=a.device)
        if self.p.bc[d] == PERIODIC:
            return a.index_select(dim, i % n)
        if kind == "face":
            src = torch.where(i < 0, -i, torch.where(i > n, 2 * n - i, i))
            sign[(i < 0) | (i > n)] = -1.0
            sign[(i == 0) | (i == n)] = 0.0
            src = torch.where(src >= n, 0, src)
        else:
            src = torch.where(i < 0, -1 - i, torch.where(i >= n, 2 * n - 1 - i, i)).clamp(0, n - 1)
            if kind == "odd":
                sign[(i < 0) | (i >= n)] = -1.0
        sh = [1, 1, 1]
        sh[dim] = i.numel()
        out = a.index_select(dim, src) * sign.reshape(sh)
        if kind == "T":
            for side in (0, 1):
                if self.p.tbc[2 * d + side] != 1:
                    continue
                m = ((i < 0) if side == 0 else (i >= n)).to(a.dtype).reshape(sh)
                e = 1 if d == 0 else 0       # the cosine runs along x, or y on x-walls
                c = torch.arange(out.shape[2 - e], device=a.device, dtype=a.dtype) - (GH if e < d else 0)
                tw = self.p.tbc_T0[2 * d + side] + self.p.tbc_dTamp[2 * d + side] * torch.cos(
                    2 * math.pi * (c + 0.5) / self.n[e])
                sw = [1, 1, 1]
                sw[2 - e] = c.numel()
                out = out * (1 - 2 * m) + 2 * m * tw.reshape(sw)
        return out

    def pad(self, a, kind):
        for d in range(3):
            a = self._pad_axis(a, d, kind)
        return a

    def pad_vel(self, a, c):
        for d in range(3):
            a = self._pad_axis(a, d, "face" if d == c else "odd")
        return a

    def at(self, P, *shifts):
        o = [GH, GH, GH]
        for d, s in shifts:
            o[d] += s
        nx, ny, nz = self.n
        return P[o[2]:o[2] + nz, o[1]:o[1] + ny, o[0]:o[0] + nx]

    # -- pieces ---------------------------------------------------------------
    @staticmethod
    def mix(al, pair):
        a = al.clamp(0, 1)
        return a * pair[1] + (1 - a) * pair[0]

    @staticmethod
    def weno(a, b, c, d, e, eps):
        b0 = 13 / 12 * (a - 2 * b + c) ** 2 + 0.25 * (a - 4 * b + 3 * c) ** 2
        b1 = 13 / 12 * (b - 2 * c + d) ** 2 + 0.25 * (b - d) ** 2
        b2 = 13 / 12 * (c - 2 * d + e) ** 2 + 0.25 * (3 * c - 4 * d + e) ** 2
        w0, w1, w2 = 0.1 / (eps + b0) ** 2, 0.6 / (eps + b1) ** 2, 0.3 / (eps + b2) ** 2
        q = w0 * (2 * a - 7 * b + 11 * c) + w1 * (-b + 5 * c + 2 * d) + w2 * (2 * c + 5 * d - e)
        return q / (6 * (w0 + w1 + w2))

    def flux(self, U, P, d, eps, *shifts):
        """U times the upwind WENO5 value of P on the low d-side at the shift."""
        v = [self.at(P, (d, m), *shifts) for m in range(-3, 3)]
        up = U >= 0
        return U * self.weno(*[torch.where(up, v[q], v[5 - q]) for q in range(5)], eps)

    @staticmethod
    def norm(sq):
        pos = sq > 0
        return torch.where(pos, torch.sqrt(torch.where(pos, sq, 1.0)), 0.0)

    def smooth(self, al):
        for _ in range(self.p.smooth_passes):
            for d in range(3):
                if self.n[d] > 1:
                    P = self.pad(al, "even")
                    al = 0.25 * (self.at(P, (d, -1)) + 2 * self.at(P) + self.at(P, (d, 1)))
        return al

    def grad(self, P):
        return [(self.at(P, (d, 1)) - self.at(P, (d, -1))) / (2 * self.h) for d in range(3)]

    def curvature(self, SP):
        h, kap = self.h, 0.0
        for d in range(3):
            nrm = []
            for s in (0, 1):
                gd = (self.at(SP, (d, s)) - self.at(SP, (d, s - 1))) / h
                sq = gd ** 2
                for t in range(3):
                    if t != d:
                        sq = sq + ((self.at(SP, (t, 1), (d, s)) - self.at(SP, (t, -1), (d, s))
                                    + self.at(SP, (t, 1), (d, s - 1)) - self.at(SP, (t, -1), (d, s - 1))) / (4 * h)) ** 2
                nrm.append(gd / (self.norm(sq) + self.eps_n))
            kap = kap + (nrm[1] - nrm[0]) / h
        return kap

    def advect(self, P, vel, eps):
        out = 0.0
        for d in range(3):
            F = [self.flux(self.at(vel[d], (d, s)), P, d, eps, (d, s)) for s in (0, 1)]
            out = out - (F[1] - F[0]) / self.h
        return out

    def advect_bounded(self, P, vel, eps, dt):
        """Zalesak's flux-corrected blend of upwind and WENO5 with bounds 0, 1."""
        h = self.h
        low, anti, div, into, outof = {}, {}, 0.0, 0.0, 0.0
        for d in range(3):
            for s in (0, 1):
                U = self.at(vel[d], (d, s))
                low[d, s] = U * torch.where(U >= 0, self.at(P, (d, s - 1)), self.at(P, (d, s)))
                anti[d, s] = self.flux(U, P, d, eps, (d, s)) - low[d, s]
            div = div + (low[d, 1] - low[d, 0]) / h
            into = into + anti[d, 0].clamp(min=0) + (-anti[d, 1]).clamp(min=0)
            outof = outof + (-anti[d, 0]).clamp(min=0) + anti[d, 1].clamp(min=0)
        td = self.at(P) - dt * div
        lim = lambda q, s: torch.where(s > 0, (q * h / dt / torch.where(s > 0, s, 1.0)).clamp(0, 1), 0.0)  # noqa: E731
        RP, RM = self.pad(lim(1 - td, into), "even"), self.pad(lim(td, outof), "even")
        out = 0.0
        for d in range(3):
            F = []
            for s in (0, 1):
                a = anti[d, s]
                pos = torch.minimum(self.at(RP, (d, s)), self.at(RM, (d, s - 1)))
                neg = torch.minimum(self.at(RP, (d, s - 1)), self.at(RM, (d, s)))
                F.append(low[d, s] + torch.where(a > 0, pos, neg) * a)
            out = out - (F[1] - F[0]) / h
        return out

    def diffuse(self, P, KP):
        out = 0.0
        for d in range(3):
            F = []
            for s in (0, 1):
                a, b = self.at(KP, (d, s - 1)), self.at(KP, (d, s))
                F.append(2 * a * b / (a + b) * (self.at(P, (d, s)) - self.at(P, (d, s - 1))) / self.h)
            out = out + (F[1] - F[0]) / self.h
        return out

    def source(self, step):
        p, dev = self.p, DEVICE
        d = []
        for q, c0 in ((0, p.q_x0 + p.q_speed * p.h * step), (1, p.q_y0)):
            x = (torch.arange(self.n[q], dtype=torch.float64, device=dev) + 0.5) * p.h - c0
            if p.bc[q] == PERIODIC:
                L = self.n[q] * p.h
                x = x - L * torch.floor(x / L + 0.5)
            d.append(x)
        r2 = p.q_radius ** 2
        return 2 / (math.pi * r2) * torch.exp(-2 * (d[0][None, :] ** 2 + d[1][:, None] ** 2) / r2)[None]

    def predictor(self, S, dt, step, dsdT, power):
        p, h = self.p, self.h
        eps = [p.weno_eps * s * s for s in p.weno_scale]
        al, T, c = S["alpha"], S["T"], S.get("c")
        vel = [self.pad_vel(S[k], d) for d, k in enumerate("uvw")]
        AP, TP, SP = self.pad(al, "even"), self.pad(T, "T"), self.pad(self.smooth(al), "even")
        sig = p.sigma0 + dsdT * (TP - p.T0)
        if c is not None:
            CP = self.pad(c, "even")
            sig = sig + p.dsigma_dc * (CP - p.c0)
        g, t, ds = self.grad(AP), self.grad(SP), self.grad(sig)
        gn = self.norm(g[0] ** 2 + g[1] ** 2 + g[2] ** 2)
        tn = self.norm(t[0] ** 2 + t[1] ** 2 + t[2] ** 2) + self.eps_n
        nds = sum(t[d] / tn * ds[d] for d in range(3))
        KP = self.pad(self.curvature(SP), "even")
        out = {}
        Ra = self.advect_bounded(AP, vel, eps[0], dt) if p.alpha_scheme else self.advect(AP, vel, eps[0])
        rcp = self.mix(al, (p.rho[0] * p.cp[0], p.rho[1] * p.cp[1]))
        RT = self.advect(TP, vel, eps[1]) + self.diffuse(TP, self.mix(AP, p.lam)) / rcp
        if p.q_power:
            RT = RT + power * self.source(step) * gn / rcp
        out["alpha"], out["T"] = al + dt * Ra, T + dt * RT
        if c is not None:
            out["c"] = c + dt * (self.advect(CP, vel, p.weno_eps * p.weno_scale_c ** 2)
                                 + self.diffuse(CP, self.mix(AP, p.diff_c)))
        mu, rho = self.mix(AP, p.mu), self.mix(AP, p.rho)
        for d, k in enumerate("uvw"):
            P, A, V = vel[d], 0.0, 0.0
            F, W = [], []
            for s in (-1, 0):
                a, b = self.at(P, (d, s)), self.at(P, (d, s + 1))
                F.append(self.flux(0.5 * (a + b), P, d, eps[2], (d, s + 1)))
                W.append(2 * self.at(mu, (d, s)) * (b - a) / h)
            A, V = A - (F[1] - F[0]) / h, V + (W[1] - W[0]) / h
            for e in range(3):
                if e == d:
                    continue
                F, W = [], []
                for s in (0, 1):
                    lo, hi = self.at(vel[e], (e, s), (d, -1)), self.at(vel[e], (e, s))
                    F.append(self.flux(0.5 * (lo + hi), P, e, eps[2], (e, s)))
                    m = 0.25 * (self.at(mu, (e, s)) + self.at(mu, (e, s), (d, -1))
                                + self.at(mu, (e, s - 1)) + self.at(mu, (e, s - 1), (d, -1)))
                    W.append(m * (self.at(P, (e, s)) - self.at(P, (e, s - 1)) + hi - lo) / h)
                A, V = A - (F[1] - F[0]) / h, V + (W[1] - W[0]) / h
            mean = lambda Q: 0.5 * (self.at(Q, (d, -1)) + self.at(Q))  # noqa: E731,B023
            fn = -mean(sig) * mean(KP) * (self.at(AP) - self.at(AP, (d, -1))) / h
            M = self.pad(gn * (ds[d] - t[d] / tn * nds), "even")
            out[k] = self.no_wall(self.at(P) + dt * (A + (V + fn + mean(M)) / mean(rho) + p.g[d]), d)
        return out

    def no_wall(self, a, d):
        if self.p.bc[d] != WALL:
            return a
        m = torch.ones(self.n[d], dtype=a.dtype, device=a.device)
        m[0] = 0
        sh = [1, 1, 1]
        sh[2 - d] = self.n[d]
        return a * m.reshape(sh)

    # -- pressure -------------------------------------------------------------
    def beta(self, al):
        rho = self.mix(al, self.p.rho)
        return [self.no_wall(2 / (rho + rho.roll(1, 2 - d)), d) for d in range(3)]

    def lap(self, x, be):
        out = torch.zeros_like(x)
        for d in range(3):
            if self.n[d] > 1:
                F = be[d] * (x - x.roll(1, 2 - d))
                out += F - F.roll(-1, 2 - d)
        return out / self.h ** 2

    def solve(self, be, b):
        """Mean-free p with L p = b - mean(b), by conjugate gradients."""
        b = b - b.mean()
        diag = sum((be[d] + be[d].roll(-1, 2 - d)) for d in range(3) if self.n[d] > 1) / self.h ** 2
        x, r = torch.zeros_like(b), b.clone()
        z = r / diag
        q, rz, bn = z.clone(), (r * z).sum(), b.norm()
        for it in range(20000):
            if it % 20 == 0 and float(r.norm()) <= 2e-15 * float(bn):
                break
            A = self.lap(q, be)
            a = rz / (q * A).sum()
            x += a * q
            r -= a * A
            z = r / diag
            new = (r * z).sum()
            q = z + (new / rz) * q
            rz = new
        return x - x.mean()

    def project(self, us, al, dt):
        be = self.beta(al)
        div = sum((u.roll(-1, 2 - d) - u) for d, u in enumerate(us)) / self.h
        pr = _Solve.apply(self, -div / dt, *be)
        return [self.no_wall(u - dt * be[d] * (pr - pr.roll(1, 2 - d)) / self.h, d) for d, u in enumerate(us)], pr

    # -- a step -----------------------------------------------------------------
    def limit(self, S):
        p, h, al = self.p, self.h, S["alpha"]
        sig = p.sigma0 + p.dsigma_dT * (S["T"] - p.T0)
        kap = (self.mix(al, p.lam) / self.mix(al, (p.rho[0] * p.cp[0], p.rho[1] * p.cp[1]))).max()
        if "c" in S:
            sig = sig + p.dsigma_dc * (S["c"] - p.c0)
            kap = max(kap, self.mix(al, p.diff_c).max())
        um = float(sum(S[k].abs().max() for k in "uvw"))
        return min(p.cfl * h / um if um else math.inf,
                   p.c_cap * math.sqrt(sum(p.rho) * h ** 3 / (4 * math.pi * float(sig.abs().max()))),
                   p.c_visc * h * h / float((self.mix(al, p.mu) / self.mix(al, p.rho)).max()),
                   p.c_therm * h * h / float(kap), p.dt_max)

    def step(self, S0, step, dt, dsdT, power):
        S0 = {k: self.no_wall(a, "uvw".index(k)) if k in "uvw" else a for k, a in S0.items()}
        X, pr = S0, None
        for a, b, c in ((0.0, 1.0, 0.0), (0.75, 0.25, 1.0), (1 / 3, 2 / 3, 0.5)):
            E = self.predictor(X, dt, step + c, dsdT, power)
            vel, pr = self.project([E[k] for k in "uvw"], X["alpha"], dt)
            E.update(zip("uvw", vel))
            X = {k: a * S0[k] + b * E[k] for k in S0}
        return X, pr


class _Solve(torch.autograd.Function):
    """p = L(beta)^+ b; backward by the same symmetric solve."""

    @staticmethod
    def forward(ctx, m, b, *be):
        pr = m.solve(be, b)
        ctx.m = m
        ctx.save_for_backward(pr, *be)
        return pr

    @staticmethod
    def backward(ctx, g):
        m, (pr, *be) = ctx.m, ctx.saved_tensors
        lam = m.solve(be, g)
        gb = [-(pr - pr.roll(1, 2 - d)) * (lam - lam.roll(1, 2 - d)) / m.h ** 2 if m.n[d] > 1 else None
              for d in range(3)]
        return (None, lam, *gb)


def exact(case, seed):
    kind, cells = case["kind"], case["nx"] * case["ny"] * case["nz"]
    # beyond these sizes the plain solve or the recorded graph takes too long
    if cells > {"adjoint": 1 << 19, "predict": 1 << 25}.get(kind, 3 << 20):
        return None
    p, s = _fields(case, seed)
    m = _Method(p)
    s = {k: a.double() for k, a in s.items()}
    if kind in ("poisson", "noalloc"):
        return [m.solve(m.beta(s["alpha"]), s["rhs"])]
    state = {k: s[k] for k in FIELDS + (("c",) if "c" in s else ())}
    if kind == "predict":
        out = m.predictor(state, _given_dt(p), 3, p.dsigma_dT, p.q_power)
        return {k: out[k] for k in FIELDS}
    if kind == "adjoint":
        th = [torch.tensor(v, dtype=torch.float64, device=DEVICE, requires_grad=True) for v in (p.dsigma_dT, p.q_power)]
        x = [state[k].requires_grad_() for k in FIELDS]
        Y, _ = m.step(dict(zip(FIELDS, x)), 2, _given_dt(p), *th)
        g = torch.autograd.grad([Y[k] for k in FIELDS], x + th, [s["lam_" + k] for k in FIELDS])
        return list(g[:5]), [float(v) for v in g[5:]]
    dt = m.limit(state)
    Y, pr = m.step(state, 3, dt, p.dsigma_dT, p.q_power)
    out = list(Y.values()) + [pr]
    if kind == "drop":
        out += [dt, float(Y["alpha"].sum() * p.h ** 3), float(m.mix(Y["alpha"], p.rho).sum() * p.h ** 3)]
    return out
