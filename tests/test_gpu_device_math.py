"""The arithmetic helpers of the double kernels (fvm_device.cuh), which stand
in for comparisons, conversions, quotients and roots of the FP64 pipe: each
against the plain operation, over all exponents and on both sides of every
branch of the helper."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

from paper_2209_09671_gb300 import _build
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dm(tmp_path_factory):
    need_gpu()
    so = str(tmp_path_factory.mktemp("dm") / "device_math.so")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "device_math.cu")
    r = subprocess.run([_build.nvcc(), *_build.ARCH, *_build.FLAGS, "--extended-lambda", "-shared",
                        "-I", _build.CSRC, "-I", os.path.join(os.path.dirname(_build.HERE), "include"),
                        src, "-o", so], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(so)


def _run(fn, ins, out_dtype=torch.float64):
    """fn(n, inputs..., out) on the device; numpy in, numpy out."""
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in ins]
    out = torch.empty(dev[0].shape, dtype=out_dtype, device="cuda")
    torch.cuda.synchronize()
    assert fn(ctypes.c_longlong(dev[0].numel()), *[ctypes.c_void_p(t.data_ptr()) for t in dev],
              ctypes.c_void_p(out.data_ptr())) == 0
    return out.cpu().numpy()


def _doubles(seed, per_exponent=8):
    """Random mantissas at every exponent of both signs, with each exponent's
    first and last mantissa, zeros, infinities and NaN."""
    rng = np.random.default_rng(seed)
    e = np.arange(2047, dtype=np.uint64)[:, None]
    m = rng.integers(0, 1 << 52, (2047, per_exponent), dtype=np.uint64)
    m[:, 0], m[:, 1] = 0, (1 << 52) - 1
    b = ((e << np.uint64(52)) | m).ravel()
    a = np.concatenate([b, b | np.uint64(1 << 63)]).view(np.float64)
    return np.concatenate([a, [0.0, -0.0, np.inf, -np.inf, np.nan, -np.nan]])


def test_clamp01(dm):
    """0 below 0, 1 above 1, infinities included; NaN stays NaN."""
    a = np.concatenate([_doubles(1), np.linspace(-1.0, 2.0, 3001), np.nextafter(1.0, [0.0, 2.0])])
    got = _run(dm.dm_clamp01, [a])
    want = np.where(a < 0.0, 0.0, np.where(a > 1.0, 1.0, a))
    assert np.array_equal(got, want, equal_nan=True)


U = 2.0 ** -53


def _near(t):
    """The numbers around t > 0: its neighbours and some more on both sides."""
    b = np.float64(t).view(np.int64) + np.array([-3, -2, -1, 0, 1, 2, 3])
    return np.concatenate([b.view(np.float64), t * np.linspace(0.5, 2.0, 301)])


def test_root(dm):
    """The approximate reciprocal root is good to 20 bits in its operand and in
    its result: a relative error d of at most 3 2^-20.  After the step on it
    the error is 3/2 d^2 + u (u = 2^-53, the rounding of the sum), which the last
    step multiplies by d: 0.33 u; with its own rounding 1.4 u of the root."""
    a = np.abs(np.concatenate([_doubles(2, 64), _near(2.0 ** -960), _near(2.0 ** 960)]))
    got = _run(dm.dm_root, [a])
    ok = np.isfinite(a)
    want = np.sqrt(a[ok].astype(np.longdouble))
    assert (np.abs(got[ok] - want) <= 1.4 * U * want).all()
    assert np.array_equal(got[~ok], np.sqrt(a[~ok]), equal_nan=True)
    edge = ok & ((a < 2.0 ** -960) | (a >= 2.0 ** 960))
    assert np.array_equal(got[edge], np.sqrt(a[edge]))
    # (the root instruction is within u of the exact root)
    assert (np.abs(got[ok] - _run(dm.dm_sqrt, [a])[ok]) <= 2.4 * U * want).all()


def test_quotient(dm):
    """|e| <= 3 2^-20 leaves e^3 = 0.21 u, the series' product and the last one
    round by u each: 2.3 u of n / d.  A result below the normal numbers is rounded
    once more, by half a unit of 2^-1074."""
    d = np.concatenate([_doubles(3, 64), _near(2.0 ** -960), -_near(2.0 ** 960)])
    rng = np.random.default_rng(4)
    for scale in (None, 0, 500, -500):
        n = rng.permutation(_doubles(5, 64))[np.arange(d.size) % 262000]
        if scale is not None:   # a quotient of about 2^scale
            n = np.ldexp(rng.uniform(1.0, 2.0, d.size), np.clip(np.frexp(d)[1] + scale, -1074, 1023))
        got = _run(dm.dm_quotient, [n, d])
        cuda = _run(dm.dm_divide, [n, d])
        inside = (np.abs(d) >= 2.0 ** -960) & (np.abs(d) < 2.0 ** 960)
        assert np.array_equal(got[~inside], cuda[~inside], equal_nan=True)
        fin = inside & np.isfinite(n) & np.isfinite(cuda) & (np.abs(cuda) < 1.7e308)
        assert fin.sum() > 1000
        want = n[fin].astype(np.longdouble) / d[fin].astype(np.longdouble)
        tol = 2.3 * U * np.abs(want) + 2.0 ** -1074
        assert (np.abs(got[fin] - want) <= tol).all()
        # (the division is within u of the exact quotient)
        assert (np.abs(got[fin] - cuda[fin]) <= tol + U * np.abs(want)).all()
        # infinities, NaN and overflow as the division has them (beyond the last
        # numbers whose quotient the 2.3 u could take over the limit)
        big = np.abs(n.astype(np.longdouble) / np.where(inside, d, 1.0).astype(np.longdouble))
        sat = inside & ~(big <= np.longdouble(2.0) ** 1024 * (1.0 + 2.0 ** -50))
        assert np.array_equal(got[sat], cuda[sat], equal_nan=True)


def test_widen(dm):
    """Every float, bit for bit."""
    differ = torch.zeros(1, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    assert dm.dm_widen_all(ctypes.c_void_p(differ.data_ptr())) == 0
    assert differ.item() == 0


def test_narrow(dm):
    """Bit for bit: every exponent, the bits below a float's last one at 0, at
    and around a tie and random, odd and even last bits; the numbers that round
    to 2^128 and the subnormal ones among them."""
    rng = np.random.default_rng(6)
    e = np.arange(2048, dtype=np.uint64)[:, None, None]
    top = np.concatenate([rng.integers(0, 1 << 23, 60, dtype=np.uint64),
                          np.array([0, 1, 2, (1 << 23) - 2, (1 << 23) - 1], dtype=np.uint64)])[:, None]
    low = np.concatenate([np.array([0, 1, (1 << 28) - 1, 1 << 28, (1 << 28) + 1, (1 << 29) - 1],
                                   dtype=np.uint64), rng.integers(0, 1 << 29, 10, dtype=np.uint64)])
    b = ((e << np.uint64(52)) | (top << np.uint64(29)) | low).ravel()
    a = np.concatenate([b, b | np.uint64(1 << 63)]).view(np.float64)
    got = _run(dm.dm_narrow, [a], torch.float32)
    cuda = _run(dm.dm_to_float, [a], torch.float32)
    assert np.array_equal(got.view(np.uint32), cuda.view(np.uint32))
    with np.errstate(over="ignore", invalid="ignore"):
        host = a.astype(np.float32)
    num = ~np.isnan(a)
    assert np.array_equal(got[num].view(np.uint32), host[num].view(np.uint32))
