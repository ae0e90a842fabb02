"""The pieces of the FP64 kernels on their own.  Arithmetic (fp64.cuh) against the
correctly rounded operations, over random mantissas, wide exponents and quotients
next to a rounding boundary; the exact solver's float start and FP64 finish, its
sampling and HLLC (riemann_f64.cuh) against the general solvers (riemann.cuh), over
states of ordinary and of extreme size, without pressure, of negative pressure or
density, and that are not numbers: the same vacua, finite where those are finite."""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    from paper_2211_12243_gb300 import build
    so = str(tmp_path_factory.mktemp("probe") / "probe.so")
    subprocess.run([build._nvcc(), "-O3", "-std=c++17", *build.ARCH, "-shared", "-Xcompiler", "-fPIC",
                    "-I", build.INCLUDE, "-I", build.CSRC, os.path.join(HERE, "fp64_probe.cu"),
                    "-o", so], check=True)
    return ctypes.CDLL(so)


N = 1 << 18
OPS = {"rcp64": 0, "rcp40": 1, "rsqrt64": 2, "sqrt64": 3, "div1": 4, "div2": 5, "div2_rounded": 6,
       "fixed64": 7}


def _arith(probe, op, a, b=None):
    import torch
    b = np.ones_like(a) if b is None else b
    x, y = (torch.as_tensor(v, dtype=torch.float64, device="cuda") for v in (a, b))
    out = torch.empty_like(x)
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    assert probe.probe_arith(OPS[op], a.size, p(x), p(y), p(out)) == 0
    return out.cpu().numpy()


def _random(seed, lo, hi):
    rng = np.random.default_rng(seed)
    return np.ldexp(1.0 + rng.random(N), rng.integers(lo, hi, N))


def _ulps(a, b):
    return np.abs(a.view(np.int64) - b.view(np.int64))


# The seeds carry 20 bits of operand and result: |e| <= 2^-19 (reciprocal) and
# 2^-18 (of x r^2).  A third-order step leaves e^3 = 2^-57 or 5/16 e^3 = 2^-55.7 and
# its roundings, half a unit at the end and, for the root, 2^-54 through x r.
@pytest.mark.parametrize("op,lo,hi,exact,ulps", [
    ("rcp64", -1000, 1000, lambda x: 1.0 / x, 1),
    ("rsqrt64", -1020, 1020, lambda x: 1.0 / np.sqrt(x.astype(np.longdouble)), 2),
    ("sqrt64", -1020, 1020, np.sqrt, 1),
])
def test_reciprocals_and_roots(probe, op, lo, hi, exact, ulps):
    x = _random(1, lo, hi)
    assert _ulps(_arith(probe, op, x), np.asarray(exact(x), dtype=np.float64)).max() <= ulps
    if op != "rcp64":
        x = np.ldexp(1.0 + np.arange(N) / N, np.arange(N) % 2)
        assert _ulps(_arith(probe, op, x), np.asarray(exact(x), dtype=np.float64)).max() <= ulps


def test_reciprocal_of_one_newton_step(probe):
    x = _random(2, -1000, 1000)
    assert np.max(np.abs(_arith(probe, "rcp40", x) * x - 1.0)) <= 2.0 ** -38


@pytest.mark.parametrize("op,ulps", [("div1", 1), ("div2", 0), ("div2_rounded", 0)])
def test_quotients(probe, op, ulps):
    a, b = _random(3, -60, 60), _random(4, -300, 300)
    q = _random(5, -40, 40)
    near = (q + 0.5 * np.spacing(q).astype(np.longdouble)) * b   # half-way between two quotients
    for num in (a, q * b, near.astype(np.float64), np.nextafter(near.astype(np.float64), np.inf)):
        assert _ulps(_arith(probe, op, num, b), num / b).max() <= ulps


def test_roots_of_special_operands(probe):
    x = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, -1.0, -5e-324, 1e-310, 2.2250738585072014e-308])
    want = np.array([0.0, 0.0, np.inf, np.nan, np.nan, np.nan, np.nan, 0.0, 2.0 ** -511])
    got = _arith(probe, "sqrt64", x)
    assert np.array_equal(got, want, equal_nan=True), got


def test_fixed_point(probe):
    t = np.concatenate([_random(6, -70, 0), [0.0, 1.0 - 2.0 ** -53, 2.0 ** -64, 2.0 ** -65, 2.0 ** -11]])
    got = _arith(probe, "fixed64", t).view(np.uint64)
    assert all(int(g) == math.floor(math.ldexp(v, 64)) for g, v in zip(got[::7], t[::7]))


def _states(kind, gamma, seed):
    rng = np.random.default_rng(seed)
    n = 1 << 16
    e = lambda s: np.exp(rng.uniform(-s, s, n))
    rho, p = np.ones(n), np.ones(n)
    mach = rng.uniform(0.0, 4.0, n)
    if kind in ("density", "both"):
        rho = 10.0 ** rng.uniform(-60, 60, n)
    if kind in ("pressure", "both"):
        p = 10.0 ** rng.uniform(-60, 60, n)
    c = np.sqrt(gamma * p / rho)
    s = np.stack([rho * e(1.5), c * mach * rng.uniform(-1, 1, n), p * e(3.0),
                  rho * e(1.5), c * mach * rng.uniform(-1, 1, n), p * e(3.0)])
    same = rng.random(n) < 0.25              # equal sides (a uniform fluid)
    s[3:, same] = s[:3, same]
    if kind == "cold":                       # pressures and velocities of zero, either sign
        z = lambda: np.copysign(0.0, rng.standard_normal(n))
        s[2] = np.where(rng.random(n) < 0.7, z(), s[2])
        s[5] = np.where(rng.random(n) < 0.7, z(), s[5])
        pick = lambda: np.where(rng.random(n) < 0.4, z(), rng.choice([-1.0, 1.0, 0.5], n))
        s[1], s[4] = pick(), pick()
    if kind == "negative":
        for q in (0, 2, 3, 5):
            s[q] *= np.where(rng.random(n) < 0.25, -1.0, 1.0)
        s[:, (s[0] < 0) & (s[3] < 0)] = 1.0  # (one density at least is positive)
    if kind == "nan":
        for q in range(6):
            s[q, rng.random(n) < 0.1] = np.nan
    return s


@pytest.mark.parametrize("gamma", [5.0 / 3.0, 1.4, 1.3, 1.05])
@pytest.mark.parametrize("kind", ["ordinary", "density", "pressure", "both", "cold", "negative", "nan"])
def test_solvers_agree_with_the_general_ones(probe, kind, gamma):
    import torch
    s = _states(kind, gamma, 11)
    n = s.shape[1]
    t = torch.as_tensor(np.ascontiguousarray(s), device="cuda")
    out = torch.empty((2, 8, n), dtype=torch.float64, device="cuda")
    flux = torch.empty((2, 5, n), dtype=torch.float64, device="cuda")
    p = lambda v: ctypes.c_void_p(v.data_ptr())
    assert probe.probe_solve(n, ctypes.c_double(gamma), p(t), p(out), p(flux)) == 0
    a, b = out.cpu().numpy()
    f, g = flux.cpu().numpy()
    fin = np.isfinite
    with np.errstate(all="ignore"):
        cs = np.sqrt(gamma * np.maximum(np.abs(s[2] / s[0]), np.abs(s[5] / s[3]))) + abs(s[1]) + abs(s[4])
        rho = np.maximum(np.abs(s[0]), np.abs(s[3]))
        assert np.array_equal(a[2], b[2])                                 # vacua
        # (HLLC's contact between sides of opposite densities is a quotient of two
        # differences that cancel: rounding, or not a number)
        real = ~(((s[0] < 0) & (s[2] < 0)) | ((s[3] < 0) & (s[5] < 0)))
        for q in (0, 1):
            assert np.array_equal(fin(a[q]), fin(b[q])), q
        for q in (6, 7):
            assert np.array_equal(fin(a[q])[real], fin(b[q])[real]), q
        assert np.array_equal(fin(a[3:6]).all(0), fin(b[3:6]).all(0))     # the sampled state
        for q in range(5):
            assert np.array_equal(fin(f[q])[real], fin(g[q])[real]), q
        # p* to the parity tolerance where a factor 1e6 above vacuum (the root of a
        # near-vacuum is ill-conditioned), u* against the fastest speed
        ok = fin(b[0]) & fin(b[1]) & (b[2] == 0) & (b[0] > 1e-6 * np.maximum(s[2], s[5]))
        assert np.all(np.abs(a[0] - b[0])[ok] <= 1e-11 * b[0][ok])
        assert np.all(np.abs(a[1] - b[1])[ok] <= 1e-11 * cs[ok])
        scale = (rho * cs, rho * cs ** 2, rho * cs ** 2, rho * cs ** 2, rho * cs ** 3)
        for q in range(5):
            ok = real & fin(g[q]) & fin(scale[q])
            assert np.all(np.abs(f[q] - g[q])[ok] <= 1e-10 * scale[q][ok]), q
