"""The FP64 reciprocal, quotient and square root of the solver's kernels against CUDA's correctly rounded ones, and
the viscosity's series against the power in quadruple or extended precision.

Each ends in one rounding of a value that is exact to about 2^-80 (the residual of the last Newton step, or the
exact remainder), so a result can differ from the correctly rounded one only where the exact value lies that
near a midpoint between two doubles: never by more than one unit in the last place, and in far fewer than one
sample of a million."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from gpu_common import scaled_close
from oracle.oracle import Oracle
from paper_2310_18916_gb300 import build as B
from paper_2310_18916_gb300 import gsis
from paper_2310_18916_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
N = 1 << 22


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("fp64") / "libfp64_probe.so")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "fp64_device_probe.cu")
    subprocess.run([B.nvcc(), *B.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", B.CSRC, src, "-o", out], check=True)
    lib = C.CDLL(out)

    def run(which, x, y=None):
        x = np.ascontiguousarray(x, dtype=np.float64)
        y = np.ones_like(x) if y is None else np.ascontiguousarray(y, dtype=np.float64)
        own, ref = np.empty_like(x), np.empty_like(x)
        ptr = lambda a: a.ctypes.data_as(C.c_void_p)  # noqa: E731
        assert lib.fp64_probe(which, len(x), ptr(x), ptr(y), ptr(own), ptr(ref)) == 0
        return own, ref

    run.lib = lib
    return run


def _values(rng, lo, hi, n=N):
    """Random mantissas with exponents spread over [lo, hi)."""
    return np.ldexp(rng.uniform(1.0, 2.0, n), rng.integers(lo, hi, n))


def _check(own, ref, what):
    assert np.isfinite(ref).all()
    ulps = np.abs(own.view(np.int64) - ref.view(np.int64))
    assert ulps.max() <= 1, f"{what}: {ulps.max()} units in the last place"
    if len(ulps) > 1000:  # (a chosen value may be such a midpoint: 1 / (1 - 2^-53) = 1 + 2^-53 + 2^-106 + ...)
        assert (ulps > 0).mean() < 1e-6, f"{what}: {(ulps > 0).sum()} of {len(ulps)} differ"


def test_reciprocal(probe):
    rng = np.random.default_rng(1)
    edges = np.array([2.0 ** -1022, np.nextafter(2.0 ** 1022, 0.0), 1.0, np.nextafter(1.0, 2.0), np.nextafter(1.0, 0.0), -3.0])
    for x, what in ((rng.uniform(0.05, 20.0, N), "near 1"), (_values(rng, -1022, 1022), "all exponents"),
                    (-_values(rng, -40, 40), "negative"), (edges, "edges")):
        _check(*probe(0, x), f"reciprocal, {what}")


def test_quotient(probe):
    rng = np.random.default_rng(2)
    # 0 <= a <= b; the guard's threshold on b at 2^-1017, and below it down to the smallest normal number
    for lo, hi in ((-4, 4), (-900, 1021), (-1022, -1012)):
        b = _values(rng, lo, hi)
        a = b * rng.uniform(0.0, 1.0, N)
        if lo == -900:
            a = np.where(a < 2.0 ** -900, b, a)
        elif lo == -1022:
            b, a = b[b < 2.0 ** -1017], b[b < 2.0 ** -1017]  # (the plain division)
        _check(*probe(1, a, b), f"quotient, exponents {lo} to {hi}")
    _check(*probe(1, np.zeros(4), np.array([1.0, 2.0 ** -1022, 2.0 ** -1017, 2.0 ** 1000])), "zero numerator")


def test_square_root(probe):
    rng = np.random.default_rng(3)
    guard = [np.array([b], dtype=np.int64).view(np.float64)[0] for b in (0x1000000000000000, 0x6000000000000000)]
    edges = np.array([v for g in guard for v in (np.nextafter(g, 0.0), g, np.nextafter(g, np.inf))] + [0.0, 5e-324, 2.0 ** -1022, 4.0])
    for x, what in ((rng.uniform(0.05, 20.0, N), "near 1"), (_values(rng, -1022, 1023), "all exponents"), (edges, "edges")):
        _check(*probe(2, x), f"square root, {what}")


def test_limiter_of_tails_below_the_normal_numbers():
    """Squares of the VDF's tails and a vanishing limiter constant: the denominators stay in the reciprocal's range."""
    p = wl.couette(n_cells=6, nv=8)
    p.vx, p.wx = wl.midpoint_grid(40, -20.0, 20.0)
    W0 = wl.perturbed_state(p, seed=5, amp=0.02)
    g = gsis.Solver(p, precision="f64", mode="dvm", kinetic_presteps=0, init_W=W0, venkat_K=1e-103)
    o = Oracle(p, W0=W0, mode=1, venkat_K=1e-103)
    for _ in range(2):
        g.step()
        o.step()
    scaled_close(g.W(), o.W(), 1e-10, "W with a vanishing limiter constant")
    assert np.isfinite(g.get_f()).all()
    g.close()


# Bound, in 2^-53: CUDA's pow 2 ulp (4), the anchor's product and the last addition 1 each, the series at most six
# roundings of a sum that is at most e - 1 times the result (12), what it leaves out 2^-3 and a fall of the
# later terms by at most 1/2 each: 20 in all.
@pytest.mark.parametrize("omega", [0.0, 0.5, 0.74, 0.81, 1.0, 1.5, -0.5, -3.0, 6.5, 12.0, 30.0, -40.0, 1e4, 3e7])
def test_viscosity_for_any_exponent(probe, omega):
    rng = np.random.default_rng(4)
    n = 1 << 18
    span = min(1.0, 300.0 / max(abs(omega), 1e-9))  # |log T| of the anchors: T^omega stays in range
    T0 = np.exp(rng.uniform(-span, span, n))
    x = np.where(np.arange(n) % 4 == 0, rng.uniform(-0.5, 0.5, n), rng.uniform(-1.0, 1.0, n) * 2.0 ** -rng.integers(5, 24, n))
    T = T0 * (1.0 + (x if abs(omega) <= 40.0 else x / abs(omega)))
    own, ref = np.empty(n), np.empty(n)
    mu0 = 0.0564
    ptr = lambda a: a.ctypes.data_as(C.c_void_p)  # noqa: E731
    assert probe.lib.fp64_probe_viscosity(C.c_double(mu0), C.c_double(omega), n, ptr(T), ptr(T0), ptr(own), ptr(ref)) == 0
    for got, at, what in ((ref, T0, "the anchor"), (own, T, "its neighbourhood")):
        want = np.longdouble(mu0) * np.power(at.astype(np.longdouble), np.longdouble(omega))
        err = float((np.abs(got - want) / want).max())
        assert err <= 20 * 2.0 ** -53, f"omega {omega}: {err * 2.0 ** 53:.1f} x 2^-53 off at {what}"


@pytest.mark.parametrize("omega", [np.nan, np.inf])
def test_viscosity_of_no_number(probe, omega):
    T = np.array([0.5, 1.0, 2.0])
    own, ref = np.empty(3), np.empty(3)
    ptr = lambda a: a.ctypes.data_as(C.c_void_p)  # noqa: E731
    assert probe.lib.fp64_probe_viscosity(C.c_double(1.0), C.c_double(omega), 3, ptr(T), ptr(T), ptr(own), ptr(ref)) == 0
    assert np.array_equal(own, np.power(T, omega), equal_nan=True) and np.array_equal(ref, own, equal_nan=True)
