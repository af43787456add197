"""The binary64 form's fixed-point Roe flux and integer slope quotient
(csrc/fv_fixed.cuh), compiled for the host: the flux against the oracle's
binary64 one, the slope against exact rationals.

Tolerance, derived before the first run: the oracle's ~130 binary64 operations
and its inputs' rounding leave at most ~16 units of 2^-53 of the flux's scale
S^a rho (S = max |u| + max c, a = 1, 2, 3), the fixed-point flux less; 4e-15
covers both."""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

import oracle
from cases.core import default_params

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2012_02925_gb300", "csrc")
WRAP = r'''
#include "fv_fixed.cuh"
extern "C" int fixed_roe(double gamma, double harten, int fix_all, const double* L, const double* R, const double* n,
                         double A, double* out) {
  const FxConsts c = fx_consts(gamma, harten);
  return c.on ? (int)fx_roe_flux(c, L, R, n[0], n[1], n[2], A, fix_all != 0, out) : -1;
}
extern "C" double half_slope(double a, double b) { return fx_vanleer_half(a, b); }
extern "C" double quotient(double n, double d) { return fx_div(n, d); }
'''


@pytest.fixture(scope="module")
def fixed(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixed")
    src, so = str(d / "w.cpp"), str(d / "libw.so")
    with open(src, "w") as f:
        f.write(WRAP)
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, src, "-o", so])
    L = ctypes.CDLL(so)
    dp = ctypes.POINTER(ctypes.c_double)
    L.fixed_roe.argtypes = [ctypes.c_double, ctypes.c_double, ctypes.c_int, dp, dp, dp, ctypes.c_double, dp]

    def call(VL, VR, n, A, gamma=1.4, harten=0.1, fix_all=0):
        a = [np.ascontiguousarray(x, dtype=np.float64) for x in (VL, VR, n)]
        out = np.full(5, np.nan)
        rc = L.fixed_roe(gamma, harten, fix_all, *(x.ctypes.data_as(dp) for x in a), A, out.ctypes.data_as(dp))
        return rc, out

    L.half_slope.argtypes = [ctypes.c_double] * 2
    L.half_slope.restype = ctypes.c_double
    call.slope = L.half_slope
    L.quotient.argtypes = [ctypes.c_double] * 2
    L.quotient.restype = ctypes.c_double
    call.quotient = L.quotient
    return call


def check(fixed, VL, VR, n, A, gamma=1.4, harten=0.1, fix_all=0):
    rc, got = fixed(VL, VR, n, A, gamma, harten, fix_all)
    if rc != 1:
        return False
    ref = oracle.roe_flux(default_params(gamma=gamma, harten=harten, fix_all=fix_all), VL, VR, np.asarray(n) * A)
    S = max(math.sqrt(V[1] ** 2 + V[2] ** 2 + V[3] ** 2) for V in (VL, VR)) + max(
        math.sqrt(gamma * V[4] / V[0]) for V in (VL, VR))
    scale = A * max(VL[0], VR[0]) * np.array([S, S * S, S * S, S * S, S ** 3])
    assert (np.abs(got - ref) <= 4e-15 * scale).all(), (VL, VR, n, A, got, ref)
    return True


def unit(v):
    v = np.asarray(v, dtype=float)
    return v / math.sqrt((v * v).sum())


@pytest.mark.parametrize("gamma", [1.3, 1.4, 5.0 / 3.0])
@pytest.mark.parametrize("mach,jump", [(0.05, 1e-6), (0.5, 0.01), (1.0, 0.1), (4.0, 0.05), (2.0, 0.3), (0.5, 0.0)])
def test_matches_the_binary64_flux(fixed, gamma, mach, jump):
    rng = np.random.default_rng(11)
    taken = 0
    for t in range(400):
        c0, r0 = 10.0 ** rng.uniform(-3, 3), 10.0 ** rng.uniform(-3, 3)
        d = unit(rng.uniform(-1, 1, 3))
        n = unit(rng.uniform(-1, 1, 3)) if t % 3 else np.eye(3)[t % 9 // 3] * (1 if t % 2 else -1)
        V = [np.concatenate([[r0 * (1 + jump * rng.uniform(-1, 1))],
                             c0 * (mach * d + jump * max(mach, 1.0) * rng.uniform(-1, 1, 3)),
                             [r0 * c0 * c0 / gamma * (1 + jump * rng.uniform(-1, 1))]]) for _ in range(2)]
        taken += check(fixed, V[0], V[1], n, 10.0 ** rng.uniform(-6, 6), gamma, 0.1 if t % 4 else 0.0, t % 2)
    assert taken >= 300 if jump < 0.3 else taken > 100


@pytest.mark.parametrize("below", [0, 1])
def test_at_the_edges_of_the_scales(fixed, below):
    """Density, area and velocity at and just below powers of two (where a
    significand's high half must not wrap), equal states, components that are
    zero, an eigenvalue inside the entropy fix."""
    eps = 1.0 - below * 2.0 ** -33
    for rho in (1.0, 2.0, 0.25, 1024.0):
        for A in (1.0, 2.0 ** -12, 4.0):
            for u in ((0.0, 0.0, 0.0), (0.5, 0.0, 0.0), (1.0, 1.0, 0.0), (math.sqrt(1.4 / rho) * 1.02, 0.0, 0.0)):
                V = np.array([rho * eps, *(x * eps for x in u), 1.0])
                W = V * np.array([1.0 + 1e-9, 1.0, 1.0, 1.0, 1.0 - 1e-9])
                for n in np.eye(3):
                    taken = check(fixed, V, V, n, A * eps) and check(fixed, V, W, n, A * eps)
                    assert taken or V[1] ** 2 + V[2] ** 2 > 64 * 1.4 * V[4] / V[0]   # Mach 8
    # a component that is zero in both states and in the normal stays zero
    rc, out = fixed([1.0, 0.3, 0.1, 0.0, 0.7], [1.1, 0.2, 0.2, 0.0, 0.8], [0.6, 0.8, 0.0], 1.0)
    assert rc == 1 and out[3] == 0.0


def test_refuses_what_does_not_fit(fixed):
    base = np.array([1.0, 0.3, 0.2, 0.1, 0.7])
    for v, bad in [(0, x) for x in (np.nan, np.inf, 0.0, -1.0, 1e-300, 8.0)] + [
            (4, x) for x in (np.nan, np.inf, 0.0, -1.0, 1e300, 1e-40)] + [
            (1, x) for x in (np.nan, np.inf, -np.inf, 1e300, 200.0)]:
        for side in (0, 1):
            V = [base.copy(), base.copy()]
            V[side][v] = bad
            assert fixed(V[0], V[1], [1.0, 0.0, 0.0], 1.0)[0] == 0, (v, bad)
    for n in ([np.nan, 0.0, 0.0], [2.5, 0.0, 0.0]):
        assert fixed(base, base, n, 1.0)[0] == 0
    for A in (0.0, np.nan, np.inf, -1.0):
        assert fixed(base, base, [1.0, 0.0, 0.0], A)[0] == 0
    assert fixed(base, base, [1.0, 0.0, 0.0], 1.0, gamma=1.1)[0] == -1
    assert fixed(base, base, [1.0, 0.0, 0.0], 1.0, harten=0.01)[0] == -1


def test_half_slope(fixed):
    """a b / (a + b) of differences with the same sign, else 0, within one
    unit in the last place of the exact quotient (rationals)."""
    from fractions import Fraction
    f = fixed.slope
    rng = np.random.default_rng(5)
    edge = [1.0, 2.0, 1.0 - 2.0 ** -53, 2.0 - 2.0 ** -52, 1.5, 1.0 + 2.0 ** -52]
    pairs = [(a * 2.0 ** i, b) for a in edge for b in edge for i in (0, 1, 10, 53, 62, 63, 64, 70)]
    pairs += [(x, y) for x, y in zip(rng.uniform(0.5, 2, 3000) * 2.0 ** rng.integers(-40, 40, 3000),
                                     rng.uniform(0.5, 2, 3000))]
    for a, b in pairs:
        for x, y in ((a, b), (b, a), (-a, -b)):
            want = Fraction(x) * Fraction(y) / (Fraction(x) + Fraction(y))
            got = f(x, y)
            assert abs(Fraction(got) - want) <= Fraction(float(np.spacing(abs(float(want))))), (x, y, got)
        assert f(a, -b) == 0.0 and f(-a, b) == 0.0
    assert f(0.0, 1.0) == 0.0 and f(1.0, 0.0) == 0.0 and f(0.0, 0.0) == 0.0
    assert f(4e-31, 4e-31) == 0.0 and f(1e-300, 1.0) <= 1e-300
    for bad in (np.nan, np.inf):
        assert np.isnan(f(bad, 1.0)) and np.isnan(f(1.0, bad))


def test_quotient(fixed):
    """n / d, d > 0, within one unit in the last place over binary64's normal
    range; zero, overflow and what is not finite."""
    f = fixed.quotient
    rng = np.random.default_rng(6)
    edge = [1.0, 2.0, 1.0 - 2.0 ** -53, 2.0 - 2.0 ** -52, 1.5, 1.0 + 2.0 ** -52]
    pairs = [(a * 2.0 ** i, b * 2.0 ** j) for a in edge for b in edge for i in (-500, 0, 500) for j in (-500, 0, 500)]
    pairs += list(zip(rng.uniform(-2, 2, 4000), rng.uniform(1e-3, 2, 4000)))
    for n, d in pairs:
        assert abs(f(n, d) - n / d) <= np.spacing(abs(n / d)), (n, d)
    assert f(0.0, 3.0) == 0.0 and f(1e300, 1e-300) == np.inf and f(-1e300, 1e-300) == -np.inf
    assert f(1e-300, 1e300) == 0.0 and f(1.7e308, 1.0) == 1.7e308
    for n, d in ((np.nan, 1.0), (1.0, np.nan), (np.inf, 1.0), (1.0, np.inf), (1.0, 0.0), (1.0, -1.0)):
        assert np.isnan(f(n, d))
