"""The integer slope and quotient (csrc/fv_fixed.cuh, compiled for the host) on
what is not finite or not normal, as the binary64 operations they stand for give
it: a NaN difference gives a NaN slope whatever the signs, an infinite one with a
number of the other sign zero, a subnormal divisor NaN."""
import ctypes
import math
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2012_02925_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("nonfinite")
    src, so = str(d / "w.cpp"), str(d / "libw.so")
    with open(src, "w") as f:
        f.write('#include "fv_fixed.cuh"\n'
                'extern "C" double half_slope(double a, double b) { return fx_vanleer_half(a, b); }\n'
                'extern "C" double quotient(double n, double d) { return fx_div(n, d); }\n')
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, src, "-o", so])
    L = ctypes.CDLL(so)
    for f in (L.half_slope, L.quotient):
        f.argtypes, f.restype = [ctypes.c_double] * 2, ctypes.c_double
    return L


@pytest.mark.parametrize("other", [-math.inf, -1e300, -1.0, -1e-40, -0.0, 0.0, 1e-40, 1.0, 1e300, math.inf, math.nan])
def test_nan_difference(lib, other):
    for nan in (math.nan, -math.nan):
        assert math.isnan(lib.half_slope(nan, other)) and math.isnan(lib.half_slope(other, nan))


def test_infinite_difference(lib):
    for x in (1e-20, 1.0, 1e300):
        assert lib.half_slope(math.inf, -x) == 0.0 and lib.half_slope(x, -math.inf) == 0.0
        assert math.isnan(lib.half_slope(math.inf, x)) and math.isnan(lib.half_slope(-math.inf, -x))


@pytest.mark.parametrize("d", [5e-324, 1e-310, 2.2250738585072009e-308])
def test_subnormal_divisor(lib, d):
    assert math.isnan(lib.quotient(1.0, d)) and math.isnan(lib.quotient(0.0, d))
