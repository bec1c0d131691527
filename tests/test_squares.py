"""The integer sum of squares of csrc/squares.cuh, compiled for the host, against exact rationals
(the start norms of single-precision Lanczos and mTPQ runs)."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1703_03637_gb300", "csrc")
SRC = """
#include "squares.cuh"
extern "C" void groups(const float* x, double* out, long n) {
  for (long i = 0; i < n; ++i) out[i] = hphi::sum_squares<8>(x + 8 * i);
}
"""


@pytest.fixture(scope="module")
def groups(tmp_path_factory):
    d = tmp_path_factory.mktemp("squares")
    (d / "s.cpp").write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "s.so"), str(d / "s.cpp")],
                   check=True)
    lib = ctypes.CDLL(str(d / "s.so"))

    def call(x):
        x = np.ascontiguousarray(x, dtype=np.float32)
        out = np.empty(len(x))
        lib.groups(x.ctypes.data_as(ctypes.c_void_p), out.ctypes.data_as(ctypes.c_void_p), ctypes.c_long(len(x)))
        return out
    return call


def _cases(what):
    rng = np.random.default_rng(7)
    x = rng.standard_normal((3000, 8)).astype(np.float32)
    if what == "spread":  # exponents far apart, zeros and subnormals among them
        x = np.ldexp(x, rng.integers(-70, 60, x.shape)).astype(np.float32)
        x[:, 3] = 0
        x[::2, 5] = 1e-41
    elif what == "close":  # a few bits apart: every shift up to the dropped bits
        x = np.ldexp(x, -rng.integers(0, 33, x.shape)).astype(np.float32)
    elif what == "small":  # either side of the lower limit, down to subnormals only
        x = np.ldexp(x, rng.integers(-150, -60, (len(x), 1))).astype(np.float32)
        x[0] = 0
    elif what == "large":
        x = np.ldexp(x, 124).astype(np.float32)
    return x


@pytest.mark.parametrize("what", ["normal", "spread", "close", "small", "large"])
def test_sum_of_squares_rounds_once(groups, what):
    """At most seven values lose less than 2^-58 of the largest square each, then one rounding: less
    than (2^-53 + 2^-55) of the sum.  Groups on the fp64 sum round at most eight times."""
    x = _cases(what)
    for got, g in zip(groups(x), x):
        exact = sum((Fraction(float(v)) ** 2 for v in g), Fraction(0))
        fast = np.max(np.abs(g)) >= 2.0 ** -63
        bound = (Fraction(1, 2 ** 53) + Fraction(1, 2 ** 55)) if fast else Fraction(8, 2 ** 53)
        assert abs(Fraction(float(got)) - exact) <= bound * exact


def test_sum_of_squares_of_non_finite_values(groups):
    x = np.ones((3, 8), dtype=np.float32)
    x[0, 2], x[1, 7], x[2, 0], x[2, 1] = np.inf, np.nan, -np.inf, np.nan
    out = groups(x)
    assert out[0] == np.inf and np.isnan(out[1]) and np.isnan(out[2])
