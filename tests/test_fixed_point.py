"""The quantisation of csrc/quant.cuh, compiled for the host, against exact rationals, and that no
kernel rounds by a copy of its own."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1703_03637_gb300", "csrc")
SRC = """
#include "quant.cuh"
extern "C" void quant(const double* x, const int* e, long long* q, long n) {
  for (long i = 0; i < n; ++i) q[i] = hphi::quant_one(x[i], e[i]);
}
"""


@pytest.fixture(scope="module")
def quant(tmp_path_factory):
    d = tmp_path_factory.mktemp("quant")
    (d / "q.cpp").write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "q.so"), str(d / "q.cpp")],
                   check=True)
    lib = ctypes.CDLL(str(d / "q.so"))

    def call(x, e):
        q = np.empty(len(x), dtype=np.int64)
        lib.quant(x.ctypes.data_as(ctypes.c_void_p), e.ctypes.data_as(ctypes.c_void_p), q.ctypes.data_as(ctypes.c_void_p),
                  ctypes.c_long(len(x)))
        return q
    return call


def test_quantisation_rounds_to_nearest(quant):
    rng = np.random.default_rng(3)
    n = 4000
    field = rng.integers(1, 2047, n)
    below = rng.integers(0, 70, n).clip(0, field - 1)  # exponents up to 70 below the scale's
    x = np.ldexp(rng.uniform(1, 2, n) * rng.choice([-1, 1], n), field - below - 1023)
    x[:200] = np.ldexp(np.round(np.ldexp(x[:200], -(field - below - 1023)[:200]) * 64) / 64, (field - below - 1023)[:200])  # halves
    q = quant(x, field.astype(np.int32))
    for xi, e, qi in zip(x.tolist(), field.tolist(), q.tolist()):
        exact = Fraction(xi) * Fraction(2) ** (1078 - e)
        size = abs(exact)
        want = int(size + Fraction(1, 2))
        assert abs(qi) == want and (qi == 0 or (qi < 0) == (xi < 0)), (xi, e)
        assert abs(qi) < 1 << 56
    assert quant(np.array([0.0, -0.0, 5e-324]), np.array([1, 900, 1], dtype=np.int32)).tolist() == [0, 0, 0]


def test_one_rounding_for_every_kernel():
    own = [f for f in sorted(os.listdir(CSRC)) if f.endswith((".cu", ".cuh")) and "<< (sh - 1)" in open(os.path.join(CSRC, f)).read()]
    assert own == ["quant.cuh"]
