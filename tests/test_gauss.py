"""The integer Box-Muller transform of csrc/gauss.cuh, compiled for the host, against the
transform in extended precision on the same fp64 uniforms (appendix A.2 / A.4 start vectors)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1703_03637_gb300", "csrc")
SRC = """
#include "gauss.cuh"
static constexpr hphi::GaussTables T = hphi::gauss_detail::make_tables();
extern "C" void pairs(const uint64_t* a, const uint64_t* b, double* g0, double* g1, long n) {
  for (long i = 0; i < n; ++i) hphi::gauss_pair(a[i], b[i], T, g0[i], g1[i]);
}
"""


@pytest.fixture(scope="module")
def pairs(tmp_path_factory):
    d = tmp_path_factory.mktemp("gauss")
    (d / "g.cpp").write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "g.so"), str(d / "g.cpp")],
                   check=True)
    lib = ctypes.CDLL(str(d / "g.so"))

    def call(a, b):
        g = np.empty((2, len(a)))
        lib.pairs(a.ctypes.data_as(ctypes.c_void_p), b.ctypes.data_as(ctypes.c_void_p),
                  g[0].ctypes.data_as(ctypes.c_void_p), g[1].ctypes.data_as(ctypes.c_void_p), ctypes.c_long(len(a)))
        return g
    return call


def _edges(what):
    rng = np.random.default_rng(5)
    top = 1 << 53
    if what == "uniform":
        return rng.integers(0, top, 200000, dtype=np.uint64)
    small = [int(rng.integers(0, 1 << int(e))) if e else 0 for e in rng.integers(0, 53, 4000)]
    if what == "ends":  # u next to 0, to 1/2 and to 1
        v = small + [top - 1 - x for x in small] + [(1 << 52) + x // 2 for x in small] + [(1 << 52) - 1 - x // 2 for x in small]
    elif what == "centres":  # the borders and centres of the logarithm's table, at every exponent
        v = [(((256 << 1) + j) << 43 >> int(e)) + d for j in range(512) for e in rng.integers(0, 30, 4) for d in (-1, 0, 1)]
    else:  # octants and the borders of the table angles
        v = [(q << 44) + (x >> 10) * (1 if x & 1 else -1) for q, x in zip(rng.integers(0, 513, 4000).tolist(), small)]
    return np.array([min(max(x, 0), top - 1) for x in v], dtype=np.uint64)


@pytest.mark.parametrize("what", ["uniform", "ends", "centres", "angles"])
def test_pairs_against_extended_precision(pairs, what):
    if np.finfo(np.longdouble).nmant < 63:
        pytest.skip("long double is no wider than double here")
    a = _edges(what)
    b = a[::-1].copy()
    g = pairs(a, b)
    L = np.longdouble
    ua, ub = ((x.astype(np.float64) + 0.5).astype(L) / L(2) ** 53 for x in (a, b))
    rad = np.sqrt(-2 * np.log1p(ua - 1))
    # angle reduced to [-1/8, 1/8] turns first, exactly
    quad = np.rint(4 * ub)
    x = (ub - quad / 4) * (2 * L("3.14159265358979323846264338327950288"))
    c, s = np.cos(x), np.sin(x)
    q = quad.astype(int) % 4
    cos = np.choose(q, [c, -s, -c, s])
    sin = np.choose(q, [s, c, -s, -c])
    for got, ref in zip(g, (rad * cos, rad * sin)):
        # one rounding to fp64, and the fixed-point error: -ln u above 2^-10 carries 2^-61.4
        # (2^-52.4 of the radius), below it the series is relative; cos and sin 2^-60
        bound = 0.5 * np.spacing(np.abs(ref).astype(np.float64)) + L(2) ** -52 * np.abs(rad)
        assert np.all(np.abs(got.astype(L) - ref) <= bound)


@pytest.mark.parametrize("what", ["uniform", "ends", "centres", "angles"])
def test_pairs_relative_to_each_number(pairs, what):
    """Each number within 3 2^-53 of itself: the final rounding, half of the 2^-52 by which the
    logarithm may be off, and 2^-60 of the radius on components of at least pi / 256 (0.64 2^-53);
    components next to an axis keep their relative accuracy."""
    if np.finfo(np.longdouble).nmant < 63:
        pytest.skip("long double is no wider than double here")
    a = _edges(what)
    for b in (a[::-1].copy(), np.roll(a, 7)):
        L = np.longdouble
        ua, ub = ((x.astype(np.float64) + 0.5).astype(L) / L(2) ** 53 for x in (a, b))
        rad = np.sqrt(-2 * np.log1p(ua - 1))
        quad = np.rint(4 * ub)
        x = (ub - quad / 4) * (2 * L("3.14159265358979323846264338327950288"))
        c, s = np.cos(x), np.sin(x)
        q = quad.astype(int) % 4
        for got, ref in zip(pairs(a, b), (rad * np.choose(q, [c, -s, -c, s]), rad * np.choose(q, [s, c, -s, -c]))):
            assert np.all(np.abs(got.astype(L) - ref) <= 3 * L(2) ** -53 * np.abs(ref))


def test_pairs_stay_inside_the_language(tmp_path):
    """Every 53-bit word is defined behaviour, the one that rounds to u = 1 (radius zero) included;
    the largest word below it is not."""
    top = (1 << 53) - 1
    words = [0, 1, top, top - 1, top - 2, 1 << 52, (1 << 52) - 1, 12345678901]
    main = SRC + "#include <cstdio>\nint main() { const uint64_t w[] = {" + ", ".join(f"{w}ull" for w in words) + "};\n" \
        "  for (uint64_t a : w) for (uint64_t b : w) { double g[2]; pairs(&a, &b, g, g + 1, 1);" \
        " std::printf(\"%d\", (g[0] != 0) + 2 * (g[1] != 0)); } }\n"
    (tmp_path / "m.cpp").write_text(main)
    exe = str(tmp_path / "m")
    subprocess.run(["g++", "-O1", "-std=c++17", "-fsanitize=undefined", "-fno-sanitize-recover=undefined", "-I", CSRC, "-o", exe, str(tmp_path / "m.cpp")], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0 and not r.stderr, r.stderr
    n = len(words)
    zero = [set(r.stdout[n * k:n * k + n]) == {"0"} for k in range(n)]
    assert zero == [w == top for w in words]
