"""Sums held as three floats (csrc/sums.cuh), compiled for the host: additions one by one and of sums, over
terms whose exponents spread as the steps of an adjoint do, against exact rational arithmetic."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1812_05264_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("sums")
    src = d / "sums.cpp"
    # lanes of n terms each, then the lanes' sums in a tree
    src.write_text('#include "sums.cuh"\nusing namespace tbk;\n'
                   'extern "C" double total(const float* x, int lanes, int n) {\n'
                   "  Sum3 s[64];\n"
                   "  for (int l = 0; l < lanes; ++l) {\n"
                   "    s[l].h = s[l].m = s[l].l = make_float2(0.f, 0.f);\n"
                   "    for (int i = 0; i < n; ++i) sum3_add(s[l], make_float2(0.f, x[l * n + i]));\n"
                   "  }\n"
                   "  for (int o = lanes / 2; o > 0; o /= 2)\n"
                   "    for (int l = 0; l < o; ++l) sum3_add(s[l], s[l + o]);\n"
                   "  return sum3_value(s[0].h.y, s[0].m.y, s[0].l.y);\n}\n")
    so = d / "libsums.so"
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, str(src), "-o",
                    str(so)], check=True)
    f = ctypes.CDLL(str(so)).total
    f.restype, f.argtypes = ctypes.c_double, [ctypes.c_void_p, ctypes.c_int, ctypes.c_int]
    return f


# An FP64 sum of N terms rounds N times; this one may round as an FP64 number once, 2^-53 of the result, beside N
# errors of 2^-72 of the magnitudes (two floats: 2^-47 of them, which these spreads reach)
@pytest.mark.parametrize("lanes,n", [(1, 1), (2, 3), (32, 1), (32, 16), (64, 257)])
@pytest.mark.parametrize("spread", [0, 10, 30, 60])
@pytest.mark.parametrize("cancel", [False, True])
def test_sum_of_three_floats(lib, lanes, n, spread, cancel):
    for seed in range(8):
        rng = np.random.default_rng(1000 * seed + spread)
        x = (rng.standard_normal(lanes * n) * 2.0 ** rng.uniform(-spread, 0, lanes * n)).astype(np.float32)
        if cancel and x.size > 1:
            x[x.size // 2:2 * (x.size // 2)] = -x[:x.size // 2]
            x[0] = np.float32(x[0] * (1 + 2.0 ** -20))
        got = lib(x.ctypes.data, lanes, n)
        exact = sum(Fraction(float(v)) for v in x)
        mag = sum(abs(Fraction(float(v))) for v in x)
        assert abs(Fraction(got) - exact) <= abs(exact) * Fraction(2.0 ** -52) + x.size * mag * Fraction(2.0 ** -71)
