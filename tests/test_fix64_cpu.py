"""The FP64 products' integer helpers (csrc/fix64.cuh, compiled for the host) against exact rational
arithmetic: nine balanced digits represent round(x 2^(P - e)), and the recombination rounds the exact
92-bit sum to FP64 once, ties to even."""
import ctypes
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = """
#define __host__
#define __device__
#define __forceinline__ inline
#include "fix64.cuh"
extern "C" {
void digits(double x, int pe, int* d) {
  const uint64_t v = qtx::fix_biased(x, pe);
  for (int i = 0; i < qtx::kDig64; ++i) d[i] = (int)qtx::digit_field(v, i) - 64;
}
int expo(double x) { return qtx::expo64(x); }
double fixsum(long long a, long long b) { return qtx::fix_sum(a, b); }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("g++ not found")
    d = tmp_path_factory.mktemp("fix64")
    (d / "f.cpp").write_text(SRC)
    so = d / "f.so"
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2606_25595_gb300", "csrc"), str(d / "f.cpp"), "-o", str(so)], check=True)
    L = ctypes.CDLL(str(so))
    L.digits.argtypes = [ctypes.c_double, ctypes.c_int, ctypes.POINTER(ctypes.c_int)]
    L.expo.argtypes = [ctypes.c_double]
    L.fixsum.argtypes = [ctypes.c_longlong, ctypes.c_longlong]
    L.fixsum.restype = ctypes.c_double
    return L


@pytest.mark.parametrize("P", [61, 62])
def test_digits_represent_the_scaled_value(lib, P):
    rng = np.random.default_rng(3)
    d = (ctypes.c_int * 9)()
    xs = np.concatenate([rng.standard_normal(400) * 2.0 ** rng.integers(-80, 80, 400),
                         [1.0, -1.0, np.nextafter(1.0, 0), -np.nextafter(2.0, 0), 5e-324, -2.2e-308, 1.7e308, 0.0, -0.0]])
    for x in xs:
        e = lib.expo(float(x))
        if x != 0:
            assert abs(Fraction(float(x))) < Fraction(2) ** e
        for gap in (0, 1, 9, 40, 200):  # the row's largest entry is 2^gap larger
            er = e + gap if x != 0 else 0
            lib.digits(float(x), P - er, d)
            assert all(-64 <= v <= 64 for v in d)
            v = sum(int(d[i]) * 128 ** (8 - i) for i in range(9))
            exact = Fraction(float(x)) * Fraction(2) ** (P - er)
            assert abs(Fraction(v) - exact) <= Fraction(1, 2), (x, gap)


def test_sum_is_rounded_once(lib):
    rng = np.random.default_rng(4)

    def rn(fr):  # round to nearest even at 53 bits (Fraction -> float is correctly rounded)
        return float(fr)

    for _ in range(4000):
        na, nb = int(rng.integers(0, 53)), int(rng.integers(0, 47))
        a = int(rng.integers(-2 ** na, 2 ** na + 1))
        b = int(rng.integers(-2 ** nb, 2 ** nb + 1))
        assert lib.fixsum(a, b) == rn(Fraction(a * 2 ** 28 + b, 2 ** 56))
    for a in (0, 1, -1, 2 ** 52, -2 ** 52 + 1, 2 ** 51 + 1):  # ties, carries and cancellations
        for b in (0, 1, -1, 2 ** 27, -2 ** 27, 2 ** 28 - 1, -2 ** 28, 2 ** 27 + 1, 2 ** 46, -2 ** 46):
            assert lib.fixsum(a, b) == rn(Fraction(a * 2 ** 28 + b, 2 ** 56)), (a, b)
