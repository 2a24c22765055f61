"""Sums of double-float slots (csrc/fsum.h, compiled for the host): against exact rationals, to the bound of a
three-word sum, which a sum kept in double-float words does not hold."""
import ctypes
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1908_07392_gb300", "csrc")
HARNESS = """
#include "fsum.h"
extern "C" long long sum3(int n, const float* x, int* e) {
  vp::Sum3 s;
  for (int i = 0; i < n; ++i) s.add(x[2 * i], x[2 * i + 1]);
  s.normalise();
  *e = s.exponent();
  return s.fixed(*e == vp::kSumZero ? 0 : *e);
}
extern "C" double sum2(int n, const float* x) {
  float hi = 0.f, lo = 0.f;
  for (int i = 0; i < 2 * n; ++i) {
    float s, e;
    vp::two_sum(hi, x[i], s, e);
    const float l = lo + e;
    hi = s + l;
    lo = l - (hi - s);
  }
  return (double)hi + (double)lo;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("fsum")
    (d / "h.cpp").write_text(HARNESS)
    subprocess.check_call([cxx, "-std=c++17", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, "-o",
                           str(d / "h.so"), str(d / "h.cpp")])
    lib = ctypes.CDLL(str(d / "h.so"))
    lib.sum3.restype, lib.sum3.argtypes = ctypes.c_longlong, [ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p]
    lib.sum2.restype, lib.sum2.argtypes = ctypes.c_double, [ctypes.c_int, ctypes.c_void_p]
    return lib


def sum3(lib, x):
    """(value, exponent, fixed-point integer) of the slots x [n][2]."""
    e = ctypes.c_int()
    v = lib.sum3(len(x), x.ctypes.data_as(ctypes.c_void_p), ctypes.byref(e))
    return Fraction(v) * Fraction(2) ** ((e.value if v else 0) - 62), e.value, v


def double_float(v):
    h = v.astype(np.float32)
    return np.stack([h, (v - h).astype(np.float32)], axis=-1)


# n slots of one size, or spread over 12 decades, or cancelling to their last digits, or tiny (the low words denormal): the
# head of fsum.h's bound, and a unit of 2^(e - 62) per word; the integer uses 62 bits, whatever lies just below a power
# of two
@pytest.mark.parametrize("kind", ["even", "spread", "cancel", "tiny"])
@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 28, 40])
def test_sum_of_slots(lib, n, kind):
    rng = np.random.default_rng(n)
    beyond = 0
    for _ in range(300):
        v = rng.standard_normal(n)
        if kind == "spread":
            v *= 10.0 ** rng.uniform(-12, 0, n)
        if kind == "cancel" and n > 1:
            v[n // 2:2 * (n // 2)] = -v[:n // 2] * (1 + 1e-9 * rng.standard_normal(n // 2))
        if kind == "tiny":
            v *= 2.0 ** -100
        x = np.ascontiguousarray(double_float(v))
        exact = sum((Fraction(float(q)) for q in x.reshape(-1)), Fraction(0))
        M = sum(abs(Fraction(float(q))) for q in x.reshape(-1))
        value, e, fixed = sum3(lib, x)
        bound = M * 8 * Fraction(n) ** 3 / 2 ** 72 + 3 * Fraction(2) ** (e - 62)
        assert abs(value - exact) <= bound
        assert 2 ** 61 - 3 <= abs(fixed) <= 2 ** 62
        beyond += abs(Fraction(lib.sum2(n, x.ctypes.data_as(ctypes.c_void_p))) - exact) > bound
    assert n <= 2 or kind == "tiny" or beyond > 30   # the bound tells a double-float sum apart


def test_powers_of_two_zero_and_overflow(lib):
    f = np.float32
    for k in (-100, -3, 0, 5, 90):
        p = f(2.0 ** k)
        for low, e in ((0.0, k + 1), (2.0 ** (k - 26), k + 1), (-2.0 ** (k - 26), k)):
            for sign in (1, -1):
                x = np.array([[sign * p, sign * low]], f)
                value, got, fixed = sum3(lib, x)
                assert got == e and value == sign * (Fraction(float(p)) + Fraction(low))
    assert sum3(lib, np.zeros((3, 2), f))[2] == 0
    assert sum3(lib, np.array([[1.5, 0], [-1.5, 0]], f))[2] == 0
    assert sum3(lib, np.array([[2.0 ** -149, 0]], f))[:2] == (Fraction(1, 2 ** 149), -148)
    for bad in ([[np.inf, 0]], [[np.nan, 0]], [[3e38, 0], [3e38, 0]]):
        assert sum3(lib, np.array(bad, f))[2] == 0
