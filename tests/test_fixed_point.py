"""Fixed-point linear maps (csrc/dg_fixed.h, host form) against exact rational arithmetic."""
import ctypes as C
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_16002_gb300", "csrc")
SHIM = r"""
#include "dg_fixed.h"
using namespace crkdg;
extern "C" double fx_dot(const double *v, const double *c, int n, int k) {
    int E = 0;
    for (int i = 0; i < n; ++i) E = fx_exp(v[i]) > E ? fx_exp(v[i]) : E;
    FxSum s{0, 0};
    for (int i = 0; i < n; ++i) fx_mac(s, fx_of(v[i], E), fx_coef(c[i], k));
    return fx_double(fx_sum(s), fx_shift(E, k));
}
"""


@pytest.fixture(scope="module")
def fx(tmp_path_factory):
    d = tmp_path_factory.mktemp("fx")
    (d / "shim.cpp").write_text(SHIM)
    so = str(d / "shim.so")
    subprocess.run(["g++", "-O2", "-shared", "-fPIC", "-I", CSRC, str(d / "shim.cpp"), "-o", so], check=True)
    lib = C.CDLL(so)
    lib.fx_dot.restype = C.c_double
    lib.fx_dot.argtypes = [C.POINTER(C.c_double)] * 2 + [C.c_int] * 2
    return lambda v, c, k: lib.fx_dot(v.ctypes.data_as(C.POINTER(C.c_double)), c.ctypes.data_as(C.POINTER(C.c_double)),
                                      len(v), k)


@pytest.mark.parametrize("n,spread", [(2, 0), (4, 3), (12, 0), (12, 6), (16, 1)])
def test_sum_error_bound(fx, n, spread):
    """|error| <= 2^-53 |sum| (the final rounding) + (n + 2) 2^-58 max|v| sum|c|: a value and a coefficient are
    rounded to 2^-58 of the largest value and of the coefficients' sum, and the low products dropped and the
    final shift add less than 2^-58 of max|v| sum|c| together."""
    rng = np.random.default_rng(n + spread)
    for _ in range(300):
        v = rng.standard_normal(n) * 10.0 ** (spread * rng.uniform(-1, 1, n)) * 2.0 ** int(rng.integers(-140, 140))
        c = rng.standard_normal(n) * 50.0
        k = 58 - int(np.ceil(np.log2(np.abs(c).sum())))
        got = fx(v, c, k)
        exact = sum(Fraction(float(a)) * Fraction(float(b)) for a, b in zip(v, c))
        bound = abs(float(exact)) * 2.0 ** -53 + (n + 2) * 2.0 ** -58 * np.abs(v).max() * np.abs(c).sum()
        assert abs(float(Fraction(got) - exact)) <= bound


def test_zeros_and_extremes(fx):
    one = np.ones(4)
    assert fx(np.zeros(4), one, 55) == 0.0
    assert fx(np.array([-0.0, 0.0, 0.0, -0.0]), one, 55) == 0.0
    assert fx(np.array([3.0, -0.0, 0.0, 0.0]), one, 55) == 3.0
    assert fx(np.array([1.0, 1e-30, -1.0, 0.0]), one, 55) in (0.0, -(2.0 ** -58), 2.0 ** -58)
    for p in (-140, 140):  # the exponent only shifts the result
        v = np.array([0.3, -1.7, 0.011, 5.0])
        assert fx(v * 2.0 ** p, one, 55) == fx(v, one, 55) * 2.0 ** p
