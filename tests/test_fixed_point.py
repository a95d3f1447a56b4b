"""Fixed-point linear maps (csrc/dg_fixed.h, host form) against exact rational arithmetic."""
import ctypes as C
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_16002_gb300", "csrc")
_LIB = []
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
extern "C" void fx_euler(const double *u, double gamma, double *f) {
    FxGas gas;
    gas.g1 = fx_limb(llrint(ldexp(gamma - 1.0, 62)));
    gas.g = fx_limb(llrint(ldexp(gamma, 61)));
    FxPoint<2> o;
    fx_point<2>(u, gas, o);
    for (int d = 0; d < 2; ++d) {
        f[4 * d] = u[1 + d];
        f[4 * d + 1 + d] = fx_value(o.q[d] + o.p, o.X);
        f[4 * d + 2 - d] = fx_value(o.c, o.X);
        f[4 * d + 3] = fx_value(fx_energy_flux<2>(o, d), o.X + o.xw[d] + 1);
    }
    f[8] = fx_value(o.r, -o.xr);
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
    lib.fx_euler.argtypes = [C.POINTER(C.c_double), C.c_double, C.POINTER(C.c_double)]
    _LIB.append(lib)
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


@pytest.mark.parametrize("kind", ["plain", "cold", "still", "light", "scaled", "inadmissible"])
def test_euler_flux_error_bound(fx, kind):
    """The fluxes within 2^-53 of themselves (the final rounding) plus 2^-57 of max(E, |m|^2 / rho) (energy: times
    |w|): eight operations that each keep 2^-60 of the largest term; the reciprocal within 2^-53 + 2^-58."""
    rng = np.random.default_rng(3)
    for _ in range(400):
        rho, w, p = np.exp(rng.normal()), rng.normal(size=2), np.exp(rng.normal())
        if kind == "cold":
            p = 1e-11
        if kind == "still":
            w = np.array([0.0, -0.0])
        if kind == "light":
            rho = 1e-12
        E = p / 0.4 + 0.5 * rho * (w @ w)
        if kind == "inadmissible":
            E *= rng.uniform(0.01, 0.5)
        u = np.array([rho, rho * w[0], rho * w[1], E]) * (2.0 ** int(rng.integers(-100, 100)) if kind == "scaled" else 1.0)
        f = np.zeros(9)
        dp = lambda x: x.ctypes.data_as(C.POINTER(C.c_double))  # noqa: E731
        _LIB[0].fx_euler(dp(u), 1.4, dp(f))
        r, mx, my, e = (Fraction(float(x)) for x in u)
        pr = Fraction(1.4 - 1.0) * (e - (mx * mx + my * my) / (2 * r))
        top = max(e, (mx * mx + my * my) / r)
        for d, m in enumerate((mx, my)):
            exact = [m, mx * m / r + (pr if d == 0 else 0), my * m / r + (pr if d == 1 else 0), (e + pr) * m / r]
            for c in range(4):
                slack = top * (abs(m) / r if c == 3 else 1) * Fraction(2) ** -57
                assert abs(Fraction(float(f[4 * d + c])) - exact[c]) <= abs(exact[c]) * Fraction(2) ** -53 + slack, (kind, c)
        assert abs(Fraction(float(f[8])) * r - 1) <= Fraction(2) ** -53 + Fraction(2) ** -58
