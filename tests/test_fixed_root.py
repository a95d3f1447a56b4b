"""The integer root of the sound speed (csrc/dg_fixed.h, host form) against integer square roots: within 2^-57 of
itself (floors of at most eight units of 2^-60, and e^3 below 2^-63), for mantissas of 1 to 62 bits."""
import ctypes as C
import math
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_16002_gb300", "csrc")
SHIM = r"""
#include "dg_fixed.h"
extern "C" long long fx_root_of(long long v, int x, int *xr) { return crkdg::fx_root(v, x, *xr); }
"""


@pytest.fixture(scope="module")
def root(tmp_path_factory):
    d = tmp_path_factory.mktemp("fx")
    (d / "shim.cpp").write_text(SHIM)
    so = str(d / "shim.so")
    subprocess.run(["g++", "-O2", "-shared", "-fPIC", "-I", CSRC, str(d / "shim.cpp"), "-o", so], check=True)
    lib = C.CDLL(so)
    lib.fx_root_of.restype = C.c_longlong
    lib.fx_root_of.argtypes = [C.c_longlong, C.c_int, C.POINTER(C.c_int)]

    def f(v, x):
        xr = C.c_int()
        return lib.fx_root_of(v, x, C.byref(xr)), xr.value

    return f


def test_root_error_bound(root):
    rng = np.random.default_rng(0)
    values = [1, 2, 3, 4, (1 << 61) - 1, 1 << 61, (1 << 62) - 1] + [1 << k for k in range(62)]
    values += [int(rng.integers(1, 1 << 62)) >> int(rng.integers(0, 62)) or 1 for _ in range(4000)]
    for v in values:
        for x in (-301, -300, 0, 1, 250):
            m, xr = root(v, x)
            # (m 2^(xr - 61))^2 = v 2^(x - 61): both as integers over 2^s
            s = 2 * (xr - 61) - (x - 61)
            exact = math.isqrt(v << (-s + 80)) if -s + 80 >= 0 else None  # root of v 2^-s, times 2^40
            assert exact is not None and abs((m << 40) - exact) <= (exact >> 57) + 1, (v, x)
    assert root(0, 5)[0] == 0
