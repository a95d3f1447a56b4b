"""The trial-step rate that setting a split-precision state posts, against the scan of the same state."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("k", [1, 2, 3])
def test_rate_near_vacuum(k):
    """A density that falls to 2^-22 .. 2^-20 of the average at one side of the cell, where the FP32 screen clears the
    point and an FP32 sum has lost up to an eighth of it: both rates take the point's FP64 evaluation, so they differ
    by FP32 roundings of the speed only (eight of 2^-24)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_16002_gb300 import build
    from paper_2412_16002_gb300.solver import Solver

    build()
    n = k + 1
    rng = np.random.default_rng(k)
    x = np.polynomial.legendre.leggauss(n)[0]
    s = Solver(2, 1, 1, k, (0.0, 1.0, 0.0, 1.0), "euler", bc=("outflow",) * 4, precision="mixed")
    for i in range(40):
        u = np.empty((4, 1, 1, n, n))
        lowest = 2.0 ** rng.uniform(-21.9, -20.1)
        u[0] = rng.uniform(1.0, 2.0) * (1.0 + (1.0 - lowest) * (x if i % 2 else x[:, None]))
        u[1], u[2], u[3] = 1e-9 * rng.normal(), 1e-9 * rng.normal(), rng.uniform(1.0, 2.0)
        s.set_state(u)
        posted = s.max_dt(0.1)
        s.set_subdomain((0, 1, 0, 1))  # drops the posted rate
        assert abs(posted / s.max_dt(0.1) - 1.0) <= 8 * 2.0 ** -24, i
