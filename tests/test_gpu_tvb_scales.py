"""The plain indicator's decisions where the averages around a cell, or a deviation and its threshold, differ by many
binades: those of FP64 arithmetic."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_16002_gb300 import build

    build()


@pytest.mark.parametrize("harvest", [False, True])
@pytest.mark.parametrize("k", [1, 2, 3])
def test_small_slopes_beside_a_large_average(k, harvest):
    """Columns with density and energy about 2^-30 and slopes of 2^-60 a cell, then a column of 1: half a slope is far
    above the threshold 2^-75 and FP64's rounding (2^-82), and below the differences of the averages on both
    sides, so no inner small cell is troubled.  In units of the large average (2^-58) the slopes vanish."""
    from paper_2412_16002_gb300.solver import Solver

    nx, ny, n = 7, 9, k + 1
    x = np.polynomial.legendre.leggauss(n)[0] / 2
    X = (np.arange(nx)[:, None] + x)[None, :, None, :]
    Y = (np.arange(ny)[:, None] + x)[:, None, :, None]
    s = 2.0 ** -30 * (1.0 + 2.0 ** -30 * (X + 0.9 * Y))
    s[:, -1] = 1.0
    U = np.stack([s, 0.5 * s, -0.25 * s, 2.0 * s])
    g = Solver(2, nx, ny, k, (0.0, 1.0 * nx, 0.0, 1.0 * ny), "euler", bc=("outflow",) * 4, indicator="tvb", tvb_M=2.0 ** -75)
    g.set_harvest(harvest)
    g.set_state(U)
    g.step(1e-60, "heun3")
    f = g.troubled_flags().reshape(ny, nx)
    assert not f[1:-1, 1:-1].any()
    assert f[:, 0].all()  # the difference to the left is zero


@pytest.mark.parametrize("k", [2, 3])
def test_constant_cells_without_a_threshold(k):
    """With M = 0 a constant cell is decided by the rounding of FP64's sums; in Q^2 and Q^3 the weights of the average and
    of both ends sum to 1 exactly, so a cell of powers of two is kept, by both kernels that decide (troubled-cell
    pass, features)."""
    from paper_2412_16002_gb300.solver import Solver

    nx, ny, n = 8, 5, k + 1
    U = np.empty((4, ny, nx, n, n))
    for c, f in enumerate((1.0, 0.5, -0.25, 2.0)):
        U[c] = f
    for harvest in (False, True):
        g = Solver(2, nx, ny, k, (0.0, 1.0 * nx, 0.0, 1.0 * ny), "euler", bc=("outflow",) * 4, indicator="tvb", tvb_M=0.0)
        g.set_harvest(harvest)
        g.set_state(U)
        g.step(1e-60, "heun3")
        assert not g.troubled_flags().any()
