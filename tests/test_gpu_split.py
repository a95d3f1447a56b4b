"""Setting and reading a split-precision state (2D Euler, one thread per cell) at meshes that end inside a
warp, a block and a row: the state read back is ubar + (dev - dbar) with dev rounded once to FP32 and dbar
its FP32 mean over up to 16 nodes, so it is within 20 * 2^-24 of the cell's largest deviation of the state
set (1 for the deviation, 1 for the difference, at most 17 for dbar, which is 0 in exact arithmetic), plus
2^-51 of the cell's magnitude for the FP64 average and sum.  Components differ by
many binades, some cells are constant, one has zero and tiny momenta."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("k", [1, 2, 3])
@pytest.mark.parametrize("nx,ny", [(1, 1), (5, 3), (33, 1), (16, 8), (43, 9)])
def test_set_get_round_trip(k, nx, ny):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_16002_gb300 import build
    from paper_2412_16002_gb300.solver import Solver

    build()
    n = k + 1
    rng = np.random.default_rng(100 * nx + 10 * ny + k)
    shape = (ny, nx, n, n)
    cell = (ny, nx, 1, 1)
    rho = 10.0 ** rng.uniform(-6, 3, cell) * (1.0 + 0.05 * rng.uniform(-1, 1, shape))
    p = 10.0 ** rng.uniform(-4, 4, cell) * (1.0 + 0.05 * rng.uniform(-1, 1, shape))
    # slow against the sound speed: nothing is limited
    w = [0.1 * np.sqrt(p / rho) * 10.0 ** rng.uniform(-9, 0, cell) * rng.uniform(-1, 1, shape) for _ in range(2)]
    for a in (rho, p):
        a[0, 0] = a[0, 0, 0, 0]
    w[0][0, 0], w[1][0, 0] = 0.0, 1e-42
    u = np.stack([rho, rho * w[0], rho * w[1], p / 0.4 + 0.5 * rho * (w[0] ** 2 + w[1] ** 2)])
    s = Solver(dim=2, nx=nx, ny=ny, k=k, flux="euler", domain=(0.0, 1.0, 0.0, 1.0), bc=("outflow",) * 4, eps=1e-13,
               precision="mixed")
    s.set_state(torch.from_numpy(u).cuda())
    out = np.asarray(s.get_state()).reshape(u.shape)
    xg, wg = np.polynomial.legendre.leggauss(n)
    w2 = np.outer(wg, wg) / 4
    bar = (u * w2).sum((-1, -2), keepdims=True)
    dev = np.abs(u - bar).max((-1, -2), keepdims=True)
    tol = 20 * 2.0 ** -24 * dev + 2.0 ** -51 * np.abs(u).max((-1, -2), keepdims=True)
    assert np.all(np.abs(out - u) <= tol)
