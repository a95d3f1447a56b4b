"""Reading a split-precision state back: the nodal values are the FP64 sums of the average and the FP32 deviations, also
where a component's average is many binades below its deviations."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("k", [1, 2, 3])
@pytest.mark.parametrize("nx,ny", [(1, 1), (43, 9)])
def test_merge_is_the_fp64_sum(k, nx, ny):
    """The momenta's averages lie 2^0 .. 2^-50 (some are zero) below their deviations; deviation and mean are
    reproduced in FP32 as the kernels take them (dev the rounded difference to the average, the mean a sum of
    rounded products in node order), and every value read is their sum with the average, rounded once."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_16002_gb300 import build
    from paper_2412_16002_gb300.solver import Solver

    build()
    n = k + 1
    rng = np.random.default_rng(10 * nx + k)
    U = np.empty((4, ny, nx, n, n))
    U[0], U[3] = 1.0, 10.0
    w = np.outer(*(2 * [np.polynomial.legendre.leggauss(n)[1]])) / 4
    for c in (1, 2):
        d = 0.01 * rng.normal(size=(ny, nx, n, n))
        d -= (d * w).sum((-1, -2), keepdims=True)
        U[c] = d + 0.01 * 2.0 ** -rng.integers(0, 51, (ny, nx, 1, 1)) * rng.uniform(-1, 1, (ny, nx, 1, 1))
    U[1, 0, 0] = 0.0
    s = Solver(2, nx, ny, k, (0.0, 1.0, 0.0, 1.0), "euler", bc=("outflow",) * 4, precision="mixed")
    s.set_state(torch.from_numpy(U).cuda())
    out = s.get_state().reshape(U.shape)
    avg = np.moveaxis(s.averages().reshape(ny, nx, 4), -1, 0)[..., None, None]
    dev = (U - avg).astype(np.float32)
    w32 = w.astype(np.float32).ravel()
    flat = dev.reshape(4, ny, nx, n * n)
    mean = np.zeros((4, ny, nx), np.float32)
    for q in range(n * n):
        mean = mean + w32[q] * flat[..., q]
    ref = avg + (dev - mean[..., None, None]).astype(np.float64)
    assert mean.dtype == np.float32 and np.array_equal(out, ref)
