"""The fixed-point G of the FP64 path: its fallback to the FP64 form and the ragged ends of its warps."""
import numpy as np
import pytest

from gpu_helpers import pair, rel_linf
from paper_2412_16002_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_16002_gb300 import build

    build()


def _apply(g, op, U):
    x = torch.from_numpy(np.ascontiguousarray(U)).cuda()
    return g.apply(op, x, torch.empty_like(x)).cpu().numpy()


@pytest.mark.parametrize("k", [1, 2, 3])
@pytest.mark.parametrize("dim,nx,ny", [(1, 1, 1), (1, 129, 1), (2, 1, 1), (2, 3, 1), (2, 13, 11), (2, 5, 33)])
def test_ragged_meshes(dim, nx, ny, k):
    """Cells that do not fill the last warp or block (tolerance of the operator parity tests)."""
    g, o = pair(dim, nx, ny, k, (0.0, 1.0, 0.0, 2.0), "euler")
    U = inputs.random_euler(dim, nx, ny, k, seed=nx + k, osc=0.3)
    for op in ("G", "F"):
        assert rel_linf(_apply(g, op, U), o.to_nodal(o.apply(op, o.to_modal(U))), o.m) < 1e-12


@pytest.mark.parametrize("k", [2, 3])
@pytest.mark.parametrize("dim", [1, 2])
def test_scaled_states(dim, k):
    """G is homogeneous: scaling the state by 2^p scales G by 2^p, to the bit while the exponents stay in the
    fixed-point range and within rounding (2^-48 of the largest value, 2^5 FP64 roundings) beyond it."""
    g, o = pair(dim, 6, 5, k, (0.0, 1.0, 0.0, 1.0), "euler")
    U = inputs.random_euler(dim, 6, 5, k, seed=k, osc=0.3)
    ref = _apply(g, "G", U)
    for p in (-120, -31, 40, 120):
        assert np.array_equal(_apply(g, "G", U * 2.0 ** p), ref * 2.0 ** p)
    for p in (-200, 200):
        assert rel_linf(_apply(g, "G", U * 2.0 ** p) * 2.0 ** -p, ref, o.m) < 2.0 ** -48


@pytest.mark.parametrize("k", [2, 3])
@pytest.mark.parametrize("dim", [1, 2])
def test_near_vacuum_and_nonfinite(dim, k):
    """Cells with a density 2^-20 below their neighbours' nodes, zero momentum, a subnormal momentum, a negative
    density and a NaN take the FP64 form: the oracle's values where they are finite, NaN where it has NaN."""
    g, o = pair(dim, 9, 4 if dim == 2 else 1, k, (0.0, 1.0, 0.0, 1.0), "euler")
    U = inputs.random_euler(dim, 9, 4 if dim == 2 else 1, k, seed=k, osc=0.2)
    cell = (lambda i: (slice(None), 0, i)) if dim == 2 else (lambda i: (slice(None), i))
    first = (0,) * dim
    U[cell(1)][(0,) + first] = 2.0 ** -22
    U[cell(3)][1] = 0.0
    U[cell(4)][(1,) + first] = 5e-310
    U[cell(6)][(0,) + first] = -0.5
    ref = o.to_nodal(o.apply("G", o.to_modal(U)))
    got = _apply(g, "G", U)
    for i in range(9):  # per cell, against the cell's own scale: the near-vacuum cells have huge fluxes
        a, b = got[cell(i)], ref[cell(i)]
        # the oracle's modal round trip moves the small density by about 2^-50 of the cell's largest, 2^-28 of
        # itself, and the flux m^3 / rho^2 by three times that
        assert np.abs(a - b).max() <= (3 * 2.0 ** -28 if i == 1 else 1e-11) * np.abs(b).max()
    U[cell(7)][(0,) + first] = np.nan
    got = _apply(g, "G", U)
    assert np.isnan(got[cell(7)]).any() and np.isfinite(got[cell(0)]).all() and np.isfinite(got[cell(8)]).all()
