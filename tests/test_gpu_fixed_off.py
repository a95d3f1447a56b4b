"""Problems outside the range of the fixed-point G (gamma >= 2, cell sizes beyond 2^100): the FP64 form for every cell,
against the oracle with the tolerance of the operator parity tests."""
import numpy as np
import pytest

from gpu_helpers import ORACLE_TABS, pair, rel_linf
from paper_2412_16002_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_16002_gb300 import build

    build()


def _same(g, o, U, limit):
    x = torch.from_numpy(np.ascontiguousarray(U)).cuda()
    for op in ("G", "F"):
        got = g.apply(op, x, torch.empty_like(x)).cpu().numpy()
        assert rel_linf(got, o.to_nodal(o.apply(op, o.to_modal(U))), o.m) < limit


@pytest.mark.parametrize("k", [1, 2, 3])
@pytest.mark.parametrize("dim,nx,ny", [(1, 67, 1), (2, 13, 11), (2, 1, 7)])
@pytest.mark.parametrize("gamma", [2.0, 2.2, 1.9999999])
def test_gamma(dim, nx, ny, k, gamma):
    bc = ("dirichlet", "reflect", "outflow", "outflow")
    kw = {"bc_state": {0: [1.1, 0.2, -0.1, 2.3] if dim == 2 else [1.1, 0.2, 2.3]}}
    g, o = pair(dim, nx, ny, k, (0.0, 1.0, 0.0, 2.0), "euler", gamma=gamma, bc=bc, **kw)
    U = inputs.random_euler(dim, nx, ny, k, seed=nx + k, osc=0.2)
    _same(g, o, U, 1e-12)
    g.set_state(U)
    o.set_state(U)
    dt = o.max_dt(0.05)
    g.step(dt, "rk4")
    assert o.step(dt, ORACLE_TABS["rk4"])[0] == 0
    assert rel_linf(g.get_state(), o.get_state(), o.m) < 1e-12


@pytest.mark.parametrize("k", [1, 2, 3])
@pytest.mark.parametrize("flux", ["euler", "burgers", "advection"])
def test_tiny_cells(flux, k):
    g, o = pair(2, 7, 5, k, (0.0, 1e-32, 0.0, 2e-32), flux, bounds=(-2.0, 2.0))
    U = inputs.random_euler(2, 7, 5, k, seed=k, osc=0.3) if flux == "euler" else inputs.random_scalar(2, 7, 5, k, seed=k, lo=-1.0, hi=1.0)
    _same(g, o, U, 1e-12)


def test_ensemble_gamma():
    """Members of an ensemble at gamma = 2.2 step as the same problems alone, to the bit."""
    from paper_2412_16002_gb300.ensemble import Ensemble
    from paper_2412_16002_gb300.solver import Solver

    sizes = [(11, 9, 2, "heun3"), (17, 6, 3, "rk4")]
    e = Ensemble([dict(nx=nx, ny=ny, k=k, tableau=t, cfl=0.05) for nx, ny, k, t in sizes], gamma=2.2)
    alone = []
    for i, (nx, ny, k, _) in enumerate(sizes):
        g = Solver(2, nx, ny, k, (0.0, 1.0, 0.0, 1.0), "euler", gamma=2.2, bc=("outflow",) * 4)
        U = inputs.random_euler(2, nx, ny, k, seed=i, osc=0.2)
        g.set_state(U)
        e.set_state(i, U)
        alone.append(g)
    for _ in range(2):
        for g, (_, _, _, t) in zip(alone, sizes):
            g.step(g.max_dt(0.05), t)
        e.step()
    for i, g in enumerate(alone):
        assert np.array_equal(e.get_state(i), g.get_state())


@pytest.mark.parametrize("k", [1, 2, 3])
def test_step_loop_gamma(k):
    """The 1D loop at gamma = 2.2 against single steps of the same size, within the rounding of their sums (the
    tolerance of the operator parity tests)."""
    from paper_2412_16002_gb300.solver import Solver

    U = inputs.random_euler(1, 70, 1, k, seed=k, osc=0.2)
    loop, single = (Solver(1, 70, 1, k, (0.0, 1.0), "euler", gamma=2.2) for _ in range(2))
    loop.set_state(U)
    single.set_state(U)
    dt = 0.2 * loop.max_dt(0.1)
    loop.advance_fixed(3, dt, 1e30, "rk4")
    for _ in range(3):
        single.step(dt, "rk4")
    assert rel_linf(loop.get_state(), single.get_state(), 3) < 1e-12
