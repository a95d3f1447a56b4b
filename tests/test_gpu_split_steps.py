"""Steps of the split path of 2D Euler (the kernels by lines and by cells) at every degree, on meshes that end inside a
warp and inside a block (64 cells in Q^1 and Q^3, 40 in Q^2), against the FP64 oracle."""
import numpy as np
import pytest

from gpu_helpers import ORACLE_TABS, pair, rel_linf
from paper_2412_16002_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
TAB = {1: "midpoint2", 2: "heun3", 3: "rk4"}


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_16002_gb300 import build

    build()


@pytest.mark.parametrize("sides", ["periodic", "closed"])
@pytest.mark.parametrize("k", [1, 2, 3])
@pytest.mark.parametrize("nx,ny", [(1, 1), (39, 1), (41, 3), (13, 11), (1, 65)])
def test_steps_match_the_oracle(nx, ny, k, sides):
    """Three steps, each within the error of the FP32 operators (2e-5 of the largest value of F, and dt F is below the
    state) of the oracle's; the averages are conserved where nothing leaves the mesh."""
    bc = ("periodic",) * 4 if sides == "periodic" else ("reflect", "outflow", "dirichlet", "reflect")
    kw = {"bc_state": {2: [1.2, 0.3, -0.2, 3.0]}} if sides == "closed" else {}
    g, o = pair(2, nx, ny, k, (0.0, 1.0 * nx, 0.0, 1.0 * ny), "euler", bc=bc, precision="mixed", **kw)
    U = inputs.random_euler(2, nx, ny, k, seed=nx + 10 * k, osc=0.1)
    g.set_state(U)
    o.set_state(U)
    m0 = [g.mass(c) for c in range(4)]
    for i in range(3):
        dt = 0.5 * o.max_dt(0.1)
        ig = g.step(dt, TAB[k])
        rc, io = o.step(dt, ORACLE_TABS[TAB[k]])
        assert rc == 0 and ig["restarts"] == io["restarts"]
        assert g.margins().min() >= 0.0
        assert rel_linf(g.get_state(), o.get_state(), 4) < 2e-5 * (i + 1)
    if sides == "periodic":
        for c in range(4):
            assert abs(g.mass(c) - m0[c]) <= 1e-13 * max(1.0, abs(m0[c]))


@pytest.mark.parametrize("n,M", [(33, 0.0), (21, 1.0)])
def test_q1_decisions_are_the_fp64_decisions(n, M):
    """Q^1: the flags that the troubled-cell pass takes from its FP32 screen are those of the FP64 feature kernel on the
    merged values, and the states keep the same bits."""
    from paper_2412_16002_gb300.solver import Solver

    wl = inputs.riemann_quadrants(3, n, 1, cfl=0.3)
    a, b = (Solver.from_workload(wl, precision="mixed", indicator="tvb", tvb_M=M) for _ in range(2))
    b.set_harvest(True)
    for s in (a, b):
        s.set_state(wl.state)
    flagged = 0
    for _ in range(12):
        dt = a.max_dt(wl.cfl)
        ia, ib = a.step(dt, "midpoint2"), b.step(dt, "midpoint2")
        fa, fb = a.troubled_flags(), b.troubled_flags()
        assert np.array_equal(fa, fb) and ia["troubled"] == ib["troubled"] == int(fa.sum())
        flagged += int(fa.sum())
    assert flagged > 0 and np.array_equal(a.get_state(), b.get_state())
