"""The face corrections of 2D meshes (one thread per face point) where a mesh is one cell wide, wraps onto itself
or ends in a boundary, and a geometry word that only one side of a face has: F against the oracle, with the
tolerance of the operator parity tests."""
import numpy as np
import pytest

from gpu_helpers import pair, rel_linf
from paper_2412_16002_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
POST = (1.2, 0.3, -0.2, 3.0)
SIDES = {"periodic": ("periodic",) * 4, "tube": ("periodic", "periodic", "reflect", "outflow"),
         "closed": ("reflect", "outflow", "dirichlet", "reflect")}


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_16002_gb300 import build

    build()


def _F(g, U):
    x = torch.from_numpy(np.ascontiguousarray(U)).cuda()
    return g.apply("F", x, torch.empty_like(x)).cpu().numpy()


@pytest.mark.parametrize("k", [1, 2, 3])
@pytest.mark.parametrize("sides", list(SIDES))
@pytest.mark.parametrize("nx,ny", [(1, 1), (1, 4), (5, 1), (13, 11)])
def test_face_corrections(nx, ny, sides, k):
    bc = SIDES[sides]
    kw = {"bc_state": {2: list(POST)}} if "dirichlet" in bc else {}
    g, o = pair(2, nx, ny, k, (0.0, 1.0, 0.0, 2.0), "euler", bc=bc, **kw)
    U = inputs.random_euler(2, nx, ny, k, seed=3 * nx + k, osc=0.3)
    assert rel_linf(_F(g, U), o.to_nodal(o.apply("F", o.to_modal(U))), o.m) < 1e-12


def test_wall_on_one_side_of_a_face():
    """A wall word on one cell's left side leaves the other cell of that face with the neighbour's trace: every
    other cell's F is the plain mesh's to the bit."""
    from paper_2412_16002_gb300.solver import Solver

    nx, ny, k = 6, 3, 2
    U = inputs.random_euler(2, nx, ny, k, seed=1, osc=0.2)
    out = []
    for wall in (False, True):
        g = Solver(2, nx, ny, k, (0.0, 1.0, 0.0, 1.0), "euler")
        if wall:
            words = np.zeros((ny, nx), dtype=np.uint32)
            words[1, 3] = 1  # side 0: reflective wall
            g.set_geometry(words.ravel(), POST, POST, 0.0, 0.0)
        out.append(_F(g, U).reshape(4, ny, nx, -1))
    same = np.ones((ny, nx), dtype=bool)
    same[1, 3] = False
    assert np.array_equal(out[0][:, same], out[1][:, same])
    assert not np.array_equal(out[0][:, 1, 3], out[1][:, 1, 3]) and np.isfinite(out[1]).all()
