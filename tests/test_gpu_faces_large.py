"""The faces' corrections in a pass of their own, which 2D meshes take from 6400 cells on (Q^1 65536): the same bits as
the final stage alone (F without a handle), on meshes one cell wide, wrapped onto themselves, bounded, and with
geometry words."""
import ctypes as C

import numpy as np
import pytest

from paper_2412_16002_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
STATE = [1.2, 0.3, -0.2, 3.0]
SIDES = {"periodic": ("periodic",) * 4, "tube": ("periodic", "periodic", "reflect", "outflow"),
         "closed": ("reflect", "outflow", "dirichlet", "reflect")}


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_16002_gb300 import build

    build()


def _sizes(k):
    return [(1, 65539), (65539, 1), (263, 251)] if k == 1 else [(1, 6403), (6403, 1), (83, 79)]


def _state(flux, nx, ny, k):
    if flux == "euler":
        return inputs.random_euler(2, nx, ny, k, seed=nx + k, osc=0.3)
    return inputs.random_scalar(2, nx, ny, k, seed=nx + k, lo=-1.0, hi=1.0)


def _F(g, U):
    x = torch.from_numpy(np.ascontiguousarray(U)).cuda()
    return g.apply("F", x, torch.empty_like(x)).cpu().numpy()


@pytest.mark.parametrize("shape", [0, 1, 2])
@pytest.mark.parametrize("k", [1, 2, 3])
@pytest.mark.parametrize("flux", ["euler", "burgers"])
@pytest.mark.parametrize("sides", list(SIDES))
def test_face_pass_has_the_bits_of_the_final_stage(sides, flux, k, shape):
    from paper_2412_16002_gb300 import _lib as L
    from paper_2412_16002_gb300.solver import Solver

    nx, ny = _sizes(k)[shape]
    bc = SIDES[sides]
    if flux == "burgers":
        bc = tuple("outflow" if b == "reflect" else b for b in bc)
    m = 4 if flux == "euler" else 1
    U = _state(flux, nx, ny, k)
    g = Solver(2, nx, ny, k, (0.0, 1.0, 0.0, 2.0), flux, bounds=(-2.0, 2.0), bc=bc, bc_state={s: STATE[:m] for s in range(4)})
    got = _F(g, U)
    mesh = L.Mesh()
    mesh.dim, mesh.nx, mesh.ny = 2, nx, ny
    mesh.x0, mesh.x1, mesh.y0, mesh.y1 = 0.0, 1.0, 0.0, 2.0
    for s in range(4):
        mesh.bc[s] = L.BC[bc[s]]
        for c in range(m):
            mesh.bc_state[s][c] = STATE[c]
    fl = L.Flux(L.FLUX[flux], 1.4, (C.c_double * 2)(1.0, 0.0))
    x = torch.from_numpy(np.ascontiguousarray(U)).cuda()
    out = torch.empty_like(x)
    rc = L.load().crkdg_apply_F_noalloc(C.byref(mesh), k, m, C.byref(fl), C.c_void_p(x.data_ptr()), C.c_void_p(out.data_ptr()),
                                        C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == L.OK
    assert np.isfinite(got).all() and np.array_equal(got, out.cpu().numpy())


@pytest.mark.parametrize("k", [2, 3])
def test_geometry_word_on_one_side(k):
    """Words on two cells of a mesh with the pass: F of a window of the mesh, too small for the pass and with the same
    cell sizes and words, has the same bits inside; other cells keep the plain mesh's."""
    from paper_2412_16002_gb300.solver import Solver

    nx, ny, i0, j0, wx, wy = 83, 79, 30, 40, 9, 7
    U = _state("euler", nx, ny, k)
    U = U.reshape(4, ny, nx, k + 1, k + 1)
    words = np.zeros((ny, nx), dtype=np.uint32)
    words[j0 + 3, i0 + 4] = 1  # side 0: reflective wall
    words[j0 + 2, i0 + 6] = 3 << 12  # side 3: state A
    h = 1.0 / 64
    full = Solver(2, nx, ny, k, (0.0, nx * h, 0.0, ny * h), "euler", bc=("outflow",) * 4)
    plain = _F(full, U)
    full.set_geometry(words.ravel(), STATE, STATE, 0.0, 0.0)
    got = _F(full, U)
    part = Solver(2, wx, wy, k, (0.0, wx * h, 0.0, wy * h), "euler", bc=("outflow",) * 4)
    part.set_geometry(words[j0:j0 + wy, i0:i0 + wx].ravel(), STATE, STATE, 0.0, 0.0)
    small = _F(part, U[:, j0:j0 + wy, i0:i0 + wx])
    inner = (slice(None), slice(1, -1), slice(1, -1))
    assert np.array_equal(got[:, j0:j0 + wy, i0:i0 + wx][inner], small.reshape(4, wy, wx, k + 1, k + 1)[inner])
    same = words == 0
    assert np.array_equal(got[:, same], plain[:, same]) and not np.array_equal(got[:, ~same], plain[:, ~same])
