"""Warps whose cells do not fill their lanes (Q^2: 27 of 32 in the FP64 kernels, 30 of 32 in the split ones): the
lanes left over shadow the last cell's last thread.  A cell's result must not depend on its place in the warp."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_2412_16002_gb300 import inputs  # noqa: E402

STATE = [1.1, 0.2, -0.1, 2.3]


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_16002_gb300 import build

    build()


def _thin(U, dim):
    """Every third cell near vacuum at one node (the FP64 form of the fluxes), its neighbours not."""
    V = U.reshape(U.shape[0], -1, (U.shape[-1] ** dim))
    V[0, ::3, -1] *= 2.0 ** -24
    return U


@pytest.mark.parametrize("k", [1, 2, 3])
@pytest.mark.parametrize("nx,ny", [(3, 1), (4, 3), (13, 11), (31, 7)])
def test_face_sums_on_every_lane(nx, ny, k):
    """F without a handle (fluxes formed in the final kernel) has the bits of F with one (stored flux sums): the
    sums are formed once per face point, from the same values in the same order."""
    from paper_2412_16002_gb300 import _lib as L
    from paper_2412_16002_gb300.solver import Solver

    lib = L.load()
    bc = ("dirichlet", "outflow", "reflect", "dirichlet")
    g = Solver(2, nx, ny, k, (0.0, 1.0, 0.0, 2.0), "euler", bc=bc, bc_state={s: STATE for s in range(4)})
    x = torch.from_numpy(_thin(inputs.random_euler(2, nx, ny, k, seed=nx + k, osc=0.2), 2)).cuda()
    ref = g.apply("F", x, torch.empty_like(x))
    mesh = L.Mesh()
    mesh.dim, mesh.nx, mesh.ny = 2, nx, ny
    mesh.x0, mesh.x1, mesh.y0, mesh.y1 = 0.0, 1.0, 0.0, 2.0
    for s in range(4):
        mesh.bc[s] = L.BC[bc[s]]
        for c in range(4):
            mesh.bc_state[s][c] = STATE[c]
    fl = L.Flux(L.FLUX["euler"], 1.4, (C.c_double * 2)(0.0, 0.0))
    out = torch.empty_like(x)
    rc = lib.crkdg_apply_F_noalloc(C.byref(mesh), k, 4, C.byref(fl), C.c_void_p(x.data_ptr()),
                                   C.c_void_p(out.data_ptr()), C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == L.OK
    assert torch.isfinite(out).all() and torch.equal(out, ref)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("k", [1, 2, 3])
@pytest.mark.parametrize("thin", [False, True])
def test_equal_cells_stay_equal(precision, k, thin):
    """A periodic mesh of equal cells: after a step all cells have the same bits."""
    from paper_2412_16002_gb300.solver import Solver

    nx, ny = 29, 11
    one = inputs.random_euler(2, 1, 1, k, seed=k, osc=0.2)
    if thin:
        one[0, 0, 0, 0, 0] *= 2.0 ** -24
    U = np.ascontiguousarray(np.broadcast_to(one, (4, ny, nx, k + 1, k + 1)))
    g = Solver(2, nx, ny, k, (0.0, 1.0, 0.0, 1.0 * ny / nx), "euler", precision=precision)
    g.set_state(torch.from_numpy(U).cuda())
    g.step(g.max_dt(0.05), "rk4")
    V = g.get_state().reshape(4, ny * nx, -1)
    assert np.isfinite(V).all() and np.array_equal(V, np.broadcast_to(V[:, :1], V.shape))
