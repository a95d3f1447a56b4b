"""Handles and ensembles on a device that is nearly full: what needs more memory than the traces (face corrections, flux
sums and radii) is left out, and the states keep their bits."""
import numpy as np
import pytest

from paper_2412_16002_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
MB = 1 << 20


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_16002_gb300 import build

    build()


class _Leave:
    """Holds all device memory but about `keep` bytes."""

    def __init__(self, keep):
        self.keep = keep

    def __enter__(self):
        torch.cuda.empty_cache()
        free = torch.cuda.mem_get_info()[0]
        self.hold = torch.empty(free - self.keep, dtype=torch.uint8, device="cuda")

    def __exit__(self, *a):
        del self.hold
        torch.cuda.empty_cache()


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_handle_without_face_corrections():
    """Q^2 with the midpoint rule (one traced stage): state and traces take 8 (3 m nn + m (1 + ntr) + m ntr + 4) bytes a
    cell, the corrections 8 m ntr more; with room for the former only, a step runs and has the bits of one with room
    for both."""
    from paper_2412_16002_gb300.solver import Solver

    n, k = 1000, 2
    U = torch.from_numpy(np.broadcast_to(inputs.random_euler(2, n, 1, k, seed=1, osc=0.2), (4, n, n, 3, 3)).copy()).cuda()
    cells, m, nn, ntr = n * n, 4, 9, 12
    need = 8 * cells * (3 * m * nn + m + m * (1 + ntr) + m * ntr + 4)
    out = []
    for keep in (need + 8 * cells * m * ntr + 512 * MB, need + 96 * MB):
        with _Leave(keep):
            g = Solver(2, n, n, k, (0.0, 1.0, 0.0, 1.0), "euler", bc=("outflow",) * 4)
            g.set_state(U)
            free = _free()
            g.step(1e-5, "midpoint2")
            used = free - _free()
        out.append((used, g.get_state()))
        g.close()
    assert out[1][0] < out[0][0] - 0.9 * 8 * cells * m * ntr  # the corrections are not there
    assert np.array_equal(out[0][1], out[1][1])


@pytest.mark.parametrize("indicator", ["off", "tvb"])
def test_ensemble_without_flux_sums(indicator):
    """Between room for the traces alone and room for everything, creating and stepping work at every amount, with the
    same bits."""
    from paper_2412_16002_gb300.ensemble import Ensemble, riemann_problem

    sizes = [(400, 3), (301, 2)]
    probs = [dict(riemann_problem(0, n, k), t_end=1e30) for n, k in sizes]
    states = [torch.from_numpy(inputs.riemann_quadrants(i, n, k).state).cuda() for i, (n, k) in enumerate(sizes)]

    def run():
        e = Ensemble(probs, indicator=indicator)
        for i, s in enumerate(states):
            e.set_state(i, s)
        e.step()
        e.step()
        used = _free()
        got = [e.get_state(i) for i in range(len(states))]
        e.close()
        return got, used

    run()  # modules are loaded
    before = _free()
    want, used = run()
    full = before - used
    extra = 0
    for n, k in sizes:
        stages = 4 if k == 3 else 2
        extra += 8 * n * n * (4 * 4 * (k + 1) + 4 * stages)
    for keep in np.linspace(full - extra + 32 * MB, full + 320 * MB, 9):
        with _Leave(int(keep)):
            got, _ = run()
        for a, b in zip(got, want):
            assert np.array_equal(a, b), keep / MB
