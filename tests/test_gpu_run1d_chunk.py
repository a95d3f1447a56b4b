"""The chunk of the 1D step loop: every size that a block holds is accepted and gives the same bits; larger ones are
refused."""
import numpy as np
import pytest

from paper_2412_16002_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("k,largest", [(1, 30), (2, 38), (3, 30)])
def test_largest_chunks(k, largest):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_16002_gb300 import build
    from paper_2412_16002_gb300._lib import CrkdgError
    from paper_2412_16002_gb300.solver import Solver

    build()
    wl = inputs.euler_blast_tube(317, k)
    out = []
    for chunk in (0, largest, largest - 1, 31 if largest > 31 else 29):
        g = Solver.from_workload(wl)
        g.set_state(wl.state)
        g.set_run1d_chunk(chunk)
        out.append((g.advance(20, wl.cfl, 1e30, wl.tableau), g.get_state().copy()))
    for run, state in out[1:]:
        assert run == out[0][0] and np.array_equal(state, out[0][1])
    for chunk in (largest + 1, -1):
        with pytest.raises(CrkdgError):
            g.set_run1d_chunk(chunk)
