"""The gradient kernel at the edges of its 64-sample tiles: one sample, a tile less and more than one
sample, several tiles per block with a ragged last one, and buffers off the 16-byte alignment.

Tolerance: every gradient entry is a sum over samples of products of sums of at most 64 FP32 terms, three
layers deep, so it is within about 3 * 64 * 2^-24 = 1.2e-5 of the sum of its terms' magnitudes; held to
1e-4 of the FP64 sum of the magnitudes' largest entry, the loss to 1e-5 of itself.  The buffers are added
to: a second call doubles them."""
import ctypes as C

import numpy as np
import pytest

from oracle import mlp

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,offset", [(1, 0), (63, 0), (64, 1), (65, 0), (300, 3), (152 * 64 * 4 + 37, 0)])
def test_gradient_tiles(n, offset):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_16002_gb300 import _lib as L
    from paper_2412_16002_gb300 import build

    build()
    lib = L.load()
    rng = np.random.default_rng(n)
    theta = mlp.init_params(9)
    X, y = rng.normal(size=(n, 44)), (rng.uniform(size=n) > 0.5).astype(float)

    def put(a):  # on the device, `offset` floats past an aligned address
        t = torch.zeros(a.size + offset, dtype=torch.float32, device="cuda")[offset:]
        return t.copy_(torch.as_tensor(np.ravel(a), dtype=torch.float32))

    tp, tx, ty, gr, ls = put(theta), put(X), put(y), put(np.zeros(mlp.NPARAM)), put(np.zeros(1))
    ptr = [C.c_void_p(t.data_ptr()) for t in (tp, tx, ty, gr, ls)]
    Xf, tf = tx.cpu().numpy().reshape(n, 44).astype(float), tp.cpu().numpy().astype(float)
    gref, lref = mlp.backward(tf, Xf, y), mlp.loss(tf, Xf, y)
    for times in (1, 2):
        assert lib.crkdg_mlp_grad(*ptr[:3], n, *ptr[3:], None) == 0
        torch.cuda.synchronize()
        assert np.abs(gr.cpu().numpy() - times * gref).max() <= 1e-4 * times * np.abs(gref).max()
        assert abs(float(ls.item()) - times * lref) <= 1e-5 * times * max(1.0, lref)
