"""The inner stages of the split path by themselves (2D Euler, csrc/dg_line.cuh): the kernel is launched on given
averages and deviations, and its traces and u* are read, which no entry point returns."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SHIM = r"""
#include "dg_line.cuh"
#include <cstring>
using namespace crkdg;
// tableau: s, A[s][s], b[s]; state and results on the device
extern "C" int stages(int n, int nx, int ny, const double *tables, int s, const double *A, const double *b, double dt,
                      double rhx, double rhy, double eps, const double *ub, const float *dv, float *dv_s, float *tr,
                      float *tavg, int *flag, unsigned long long *nlim, unsigned long long *thmin) {
    if (n < 2 || n > 4 || s < 1 || s > MAXS) return -1;
    if (cudaMemcpyToSymbol(c_tab, tables, sizeof(NodalTables) * 3) != cudaSuccess) return -2;
    Params P;
    memset(&P, 0, sizeof(P));
    P.nx = nx, P.ny = ny, P.ncell = nx * ny;
    P.rhx = rhx, P.rhy = rhy, P.gamma = 1.4, P.eps = eps, P.dt = dt;
    P.s = s;
    for (int i = 0; i < s; ++i) {
        P.b[i] = b[i];
        for (int j = 0; j < s; ++j) P.A[i][j] = A[i * s + j];
        P.slot[i] = b[i] != 0.0 ? P.nslot++ : -1;
    }
    P.mode = MODE_STEP;
    tvb_thresholds(P);
    screen_bounds(P);
    fill_f32(P);
    MixBufs X;
    memset(&X, 0, sizeof(X));
    X.ub = ub, X.dv = dv, X.dv_s = dv_s, X.tr = tr, X.tavg = tavg, X.flag = flag, X.nlim = nlim, X.thmin = thmin;
    auto run = [&](auto k, int cpb, int smem) {
        if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) return -3;
        k<<<(P.ncell + cpb - 1) / cpb, pc::LT, smem>>>(P, X);
        return cudaGetLastError() == cudaSuccess && cudaDeviceSynchronize() == cudaSuccess ? 0 : -4;
    };
    if (n == 2) return run(k_inner_l<2>, pc::Line<2>::CPB, (int)sizeof(pc::LineSmem<2>));
    if (n == 3) return run(k_inner_l<3>, pc::Line<3>::CPB, (int)sizeof(pc::LineSmem<3>));
    return run(k_inner_l<4>, pc::Line<4>::CPB, (int)sizeof(pc::LineSmem<4>));
}
extern "C" int table_bytes() { return (int)(sizeof(NodalTables) * 3); }
"""
TABS = {"midpoint2": ([[0.0, 0.0], [0.5, 0.0]], [0.0, 1.0]), "euler1": ([[0.0]], [1.0])}


@pytest.fixture(scope="module")
def stages(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_16002_gb300 import _lib, build

    build()
    from paper_2412_16002_gb300.build import ARCH, CSRC, FLAGS, _nvcc

    d = tmp_path_factory.mktemp("stage")
    (d / "shim.cu").write_text(SHIM)
    so = str(d / "shim.so")
    r = subprocess.run([_nvcc(), *ARCH, *FLAGS, "-shared", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                        str(d / "shim.cu"), "-o", so], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    lib = C.CDLL(so)
    host = _lib.load()
    tables = (C.c_char * lib.table_bytes())()
    host._Z18crkdg_build_tablesPN5crkdg11NodalTablesE(tables)

    def run(k, nx, ny, tab, dt, rh, eps, ub, dv):
        """ub [4][ncell] float64, dv [4][ncell][nn] float32 -> u*'s deviations, traces [slot][4][ncell][4n], flag, limited"""
        n, A, b = k + 1, *TABS[tab]
        slots = sum(x != 0.0 for x in b)
        g = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
        u, v = g(ub), g(dv)
        out = torch.full_like(v, float("nan"))
        tr = torch.full((slots, 4, nx * ny, 4 * n), float("nan"), dtype=torch.float32, device="cuda")
        av = torch.full((slots, 4, nx * ny), float("nan"), dtype=torch.float32, device="cuda")
        sc = torch.zeros(4, dtype=torch.int64, device="cuda")
        A_, b_ = (np.ascontiguousarray(x, dtype=np.float64) for x in (A, b))
        p = lambda t: C.c_void_p(t.data_ptr())  # noqa: E731
        f = C.c_double
        rc = lib.stages(n, nx, ny, tables, len(b), A_.ctypes.data_as(C.c_void_p), b_.ctypes.data_as(C.c_void_p), f(dt),
                        f(rh[0]), f(rh[1]), f(eps), p(u), p(v), p(out), p(tr), p(av), p(sc), C.c_void_p(sc.data_ptr() + 8),
                        C.c_void_p(sc.data_ptr() + 16))
        assert rc == 0
        return out.cpu().numpy(), tr.cpu().numpy(), int(sc[0]), int(sc[1])

    return run


def _near_vacuum(k, ncell, seed):
    """Averages and deviations of nearly still gas whose density polynomial dips below eps in every cell."""
    rng = np.random.default_rng(seed)
    n = k + 1
    w = np.outer(*(2 * [np.polynomial.legendre.leggauss(n)[1]])).ravel() / 4
    ub = np.stack([rng.uniform(0.5, 2.0, ncell), 1e-9 * rng.normal(size=ncell), 1e-9 * rng.normal(size=ncell),
                   rng.uniform(1.0, 3.0, ncell)])
    dv = rng.normal(size=(4, ncell, n * n))
    dv -= (dv @ w)[..., None]
    dv[0] *= -2.0 * ub[0][:, None] / np.take_along_axis(dv[0], np.abs(dv[0]).argmax(-1)[:, None], -1)
    dv[1:3] *= 1e-10
    dv[3] *= 1e-3
    return ub, dv.astype(np.float32)


@pytest.mark.parametrize("k", [1, 2, 3])
@pytest.mark.parametrize("nx,ny", [(1, 1), (41, 3), (997, 11)])
def test_limited_traces_are_in_bounds(stages, k, nx, ny):
    """The traces of a limited stage are S_K points that the limiter verified: their density is the rounded value
    of one >= eps where the FP32 sum is ill-conditioned, positive elsewhere; and it is never put to eps, as
    the bound for points that were not verified would."""
    eps = 1e-13
    ub, dv = _near_vacuum(k, nx * ny, nx + k)
    _, tr, flag, limited = stages(k, nx, ny, "midpoint2", 1e-12, (2.0, 2.0), eps, ub, dv)
    rho = tr[0, 0]
    assert flag == 0 and limited > 0.9 * nx * ny and np.isfinite(tr).all()
    assert rho.min() >= np.float32(eps)
    assert not ((rho > 0) & (rho < 1.01 * eps)).any()
