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


def _line(n):
    """Dhat, the end values of the basis and the Gauss weights on [-1, 1]."""
    x, w = np.polynomial.legendre.leggauss(n)
    inv = np.linalg.inv(np.polynomial.legendre.legvander(x, n - 1))
    at = lambda y: np.polynomial.legendre.legvander(np.array([y]), n - 1)[0] @ inv  # noqa: E731
    der = np.stack([np.polynomial.legendre.legval(x, np.polynomial.legendre.legder(np.eye(n)[j])) for j in range(n)], 1) @ inv
    return der.T * w[None, :] / w[:, None], at(-1.0), at(1.0), w


def _flux(u, d):
    w = u[1 + d] / u[0]
    p = 0.4 * (u[3] - 0.5 * (u[1] ** 2 + u[2] ** 2) / u[0])
    return np.stack([u[1 + d], u[1] * w + (p if d == 0 else 0), u[2] * w + (p if d == 1 else 0), (u[3] + p) * w])


@pytest.mark.parametrize("k,node", [(2, 4), (3, 5), (3, 10)])
def test_flux_of_an_ill_conditioned_node(stages, k, node):
    """A node with density 2^-30 and momentum 2^-16 beside averages of about 1: its flux is that of the FP64 state, so
    u* is within 64 roundings of 2^-24 of the terms' magnitudes of the FP64 evaluation (2 n + 4 products, n^2 terms
    of the mean, and the well-conditioned fluxes' own roundings); an FP32 momentum there is wrong by 2^-9."""
    n, ncell, rh = k + 1, 300, (2.0, 3.0)
    rng = np.random.default_rng(node)
    dv = 0.1 * rng.normal(size=(4, ncell, n * n))
    dv[0] = 0.6 + 0.05 * rng.normal(size=dv[0].shape)
    dv = dv.astype(np.float32)
    dv[:3, :, node] = -rng.uniform(0.5, 0.99, (3, ncell)).astype(np.float32)
    ub = np.empty((4, ncell))
    ub[0] = -dv[0, :, node].astype(np.float64) + 2.0 ** -30 * rng.uniform(1.0, 2.0, ncell)
    ub[1:3] = -dv[1:3, :, node].astype(np.float64) + 2.0 ** -16 * rng.uniform(0.5, 1.0, (2, ncell))
    ub[3] = rng.uniform(2.0, 3.0, ncell)
    got, _, _, _ = stages(k, 60, 5, "euler1", 1.0, rh, 1e-13, ub, dv)
    D, lm, lp, w = _line(n)
    u = (ub[..., None] + dv).reshape(4, ncell, n, n)  # [b][a]
    G, S = np.zeros_like(u), np.zeros_like(u)
    for d in range(2):
        at = (lambda M, v: v @ M.T) if d == 0 else (lambda M, v: np.moveaxis(np.moveaxis(v, -2, -1) @ M.T, -1, -2))
        ends = (lambda l: u @ l) if d == 0 else (lambda l: np.moveaxis(u, -2, -1) @ l)
        spread = (lambda f, l: f[..., None] * l) if d == 0 else (lambda f, l: f[..., None, :] * l[:, None])
        f, fm, fp = _flux(u, d), _flux(ends(lm), d), _flux(ends(lp), d)
        G += rh[d] * (at(D, f) + spread(fm, lm / w) - spread(fp, lp / w))
        S += rh[d] * (at(np.abs(D), np.abs(f)) + spread(np.abs(fm), np.abs(lm / w)) + spread(np.abs(fp), np.abs(lp / w)))
    w2 = np.outer(w, w) / 4
    mean = lambda v: (v * w2).sum((-1, -2), keepdims=True)  # noqa: E731
    ref = dv + (G - mean(G)).reshape(dv.shape)
    tol = 64 * 2.0 ** -24 * (np.abs(dv) + (S + mean(S)).reshape(dv.shape))
    assert np.isfinite(got).all() and (np.abs(got - ref) <= tol).all()
