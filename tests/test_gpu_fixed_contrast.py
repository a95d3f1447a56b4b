"""Cells whose values differ by many binades: the fixed-point G and lift of the FP64 path share one exponent per cell,
FP64 rounds a sum by its own row and column.  Against extended precision, at the nodes whose row and column hold
small values only: 64 roundings of 2^-53 of the magnitudes of their own terms (12 products, fluxes of eight
operations, and tables that are Lagrange quotients of rounded nodes)."""
import numpy as np
import pytest

from paper_2412_16002_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
LD = np.longdouble


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_16002_gb300 import build

    build()


def _tables(n):
    x = np.polynomial.legendre.leggauss(n)[0].astype(LD)
    P = lambda x: [np.ones_like(x), x, (3 * x * x - 1) / 2, (5 * x ** 3 - 3 * x) / 2, (35 * x ** 4 - 30 * x * x + 3) / 8]  # noqa: E731
    for _ in range(4):  # Newton on P_n: P_n' = n (x P_n - P_{n-1}) / (x^2 - 1)
        d = n * (x * P(x)[n] - P(x)[n - 1]) / (x * x - 1)
        x = x - P(x)[n] / d
    w = 2 / ((1 - x * x) * (n * (x * P(x)[n] - P(x)[n - 1]) / (x * x - 1)) ** 2)

    def lag(a, t):
        v = LD(1)
        for b in range(n):
            if b != a:
                v = v * (t - x[b]) / (x[a] - x[b])
        return v

    def dlag(a, q):
        s = LD(0)
        for c in range(n):
            if c != a:
                v = 1 / (x[a] - x[c])
                for b in range(n):
                    if b not in (a, c):
                        v = v * (x[q] - x[b]) / (x[a] - x[b])
                s = s + v
        return s

    D = np.array([[w[q] * dlag(a, q) / w[a] for q in range(n)] for a in range(n)])
    return D, np.array([lag(a, LD(-1)) for a in range(n)]), np.array([lag(a, LD(1)) for a in range(n)]), w


def _flux(flux, u, d):
    """flux, magnitude of the terms that form it, spectral radius"""
    if flux == "burgers":
        return u * u / 2, u * u / 2, np.abs(u[0])
    if flux == "advection":
        v = LD((0.7, -1.3)[d])
        return v * u, np.abs(v * u), np.abs(v) + 0 * u[0]
    w = u[1 + d] / u[0]
    gm1 = LD(1.4 - 1.0)
    kin = (u[1] ** 2 + u[2] ** 2) / (2 * u[0])
    p, pm = gm1 * (u[3] - kin), gm1 * (np.abs(u[3]) + kin)
    f = [u[1 + d], u[1] * w + (p if d == 0 else 0), u[2] * w + (p if d == 1 else 0), (u[3] + p) * w]
    m = [np.abs(u[1 + d]), np.abs(u[1] * w) + pm, np.abs(u[2] * w) + pm, (np.abs(u[3]) + pm) * np.abs(w)]
    c = np.sqrt(np.maximum(LD(1.4) * p / u[0], 0))
    return np.stack(f), np.stack(m), np.abs(w) + c


def _parts(U, n, d):
    """Line operators along direction d of [m][..][b][a]."""
    D, lm, lp, w = _tables(n)
    if d == 0:
        return (lambda M, v: v @ M.T), (lambda l: U @ l), (lambda f, l: f[..., None] * l), D, lm, lp, w
    T = lambda v: np.moveaxis(v, -2, -1)  # noqa: E731
    return (lambda M, v: T(T(v) @ M.T)), (lambda l: T(U) @ l), (lambda f, l: f[..., None, :] * l[:, None]), D, lm, lp, w


def _G(flux, U, n, rh):
    """G of [m][ny][nx][b][a] and the magnitude of each node's own terms."""
    G, S = np.zeros(U.shape, dtype=LD), np.zeros(U.shape, dtype=LD)
    for d in range(2):
        at, ends, spread, D, lm, lp, w = _parts(U, n, d)
        f, m, _ = _flux(flux, U, d)
        G += rh[d] * at(D, f)
        S += rh[d] * at(np.abs(D), m)
        for l, sign in ((lm, 1), (lp, -1)):
            t, tm = ends(l), _parts(np.abs(U), n, d)[1](np.abs(l))
            f = _flux(flux, t, d)[0]
            # the trace's own rounding: the flux at a state of the size of its terms
            m = _flux(flux, np.concatenate([np.minimum(np.abs(t[:1]), tm[:1]), tm[1:]]) if flux == "euler" else tm, d)[1]
            G += rh[d] * sign * spread(f, l / w)
            S += rh[d] * spread(m, np.abs(l / w))
    return G, S


def _solver(flux, k, nx, ny):
    from paper_2412_16002_gb300.solver import Solver

    return Solver(2, nx, ny, k, (0.0, 1.0 * nx, 0.0, 1.0 * ny), flux, velocity=(0.7, -1.3), bounds=(-2.0, 2.0), bc=("outflow",) * 4)


def _base(flux, k, nx, ny, seed):
    if flux == "euler":
        return inputs.random_euler(2, nx, ny, k, seed=seed, osc=0.1)
    return inputs.random_scalar(2, nx, ny, k, seed=seed, lo=0.5, hi=1.0)


def _apply(g, op, U):
    x = torch.from_numpy(np.ascontiguousarray(U)).cuda()
    return g.apply(op, x, torch.empty_like(x)).cpu().numpy()


@pytest.mark.parametrize("k", [1, 2, 3])
@pytest.mark.parametrize("flux", ["euler", "burgers", "advection"])
@pytest.mark.parametrize("binades", [3, 9, 19])
def test_G_beside_a_large_corner(flux, k, binades):
    nx, ny = 13, 3
    U = _base(flux, k, nx, ny, k)
    U[..., :-1, :-1] *= 2.0 ** -binades
    U[..., -1, :-1] *= 2.0 ** -binades  # all but the last node of the last row
    U[..., :-1, -1] *= 2.0 ** -binades
    got = _apply(_solver(flux, k, nx, ny), "G", U)
    G, S = _G(flux, U.astype(LD), k + 1, (LD(2), LD(2)))
    small = (slice(None),) * 3 + (slice(0, k), slice(0, k))
    assert (np.abs(got - G) <= 64 * LD(2) ** -53 * S)[small].all()


@pytest.mark.parametrize("k", [1, 2, 3])
@pytest.mark.parametrize("flux", ["euler", "burgers", "advection"])
@pytest.mark.parametrize("binades", [3, 9, 19])
def test_lift_beside_a_large_face_point(flux, k, binades):
    """Two cells, the first small throughout, the second large in its last row: in the first one only the last row's
    right face point takes a large correction, so the other rows' F is rounded by their own terms.  (Euler: the
    last row large in density and energy alike keeps the radius of the face, the largest over its points, ordinary.)"""
    U = _base(flux, k, 2, 1, 7 + k)
    U *= 2.0 ** -binades
    U[:, 0, 1, -1, :] *= 2.0 ** binades
    n = k + 1
    got = _apply(_solver(flux, k, 2, 1), "F", U)
    V = U.astype(LD)
    G, S = _G(flux, V, n, (LD(2), LD(2)))
    _, lm, lp, w = _tables(n)
    left, right = V[:, 0, 0] @ lp, V[:, 0, 1] @ lm  # the shared face's traces [m][pos]
    (fl, ml, al), (fr, mr, ar) = _flux(flux, left, 0), _flux(flux, right, 0)
    tl, tr = np.abs(V[:, 0, 0]) @ np.abs(lp), np.abs(V[:, 0, 1]) @ np.abs(lm)
    alpha = np.maximum(al.max(), ar.max())
    dc = (fr - fl) / 2 - alpha * (right - left) / 2
    mag = (ml + mr) / 2 + alpha * (tl + tr) / 2
    F, SF = G[:, 0, 0].copy(), S[:, 0, 0].copy()
    F -= 2 * dc[..., None] * (lp / w)
    SF += 2 * mag[..., None] * np.abs(lp / w)
    # the three boundary faces: the cell average outside
    for d, l, sign in ((0, lm, 1), (1, lm, 1), (1, lp, -1)):
        c = V[:, 0, 0]
        avg = (c * np.outer(w, w) / 4).sum((-1, -2))[:, None] + 0 * tl
        t = c @ l if d == 0 else np.moveaxis(c, -2, -1) @ l
        tm = np.abs(c) @ np.abs(l) if d == 0 else np.moveaxis(np.abs(c), -2, -1) @ np.abs(l)
        (fi, mi, ai), (fe, me, ae) = _flux(flux, t, d), _flux(flux, avg, d)
        al = np.maximum(ai.max(), ae.max())
        dcb = (fe - fi) / 2 + sign * al * (avg - t) / 2
        mb = (mi + me) / 2 + al * (tm + np.abs(avg)) / 2
        sp = (lambda f, v: f[..., None] * v) if d == 0 else (lambda f, v: f[..., None, :] * v[:, None])
        F += 2 * sign * sp(dcb, l / w)
        SF += 2 * sp(mb, np.abs(l / w))
    rows = (slice(None), slice(0, k), slice(None))
    assert (np.abs(got[:, 0, 0] - F) <= 64 * LD(2) ** -53 * SF)[rows].all()
