"""GPU tests of the all-FP64 passes against extended precision, bond by bond bounds: the
displacements are multiples of a power of two of the spacing, so that the relative
displacements the kernels form are exact and only their own roundings are left.

u = 2^-53. A bond's num = |y|^2 - |d|^2 takes at most six roundings of partial sums no
larger than P = sum_c (e_c^2 + 2 |d_c e_c|); |y|^2, the root, the quotient and the products
after it stay below 26 more of the term; S additions follow. So each sum's error is at
most (32 + S) u times the sum of its terms' magnitudes, with P in the place of |num|."""
import itertools

import numpy as np
import pytest

from paper_1806_06917_gb300 import workloads as W

pytestmark = pytest.mark.gpu

U = 2.0 ** -53
H = 2.0 ** -6
LD = np.longdouble


@pytest.fixture(scope="module")
def pd():
    import torch

    torch.cuda.set_device(0)
    from paper_1806_06917_gb300 import pd as _pd

    return _pd


def _bonds(grid):
    """(d, i, j) per stencil offset: the user indices of the points that have the neighbour and of it."""
    n = [np.arange(k) for k in grid.n]
    z, y, x = np.meshgrid(n[2], n[1], n[0], indexing="ij")
    i = np.arange(grid.npoints)
    c = [a.ravel() for a in (x, y, z)]
    r = range(-grid.m, grid.m + 1)
    for d in itertools.product(r, r, r if grid.dim == 3 else (0,)):
        if not 0 < sum(k * k for k in d) <= grid.m ** 2:
            continue
        p = [c[a] + d[a] for a in range(3)]
        ok = np.all([(p[a] >= 0) & (p[a] < grid.n[a]) for a in range(3)], axis=0)
        if ok.any():
            yield np.array(d[:grid.dim], dtype=LD), i[ok], (p[0] + grid.n[0] * (p[1] + grid.n[1] * p[2]))[ok]


def _field(grid, rho, seed):
    """Displacements / h: every bond shrunk to rho of its length, and a perturbation well below it."""
    rng = np.random.default_rng(seed)
    X = np.round(grid.positions() / grid.h)
    noise = rng.integers(-2 ** 8, 2 ** 8 + 1, size=X.shape) * (2.0 ** -13 * rho * 2.0 ** -8)
    return (rho - 1.0) * X + noise


def _geometry(e, d):
    y, r0 = d + e, np.sqrt((d * d).sum())
    r = np.sqrt((y * y).sum(1))
    num = (e * (y + d)).sum(1)
    P = (e * e + 2 * np.abs(d * e)).sum(1)
    return y, r0, r, num, P


# |y| / |d|: near the reference, and down to where |d|^2 + num rounds to zero
RHOS = [1.0, 0.5, 2.0 ** -3, 2.0 ** -7, 2.0 ** -27]
GRIDS = [((21, 18, 1), 3), ((13, 9, 1), 5), ((9, 8, 7), 2)]


@pytest.mark.parametrize("n,m", GRIDS)
@pytest.mark.parametrize("rho", RHOS)
def test_force_and_tangent_of_compressed_bonds(pd, n, m, rho):
    g = W.Grid(dim=3 if n[2] > 1 else 2, n=n, h=H, m=m)
    sim = pd.pd_create(*pd.describe(g, W.Material(model=W.PMB, E=72e9, rho=2440.0), precision=pd.PD_FP64))
    pd.pd_build_neighbors(sim)
    u = _field(g, rho, 3)
    w = np.random.default_rng(4).integers(-2 ** 20, 2 ** 20, size=u.shape) * 2.0 ** -20
    f, k = pd.pd_force(sim, u=u * H), pd.pd_jvp(sim, w, u_lin=u * H)
    sim.close()
    e_ = LD(72e9)
    delta = LD(m) * H
    if g.dim == 3:
        c, V = 18 * (e_ / LD(1.5)) / (LD(np.pi) * delta ** 4), LD(H) ** 3
    else:
        c, V = 9 * e_ / (LD(np.pi) * delta ** 3), LD(H) ** 2
    F, FM, K, KM = (np.zeros(u.shape, dtype=LD) for _ in range(4))
    S = 0
    ul, wl = u.astype(LD), w.astype(LD)
    for d, i, j in _bonds(g):
        y, r0, r, num, P = _geometry(ul[j] - ul[i], d)
        S += 1
        dw = wl[j] - wl[i]
        sr, srm = num / (r0 * (r + r0) * r), P / (r0 * (r + r0) * r)
        nd, ndm = (y * dw).sum(1), np.abs(y * dw).sum(1)
        F[i] += sr[:, None] * y
        FM[i] += srm[:, None] * np.abs(y)
        K[i] += (nd / r ** 3)[:, None] * y + sr[:, None] * dw
        KM[i] += (ndm / r ** 2 * (1 / r0 + srm))[:, None] * np.abs(y) + srm[:, None] * np.abs(dw)
    # pi and the constants in front are doubles of the library's own
    for got, ref, mag, scale in ((f, F, FM, c * V), (k, K, KM, c * V / H)):
        err = np.abs(got - scale * ref)
        bound = (32 + S) * U * scale * mag
        assert np.isfinite(got).all()
        assert (err <= bound).all(), "error / bound up to %.2e" % float((err / np.where(mag > 0, bound, 1)).max())


@pytest.mark.parametrize("rho", RHOS)
def test_lps_of_compressed_bonds(pd, rho):
    g = W.Grid(dim=3, n=(9, 8, 7), h=H, m=2)
    mat = W.Material(model=W.LPS, E=72e9, rho=2440.0, K=40e9, mu=30e9)
    sim = pd.pd_create(*pd.describe(g, mat, precision=pd.PD_FP64))
    pd.pd_build_neighbors(sim)
    u = _field(g, rho, 5)
    th, f = pd.pd_dilatation(sim, u=u * H), pd.pd_force(sim, u=u * H)
    sim.close()
    ul = u.astype(LD)
    bonds = list(_bonds(g))
    S, N = len(bonds), g.npoints
    mt, T, TM = np.zeros(N, dtype=LD), np.zeros(N, dtype=LD), np.zeros(N, dtype=LD)
    for d, i, j in bonds:
        y, r0, r, num, P = _geometry(ul[j] - ul[i], d)
        mt[i] += r0 * r0
        T[i] += r0 * num / (r + r0)
        TM[i] += r0 * P / (r + r0)
    T, TM = 3 * T / mt, 3 * TM / mt
    err = np.abs(th - T)
    assert (err <= (32 + S) * U * TM).all(), "dilatation: error / bound up to %.2e" % float((err / ((32 + S) * U * TM)).max())
    A, B = LD(3 * mat.K - 5 * mat.mu), LD(15 * mat.mu)
    F, FM = np.zeros(u.shape, dtype=LD), np.zeros(u.shape, dtype=LD)
    for d, i, j in bonds:
        y, r0, r, num, P = _geometry(ul[j] - ul[i], d)
        t = A * r0 * (T[i] / mt[i] + T[j] / mt[j]) + B * num / (r + r0) * (1 / mt[i] + 1 / mt[j])
        tm = np.abs(A) * r0 * (TM[i] / mt[i] + TM[j] / mt[j]) + B * P / (r + r0) * (1 / mt[i] + 1 / mt[j])
        F[i] += (t / r)[:, None] * y
        FM[i] += (tm / r)[:, None] * np.abs(y)
    err = np.abs(f - F / H)
    bound = 2 * (32 + S) * U * FM / H       # the dilatation's error, and the sum's own
    assert np.isfinite(f).all()
    assert (err <= bound).all(), "force: error / bound up to %.2e" % float((err / bound).max())
