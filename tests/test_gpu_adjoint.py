"""The adjoint product against its definition, <v, K w> = <K^T v, w>, for two independent
vectors, with bonds of a notch broken: it holds whether or not K is symmetric, and fails
for a mask, a sign or a coefficient that differs between the two ends of a bond.

Each component of a product is a sum of S + 32 roundings at most of its terms, and a term
is below 2 (c V / h) / |d| (|w_i| + |w_j|) at strains this small (1 + s/r |d| < 2)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1806_06917_gb300 import workloads as W
from tests.helpers import gpu_sim, oracle_pairs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pd():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1806_06917_gb300 import pd as _pd
    return _pd


@pytest.mark.parametrize("precision,unit", [("fp64", 2.0 ** -53), ("fp32c", 2.0 ** -24)])
@pytest.mark.parametrize("n,m,vc", [((21, 18, 1), 3, 0), ((40, 37, 1), 5, 1), ((11, 9, 10), 2, 1), ((13, 17, 9), 3, 0)])
def test_adjoint_of_the_tangent(pd, n, m, vc, precision, unit):
    dim = 3 if n[2] > 1 else 2
    grid = W.Grid(dim=dim, n=n, h=0.01, m=m)
    mat = W.Material(model=W.PMB, E=72e9, rho=2440.0, vol_corr=vc)
    notch = W.Notch(axis=0, pos=n[0] // 2 - 0.5, lo=(0.0, -0.5, -0.5), hi=(0.0, n[1] / 2.0, n[2] / 2.0))
    sim = gpu_sim(pd, grid, mat, precision, notch=notch)
    assert pd.pd_get_broken(sim).any()
    u = W.random_field(grid, 1e-3 * grid.h, seed=1)
    v, w = W.random_field(grid, 1.0, seed=2), W.random_field(grid, 1.0, seed=3)
    kw, ktv = pd.pd_jvp(sim, w, u_lin=u), pd.pd_vjp(sim, v, u_lin=u)
    sim.close()
    bonds = O.neighbors(grid)
    i, j = oracle_pairs(bonds)
    x = grid.coords()[:, :dim]
    r0 = np.sqrt(((x[i] - x[j]) ** 2).sum(1))
    V = grid.h ** 3 if dim == 3 else grid.h ** 2 * mat.thickness
    k = 2 * O.micromodulus(grid, mat) * V / grid.h / r0
    S = np.bincount(i).max()

    def roundings(a, b):
        """Rounding bound of <a, K b>: every bond's term, and the dot product's own sum in FP64."""
        terms = k * np.abs(a[i]).sum(1) * (np.abs(b[i]).sum(1) + np.abs(b[j]).sum(1))
        return (S + 32) * unit * terms.sum()

    assert abs((v * kw).sum() - (ktv * w).sum()) <= roundings(v, w) + roundings(w, v)
    # (the bound means something: the two products are far larger)
    assert np.abs(v * kw).sum() > 50 * (roundings(v, w) + roundings(w, v))
