"""The all-FP64 passes where their algebra differs from the definition: the tangent
product's coefficient of n n^T (1 / |y|), its adjoint and the partial volume, against
central differences of the force; the NP exponential on both sides of its series' range."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1806_06917_gb300 import workloads as W
from tests.helpers import gpu_sim, rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pd():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1806_06917_gb300 import pd as _pd
    return _pd


@pytest.mark.parametrize("n,m,vc", [((21, 18, 1), 3, 0), ((19, 23, 1), 4, 1), ((9, 11, 10), 2, 1), ((13, 9, 12), 3, 0)])
def test_fp64_tangent_is_the_force_derivative(pd, n, m, vc):
    grid = W.Grid(dim=3 if n[2] > 1 else 2, n=n, h=0.01, m=m)
    mat = W.Material(model=W.PMB, vol_corr=vc)
    sim = gpu_sim(pd, grid, mat, pd.PD_FP64)
    u = W.random_field(grid, 0.05 * grid.h, seed=1)
    w = W.random_field(grid, 1.0, seed=2)
    kw = pd.pd_jvp(sim, w, u_lin=u)
    eps = 1e-6 * grid.h         # truncation (1e-6)^2, rounding 1e-16 / 1e-6
    fd = (pd.pd_force(sim, u=u + eps * w) - pd.pd_force(sim, u=u - eps * w)) / (2 * eps)
    assert rel_l2(kw, fd) <= 1e-8
    assert rel_l2(pd.pd_vjp(sim, w, u_lin=u), kw) <= 1e-12       # K is symmetric
    sim.close()


@pytest.mark.parametrize("scale", [1e-4, 0.125, 0.5])
def test_fp64_np_force_on_both_sides_of_the_series(pd, scale):
    # beta |xi| S^2 reaches about (3 scale)^2: 1e-7, 0.14 and 2.3, the series ends at 2^-6
    grid = W.Grid(dim=2, n=(33, 29, 1), h=0.3, m=4)
    mat = W.Material(model=W.NP, rho=1.0, psi_c=1.0, psi_beta=1.0)
    sim = gpu_sim(pd, grid, mat, pd.PD_FP64, dt=1e-5)
    u = W.random_field(grid, scale * grid.h, seed=3)
    assert rel_l2(pd.pd_force(sim, u=u), O.internal_force(grid, mat, O.neighbors(grid), u)[0]) <= 1e-10
    sim.close()
