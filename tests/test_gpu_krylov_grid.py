"""GMRES with the cached tangent (a cycle in one launch) against GMRES with the JVP tangent
(a kernel per operation) after the same number of iterations: both are stable solves of
Krylov spaces that differ by rounding, 1e-16 times a condition number below 1e6 (the
number of points along the plate, squared)."""
import numpy as np
import pytest

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


# fewer unknowns than slices; a last slice cut short; several cycles; 3D; more dots than
# blocks (restart 200); slices of several warps a dot (300^2, 1,190 unknowns each)
@pytest.mark.parametrize("n,m,restart,iters", [((9, 4, 1), 2, 50, 12), ((73, 61, 1), 3, 50, 64), ((37, 22, 1), 4, 7, 30),
                                             ((13, 9, 8), 2, 20, 33), ((60, 40, 1), 3, 200, 200),
                                             ((300, 300, 1), 3, 20, 24)])
def test_gmres_cycle_in_one_launch_matches_the_kernels(pd, n, m, restart, iters):
    grid = W.Grid(dim=3 if n[2] > 1 else 2, n=n, h=1.0 / n[0], m=m)
    mat = W.Material(model=W.PMB, E=72e9, rho=2440.0)
    kind = np.zeros((grid.npoints, grid.dim), dtype=np.uint8)
    kind[W.collar_mask(grid, 0, -1)] = W.BC_DISPLACEMENT
    kind[W.collar_mask(grid, 0, +1), 0] = W.BC_DISPLACEMENT
    val = np.where(kind != 0, 1e-4 * grid.positions()[:, :1], 0.0)
    out = []
    for tangent in (pd.PD_TANGENT_CACHED, pd.PD_TANGENT_JVP):
        sim = gpu_sim(pd, grid, mat, pd.PD_FP64)
        z = np.zeros((grid.npoints, grid.dim))
        pd.pd_set_state(sim, u=z, v=z)
        pd.pd_set_bc(sim, kind, val)
        st = pd.pd_solve_static(sim, pd.newton_opts(krylov=pd.PD_KRYLOV_GMRES, restart=restart, max_linear_iters=iters,
                                                    max_newton_iters=1, linear_rtol=1e-13, tangent=tangent))
        out.append((pd.pd_get_state(sim)[0], st["linear_iters"]))
        sim.close()
    assert abs(out[0][1] - out[1][1]) <= 1      # the residual meets the target at rounding level
    assert rel_l2(out[0][0], out[1][0]) <= 1e-9
