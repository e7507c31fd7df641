"""The row-wise FP32C passes (2^9-point tiles, from 304 tiles on; the LPS force pass
from 153): forces and dilatation against the oracle on ragged grids on both sides of
those counts, with the table in shared memory and (2048 tiles) as a kernel parameter,
one and two parts of the sum, and partial volume. FP32C bars: 1e-5 relative L2."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1806_06917_gb300 import workloads as W
from tests.helpers import gpu_sim, rel_l2

pytestmark = pytest.mark.gpu

TOL = 1e-5


@pytest.fixture(scope="module")
def pd():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1806_06917_gb300 import pd as _pd
    return _pd


CASES = [
    # (n, m, model, partial volume, pair_threads): tiles
    ((57, 65, 33), 3, W.PMB, 0, 0),         # 360
    ((57, 65, 33), 3, W.PMB, 1, 2),
    ((61, 58, 40), 2, W.PMB, 0, 0),         # 320, one mask word
    ((57, 59, 36), 4, W.PMB, 0, 0),         # 320, eight mask words
    ((121, 98, 89), 3, W.PMB, 0, 0),        # 2496
    ((57, 65, 30), 3, W.LPS, 0, 0),         # 288: force pass alone
    ((61, 58, 40), 1, W.LPS, 0, 0),         # 320, one part
    ((57, 59, 36), 4, W.LPS, 1, 0),
    ((121, 98, 89), 3, W.LPS, 0, 0),
]


@pytest.mark.parametrize("n,m,model,vc,pt", CASES)
def test_row_wise_forces_match_oracle(pd, n, m, model, vc, pt):
    grid = W.Grid(dim=3, n=n, h=1.0 / 128, m=m)
    mat = W.Material(model=model, E=72e9, K=40e9, mu=30e9, vol_corr=vc)
    sim = gpu_sim(pd, grid, mat, pd.PD_FP32C, pair_threads=pt)
    bonds = O.neighbors(grid)
    u = (1e-4 / 3) * grid.positions() + W.random_field(grid, 1e-4 * grid.h, seed=11)
    f = pd.pd_force(sim, u=u)
    if model == W.PMB:
        want = O.pmb_force(grid, mat, bonds, u)
    else:
        mv = O.weighted_volume(grid, mat, bonds)
        th = O.dilatation(grid, mat, bonds, mv, u)
        assert rel_l2(pd.pd_dilatation(sim, u=u), th) <= TOL
        want = O.lps_force(grid, mat, bonds, mv, th, u)
    assert rel_l2(f, want) <= TOL
    # one step from rest at u moves v by dt f / rho
    pd.pd_set_state(sim, u, np.zeros_like(u))
    pd.pd_step_explicit(sim, 1)
    moved, _ = pd.pd_get_state(sim, want_v=False)
    dt = pd.pd_get_dt(sim)
    assert rel_l2(moved - u, dt * dt / 2 * want / mat.rho) <= 2 * TOL
    sim.close()
