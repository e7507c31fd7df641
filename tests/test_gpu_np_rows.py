"""NP and LP in 2D at wide horizons (two x-adjacent point pairs per thread, by stencil
rows): force against the FP64 oracle, two steps' velocities (from rest, so they are the
forces summed) against the FP64 passes. FP32 bonds: 1e-5."""
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


# tiles of 16 x 8, 16 x 16, 32 x 16 points; 2 and 4 ranges of words; odd and even horizons,
# within a tile and over several; grids that end inside a tile
@pytest.mark.parametrize("n,m,tile", [((61, 47, 1), 9, 7), ((57, 71, 1), 18, 7), ((53, 49, 1), 11, 8), ((75, 66, 1), 17, 9),
                                    ((97, 59, 1), 20, 9), ((81, 83, 1), 24, 9)])
@pytest.mark.parametrize("model", [W.NP, W.LP])
def test_np_rows_match_the_oracle(pd, n, m, tile, model):
    grid = W.Grid(dim=2, n=n, h=0.3, m=m)
    mat = W.Material(model=model, rho=1.0, psi_c=1.0, psi_beta=1.0, K=1.0, mu=1.0)
    u = W.random_field(grid, 0.02 * grid.h, seed=5)
    sim = gpu_sim(pd, grid, mat, pd.PD_FP32C, dt=1e-3, tile_log2=tile)
    f = O.internal_force(grid, mat, O.neighbors(grid), u)[0]
    assert rel_l2(pd.pd_force(sim, u=u), f) <= 1e-5
    v = []
    for s in (sim, gpu_sim(pd, grid, mat, pd.PD_FP64, dt=1e-3)):
        pd.pd_set_state(s, u=u, v=np.zeros_like(u))
        pd.pd_step_explicit(s, 2)
        v.append(pd.pd_get_state(s)[1])
        s.close()
    assert rel_l2(v[0], v[1]) <= 1e-5
