"""FP32C forces and dilatation on both sides of the rules that choose a kernel and its
staging in 3D: by columns or by pairs (ragged grids of few tiles, grids of many, breaking
or not, by horizon), row-wise or word-wise. Against the oracle, FP32C bar 1e-5 relative L2;
no bond reaches s_c here."""
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


FEW, MANY, FIVE = (21, 30, 26), (57, 65, 33), (65, 72, 67)      # 48, 360 and 729 tiles
CASES = [(FEW, m, W.PMB, s_c, 0) for m in (1, 2, 3, 4) for s_c in (0.0, 0.1)]
CASES += [(MANY, m, W.PMB, 0.1, 0) for m in (1, 2, 3, 4, 5)]
CASES += [((24, 32, 16), 3, W.PMB, 0.1, 0), (FIVE, 3, W.PMB, 0.0, 0), (MANY, 3, W.PMB, 0.0, 4)]
CASES += [(FEW, 3, W.LPS, 0.0, 0), (FEW, 5, W.LPS, 0.0, 0), ((45, 47, 42), 5, W.LPS, 0.0, 0), (MANY, 5, W.LPS, 0.0, 0),
          (MANY, 1, W.LPS, 0.0, 0)]


@pytest.mark.parametrize("n,m,model,s_c,pt", CASES)
def test_every_route_matches_the_oracle(pd, n, m, model, s_c, pt):
    grid = W.Grid(dim=3, n=n, h=1.0 / 64, m=m)
    mat = W.Material(model=model, E=72e9, K=40e9, mu=30e9, s_c=s_c)
    sim = gpu_sim(pd, grid, mat, pd.PD_FP32C, pair_threads=pt)
    bonds = O.neighbors(grid)
    u = (1e-4 / 3) * grid.positions() + W.random_field(grid, 1e-4 * grid.h, seed=11)
    f = pd.pd_force(sim, u=u, flags=pd.PD_FORCE_UPDATE_BREAKING if s_c else 0)
    if model == W.PMB:
        want = O.pmb_force(grid, mat, bonds, u)
        assert not pd.pd_get_broken(sim).any()
    else:
        mv = O.weighted_volume(grid, mat, bonds)
        th = O.dilatation(grid, mat, bonds, mv, u)
        assert rel_l2(pd.pd_dilatation(sim, u=u), th) <= TOL
        want = O.lps_force(grid, mat, bonds, mv, th, u)
    sim.close()
    assert rel_l2(f, want) <= TOL
