"""The neighbour build by tile against brute force, where its classes and positions can
go wrong: axes shorter than, equal to and one above 2m + 1 points, partial tiles, the
widest halo a tile allows, and grids whose tiles' rows several CTAs share."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1806_06917_gb300 import workloads as W
from tests.helpers import gpu_csr_in_user_numbering, gpu_sim, oracle_pairs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pd():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1806_06917_gb300 import pd as _pd
    return _pd


@pytest.mark.parametrize("n,m,vc", [((6, 7, 8), 3, 0), ((7, 7, 7), 3, 1), ((8, 9, 17), 4, 0), ((16, 8, 24), 3, 1),
                                    ((33, 16, 1), 16, 0), ((66, 31, 1), 5, 1), ((40, 40, 40), 2, 0)])
def test_lists_masks_and_sums_match_brute_force(pd, n, m, vc):
    grid = W.Grid(dim=3 if n[2] > 1 else 2, n=n, h=0.01, m=m)
    mat = W.Material(model=W.LPS if n[2] > 1 else W.PMB, K=40e9, mu=30e9, vol_corr=vc)
    sim = gpu_sim(pd, grid, mat, pd.PD_FP64)
    bonds = O.neighbors(grid)
    rows, cols, _, (row_ptr, col, _) = gpu_csr_in_user_numbering(pd, sim)
    want_rows, want_cols = oracle_pairs(bonds)
    assert pd.pd_bond_count(sim) == len(want_cols)
    order = np.lexsort((want_cols, want_rows))
    assert np.array_equal(rows, want_rows[order]) and np.array_equal(cols, want_cols[order])
    starts = np.zeros(len(col), bool)
    starts[row_ptr[:-1][np.diff(row_ptr) > 0]] = True
    assert np.all((np.diff(col) > 0) | starts[1:])               # every row ascends
    assert not pd.pd_get_broken(sim).any()                       # every bond's mask bit is set
    u = W.random_field(grid, 1e-3 * grid.h, seed=4)
    if n[2] > 1:                                                 # the weighted volume, through theta
        mv = O.weighted_volume(grid, mat, bonds)
        th = O.dilatation(grid, mat, bonds, mv, u)
        assert np.allclose(pd.pd_dilatation(sim, u=u), th, rtol=1e-10, atol=1e-13)
    sim.close()
