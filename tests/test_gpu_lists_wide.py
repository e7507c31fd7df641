"""The neighbour build by tile where a tile's mask words stay in global memory (more than
4096 of them: wide horizons on 2^9-point tiles), on the small tiles that FP64 grids take by
themselves, and the cell-list build of horizons wider than a tile: CSR, masks and step
bound against the oracle."""
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


# (sides, m, precision, tile_log2): 2D 32 x 16 and 3D 8 x 8 x 8 tiles, words per tile 6144,
# 12800 and 8704, ragged in every direction; one axis shorter than 2 m + 1; then 8 x 8 and
# 4 x 4 x 4 tiles; then horizons wider than the tile (cell list)
FORMS = [((75, 41, 1), 11, "fp32c", 9), ((97, 50, 1), 16, "fp32c", 9), ((40, 23, 1), 16, "fp64", 9),
         ((19, 26, 13), 5, "fp32c", 9), ((9, 21, 17), 5, "fp32c", 9),
         ((37, 29, 1), 8, "fp64", 0), ((13, 10, 9), 4, "fp64", 0),
         ((33, 16, 1), 16, "fp64", 0), ((75, 41, 1), 17, "fp32c", 9)]


@pytest.mark.parametrize("n,m,precision,L", FORMS)
def test_lists_of_every_form_of_the_build(pd, n, m, precision, L):
    grid = W.Grid(dim=3 if n[2] > 1 else 2, n=n, h=0.01, m=m)
    mat = W.Material(model=W.PMB, E=72e9, rho=2440.0)
    sim = gpu_sim(pd, grid, mat, precision, tile_log2=L)
    bonds = O.neighbors(grid)
    rows, cols, _, (row_ptr, col, _) = gpu_csr_in_user_numbering(pd, sim)
    want_rows, want_cols = oracle_pairs(bonds)
    order = np.lexsort((want_cols, want_rows))
    assert np.array_equal(rows, want_rows[order]) and np.array_equal(cols, want_cols[order])
    starts = np.zeros(len(col), bool)
    starts[row_ptr[:-1][np.diff(row_ptr) > 0]] = True
    assert np.all((np.diff(col) > 0) | starts[1:])               # every row ascends
    assert not pd.pd_get_broken(sim).any()                       # every bond's mask bit is set
    assert pd.pd_get_dt(sim) == pytest.approx(0.5 * O.stable_dt(grid, mat, bonds), rel=1e-12)
    sim.close()
