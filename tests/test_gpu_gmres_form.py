"""The two forms of GMRES with the cached tangent, chosen by name: the same Krylov iterates
but for rounding, and a wait of the one-launch form that runs out. The stall leaves one
block out of the launch, so that the others give up after the limit and the kernel ends."""
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


def _plate(pd, n, m, precision="fp64"):
    grid = W.Grid(dim=3 if n[2] > 1 else 2, n=n, h=1.0 / n[0], m=m)
    sim = gpu_sim(pd, grid, W.Material(model=W.PMB, E=72e9, rho=2440.0), precision)
    kind = np.zeros((grid.npoints, grid.dim), dtype=np.uint8)
    kind[W.collar_mask(grid, 0, -1)] = W.BC_DISPLACEMENT
    kind[W.collar_mask(grid, 0, +1), 0] = W.BC_DISPLACEMENT
    pd.pd_set_bc(sim, kind, np.where(kind != 0, 1e-4 * grid.positions()[:, :1], 0.0))
    return sim, np.zeros((grid.npoints, grid.dim))


def _solve(pd, sim, zero, form, **kw):
    opts = dict(restart=20, max_linear_iters=400, max_newton_iters=1, linear_rtol=1e-10)
    opts.update(kw)
    limit = opts.pop("limit", 0)
    stall = opts.pop("stall", 0)
    pd.pd_set_state(sim, u=zero, v=zero)
    pd.pd_set_gmres_form(sim, form, limit, stall)
    st = pd.pd_solve_static(sim, pd.newton_opts(krylov=pd.PD_KRYLOV_GMRES, **opts))
    return pd.pd_get_state(sim)[0], st


# after 24 steps (two cycles) the forms differ by the products' rounding, 1e-16 in FP64 and
# 6e-8 in FP32, times the condition of 24 Krylov vectors, below the number of points along
# the plate squared
@pytest.mark.parametrize("n,m", [((30, 22, 1), 3), ((13, 9, 8), 2), ((61, 40, 1), 2)])
@pytest.mark.parametrize("precision,unit", [("fp64", 2.0 ** -53), ("fp32c", 2.0 ** -24)])
def test_both_forms_take_the_same_steps(pd, n, m, precision, unit):
    sim, zero = _plate(pd, n, m, precision)
    kw = dict(max_linear_iters=24, restart=12, linear_rtol=1e-30)
    (a, sa), (b, sb), (c, _) = (_solve(pd, sim, zero, f, **kw) for f in (pd.PD_GMRES_GRID, pd.PD_GMRES_GRAPH, pd.PD_GMRES_AUTO))
    sim.close()
    assert sa["linear_iters"] == sb["linear_iters"] == 24
    assert np.abs(a).max() > 0
    assert rel_l2(a, b) <= 4 * unit * n[0] ** 2
    assert (c == a).all()


def test_a_wait_that_runs_out(pd):
    sim, zero = _plate(pd, (40, 30, 1), 3)
    want, st = _solve(pd, sim, zero, pd.PD_GMRES_GRAPH)
    grid, _ = _solve(pd, sim, zero, pd.PD_GMRES_GRID)
    with pytest.raises(pd.PdError) as e:
        _solve(pd, sim, zero, pd.PD_GMRES_GRID, limit=20, stall=1)
    assert e.value.code == pd.PD_ETIMEOUT
    # by itself the solve goes on kernel by kernel, from the cycle that failed
    got, s2 = _solve(pd, sim, zero, pd.PD_GMRES_AUTO, limit=20, stall=1)
    assert (got == want).all() and s2 == st
    # and the launch works again afterwards
    assert (_solve(pd, sim, zero, pd.PD_GMRES_AUTO)[0] == grid).all()
    for bad in ((3, 0, 0), (-1, 0, 0), (0, -1, 0), (0, 0, 2)):
        with pytest.raises(pd.PdError):
            pd.pd_set_gmres_form(sim, *bad)
    sim.close()
