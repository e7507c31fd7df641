"""GPU tests of the last bits of the all-FP64 passes, on one bond whose quantities are
exact: the spacing is a power of two, the bond's strain e a multiple of 2^-20, so that
y = 1 + e, |y|^2 and |y|^2 - 1 have at most 42 bits."""
from fractions import Fraction

import numpy as np
import pytest

from paper_1806_06917_gb300 import workloads as W

pytestmark = pytest.mark.gpu

H = 2.0 ** -6
PAIR = W.Grid(dim=3, n=(2, 1, 1), h=H, m=1)
STRAINS = np.random.default_rng(7).integers(-900_000, 2_000_000, size=150) * 2.0 ** -20


@pytest.fixture(scope="module")
def pd():
    import torch

    torch.cuda.set_device(0)
    from paper_1806_06917_gb300 import pd as _pd

    return _pd


def _sim(pd, mat):
    sim = pd.pd_create(*pd.describe(PAIR, mat, precision=pd.PD_FP64))
    pd.pd_build_neighbors(sim)
    return sim


def _pull(e):
    return np.array([[0.0, 0.0, 0.0], [e * H, 0.0, 0.0]])


def test_dilatation_rounds_root_and_quotient_once(pd):
    """theta = 3 (|y|^2 - 1) / (|y| + 1) = 3 e: the root, the quotient and the product are
    representable, so a root and a quotient with no error but their rounding return them."""
    sim = _sim(pd, W.Material(model=W.LPS, E=72e9, rho=2440.0, K=40e9, mu=30e9))
    th = np.array([pd.pd_dilatation(sim, u=_pull(e)) for e in STRAINS])
    sim.close()
    assert (th == 3.0 * STRAINS[:, None]).all(), "%d of %d differ" % ((th != 3.0 * STRAINS[:, None]).sum(), th.size)


def test_energy_divides_and_takes_roots_in_ieee_arithmetic(pd):
    """The strain energy of the pair is K s^2 with s = (q - 1) / (q rs + 1), rs = 1 / sqrt(q);
    K comes from e = 1, where s = 1. Whether q rs + 1 is one rounding or two is the compiler's."""
    sim = _sim(pd, W.Material(model=W.PMB, E=72e9, rho=2440.0))

    def energy(e):
        pd.pd_set_state(sim, u=_pull(e), v=np.zeros((2, 3)))
        return pd.pd_energy(sim)[1]

    k = energy(1.0)
    got = np.array([energy(e) for e in STRAINS])
    sim.close()
    q = (1.0 + STRAINS) ** 2
    rs = 1.0 / np.sqrt(q)
    fused = np.array([float(Fraction(a) * Fraction(b) + 1) for a, b in zip(q.tolist(), rs.tolist())])
    want = []
    for den in (q * rs + 1.0, fused):
        s = (q - 1.0) / den
        want.append(k * (s * s))
    assert any((got == w).all() for w in want), [int((got != w).sum()) for w in want]


@pytest.mark.parametrize("model", [W.NP, W.LP])
def test_points_at_the_horizon_do_not_act(pd, model):
    """J = 0 at |xi| = delta (NP, LP): a displacement without bound there leaves the force
    alone. (5, 5) is no tile's reference point; those at a distance below 3 do see it."""
    g = W.Grid(dim=2, n=(17, 15, 1), h=0.25, m=3)
    sim = pd.pd_create(*pd.describe(g, W.Material(model=model, rho=1.0, psi_c=1.0, psi_beta=1.0),
                                    precision=pd.PD_FP64, dt=1e-5))
    pd.pd_build_neighbors(sim)
    u = W.random_field(g, 0.01 * g.h, seed=2)
    f0 = pd.pd_force(sim, u=u)
    c = g.coords()[:, :2]
    r2 = ((c - [5, 5]) ** 2).sum(1)
    u[r2 == 0] = np.inf
    f = pd.pd_force(sim, u=u)
    sim.close()
    assert (r2 == 9).sum() == 4
    assert (f[r2 >= 9] == f0[r2 >= 9]).all()
