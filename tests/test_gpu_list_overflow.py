"""Lists that outgrow their capacity in the middle of a launch of many steps: those NPs
are summed from the cells, whose arrays the same launch writes; the same bits as the
separate kernels, and the float64 oracle's forces."""
import numpy as np
import pytest

import oracle
import workloads as wl
from gpu_helpers import FORCE_TOL, cutoff_ambiguous, force_error, library

pytestmark = pytest.mark.gpu
SKIN = 0.3


@pytest.fixture(scope="module")
def P():
    return library()


def _lattice(coulomb, m):
    """A simple cubic lattice whose list radius lies between its shells of 32 and 56
    partners (2 and sqrt(5) spacings): 32 entries per NP, the capacity at creation; hot
    enough that the next shell moves in and the lists are built anew several times."""
    cut = 4.0 if coulomb else 2.5
    a = (cut + SKIN) / 2.1
    g = (np.arange(m) - (m - 1) / 2) * a
    x = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
    x = x.astype(np.float32).astype(np.float64)
    n = len(x)
    q = (1.0, -1.0) if coulomb else (0.0, 0.0)
    t = [wl.TypeSpec(sigma=1.0, eps=1.0, mass=1.0, charge=c, gamma=1.0, k_wall=100.0) for c in q]
    sc = wl.Scenario(name="lattice", types=t, n=n, seed=4, dt=1e-3, kT=20.0, R0=2 * a * m,
                     lj_mode=2, lj_cut=2.5, coulomb=coulomb, coulomb_cut=cut if coulomb else 0.0,
                     bjerrum=0.7)
    return sc, x, (np.arange(n) % 2).astype(np.int32)


# a few CTAs; more slots than one CTA per SM holds
@pytest.mark.parametrize("m", [11, 35])
@pytest.mark.parametrize("coulomb", [False, True])
def test_overflow_inside_a_launch(P, coulomb, m):
    sc, x, types = _lattice(coulomb, m)
    with P.Sim(sc, x, None, types) as a, P.Sim(sc, x, None, types) as b:
        b.profile(True)  # one launch per kernel
        assert a.nbr_info()[0] == 32
        builds = a.nbr_info()[2]
        for k in (200, 1, 64):  # the lists grow between the calls
            a.step(k)
            b.step(k)
            for got, ref in zip(a.state(), b.state()):
                assert np.array_equal(got, ref), k
            if k == 200:
                assert a.nbr_info()[0] > 32 and a.nbr_info()[2] >= builds + 3
        assert a.nbr_info()[2] == b.nbr_info()[2]


@pytest.mark.parametrize("coulomb", [False, True])
def test_forces_summed_from_the_cells(P, coulomb):
    """The forces a launch of many steps leaves while lists are too short."""
    sc, x, types = _lattice(coulomb, 11)
    with P.Sim(sc, x, None, types) as sim:
        sim.step(200)
        x1, _, F, _ = sim.state()
        xh = x1.astype(np.float32).astype(np.float64)
    ref = oracle.pair_forces(xh, types, [t.sigma for t in sc.types], [t.eps for t in sc.types],
                             [t.charge for t in sc.types], sc.bjerrum, lj_cut=sc.lj_cut,
                             coulomb=coulomb, coulomb_cut=sc.coulomb_cut)
    keep = ~cutoff_ambiguous(xh, types, sc)
    assert keep.mean() > 0.99
    assert force_error(F, ref)[keep].max() <= FORCE_TOL
