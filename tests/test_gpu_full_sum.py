"""sum_neutral with LJ in the pair sum: the Coulomb term is evaluated for pairs without a
charge product too, by every launch shape."""
import numpy as np
import pytest

import oracle
import workloads as wl
from gpu_helpers import FORCE_TOL, cutoff_ambiguous, force_error, library, small, with_

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    return library()


def _shapes(P, monkeypatch, sc, state):
    types, x, v = state
    for idx in range(P.npsim_allpairs_num_configs()):
        monkeypatch.setenv("NPSIM_AUTOTUNE", f"1:{idx}")
        with P.Sim(sc, x, v, types) as sim:
            if sim.allpairs_config()["index"] == idx:
                yield idx, sim


def _scenario(n, full):
    types = [wl.stokes_type(1.0, 1.0, frac=0.4), wl.stokes_type(1.5, 0.0, frac=0.3),
             wl.stokes_type(1.0, -0.5, frac=0.3)]
    return with_(small(wl.config2(), n), types=types, sum_neutral=full)


# one row tile; several
@pytest.mark.parametrize("n", [700, 5003])
def test_forces(P, monkeypatch, n):
    sc = _scenario(n, True)
    state = types, x, v = wl.initial_state(sc, fp32_positions=True)
    ref = oracle.pair_forces(x, types, [t.sigma for t in sc.types], [t.eps for t in sc.types],
                             [t.charge for t in sc.types], sc.bjerrum, lj_cut=sc.lj_cut)
    keep = ~cutoff_ambiguous(x, types, sc)
    ran = 0
    for idx, sim in _shapes(P, monkeypatch, sc, state):
        ran += 1
        assert force_error(sim.forces(1), ref)[keep].max() <= FORCE_TOL, idx
    assert ran > 6


@pytest.mark.parametrize("full", [True, False])
@pytest.mark.parametrize("n", [700, 5003])
def test_neutral_pairs_are_evaluated(P, monkeypatch, n, full):
    """A neutral NP beyond the float32 range (zero times an infinite distance: not a
    number) shows which pairs are evaluated: with sum_neutral it reaches the Coulomb force
    of every charged NP.  LJ does not act between charged and neutral types.  The default
    sum may leave such pairs out; the kernels that evaluate each pair once do."""
    eps = np.array([[1.0, 0.0, 1.0], [0.0, 1.0, 0.0], [1.0, 0.0, 1.0]])
    sc = with_(_scenario(n, full), eps_override=eps)
    state = types, x, v = wl.initial_state(sc, fp32_positions=True)
    charged = types != 1
    far = x.copy()
    far[np.flatnonzero(types == 1)[7]] = [1e300, 0.0, 0.0]
    ran = 0
    for idx, sim in _shapes(P, monkeypatch, sc, state):
        sim.set_state(far, v, 0)
        F = sim.forces(1)[charged]
        if full:
            assert np.isnan(F).any(1).all(), idx
        elif sim.allpairs_config()["packed"] == 3 and sim.allpairs_config()["j_tile"] <= 128:
            assert np.isfinite(F).all(), idx
        ran += 1
    assert ran > 6
