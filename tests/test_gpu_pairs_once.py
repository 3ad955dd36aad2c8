"""The all-pairs kernels that evaluate each pair once: every launch shape against
the FP64 oracle at sizes around the tiles' and groups' edges, for charge products
on both sides of the sums' unit (ordinary, far below it, zero)."""
import numpy as np
import pytest

import oracle
import workloads as wl
from gpu_helpers import FORCE_TOL, cutoff_ambiguous, force_error, library, small, with_

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    return library()


def _pair(sc, x, types, lj=True, coul=True):
    return oracle.pair_forces(x, types, [t.sigma for t in sc.types], [t.eps for t in sc.types],
                              [t.charge for t in sc.types], sc.bjerrum, lj_cut=sc.lj_cut,
                              lj=lj and sc.lj_mode != 0, coulomb=coul and sc.coulomb)


# around the 64-partner segment, the 256-position block, the 512-position group
# padding, the 1024-row tile, and several row tiles with a ragged end
@pytest.mark.parametrize("n", [1, 2, 65, 257, 513, 1025, 2700])
@pytest.mark.parametrize("charges", [(1.0, -1.0), (0.7, 2e-5), (3e-4, 0.0), (0.0, 0.0)])
def test_every_shape_at_tile_edges(P, monkeypatch, n, charges):
    sc = small(wl.config2(), n)
    sc = with_(sc, types=[wl.stokes_type(1.0, charges[0], frac=0.6),
                          wl.stokes_type(2.0, charges[1], eps=0.5, frac=0.4)])
    types, x, v = wl.initial_state(sc, fp32_positions=True)
    for lj_mode in (1, 0):  # LJ + Coulomb, Coulomb only
        s = with_(sc, lj_mode=lj_mode)
        ref = [_pair(s, x, types), _pair(s, x, types, coul=False), _pair(s, x, types, lj=False)]
        keep = ~cutoff_ambiguous(x, types, s)
        ran = 0
        for idx in range(P.npsim_allpairs_num_configs()):
            monkeypatch.setenv("NPSIM_AUTOTUNE", f"1:{idx}")
            with P.Sim(s, x, v, types) as sim:
                if sim.allpairs_config()["index"] != idx:
                    continue
                ran += 1
                for what, r in zip((1, 2, 3), ref):
                    F = sim.forces(what)
                    if not np.any(r):
                        assert np.all(F == 0), (idx, what)
                        continue
                    assert force_error(F, r)[keep].max() <= FORCE_TOL, (idx, what)
                    assert np.array_equal(F, sim.forces(what)), (idx, what)
        assert ran > 0


@pytest.mark.parametrize("n", [700, 3001, 20011])
def test_full_sum_keeps_to_the_kernels_that_evaluate_every_pair(P, n):
    """sum_neutral asks for the Coulomb term of all N(N-1) pairs: the LJ + Coulomb
    kernels (packed 3), which pass over type pairs without a charge product, are not
    chosen for it."""
    sc = with_(small(wl.config3(), n), sum_neutral=True)
    types, x, v = wl.initial_state(sc, fp32_positions=True)
    with P.Sim(sc, x, v, types) as sim:
        assert sim.allpairs_config()["packed"] != 3
