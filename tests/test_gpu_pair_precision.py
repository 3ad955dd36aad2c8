"""Rounding of the each-pair-once kernels against float64, by thirds of the order in which
the NPs are summed (late NPs get most of their force as partners): no worse than that of
the one-sided kernels with tiles of 256 partners, which add 128 terms before each
compensated sum, and for a long Coulomb sum with tiles of 512."""
import numpy as np
import pytest

import oracle
import workloads as wl
from gpu_helpers import library, small, with_

pytestmark = pytest.mark.gpu
# both sides are rms values over 4000 or more components of a third: 1.1 % sampling error
# each for a normal distribution; 5 % allowed
TOL = 1.05


@pytest.fixture(scope="module")
def P():
    return library()


def _errors(P, monkeypatch, sc, state, ref, thirds, shape):
    """Launch shape and rms errors by thirds (shape None: the autotuner's)."""
    types, x, v = state
    if shape is None:
        monkeypatch.delenv("NPSIM_AUTOTUNE", raising=False)
    else:
        monkeypatch.setenv("NPSIM_AUTOTUNE", f"1:{shape}")
    with P.Sim(sc, x, v, types) as sim:
        cfg = sim.allpairs_config()
        if shape is not None and cfg["index"] != shape:
            return cfg, None
        e = sim.forces(3) - ref
    return cfg, [np.sqrt((e[t] ** 2).mean()) for t in thirds]


@pytest.mark.parametrize("n,tile", [(4000, 256), (16384, 256), (22801, 512), (33001, 512)])
def test_partner_sums_round_no_more_than_row_sums(P, monkeypatch, n, tile):
    sc = with_(small(wl.config2(), n), lj_mode=0)
    state = types, x, v = wl.initial_state(sc, fp32_positions=True)
    ref = oracle.pair_forces(x, types, [t.sigma for t in sc.types], [t.eps for t in sc.types],
                             [t.charge for t in sc.types], sc.bjerrum, lj=False)
    order = np.argsort(types, kind="stable")  # Coulomb alone: index order inside a type
    thirds = [order[k * n // 3:(k + 1) * n // 3] for k in range(3)]
    args = P, monkeypatch, sc, state, ref, thirds
    shapes = {i: _errors(*args, i) for i in range(P.npsim_allpairs_num_configs())}
    allowed = [r for c, r in shapes.values()
               if r and c["packed"] == 1 and c["j_tile"] == tile][0]
    # every LJ + Coulomb kernel, whatever the length, and the one the autotuner picks
    got = [(c, r) for c, r in shapes.values() if r and c["packed"] == 3 and c["j_tile"] <= 128]
    assert len(got) >= 5
    got.append(_errors(*args, None))
    for c, r in got:
        for a, b in zip(r, allowed):
            assert a <= TOL * b, (c, r, allowed)
