"""Scratch of the launch-shape tuners: where the largest does not fit only the shapes that
need it drop out, such a choice is not kept for later objects, and tiles of few rows are no
candidates where their partner sums grow large."""
import re

import numpy as np
import pytest

import oracle
import workloads as wl
from gpu_helpers import FORCE_TOL, force_error, library, small, with_

pytestmark = pytest.mark.gpu
MB = 1 << 20


@pytest.fixture(scope="module")
def P():
    return library()


@pytest.fixture
def timed(monkeypatch, capfd):
    """A function that creates an object and returns it with the shapes the tuner timed
    (rows per tile by index)."""
    monkeypatch.setenv("NPSIM_AUTOTUNE_LOG", "1")
    monkeypatch.delenv("NPSIM_AUTOTUNE", raising=False)
    monkeypatch.delenv("NPSIM_ENS_SHAPE", raising=False)

    def make(create, limit=None):
        if limit is None:
            monkeypatch.delenv("NPSIM_TUNE_BYTES", raising=False)
        else:
            monkeypatch.setenv("NPSIM_TUNE_BYTES", str(limit))
        capfd.readouterr()
        obj = create()
        log = capfd.readouterr().err
        return obj, {int(i): int(b) * int(k) for i, b, k in
                     re.findall(r"shape (\d+) <(\d+),(\d+),\d+>", log)}

    return make


def _droplet(n, seed=1):
    sc = with_(small(wl.config2(seed=seed), n), lj_mode=0)
    return (sc,) + wl.initial_state(sc, fp32_positions=True)


def test_single_droplet(P, timed):
    sc, types, x, v = _droplet(61003)
    create = lambda: P.Sim(sc, x, v, types)
    rows = np.arange(0, len(x), 211, dtype=np.int64)
    ref = oracle.pair_forces(x, types, [t.sigma for t in sc.types], [t.eps for t in sc.types],
                             [t.charge for t in sc.types], sc.bjerrum, lj=False, sel=rows)
    rms = np.sqrt((ref ** 2).sum(1).mean())
    seen = []
    for limit in (160 * MB, 100 * MB, 40 * MB):
        sim, shapes = timed(create, limit)
        with sim:
            cfg = sim.allpairs_config()
            err = np.linalg.norm(sim.forces(3)[rows] - ref, axis=1)
        assert (err <= FORCE_TOL * np.maximum(np.linalg.norm(ref, axis=1), rms)).all()
        seen.append((shapes, cfg))
    full, all_shapes = timed(create)
    full.close()
    assert all_shapes, "a choice from a part of the shapes was kept"
    parts = [(s, c) for s, c in seen if s and set(s) < set(all_shapes)]
    assert parts
    # each-pair-once shapes (j-tiles of at most 128) among what still fits
    assert any(c["packed"] >= 2 and c["j_tile"] <= 128 for _, c in parts)
    again, shapes = timed(create)
    again.close()
    assert not shapes  # the full choice is kept


def test_ensemble(P, timed):
    drops = [_droplet(n, 2 + n) for n in (21007, 3001)]
    drops = [(with_(sc, lj_mode=1), x, v, types) for sc, types, x, v in drops]
    create = lambda: P.Ensemble(drops)
    seen = []
    for limit in (60 * MB, 56 * MB, 52 * MB, 48 * MB, 44 * MB, 40 * MB):
        try:
            ens, shapes = timed(create, limit)
        except P.NpsimError as e:  # not even the smallest
            assert e.code == -5
            continue
        with ens:
            seen.append((shapes, ens.config()))
            F = ens.forces(0)
        assert np.isfinite(F).all()
    ens, all_shapes = timed(create)
    ens.close()
    assert all_shapes
    parts = [(s, c) for s, c in seen if s and set(s) < set(all_shapes)]
    assert any(c["j_tile"] <= 128 for _, c in parts)
    ens, shapes = timed(create)
    ens.close()
    assert not shapes


def test_small_tiles_of_a_large_droplet(P, timed):
    """Partner sums of 128-row tiles: 6 n^2 / 128 bytes, above 512 MiB from 107000 NPs."""
    sc, types, x, v = _droplet(110003)
    sim, shapes = timed(lambda: P.Sim(sc, x, v, types))
    sim.close()
    once = [r for i, r in shapes.items() if r >= 256]
    assert once and 128 not in shapes.values()
    ens, shapes = timed(lambda: P.Ensemble([(with_(sc, lj_mode=1), x, v, types)]))
    ens.close()
    assert max(shapes.values()) == 1024 and 128 not in shapes.values()
