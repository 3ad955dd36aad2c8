"""Failure path of the list kernels' grid barrier, without a stuck GPU: with the bound
of its waits cut short in one simulation, the launch that meets it gives up, the launches
queued behind it leave the lists alone, every call that may build lists reports
NPSIM_ERR_TIMEOUT, and after npsim_set_state the simulation is as good as a new one."""
import numpy as np
import pytest

import workloads as wl
from gpu_helpers import library, small, with_

pytestmark = pytest.mark.gpu
TIMEOUT = -4


@pytest.fixture(scope="module")
def P():
    return library()


# many steps per launch; one launch per kernel (the path while kernels are timed apart);
# too many NPs for the former; with an all-pairs sum beside the lists.  Hot enough that
# the lists are built anew within a few steps.
CASES = {"fused": (wl.config1, 1000), "separate": (wl.config1, 1000),
         "large": (wl.config1, 70001), "paper": (wl.config3, 3001)}


def _make(P, name):
    make, n = CASES[name]
    sc = with_(small(make(), n), kT=20.0)
    types, x, v = wl.initial_state(sc)
    sim = P.Sim(sc, x, v, types)
    if name == "separate":
        sim.profile(True)
    return sim, x, v


def _expires(P, call, *args):
    with pytest.raises(P.NpsimError) as e:
        call(*args)
    assert e.value.code == TIMEOUT


def _as_new(P, name, sim, x, v):
    P.npsim_test_list_wait(sim.h, -1)
    sim.set_state(x, v, 0)
    fresh = _make(P, name)[0]
    with fresh:
        for k in (0, 1, 40):
            sim.step(k)
            fresh.step(k)
            for got, ref in zip(sim.state(), fresh.state()):
                assert np.array_equal(got, ref), k
            assert np.array_equal(sim.forces(1), fresh.forces(1)), k


@pytest.mark.parametrize("name", list(CASES))
def test_every_call_reports_it_and_a_new_state_recovers(P, name):
    sim, x, v = _make(P, name)
    with sim:
        sim.step(3)
        P.npsim_test_list_wait(sim.h, 0)
        _expires(P, sim.step, 600)  # several launches queued behind the one that gives up
        # steps of many per launch that were not finished are not counted
        assert sim.state()[3] == (3 if name == "fused" else 603)
        _expires(P, sim.forces, 1)
        # 903 steps so far: the cell grid, which follows the droplet every 1024 steps, is
        # still the one of a new simulation
        _expires(P, sim.record, 300, 150)
        _expires(P, sim.set_state, x, v, 0)
        _as_new(P, name, sim, x, v)


@pytest.mark.parametrize("polls", [1, 30, 200])
@pytest.mark.parametrize("name", list(CASES))
def test_some_blocks_give_up(P, name, polls):
    """A bound that some blocks of a launch may meet and others not."""
    sim, x, v = _make(P, name)
    with sim:
        P.npsim_test_list_wait(sim.h, polls)
        try:
            sim.step(600)
        except P.NpsimError as e:
            assert e.code == TIMEOUT
        _as_new(P, name, sim, x, v)


@pytest.mark.parametrize("name", ["fused", "separate"])
def test_reported_before_a_non_finite_position(P, name):
    """Both bits in the error word: the barrier is put right all the same."""
    sim, x, v = _make(P, name)
    with sim:
        bad = x.copy()
        bad[5] = [1e300, 0.0, 0.0]  # beyond float32
        sim.set_state(bad, v, 0)
        P.npsim_test_list_wait(sim.h, 0)
        _expires(P, sim.step, 2)
        _as_new(P, name, sim, x, v)


def test_bound_out_of_range(P):
    sim = _make(P, "fused")[0]
    with sim:
        for polls in (-2, 1 << 32):
            with pytest.raises(P.NpsimError) as e:
                P.npsim_test_list_wait(sim.h, polls)
            assert e.value.code == -1
    sc = small(wl.config2(), 600)  # no lists
    types, x, v = wl.initial_state(sc)
    with P.Sim(sc, x, v, types) as sim:
        with pytest.raises(P.NpsimError):
            P.npsim_test_list_wait(sim.h, 0)
