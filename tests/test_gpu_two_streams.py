"""Simulations on neighbour lists stepped from several threads at once, each on a stream of
its own: their launches of many steps and their list builds hold grid barriers, and whatever
else runs, every block of such a launch has to be resident.  The same bits as one after
another."""
import threading

import numpy as np
import pytest

import workloads as wl
from gpu_helpers import library, small, with_

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def P():
    return library()


def _run(P, sc, state, out, k):
    types, x, v = state
    with P.Sim(sc, x, v, types, stream=torch.cuda.Stream()) as sim:
        for steps in (7, 300, 300, 1):
            sim.step(steps)
        out[k] = sim.state() + (sim.forces(1),)


# launches of many steps (one CTA and two per SM); builds inside captured graphs, alone and
# beside all-pairs sums.  Hot: a build every few steps
@pytest.mark.parametrize("sizes", [((wl.config1, 1000), (wl.config1, 45001)),
                                   ((wl.config1, 60001), (wl.config1, 50003)),
                                   ((wl.config1, 30001), (wl.config1, 70001), (wl.config3, 6001))])
def test_at_once_as_one_after_another(P, sizes):
    scs = [with_(small(make(), n), kT=5.0) for make, n in sizes]
    states = [wl.initial_state(sc) for sc in scs]
    alone, at_once = {}, {}
    for k, sc in enumerate(scs):
        _run(P, sc, states[k], alone, k)
    for _ in range(2):
        at_once.clear()
        threads = [threading.Thread(target=_run, args=(P, sc, states[k], at_once, k))
                   for k, sc in enumerate(scs)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        assert sorted(at_once) == sorted(alone)  # none of them raised
        for k in alone:
            for a, b in zip(alone[k], at_once[k]):
                assert np.array_equal(a, b), k
