"""Launches per step as the dispatch has them."""
import pytest

import workloads as wl
from gpu_helpers import library, small, with_

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,n,separate", [
    ("lists", 1000, 3),    # build, list forces, integrator; else many steps a launch
    ("free", 1000, 1),
])
def test_many_steps_per_launch_only_without_profiling(name, n, separate):
    P = library()
    sc = small(wl.config1(), n)
    if name == "free":
        sc = with_(sc, lj_mode=0)
    types, x, v = wl.initial_state(sc)
    with P.Sim(sc, x, v, types) as sim:
        assert sim.launches_per_step() == 1
        sim.profile(True)
        assert sim.launches_per_step() == separate
        sim.profile(False)
        assert sim.launches_per_step() == 1


def test_separate_kernels():
    P = library()
    for make, n, most in ((wl.config1, 70000, 3), (wl.config3, 3000, 5)):
        sc = small(make(), n)
        types, x, v = wl.initial_state(sc)
        with P.Sim(sc, x, v, types) as sim:
            assert 3 <= sim.launches_per_step() <= most
