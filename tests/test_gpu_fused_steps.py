"""Many steps per launch, for small droplets on neighbour lists and for NPs without
pair forces: the same bits as the separate kernels (the path taken while the kernels
are timed apart), across list builds, list growth and a regrid, for every integrator
and both list force terms."""
import numpy as np
import pytest

import workloads as wl
from gpu_helpers import library, small, with_

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    return library()


def _scenario(name, n):
    if name == "lj":
        return small(wl.config1(), n)
    if name == "overdamped":
        return with_(small(wl.config1(), n), integrator=1, dt=1e-4)
    if name == "hot":  # moves half a skin in a few steps: a build every few steps
        return with_(small(wl.config1(), n), kT=20.0)
    sc = with_(small(wl.config3(), n), coulomb_cut=4.0)
    return with_(sc, integrator=2, v_kick=0.05, wall_band=True) if name == "printed" else sc


# one NP, a warp's edges, several CTAs, more slots than one CTA per SM holds
@pytest.mark.parametrize("n", [1, 31, 33, 1000, 5003, 40001])
@pytest.mark.parametrize("name", ["lj", "overdamped", "hot", "truncated", "printed"])
def test_same_bits_as_separate_kernels(P, name, n):
    sc = _scenario(name, n)
    types, x, v = wl.initial_state(sc)
    calls = (1, 2, 5, 33) if n > 10000 else (1, 2, 5, 64, 259)
    with P.Sim(sc, x, v, types) as a, P.Sim(sc, x, v, types) as b:
        b.profile(True)  # one launch per kernel
        for k in calls:
            a.step(k)
            b.step(k)
            for got, ref in zip(a.state(), b.state()):
                assert np.array_equal(got, ref), (k,)
            assert np.array_equal(a.forces(1), b.forces(1)), (k,)
        assert a.nbr_info()[2] == b.nbr_info()[2]  # as many list builds


@pytest.mark.parametrize("n", [1, 257, 5000])
@pytest.mark.parametrize("integrator", [0, 1, 2])
@pytest.mark.parametrize("wall", [0, 1, 2])
def test_free_steps_same_bits(P, n, integrator, wall):
    """Without pair forces; steps around the 64 of one launch, up to and past the
    time at which the droplet has gone (R(t) = 0)."""
    sc = small(wl.config3(), n)
    sc = with_(sc, coulomb=False, lj_mode=0, integrator=integrator, g=0.3, omega=0.2, rot_mode=1,
               v_kick=0.02, wall=wall > 0, wall_band=wall == 2)
    sc = with_(sc, k_evap=sc.R0 ** 2 / (200 * sc.dt))
    types, x, v = wl.initial_state(sc)
    with P.Sim(sc, x, v, types) as a, P.Sim(sc, x, v, types) as b:
        b.profile(True)
        for k in (1, 63, 64, 65, 130):
            codes = []
            for s in (a, b):
                try:
                    s.step(k)
                    codes.append(0)
                except P.NpsimError as e:  # an NP left behind by the interface
                    codes.append(e.code)
            assert codes[0] == codes[1]
            for got, ref in zip(a.state(), b.state()):
                assert np.array_equal(got, ref), (k,)
            assert np.array_equal(a.forces(0), b.forces(0)), (k,)


def test_across_a_regrid_and_recorded_frames(P):
    """1100 steps with a regrid at step 1024 in one call equal the separate kernels';
    frames recorded every third step equal the states of single steps."""
    sc = small(wl.config1(), 700)
    types, x, v = wl.initial_state(sc)
    with P.Sim(sc, x, v, types) as a, P.Sim(sc, x, v, types) as b:
        b.profile(True)
        a.step(1100)
        b.step(1100)
        assert a.cell_grid() == b.cell_grid()
        for got, ref in zip(a.state(), b.state()):
            assert np.array_equal(got, ref)
        frames = a.record(9, every=3)
        for f in frames:
            b.step(3)
            assert np.array_equal(f[:, :3], b.state()[0].astype(np.float32))
