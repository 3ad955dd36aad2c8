"""The pair histogram's float32 classification and the box counts of several scales
per launch against the oracle's float64 integers, where they can go wrong: distances
on bin boundaries, coordinates large against the bin width, one to thousands of bins,
a range beyond the whole cloud, and coincident positions."""
import numpy as np
import pytest

import oracle
import workloads as wl
from gpu_helpers import library

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    return library()


def _cloud(kind, n):
    rng = np.random.default_rng(n + len(kind))
    if kind == "lattice":  # every distance sqrt(k) / 2, many of them on bin boundaries
        m = int(np.ceil(n ** (1.0 / 3.0)))
        g = np.stack(np.meshgrid(*[np.arange(m) * 0.5] * 3, indexing="ij"), -1).reshape(-1, 3)
        return g[:n] - 0.25 * m
    if kind == "far":  # lo words of 1e-5: the hi words alone misplace the pairs
        return rng.uniform(-2.0, 2.0, (n, 3)) + np.array([400.0, -300.0, 350.0])
    x = rng.uniform(-6.0, 6.0, (n, 3))
    x[n // 2:] = x[:n - n // 2]  # coincident pairs
    return x


@pytest.mark.parametrize("kind", ["lattice", "far", "coincident"])
@pytest.mark.parametrize("n", [1, 2, 129, 1500])
def test_counts_equal_the_oracle(P, kind, n):
    x = _cloud(kind, n)
    t = wl.TypeSpec(sigma=1.0, eps=1.0, mass=1.0, charge=0.0, gamma=1.0, k_wall=0.0)
    sc = wl.Scenario(name="cloud", types=[t], n=n, R0=1000.0, wall=False, lj_mode=0,
                     coulomb=False)
    with P.Sim(sc, x, None, np.zeros(n, np.int32)) as sim:
        xg = sim.state()[0]
        for r_max, bins in ((4.0, 128), (4.0, 1), (0.3, 7), (50.0, 1100), (3.0, 2500),
                            (6.0, 5000), (2.0, 200000)):
            st = sim.stats(r_max=r_max, n_bins=bins, radial_bins=3, boxcount=True)
            assert np.array_equal(st["rdf_counts"], oracle.pair_hist(xg, r_max, bins)), (r_max, bins)
        if n > 2:
            Rg, _, _ = oracle.rg(xg, 1.0)
            assert np.array_equal(st["nbox"], oracle.boxcount_df(xg, 1.0, Rg)[1])
