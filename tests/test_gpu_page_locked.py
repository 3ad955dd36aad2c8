"""Results into host arrays that lie back to back but are page-locked one by one: no copy
may span two of them."""
import mmap

import numpy as np
import pytest

import workloads as wl
from gpu_helpers import library, small

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
PAGE = 65536  # a multiple of every page size


class Parts:
    """`count` parts of `size` bytes of one mapping, each registered by itself."""

    def __init__(self, size, count):
        assert size % PAGE == 0
        self.m = mmap.mmap(-1, size * count + PAGE)
        whole = np.frombuffer(self.m, np.uint8)
        o = -whole.ctypes.data % PAGE
        self.parts = [whole[o + k * size:o + (k + 1) * size] for k in range(count)]
        self.rt = torch.cuda.cudart()

    def __enter__(self):
        torch.zeros(1, device="cuda")
        for p in self.parts:
            assert int(self.rt.cudaHostRegister(p.ctypes.data, p.nbytes, 0)) == 0
        return self.parts

    def __exit__(self, *exc):
        for p in self.parts:
            self.rt.cudaHostUnregister(p.ctypes.data)


@pytest.fixture(scope="module")
def P():
    return library()


def test_state(P):
    n = 8192  # 24 n bytes a part
    sc = small(wl.config1(), n)
    types, x, v = wl.initial_state(sc)
    with P.Sim(sc, x, v, types) as sim, Parts(24 * n, 3) as parts:
        sim.step(3)
        out = tuple(p.view(np.float64).reshape(n, 3) for p in parts)
        got, want = P.npsim_get_state(sim.h, n, out), sim.state()
        for a, b in zip(got, want):
            assert np.array_equal(a, b)
        sim.step(1)  # no error is left behind


def test_prediction(P):
    B, n_out = 256, 64  # 65536 bytes a part
    X = np.random.default_rng(3).standard_normal((B, 8)).astype(np.float32)
    with P.Surrogate(8, 64, 2, n_out, n_nets=3, seed=1) as s, Parts(4 * B * n_out, 2) as parts:
        want = s.predict(X)
        mean, spread = (p.view(np.float32).reshape(B, n_out) for p in parts)
        f = P.C.POINTER(P.C.c_float)
        rc = P.lib().npsim_surr_predict(s.h, X.ctypes.data_as(f), B, mean.ctypes.data_as(f),
                                        spread.ctypes.data_as(f))
        assert rc == 0, P.lib().npsim_last_error()
        assert np.array_equal(mean, want[0]) and np.array_equal(spread, want[1])
        assert np.array_equal(s.predict(X)[0], want[0])
