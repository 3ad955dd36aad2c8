"""The surrogate's products at the widths where their tiles change: columns that fill
64-column tiles or not, one or several 64-column chunks along K (the last one ragged),
minibatches of one or several 128-row tiles, one network alone or others beside it."""
import numpy as np
import pytest

from oracle import mlp
from gpu_helpers import library

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    return library()


def _pad(X, w):
    out = np.zeros((X.shape[0], w))
    out[:, :X.shape[1]] = X
    return out


@pytest.mark.parametrize("rows", [1, 128, 300])
@pytest.mark.parametrize("n_in,hidden,n_out", [(3, 16, 1), (20, 48, 64), (8, 64, 65), (64, 80, 16),
                                               (8, 192, 130), (33, 256, 256)])
def test_gradients_and_a_step_at_tile_edges(P, n_in, hidden, n_out, rows):
    """BF16 products with FP32 sums against the oracle's float64 network with the same
    rounding points: a value lies a few BF16 steps (2^-8 relative) off where an
    intermediate rounds the other way, so norms agree to 1e-2.  A step of one
    minibatch with every network leaves the AdamW parameters of those gradients."""
    rng = np.random.default_rng(1000 * hidden + rows)
    X = rng.standard_normal((rows, n_in)).astype(np.float32)
    Y = rng.standard_normal((rows, n_out)).astype(np.float32)
    r16 = lambda v: (v + 15) // 16 * 16
    ip, op = r16(n_in), r16(n_out)
    dims = [(hidden, ip), (hidden, hidden), (op, hidden)]
    lr, wd = 1e-3, 1e-2
    with P.Surrogate(n_in=n_in, n_hidden=hidden, n_layers=2, n_out=n_out, n_nets=3, seed=3) as s:
        p0 = [s.get_params(k)[0] for k in range(3)]
        _, loss, yh = s.grads(1, X, Y)
        s.train(X, Y, epochs=1, batch=rows, lr=lr, wd=wd, seed=0)
        after = [s.get_params(k) for k in range(3)]
    for k in range(3):
        flat, (p1, g) = p0[k], after[k]
        lo, go, yo = mlp.loss_and_grads(mlp.unflatten(flat, dims), _pad(X, ip), _pad(Y, op),
                                        n_valid=n_out, m_valid=rows, bf=True)
        if k == 1:
            assert np.abs(yh - yo[:, :n_out]).max() <= 1e-2 * max(1.0, np.abs(yo).max())
            assert loss == pytest.approx(lo, rel=1e-2)
        for l, ((gW, gb), (oW, ob)) in enumerate(zip(mlp.unflatten(g, dims), go)):
            assert np.linalg.norm(gW - oW) <= 1e-2 * np.linalg.norm(oW), (k, l)
            assert np.linalg.norm(gb - ob) <= 1e-2 * np.linalg.norm(ob) + 1e-12, (k, l)
        dec = np.concatenate([np.r_[np.full(o * i, wd), np.zeros(o)] for o, i in dims])
        w1, _, _ = mlp.adamw(flat.astype(np.float64), g.astype(np.float64), 0.0, 0.0, 1, lr, wd=dec)
        live = (flat != 0) | (g != 0)
        sel = live & (np.abs(g) > 1e-6)
        assert np.abs(p1[sel] - w1[sel]).max() <= 1e-3 * lr + 1e-6 * np.abs(flat[sel]).max()
        assert np.all(p1[~live] == 0)


@pytest.mark.parametrize("nets", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("scale", [1e-25, 1.0, 1e12])
def test_mean_and_spread_over_the_networks(P, nets, scale):
    """Against float64 statistics of each network's own float32 predictions (one
    network alone with the same parameters gives its outputs, and a spread of what
    rounding leaves of v^2 - v v, below 2^-26 of v).  The
    outputs differ by an offset of about their own size, so neither the mean nor the
    spread cancels; the float32 rounding of the single outputs (2^-24) moves the mean
    and the spread by at most 4 x 2^-24 of the largest output."""
    rng = np.random.default_rng(nets)
    X = rng.standard_normal((200, 5)).astype(np.float32)
    kw = dict(n_in=5, n_hidden=32, n_layers=2, n_out=7)
    ym = (scale * rng.standard_normal(7)).astype(np.float32)
    ys = (scale * (1 + rng.random(7))).astype(np.float32)
    one = (np.zeros(5, np.float32), np.ones(5, np.float32), ym, ys)
    with P.Surrogate(n_nets=nets, seed=9, **kw) as s:
        s.set_norm(*one)
        m, sp = s.predict(X)
        flats = [s.get_params(k)[0] for k in range(nets)]
    outs = []
    for f in flats:
        with P.Surrogate(n_nets=1, seed=1, **kw) as s:
            s.set_norm(*one)
            s.set_params(0, f)
            y, z = s.predict(X)
            assert np.all(z <= 2.0 ** -26 * np.abs(y))
            outs.append(y.astype(np.float64))
    outs = np.array(outs)
    tol = 4 * 2.0 ** -24 * np.abs(outs).max()
    assert np.abs(m - outs.mean(0)).max() <= tol
    assert np.abs(sp - outs.std(0)).max() <= tol
