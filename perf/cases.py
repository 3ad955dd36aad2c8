"""Timed workloads of the nanoparticle library, through its Python binding.

Each case is one call sequence of a user's program on prepared inputs: steps of a
droplet followed by a read of the state, forces at one configuration, recorded
frames, statistics of an aggregate, an ensemble of droplets, training and
prediction of the surrogate.  Physics, compositions and sizes are those of the
repository's workloads (one-type LJ droplet of 1000 NPs, two-type charged droplet
of 16384, three-type droplet of 250000, ensembles with N log-uniform up to 32768,
surrogate 8 -> 4 x 256 -> 65) and the ranges around them.

Positions and velocities are made representable in float32, as after a restart from
recorded frames.  The device keeps velocities as float32 and positions and forces as
float32 (hi, lo) pairs, so states are returned as float32 words.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2501_04456_gb300 as P

BJERRUM = 0.7
SLOW = 400000  # steps of the whole evaporation: a pass sees a small part of it


# ---------------------------------------------------------------------------
# Cases


def listed():
    return [
        # the plain model's droplet: launches and latency are all there is
        {"name": "lj1000", "kind": "lj", "n": 1000, "steps": 100, "integrator": 0},
        # two charged types, LJ and Coulomb in one all-pairs sum
        {"name": "ljc16384", "kind": "ljc", "n": 16384, "steps": 64, "integrator": 0},
        # the paper-scale droplet: all-pairs Coulomb, LJ from neighbour lists
        {"name": "paper250000", "kind": "paper", "n": 250000, "steps": 8, "integrator": 0,
         "sum_neutral": False},
        # a dried aggregate under LJ alone: about 90 list partners per NP
        {"name": "dense262144", "kind": "dense", "n": 262144, "steps": 64, "integrator": 0},
        # the printed interaction model (truncated Coulomb, band wall, fixed kick) with
        # every tenth frame recorded to the host
        {"name": "printed250000", "kind": "printed", "n": 250000, "steps": 100, "every": 10},
        # the integrator alone on a state larger than L2, last frame recorded
        {"name": "free4000000", "kind": "free", "n": 4000000, "steps": 200, "every": 200,
         "integrator": 0},
        # pair forces of one configuration, all terms together and each alone, odd size
        {"name": "forces30011", "kind": "forces", "n": 30011, "model": "ljc"},
        # many small droplets in one launch
        {"name": "ens16_small", "kind": "ens", "drops": 16, "n_min": 512, "n_max": 4096,
         "steps": 32},
        # droplets of uneven size, the largest as in the full ensemble
        {"name": "ens48", "kind": "ens", "drops": 48, "n_min": 512, "n_max": 32768, "steps": 32},
        # RDF, concentration, R_g and box counting of a final aggregate
        {"name": "stats200000", "kind": "stats", "n": 200000, "dense": True, "r_max": 10.0,
         "bins": 128, "radial": 64},
        # a what-if query of the surrogate
        {"name": "predict4096", "kind": "predict", "batch": 4096, "nets": 4},
        # training of the surrogate's networks
        {"name": "train2048", "kind": "train", "samples": 2048, "batch": 256, "nets": 4,
         "epochs": 2},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lj", "ljc", "paper", "dense", "printed", "free", "forces", "ens", "stats",
                       "predict", "train"])
    if kind == "lj":
        return {"kind": kind, "n": _log(rng, 300, 100000), "steps": rng.randint(40, 100),
                "integrator": rng.choice([0, 0, 1])}
    if kind == "ljc":
        return {"kind": kind, "n": _log(rng, 500, 20000), "steps": rng.randint(16, 64),
                "integrator": rng.choice([0, 0, 1])}
    if kind == "paper":
        neutral = rng.random() < 0.25
        return {"kind": kind, "n": _log(rng, 4000, 80000 if neutral else 250000),
                "steps": rng.randint(4, 8), "integrator": 0, "sum_neutral": neutral}
    if kind == "dense":
        return {"kind": kind, "n": _log(rng, 5000, 262144), "steps": rng.randint(16, 64),
                "integrator": rng.choice([0, 0, 1])}
    if kind == "printed":
        every = rng.choice([5, 7, 10, 20])
        return {"kind": kind, "n": _log(rng, 5000, 250000), "steps": every * rng.randint(3, 5),
                "every": every}
    if kind == "free":
        steps = rng.randint(50, 200)
        return {"kind": kind, "n": _log(rng, 100000, 4000000), "steps": steps, "every": steps,
                "integrator": rng.choice([0, 1])}
    if kind == "forces":
        return {"kind": kind, "n": _log(rng, 700, 60000), "model": rng.choice(["ljc", "paper"])}
    if kind == "ens":
        lo = _log(rng, 300, 1500)
        return {"kind": kind, "drops": rng.randint(3, 48), "n_min": lo,
                "n_max": _log(rng, 2 * lo, 24000), "steps": rng.randint(8, 32)}
    if kind == "stats":
        return {"kind": kind, "n": _log(rng, 2000, 200000), "dense": rng.random() < 0.6,
                "r_max": round(rng.uniform(4.0, 10.0), 2), "bins": rng.choice([64, 100, 128, 200]),
                "radial": rng.choice([0, 50, 64])}
    if kind == "predict":
        return {"kind": kind, "batch": _log(rng, 1, 8192), "nets": rng.choice([1, 4, 5])}
    return {"kind": kind, "samples": _log(rng, 300, 2048), "batch": rng.choice([64, 200, 256, 512]),
            "nets": rng.choice([1, 4]), "epochs": rng.randint(1, 2)}


# ---------------------------------------------------------------------------
# Inputs


def _type(sigma, charge=0.0, eps=1.0, gamma=None, k_wall=100.0, frac=1.0):
    """NP type of uniform density with Stokes friction (mass sigma^3, m gamma = sigma)."""
    m = sigma ** 3
    return SimpleNamespace(sigma=sigma, eps=eps, mass=m, charge=charge,
                           gamma=sigma / m if gamma is None else gamma, k_wall=k_wall, frac=frac)


def _scenario(types, **kw):
    sc = dict(types=types, seed=1, dt=5e-4, kT=1.0, R0=10.0, k_evap=0.0, g=0.0, omega=0.0,
              rot_mode=0, bjerrum=0.0, lj_cut=2.5, coulomb=False, lj_mode=1, integrator=0,
              wall=True, wall_band=False, v_kick=0.0, coulomb_cut=0.0, eps_override=None,
              sum_neutral=False)
    sc.update(kw)
    return SimpleNamespace(**sc)


def _f32(a):
    return np.asarray(a, np.float64).astype(np.float32).astype(np.float64)


def _assign(types, n):
    t = np.full(n, len(types) - 1, np.int32)
    start = 0
    for a, ty in enumerate(types[:-1]):
        cnt = int(round(ty.frac * n))
        t[start:start + cnt] = a
        start += cnt
    return t


def _cubic_sites(a, R):
    m = int(R / a) + 1
    k = np.arange(-m, m + 1) * a
    g = np.stack(np.meshgrid(k, k, k, indexing="ij"), -1).reshape(-1, 3) + 0.5 * a
    return g[(g * g).sum(1) <= R * R]


def _dilute(rng, types, t, R):
    """Random positions in the ball without overlaps: jittered sites of a cubic lattice,
    taken in random order (no relation between index and place)."""
    n = len(t)
    smax = max(ty.sigma for ty in types)
    a = (4.0 / 3.0 * math.pi * R ** 3 / n) ** (1.0 / 3.0)
    sites = _cubic_sites(a, R - 0.5 * smax)
    while len(sites) < n:
        a *= 0.985
        sites = _cubic_sites(a, R - 0.5 * smax)
    x = sites[rng.permutation(len(sites))[:n]]
    j = max(0.0, 0.5 * (a - 0.95 * smax))
    return x + rng.uniform(-j, j, (n, 3))


def _aggregate(rng, types, t):
    """A compact ball of the types in concentric shells, the largest NPs inside, each shell a
    slightly expanded FCC lattice; returns positions and the ball's radius."""
    x = np.zeros((len(t), 3))
    r_in, prev = 0.0, 0.0
    for a in sorted(range(len(types)), key=lambda k: -types[k].sigma):
        idx = np.nonzero(t == a)[0]
        if not len(idx):
            continue
        s = types[a].sigma
        c = 1.1 * s * math.sqrt(2.0)  # cubic cell edge, nearest neighbours at 1.1 sigma
        r0 = r_in + (0.55 * (prev + s) if prev else 0.0)
        R = (r0 ** 3 + 1.3 * len(idx) * c ** 3 / 4.0 / (4.0 / 3.0 * math.pi)) ** (1.0 / 3.0) + 2 * c
        cub = _cubic_sites(c, R)
        f = np.array([[0, 0, 0], [.5, .5, 0], [.5, 0, .5], [0, .5, .5]]) * c
        sites = (cub[:, None, :] + f[None]).reshape(-1, 3)
        r = np.sqrt((sites * sites).sum(1))
        sites, r = sites[r >= r0], r[r >= r0]
        order = np.argsort(r, kind="stable")[:len(idx)]
        sites, r = sites[order], r[order]
        x[rng.permutation(idx)] = sites + rng.uniform(-0.03 * s, 0.03 * s, sites.shape)
        r_in, prev = float(r[-1]), s
    return x, r_in + prev


def _evaporation(R0, Rf, n_steps, dt):
    return (R0 * R0 - Rf * Rf) / (n_steps * dt)


def _droplet(rng, kind, n, integrator=0, sum_neutral=False):
    """(scenario, x, v, types) of one droplet of the named composition."""
    seed = int(rng.integers(1 << 40))
    if kind == "lj":  # one type, R0 = 30 at 1000 NPs
        types = [_type(1.0)]
        R = 30.0 * (n / 1000.0) ** (1.0 / 3.0)
        sc = _scenario(types, dt=1e-3, R0=R, k_evap=_evaporation(R, 2 * R / 3, SLOW, 1e-3),
                       lj_mode=2)
    elif kind == "ljc":  # two charged types, R0 = 80 at 16384 NPs
        types = [_type(1.0, +1.0, frac=0.75), _type(2.0, -1.0, frac=0.25)]
        R = 80.0 * (n / 16384.0) ** (1.0 / 3.0)
        sc = _scenario(types, R0=R, k_evap=_evaporation(R, 0.375 * R, SLOW, 5e-4), g=0.01,
                       omega=0.05, rot_mode=1, bjerrum=BJERRUM, coulomb=True, lj_mode=1)
    elif kind in ("paper", "printed"):  # three types, R0 = 200 at 250000 NPs
        types = [_type(1.0, 0.0, frac=0.6), _type(1.5, +0.5, frac=0.3),
                 _type(3.0, -0.5, frac=0.1)]
        R = 200.0 * (n / 250000.0) ** (1.0 / 3.0)
        sc = _scenario(types, R0=R, k_evap=_evaporation(R, 0.3 * R, SLOW, 5e-4),
                       bjerrum=BJERRUM, coulomb=True, lj_mode=2, sum_neutral=sum_neutral)
        if kind == "printed":
            sc.coulomb_cut, sc.integrator, sc.v_kick, sc.wall_band = 4.0, 2, 0.03, True
    elif kind == "dense":  # LJ only, dried
        types = [_type(1.0, frac=0.6), _type(1.5, frac=0.3), _type(3.0, frac=0.1)]
        sc = _scenario(types, lj_mode=2)
    else:  # free NPs: gravity, spring and noise only
        types = [_type(1.0, frac=0.6), _type(1.5, frac=0.3), _type(3.0, frac=0.1)]
        R = 200.0 * (n / 250000.0) ** (1.0 / 3.0)
        sc = _scenario(types, R0=R, k_evap=_evaporation(R, 0.3 * R, SLOW, 5e-4), g=0.01,
                       lj_mode=0)
    if kind != "printed":
        sc.integrator = integrator
        if integrator == 1 and kind != "free":
            sc.dt *= 0.1  # overdamped steps against the stiff LJ core are shorter
    sc.seed = seed
    t = _assign(types, n)
    if kind == "dense":
        x, sc.R0 = _aggregate(rng, types, t)
    elif kind == "free":
        u = rng.standard_normal((n, 3))
        u *= (sc.R0 * rng.random(n) ** (1.0 / 3.0) / np.linalg.norm(u, axis=1))[:, None]
        x = u
    else:
        x = _dilute(rng, types, t, sc.R0)
    m = np.array([ty.mass for ty in types])[t]
    v = rng.standard_normal((n, 3)) * np.sqrt(sc.kT / m)[:, None]
    return sc, _f32(x), _f32(v), t


def _ens_sizes(case):
    """Sizes spread evenly over the logarithm of the range, its ends included."""
    lo, hi, m = math.log(case["n_min"]), math.log(case["n_max"]), case["drops"]
    return [int(round(math.exp(lo + (hi - lo) * k / (m - 1)))) for k in range(m)]


def _ensemble(rng, case):
    out = []
    sizes = _ens_sizes(case)
    for k in rng.permutation(len(sizes)):
        n = sizes[k]
        q, eps = float(rng.uniform(0, 1)), float(rng.uniform(0.5, 2.0))
        types = [_type(1.0, +q, eps=eps, frac=0.75), _type(2.0, -q, eps=eps, frac=0.25)]
        vol = n * sum(ty.frac * math.pi / 6.0 * ty.sigma ** 3 for ty in types)
        R = (vol / 0.01 / (4.0 / 3.0 * math.pi)) ** (1.0 / 3.0)
        sc = _scenario(types, seed=int(rng.integers(1 << 40)), R0=R,
                       k_evap=_evaporation(R, float(rng.uniform(0.2, 0.6)) * R, SLOW, 5e-4),
                       g=0.01, omega=0.05, rot_mode=1, bjerrum=BJERRUM, coulomb=True, lj_mode=1)
        t = _assign(types, n)
        x = _dilute(rng, types, t, R)
        v = rng.standard_normal((n, 3)) / np.sqrt(np.array([ty.mass for ty in types])[t])[:, None]
        out.append((sc, _f32(x), _f32(v), t))
    return out


NET_IN, NET_HIDDEN, NET_LAYERS, NET_OUT = 8, 256, 4, 65


def _net_shapes():
    dims = [NET_IN] + [NET_HIDDEN] * NET_LAYERS + [NET_OUT]
    return [(o, i, -(-o // 16) * 16, -(-i // 16) * 16) for i, o in zip(dims[:-1], dims[1:])]


def _net_weights(rng):
    """One network's (W, b) per layer and the padded flat vector of the binding."""
    layers, flat = [], []
    for o, i, op, ip in _net_shapes():
        lim = math.sqrt(6.0 / i)
        W = rng.uniform(-lim, lim, (o, i)).astype(np.float32)
        b = rng.uniform(-0.1, 0.1, o).astype(np.float32)
        Wp, bp = np.zeros((op, ip), np.float32), np.zeros(op, np.float32)
        Wp[:o, :i], bp[:o] = W, b
        layers.append((W, b))
        flat += [Wp.ravel(), bp]
    return layers, np.concatenate(flat)


def _surrogate_inputs(rng, case):
    nets = [_net_weights(rng) for _ in range(case["nets"])]
    xm, xs = rng.uniform(-1, 1, NET_IN), rng.uniform(0.5, 2.0, NET_IN)
    ym, ys = rng.uniform(-1, 1, NET_OUT), rng.uniform(0.5, 2.0, NET_OUT)
    norm = [a.astype(np.float32) for a in (xm, xs, ym, ys)]
    rows = case["batch"] if case["kind"] == "predict" else case["samples"]
    X = (xm + xs * rng.standard_normal((rows, NET_IN))).astype(np.float32)
    A = rng.standard_normal((NET_IN, NET_OUT))
    Z = (X - norm[0]) / norm[1]
    Y = (ym + ys * np.tanh(Z @ A * 0.3)).astype(np.float32)
    return nets, norm, X, Y


def _pinned(n):
    """x, v and F buffers in page-locked memory for repeated state reads."""
    if torch.cuda.is_available():
        return tuple(torch.empty((n, 3), dtype=torch.float64, pin_memory=True).numpy()
                     for _ in range(3))
    return tuple(np.empty((n, 3)) for _ in range(3))


def prepare(case, seed):
    rng = np.random.default_rng([int(seed), 20250108])
    kind = case["kind"]
    s = SimpleNamespace(case=case, kind=kind)
    if kind in ("lj", "ljc", "paper", "dense", "printed", "free"):
        sc, x, v, t = _droplet(rng, kind, case["n"], case.get("integrator", 0),
                               case.get("sum_neutral", False))
        s.sim = P.Sim(sc, x, v, t)
        if kind in ("printed", "free"):
            s.frames = P.frame_buffer(case["steps"] // case["every"], case["n"])
        else:
            s.out = _pinned(case["n"])
            s.words = [np.empty((case["n"], 3), np.float32) for _ in range(3)]
    elif kind == "forces":
        s.sim = P.Sim(*_droplet(rng, case["model"], case["n"]))
    elif kind == "stats":
        s.sim = P.Sim(*_droplet(rng, "dense" if case["dense"] else "lj", case["n"]))
    elif kind == "ens":
        s.ens = P.Ensemble(_ensemble(rng, case))
    else:
        nets, norm, s.X, s.Y = _surrogate_inputs(rng, case)
        s.net = P.Surrogate(NET_IN, NET_HIDDEN, NET_LAYERS, NET_OUT, case["nets"], seed=int(seed))
        s.net.set_norm(*norm)
        for k, (_, flat) in enumerate(nets):
            s.net.set_params(k, flat)
    return s


# ---------------------------------------------------------------------------
# One pass


def run(s):
    c = s.case
    if s.kind in ("lj", "ljc", "paper", "dense"):
        s.sim.step(c["steps"])
        x, v, F, step = P.npsim_get_state(s.sim.h, s.sim.n, s.out)
        for w, a in zip(s.words, (x, v, F)):
            np.copyto(w, a, casting="same_kind")
        return {"x": s.words[0], "v": s.words[1], "F": s.words[2]}
    if s.kind in ("printed", "free"):
        return s.sim.record(c["steps"], c["every"], s.frames)
    if s.kind == "forces":
        return [s.sim.forces(what).astype(np.float32) for what in (1, 2, 3)]
    if s.kind == "stats":
        return s.sim.stats(r_max=c["r_max"], n_bins=c["bins"], radial_bins=c["radial"])
    if s.kind == "ens":
        s.ens.step(c["steps"])
        st = [s.ens.state(d) for d in range(c["drops"])]
        return {k: np.concatenate([a[j] for a in st]).astype(np.float32)
                for j, k in enumerate(("x", "v", "F"))}
    if s.kind == "predict":
        return s.net.predict(s.X)
    loss = s.net.train(s.X, s.Y, epochs=c["epochs"], batch=c["batch"], lr=1e-3, wd=1e-4, seed=7)
    return {"loss": np.float32(loss), "params": [s.net.get_params(k)[0] for k in range(c["nets"])]}


# ---------------------------------------------------------------------------
# Work of one pass: what the path cannot do without


# position (hi, lo) and velocity of one NP, read and written by one step
STEP_BYTES = 72
# one unordered Coulomb pair: difference 3, r^2 5, 1/r^3 3, both sides' sums 9
COUL_FLOPS = 20
# one unordered LJ pair within the cutoff: difference 3, r^2 5, force over r 7, both sums 9
LJ_FLOPS = 24


def _list_pairs(kind, n):
    """Unordered pairs within the cutoff: about 70 partners per NP in an aggregate, a few in a
    dilute droplet."""
    return n * (35.0 if kind == "dense" else 1.0)


def work(case):
    k = case["kind"]
    if k in ("lj", "ljc", "paper", "dense", "printed", "free"):
        n, st = case["n"], case["steps"]
        flops = st * n * 60.0  # noise and update
        if k in ("ljc", "paper"):
            m = n if k == "ljc" or case.get("sum_neutral") else 0.4 * n
            flops += st * 0.5 * m * (m - 1) * COUL_FLOPS
        if k != "free":
            flops += st * _list_pairs(k, n) * LJ_FLOPS
        out = 16 * n * (st // case["every"]) if "every" in case else 36 * n
        return {"bytes": st * n * STEP_BYTES + out, "flops": flops}
    if k == "forces":
        n = case["n"]
        m = n if case["model"] == "ljc" else 0.4 * n
        return {"bytes": 3 * n * 28, "flops": 2 * 0.5 * m * (m - 1) * COUL_FLOPS}
    if k == "ens":
        n1, n2 = sum(_ens_sizes(case)), sum(n * (n - 1) for n in _ens_sizes(case))
        return {"bytes": n1 * (case["steps"] * STEP_BYTES + 36.0),
                "flops": case["steps"] * (0.5 * n2 * COUL_FLOPS + n1 * 60.0)}
    if k == "stats":
        n = case["n"]
        dens = 0.18 if case["dense"] else 0.0089  # NPs per unit volume, all types
        return {"bytes": 24.0 * n,
                "flops": 0.5 * n * dens * 4.19 * case["r_max"] ** 3 * 10.0}
    weights = sum(o * i for o, i, _, _ in _net_shapes())
    if k == "predict":
        b = case["batch"]
        return {"bytes": b * (NET_IN + 2 * NET_OUT) * 4.0 + case["nets"] * weights * 2.0,
                "flops": 2.0 * b * weights * case["nets"]}
    rows = case["samples"] * case["epochs"] * case["nets"]
    updates = -(-case["samples"] // case["batch"]) * case["epochs"] * case["nets"]
    return {"bytes": rows * (NET_IN + NET_OUT) * 4.0 + updates * weights * 24.0,
            "flops": 6.0 * rows * weights}


# ---------------------------------------------------------------------------
# The same in float64, in plain torch and numpy

EXACT_PAIRS = 4e10  # pair evaluations that take a few seconds


def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _pair_forces(sc, x, t, lj=True, coul=True):
    """Brute-force LJ and Coulomb forces (n x 3, float64)."""
    n = x.shape[0]
    sig = torch.tensor([ty.sigma for ty in sc.types], dtype=torch.float64, device=x.device)[t]
    eps = torch.tensor([ty.eps for ty in sc.types], dtype=torch.float64, device=x.device)[t]
    q = torch.tensor([ty.charge for ty in sc.types], dtype=torch.float64, device=x.device)[t]
    coul = coul and sc.coulomb
    lj = lj and sc.lj_mode != 0
    F = torch.zeros_like(x)
    if not (lj or coul):
        return F
    rows = max(1, int(3e7) // n)
    for a in range(0, n, rows):
        b = min(n, a + rows)
        d = x[a:b, None, :] - x[None, :, :]
        r2 = (d * d).sum(-1)
        r2[torch.arange(b - a), torch.arange(a, b)] = math.inf
        f = torch.zeros_like(r2)
        s_ab = 0.5 * (sig[a:b, None] + sig[None, :])
        if lj:
            s6 = (s_ab * s_ab / r2) ** 3
            e = torch.sqrt(eps[a:b, None] * eps[None, :])
            w = 24.0 * e * (2.0 * s6 * s6 - s6) / r2
            f += torch.where(r2 < (sc.lj_cut * s_ab) ** 2, w, torch.zeros_like(w))
        if coul:
            w = sc.bjerrum * q[a:b, None] * q[None, :] / (r2 * torch.sqrt(r2))
            if sc.coulomb_cut > 0:
                w = torch.where(r2 < (sc.coulomb_cut * s_ab) ** 2, w, torch.zeros_like(w))
            f += w
        F[a:b] = (f[:, :, None] * d).sum(1)
    return F


def _total_forces(sc, x, t, step):
    F = _pair_forces(sc, x, t)
    par = lambda k: torch.tensor([getattr(ty, k) for ty in sc.types], dtype=torch.float64,  # noqa: E731
                                 device=x.device)[t]
    m, sig, kw = par("mass"), par("sigma"), par("k_wall")
    R2 = sc.R0 ** 2 - sc.k_evap * step * sc.dt
    r = torch.linalg.norm(x, dim=1)
    if sc.wall:
        s = r - ((math.sqrt(R2) if R2 > 0 else 0.0) - 0.5 * sig)
        on = s > 0
        if sc.wall_band:
            on &= s < sig
        F = F - torch.where(on, kw * s / r, torch.zeros_like(s))[:, None] * x
    F[:, 2] -= m * sc.g
    if sc.rot_mode:
        k = 2 if sc.rot_mode == 1 else 3
        F[:, :k] += (m * sc.omega ** 2)[:, None] * x[:, :k]
    return F


def _normals(seed, step, n):
    """Three standard normals per NP from Philox4x32-10, counter (i, step, 0)."""
    mask = np.uint64(0xFFFFFFFF)
    c = [np.arange(n, dtype=np.uint64), np.full(n, step & 0xFFFFFFFF, np.uint64),
         np.full(n, step >> 32, np.uint64), np.zeros(n, np.uint64)]
    k0, k1 = seed & 0xFFFFFFFF, seed >> 32
    for _ in range(10):
        p0, p1 = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & mask,
             (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), p0 & mask]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    u = [(w.astype(np.float64) + 0.5) * 2.0 ** -32 for w in c]
    r1, r2 = np.sqrt(-2.0 * np.log(u[0])), np.sqrt(-2.0 * np.log(u[2]))
    return np.stack([r1 * np.cos(2 * np.pi * u[1]), r1 * np.sin(2 * np.pi * u[1]),
                     r2 * np.cos(2 * np.pi * u[3])], 1)


def _trajectory(sc, x, v, t, steps, every=0):
    """Positions, velocities and forces after `steps` steps, and every every-th position."""
    dev = _dev()
    x, v = torch.tensor(x, device=dev), torch.tensor(v, device=dev)
    t = torch.tensor(t, dtype=torch.long, device=dev)
    par = lambda k: torch.tensor([getattr(ty, k) for ty in sc.types], dtype=torch.float64,  # noqa: E731
                                 device=dev)[t][:, None]
    m, gam, dt = par("mass"), par("gamma"), sc.dt
    c1 = torch.exp(-gam * dt)
    sd = torch.sqrt((1.0 - c1 * c1) * sc.kT / m)
    F = _total_forces(sc, x, t, 0)
    frames = []
    for k in range(steps):
        z = torch.tensor(_normals(sc.seed, k, x.shape[0]), device=dev)
        if sc.integrator == 0:
            v = v + 0.5 * dt * F / m
            x = x + 0.5 * dt * v
            v = c1 * v + sd * z
            x = x + 0.5 * dt * v
        elif sc.integrator == 1:
            x = x + F * dt / (m * gam) + torch.sqrt(2.0 * sc.kT * dt / (m * gam)) * z
        else:
            v = v + dt * (F / m - gam * v)
            v = v + sc.v_kick * z / torch.linalg.norm(z, dim=1, keepdim=True)
            x = x + dt * v
        F = _total_forces(sc, x, t, k + 1)
        if sc.integrator == 0:
            v = v + 0.5 * dt * F / m
        if every and (k + 1) % every == 0:
            frames.append(x.cpu().numpy())
    return x.cpu().numpy(), v.cpu().numpy(), F.cpu().numpy(), frames


def _exact_stats(sc, x, t, case):
    n, dr = len(x), case["r_max"] / case["bins"]
    sig = np.array([ty.sigma for ty in sc.types])[t]
    R, V = sc.R0, 4.0 / 3.0 * math.pi * sc.R0 ** 3
    c = x.mean(0)
    rg = math.sqrt(((x - c) ** 2).sum(1).mean())
    d = sig.mean()
    eps, nbox = [], []
    while len(eps) < 32 and d * 2.0 ** len(eps) <= 2.0 * rg:
        eps.append(d * 2.0 ** len(eps))
        b = np.floor((x - x.min(0)) / eps[-1]).astype(np.int64)
        nbox.append(len(np.unique((b[:, 2] << 42) | (b[:, 1] << 21) | b[:, 0])))
    df = -np.polyfit(np.log(eps[1:]), np.log(nbox[1:]), 1)[0] if len(eps) >= 3 else None
    r = np.sqrt((x[:, 0] ** 2 + x[:, 1] ** 2) + x[:, 2] ** 2)
    counts = g = None
    if n <= 30000:
        p = torch.tensor(x, device=_dev())
        h = torch.zeros(case["bins"] + 1, dtype=torch.int64, device=p.device)
        for a in range(0, n, 1000):
            e = [p[a:a + 1000, None, k] - p[None, :, k] for k in range(3)]
            q = torch.sqrt(e[0] * e[0] + e[1] * e[1] + e[2] * e[2]) / dr
            h += torch.bincount(q.floor().clamp_(max=case["bins"]).long().ravel(),
                                minlength=case["bins"] + 1)
        counts = h[:case["bins"]].cpu().numpy()
        counts[0] -= n  # every NP with itself
        e = np.arange(case["bins"] + 1) * dr
        g = counts / n / ((n - 1) * (4.0 / 3.0 * math.pi * np.diff(e ** 3)) / V)
    rb, rad = case["radial"], np.zeros(0, np.int64)
    if rb:
        rad = np.bincount(np.minimum(np.floor(r / (R / rb)), rb).astype(int), minlength=rb + 1)[:rb]
    e = np.arange(rb + 1) * (R / rb if rb else 0.0)
    return {"R": R, "d_mean": d, "Rg": rg, "Df_rg": math.log(n / 1.593) / math.log(2 * rg / d),
            "Df_box": df, "center": c, "nbox": np.array(nbox, np.int64),
            "n_surf": int((np.abs(r - R) < 0.5 * sig).sum()), "rdf_counts": counts, "rdf_g": g,
            "radial_counts": rad,
            "radial_c": rad / n / (4.0 / 3.0 * math.pi * np.diff(e ** 3) / V)}


def _exact_predict(nets, norm, X):
    xm, xs, ym, ys = [a.astype(np.float64) for a in norm]
    outs = []
    for layers, _ in nets:
        h = (X.astype(np.float64) - xm) / xs
        for k, (W, b) in enumerate(layers):
            h = h @ W.astype(np.float64).T + b
            if k + 1 < len(layers):
                h = h / (1.0 + np.exp(-h))
        outs.append(h * ys + ym)
    a = np.stack(outs)
    # one network has no spread: what comes back is rounding
    return [a.mean(0), a.std(0) if len(nets) > 1 else None]


def exact(case, seed):
    rng = np.random.default_rng([int(seed), 20250108])
    k = case["kind"]
    if k in ("lj", "ljc", "paper", "dense", "printed", "free"):
        n = case["n"]
        if (0.0 if k == "free" else n * n) * (case["steps"] + 1) > EXACT_PAIRS or n > 500000:
            return None
        sc, x, v, t = _droplet(rng, k, n, case.get("integrator", 0),
                               case.get("sum_neutral", False))
        xe, ve, Fe, frames = _trajectory(sc, x, v, t, case["steps"], case.get("every", 0))
        if k in ("printed", "free"):
            q = np.array([ty.charge for ty in sc.types])[t]
            return np.stack([np.concatenate([f, q[:, None]], 1) for f in frames])
        return {"x": xe, "v": ve, "F": Fe}
    if k == "forces":
        sc, x, v, t = _droplet(rng, case["model"], case["n"])
        xt = torch.tensor(x, device=_dev())
        tt = torch.tensor(t, dtype=torch.long, device=xt.device)
        lj = _pair_forces(sc, xt, tt, coul=False)
        co = _pair_forces(sc, xt, tt, lj=False)
        return [a.cpu().numpy() for a in (lj + co, lj, co)]
    if k == "ens":
        drops = _ensemble(rng, case)
        if sum(len(d[1]) ** 2 for d in drops) * (case["steps"] + 1) > EXACT_PAIRS:
            return None
        st = [_trajectory(*d, case["steps"]) for d in drops]
        return {key: np.concatenate([a[j] for a in st]) for j, key in enumerate(("x", "v", "F"))}
    if k == "stats":
        sc, x, v, t = _droplet(rng, "dense" if case["dense"] else "lj", case["n"])
        return _exact_stats(sc, x, t, case)
    if k == "predict":
        nets, norm, X, _ = _surrogate_inputs(rng, case)
        return _exact_predict(nets, norm, X)
    return None
