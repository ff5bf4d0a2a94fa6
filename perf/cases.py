"""What this library is used for, as measurable cases.

Every case goes through the public binding (`paper_1502_06447_gb300.ecmc`): a
melt in hand, one call or a few calls of the kind a simulation makes in its
loop, and the frame or the observables it takes away.  A melt case ends with
the positions and image counters copied into the caller's pinned buffers, as
a simulation that keeps trajectory frames does.

Positions of a run are whole answers (the event sequence is a function of the
start and the seed), so the melt cases have no separate 64-bit value; the
observables and the chain structure have one, from plain numpy and torch.
The counters that tell how the search worked inside (FP64 confirmations,
exhaustive evaluations) and the device times are no results and are left out.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1502_06447_gb300 import ecmc
from paper_1502_06447_gb300.configs import replica_specs

BASE_SEED = 0xEC0000
FP64, FP32F = "fp64", "fp32f"


def _melt(name, dims, spacing, N, **kw):
    c = dict(kind="melt", name=name, d0=dims[0], d1=dims[1], d2=dims[2], spacing=spacing, N=N,
             jitter=0.01, b_max=1.2, ell=10.0, prec=FP32F, t0=3, t1=3, t2=3, lanes=8, ecs=1,
             block_tiles=0, cell_side=0.0, tight=0.0, p_swap=0.0, swap_rate=0.0, k_spring=0.0,
             melt=4, sweeps=1, frame_in=False, g1_P=0, g1_K=0, obs=False)
    c.update(kw)
    return c


def listed():
    return [
        # undecomposed serial chains of a small melt (64 chains of 10), plain
        # FP64: the reference run of the method, one event after another
        dict(name="serial_640", kind="serial", d0=8, d1=8, d2=10, spacing=1.05, N=10, jitter=0.01,
             ell=5.0, prec=FP64, n_ec=400),
        # one call per sweep on a small melt with every launch option left at
        # its default: an interactive study that looks at the observables
        # after each sweep (latency and launches)
        _melt("default_call_4k", (16, 16, 16), 1.05, 8, ell=4.0, lanes=0, sweeps=1, obs=True),
        # a small melt (27 tiles) over many sweeps, a swap proposed at every
        # contact: the long runs that relax chain statistics
        _melt("swap_small_1728", (12, 12, 12), 1.05, 16, ell=5.0, p_swap=1.0, sweeps=60),
        # the reptation melt's size and density (20 chains of 500, tethers of
        # 1.4), sweeps with the g1 table kept on the device
        _melt("reptation_10k", (20, 20, 25), 1.2068, 500, b_max=1.4, ell=10.0, t0=6, t1=6, t2=7,
              ecs=2, sweeps=24, g1_P=4, g1_K=8),
        # plain FP64 domain sweeps, 4096 chains of 64
        _melt("fp64_262k", (64, 64, 64), 1.05, 64, prec=FP64, lanes=16, t0=16, t1=16, t2=16,
              sweeps=2),
        # dense melt (phi = 0.50), screened: a frame handed in, a sweep, the
        # frame taken back (restarts, exchange of frames with another program)
        _melt("frame_512k", (80, 80, 80), 1.0156, 256, jitter=0.005, t0=20, t1=20, t2=20, ecs=2,
              sweeps=1, frame_in=True),
        # the largest single melt: 1000 chains of 1000 with 0.1 swap attempts
        # per bead and sweep, in the benchmark's launch setting
        _melt("swap_1m", (100, 100, 100), 1.05, 1000, ell=20.0, t0=25, t1=25, t2=25, ecs=8,
              block_tiles=8, cell_side=1.05, tight=1.0, swap_rate=0.1, melt=10, sweeps=1),
        # replicas of uneven N, bead count and density in one graph-replayed
        # launch sequence per sweep
        dict(name="batch_64", kind="batch", replicas=64, draw_seed=0xEC0004, jitter=0.005, ell=5.0,
             prec=FP32F, lanes=8, tile_side=3.4, ecs=8, melt=2, sweeps=4),
        # bead-spring chains (k = 30) at the paper's System I size and density
        _melt("springs_48k", (40, 40, 30), 1.103, 120, k_spring=30.0, t0=10, t1=10, t2=7, ecs=4,
              sweeps=4),
        # a start made as the paper makes it: phantom chains, slow push-off
        dict(name="pushoff_2k", kind="pushoff", n_chains=40, N=60, eta=0.30, b_max=1.4, c=1.9,
             stages=5, ell=2.0, k_spring=30.0, lanes=32, tile_side=4.4),
        # what a trajectory analysis asks of every kept frame of the largest
        # melt: bonds, R_e^2, overlaps, contact pressure ...
        dict(name="observables_1m", kind="observables", d0=100, d1=100, d2=100, spacing=1.05,
             N=1000, jitter=0.02),
        # ... and gyration tensor, shape, R^2(n) and the end-to-end histogram
        dict(name="structure_1m", kind="structure", d0=100, d1=100, d2=100, spacing=1.05, N=1000,
             jitter=0.02, dR=1.0, nbins=200),
    ]


# ------------------------------------------------------------------ drawing
def _log(rng, a, b):
    return math.exp(rng.uniform(math.log(a), math.log(b)))


def _dims(rng, lo, hi, N, beads_hi):
    """Uneven lattice dims in [lo, hi] with N | d0 d1 d2."""
    for _ in range(1000):
        d = [int(round(_log(rng, lo, hi))) for _ in range(3)]
        for up in range(N):
            if d[0] * d[1] * (d[2] + up) % N == 0:
                d[2] += up
                break
        n = d[0] * d[1] * d[2]
        if n % N == 0 and d[2] <= hi and n <= beads_hi:
            return d
    return [lo, lo, N if N >= lo else N * (lo // N + 1)]


def _tiles(d, spacing, side, joint):
    """Tiles per axis of about `side`, each tile plus halo below half a box."""
    t = []
    for k in d:
        L = k * spacing
        D = max(3, int(L / side))
        while L / D - joint + 2.01 * joint >= 0.5 * L:
            D += 1
        t.append(D)
    return t


def draw(rng):
    kind = rng.choice(["serial", "default", "swap", "screened", "fp64", "springs", "reptation",
                       "batch", "pushoff", "observables", "structure"])
    if kind == "serial":
        d = _dims(rng, 7, 13, 10, 1100)
        return dict(kind="serial", d0=d[0], d1=d[1], d2=d[2], spacing=rng.uniform(1.05, 1.15), N=10,
                    jitter=0.01, ell=rng.uniform(3.0, 8.0), prec=rng.choice([FP64, FP64, FP32F]),
                    n_ec=int(_log(rng, 100, 400)))
    if kind == "batch":
        return dict(kind="batch", replicas=int(_log(rng, 8, 64)), draw_seed=rng.randrange(1 << 30),
                    jitter=0.005, ell=rng.uniform(3.0, 5.0), prec=FP32F, lanes=rng.choice([8, 8, 16]),
                    tile_side=rng.uniform(3.4, 4.6), ecs=rng.choice([1, 2, 4, 8]), melt=2, sweeps=2)
    if kind == "pushoff":
        return dict(kind="pushoff", n_chains=rng.randint(24, 48), N=rng.randint(30, 60),
                    eta=rng.uniform(0.22, 0.30), b_max=1.4, c=1.9, stages=5, ell=2.0, k_spring=30.0,
                    lanes=rng.choice([16, 32]), tile_side=4.4)
    if kind in ("observables", "structure"):
        N = rng.choice([10, 25, 64, 120, 250, 500, 1000])
        d = _dims(rng, 12, 100, N, 1_000_000)
        c = dict(kind=kind, d0=d[0], d1=d[1], d2=d[2], spacing=rng.uniform(1.05, 1.12), N=N,
                 jitter=0.02)
        if kind == "structure":
            c.update(dR=rng.uniform(0.3, 2.0), nbins=rng.randint(20, 300))
        return c
    N = {"springs": 120, "reptation": 500}.get(kind) or rng.choice([8, 16, 27, 64, 120, 256, 1000])
    hi, beads = {"default": (18, 6000), "swap": (24, 14000), "reptation": (40, 30000),
                 "springs": (48, 60000), "fp64": (64, 262144), "screened": (100, 700000)}[kind]
    d = _dims(rng, 11, hi, N, beads)
    lo_a, b_max = (1.10, 1.4) if kind == "reptation" else (1.03, 1.2)
    a = rng.uniform(1.06, 1.12) if kind == "springs" else rng.uniform(lo_a, min(b_max - 0.06, 1.21))
    side = rng.uniform(4.0 if kind == "reptation" else 3.6, 5.4)
    t = _tiles(d, a, side, b_max)
    c = _melt("", d, a, N, b_max=b_max, ell=_log(rng, 4.0, 20.0), t0=t[0], t1=t[1], t2=t[2],
              ecs=rng.choice([1, 2, 4, 8]), lanes=rng.choice([8, 8, 8, 4, 16]))
    del c["name"]
    if kind == "default":
        c.update(lanes=0, ecs=1, obs=True)
    elif kind == "swap":
        c.update(p_swap=rng.choice([1.0, rng.uniform(0.05, 0.5)]), sweeps=rng.randint(5, 30))
    elif kind == "reptation":
        c.update(ecs=rng.choice([1, 2]), sweeps=rng.randint(8, 24), g1_P=rng.randint(3, 8),
                 g1_K=rng.randint(3, 8))
    elif kind == "fp64":
        c.update(prec=FP64, lanes=rng.choice([8, 16, 16, 32]), ecs=rng.choice([1, 2]))
    elif kind == "springs":
        c.update(k_spring=rng.uniform(20.0, 40.0), prec=rng.choice([FP32F, FP32F, FP64]),
                 ecs=rng.choice([1, 2, 4]), sweeps=2)
    else:
        c.update(swap_rate=rng.choice([0.0, 0.1]), frame_in=rng.random() < 0.3)
    return c


# ------------------------------------------------------------------ inputs
def _seed(seed):
    return BASE_SEED + 7919 * int(seed)


def _pinned(n):
    return (torch.empty((n, 3), dtype=torch.float64, pin_memory=True).numpy(),
            torch.empty((n, 3), dtype=torch.int32, pin_memory=True).numpy())


def _beads(c):
    if c["kind"] == "batch":
        return sum(m.n for m in replica_specs(c["replicas"], c["draw_seed"]))
    if c["kind"] == "pushoff":
        return c["n_chains"] * c["N"]
    return c["d0"] * c["d1"] * c["d2"]


def _snake(c, seed):
    """Jittered simple-cubic sites visited in a snake (the order in which the
    library's lattice strings its chains), and the box."""
    n0, n1, n2 = c["d0"], c["d1"], c["d2"]
    z, y, x = np.meshgrid(np.arange(n2), np.arange(n1), np.arange(n0), indexing="ij")
    ys = np.where(z % 2 == 0, y, n1 - 1 - y)
    xs = np.where((z * n1 + y) % 2 == 0, x, n0 - 1 - x)
    site = np.stack([xs, ys, z], -1).reshape(-1, 3)
    rng = np.random.default_rng(_seed(seed))
    r = (site + 0.5) * c["spacing"] + c["jitter"] * rng.uniform(-1.0, 1.0, site.shape)
    return r, np.array([n0, n1, n2]) * c["spacing"]


def _prec(c):
    return ecmc.PREC_FP64 if c["prec"] == FP64 else ecmc.PREC_FP32F


def prepare(case, seed):
    c, s = case, _seed(seed)
    st = {"case": c, "seed": s}
    if c["kind"] == "batch":
        specs = [dict(dims=m.dims, spacing=m.spacing, N=m.N)
                 for m in replica_specs(c["replicas"], c["draw_seed"])]
        b = ecmc.Batch(specs, jitter=c["jitter"], seed=s)
        b.configure(dir_mode=ecmc.DIR_ISO, precision=_prec(c), lanes=c["lanes"],
                    tile_side=c["tile_side"], ecs_per_tile=c["ecs"])
        b.run(c["ell"], seed=s, n_sweeps=c["melt"], graph=True)
        st["batch"] = b
        return st
    if c["kind"] == "pushoff":
        n = c["n_chains"] * c["N"]
        st["L"] = (n * math.pi / (6.0 * c["eta"])) ** (1.0 / 3.0)
        st["out"] = _pinned(n)
        return st
    if c["kind"] in ("observables", "structure"):
        ctx = ecmc.Context.create_lattice((c["d0"], c["d1"], c["d2"]), c["spacing"], c["N"],
                                          b_max=1.2)
        ctx.set_positions(_snake(c, seed)[0])
        st["ctx"] = ctx
        return st
    ctx = ecmc.Context.create_lattice((c["d0"], c["d1"], c["d2"]), c["spacing"], c["N"],
                                      b_max=c.get("b_max", 1.2), jitter=c["jitter"], seed=s)
    st["ctx"], st["out"] = ctx, _pinned(ctx.n)
    if c["kind"] == "serial":
        ctx.configure(mode=ecmc.MODE_SERIAL, dir_mode=ecmc.DIR_CART3, precision=_prec(c))
        ctx.run(c["ell"], chains_per_sweep=100, seed=s)
        return st
    ctx.configure(mode=ecmc.MODE_DOMAIN, dir_mode=ecmc.DIR_ISO, precision=_prec(c),
                  tiles=(c["t0"], c["t1"], c["t2"]), lanes=c["lanes"], ecs_per_tile=c["ecs"],
                  block_tiles=c["block_tiles"], cell_side=c["cell_side"], tight_factor=c["tight"],
                  p_swap=c["p_swap"], k_spring=c["k_spring"])
    ctx.run(c["ell"], seed=s, n_sweeps=c["melt"])  # the lattice start melts first
    if c["swap_rate"]:
        ctx.swap(c["swap_rate"])
    if c["g1_P"]:
        ctx.g1_track(c["g1_P"], c["g1_K"])
    if c["frame_in"]:
        st["in"] = _pinned(ctx.n)
        ctx.get_positions(out=st["in"])
    return st


# ------------------------------------------------------------------ one pass
OBS = ("re2_mean", "bond_max", "bond_min", "bond_mean", "overlaps", "tether_violations",
       "contact_pairs", "taut_bonds", "pressure_contact")
EVENTS = ecmc.EV_NAMES + ("events_total", "ecs", "sweeps", "swap_tried", "lift_sum", "refl_sum")


def run(state):
    c, s = state["case"], state["seed"]
    if c["kind"] == "batch":
        b = state["batch"]
        b.run(c["ell"], seed=s, n_sweeps=c["sweeps"], graph=True)
        frames = [b.get_positions(r) for r in range(b.n)]
        t = b.stats()
        return {"r": np.concatenate([f[0] for f in frames]),
                "img": np.concatenate([f[1] for f in frames]),
                "events": t["events_total"], "ecs": t["ecs"]}
    if c["kind"] == "pushoff":
        L = (state["L"],) * 3
        with ecmc.Context.create_phantom(L, c["n_chains"], c["N"], bond=1.0, c=c["c"], seed=s,
                                         b_max=c["b_max"]) as ctx:
            D = max(3, int(state["L"] / c["tile_side"]))
            ctx.configure(mode=ecmc.MODE_DOMAIN, dir_mode=ecmc.DIR_ISO, precision=ecmc.PREC_FP64,
                          tiles=(D, D, D), lanes=c["lanes"], k_spring=c["k_spring"])
            n = ctx.pushoff(f0=0.5, stages=c["stages"], ell=c["ell"], seed=s, max_sweeps=40000)
            r, img = ctx.get_positions(out=state["out"])
        return {"r": r, "img": img, "sweeps": n}
    ctx = state["ctx"]
    if c["kind"] == "observables":
        o = ctx.observables()
        return {k: list(o[k]) if isinstance(o[k], tuple) else o[k] for k in OBS}
    if c["kind"] == "structure":
        o, r2n, hist = ctx.structure(dR=c["dR"], nbins=c["nbins"])
        return {"sums": {k: list(v) if isinstance(v, tuple) else v for k, v in o.items()},
                "r2n": r2n, "hist": hist}
    if c["kind"] == "serial":
        ctx.run(c["ell"], chains_per_sweep=c["n_ec"], seed=s)
    else:
        if c["frame_in"]:
            ctx.set_positions(*state["in"])
        ctx.run(c["ell"], seed=s, n_sweeps=c["sweeps"])
    r, img = ctx.get_positions(out=state["out"])
    out = {"r": r, "img": img}
    if c.get("obs"):
        o = ctx.observables()
        out.update({k: list(o[k]) if isinstance(o[k], tuple) else o[k] for k in OBS + EVENTS})
    if c.get("g1_P"):
        lags, g1, cnt = ctx.g1_table()
        out.update(lags=lags, g1=g1, origins=cnt)
    return out


# ------------------------------------------------------------------ work
def work(case):
    """Bytes: the state read once and written once (positions 24 B, images
    12 B per bead).  Flops: the events of the pass (about 15 per sigma of
    displacement in these melts) times one exact contact distance and move
    (13 FP64 operations for the distance with its square root, 9 for the move
    and the bookkeeping of the flight)."""
    c, n = case, _beads(case)
    per_event = 22.0
    if c["kind"] == "observables":
        # per bead: one bond (14) and the 13 half-neighbours within reach (8)
        return {"bytes": 24.0 * n, "flops": n * (14.0 + 13 * 8.0)}
    if c["kind"] == "structure":
        N = c["N"]
        return {"bytes": 24.0 * n, "flops": n * 30.0 + (n / N) * (N * (N - 1) / 2) * 9.0}
    if c["kind"] == "serial":
        return {"bytes": 72.0 * n, "flops": c["n_ec"] * c["ell"] * 15.0 * per_event}
    if c["kind"] == "pushoff":
        # every bead is flagged against its neighbours and moved a few times
        return {"bytes": 72.0 * n, "flops": n * c["stages"] * c["ell"] * 15.0 * per_event}
    if c["kind"] == "batch":
        tiles = n / 0.85 / c["tile_side"] ** 3
    else:
        tiles = c["t0"] * c["t1"] * c["t2"]
    return {"bytes": 72.0 * n,
            "flops": tiles * c["ecs"] * c["ell"] * 15.0 * per_event * c["sweeps"]}


# ------------------------------------------------------------------ 64 bits
def exact(case, seed):
    if case["kind"] == "observables":
        return _exact_observables(case, seed)
    if case["kind"] == "structure":
        return _exact_structure(case, seed)
    return None


def _bonds(r, L, N):
    u = r.reshape(-1, N, 3)
    d = u[:, 1:] - u[:, :-1]
    return d - L * np.round(d / L)


def _exact_observables(c, seed):
    sigma, b_max, delta = 1.0, 1.2, 0.02
    r, L = _snake(c, seed)
    r = r % L
    N, n = c["N"], len(r)
    d = _bonds(r, L, N)
    re2 = (d.sum(1) ** 2).sum(1)
    dd = (d ** 2).sum(2)
    b = np.sqrt(dd)
    taut = [int(((dd > (b_max - delta) ** 2) & (dd <= b_max ** 2 * (1 + 1e-10))).sum()),
            int(((dd > (b_max - 2 * delta) ** 2) & (dd <= (b_max - delta) ** 2)).sum())]
    # pairs: jittered lattice sites closer than 1.04 sigma are lattice neighbours
    grid = np.empty((c["d2"], c["d1"], c["d0"], 3))
    site = np.floor(r / c["spacing"]).astype(np.int64)
    grid[site[:, 2], site[:, 1], site[:, 0]] = r
    over, pairs = 0, [0, 0]
    for ax in range(3):
        q = np.roll(grid, -1, axis=ax) - grid
        q = q - L * np.round(q / L)
        s = (q ** 2).sum(-1)
        over += int((s < 1.0 - 1e-10).sum())
        pairs[0] += int(((s >= 1.0 - 1e-10) & (s < (sigma + delta) ** 2)).sum())
        pairs[1] += int(((s >= (sigma + delta) ** 2) & (s < (sigma + 2 * delta) ** 2)).sum())
    fs = (1.5 * pairs[0] - 0.5 * pairs[1]) / delta
    fb = (1.5 * taut[0] - 0.5 * taut[1]) / delta
    return {"re2_mean": float(re2.mean()), "bond_max": float(b.max()), "bond_min": float(b.min()),
            "bond_mean": float(b.mean()), "overlaps": over,
            "tether_violations": int((dd > b_max ** 2 * (1 + 1e-10)).sum()),
            "contact_pairs": pairs, "taut_bonds": taut,
            "pressure_contact": 1.0 + (sigma * fs - b_max * fb) / (3.0 * n)}


def _exact_structure(c, seed):
    r, L = _snake(c, seed)
    N = c["N"]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    d = torch.from_numpy(_bonds(r % L, L, N)).to(dev)
    u = torch.cat([torch.zeros_like(d[:, :1]), torch.cumsum(d, 1)], 1)
    w = u - u.mean(1, keepdim=True)
    S = torch.einsum("cja,cjb->cab", w, w) / N
    lam = torch.linalg.eigvalsh(S.cpu())
    l0, l1, l2 = lam[:, 0], lam[:, 1], lam[:, 2]
    T = lam.sum(1)
    P = l0 * l1 + l1 * l2 + l2 * l0
    re2 = (u[:, -1] ** 2).sum(1)
    r2n = torch.zeros(N, dtype=torch.float64)
    for k in range(1, N):
        r2n[k] = ((u[:, k:] - u[:, :-k]) ** 2).sum(2).mean().item()
    bins = torch.clamp(torch.floor(torch.sqrt(re2) / c["dR"]).to(torch.int64), max=c["nbins"] - 1)
    hist = torch.bincount(bins.cpu(), minlength=c["nbins"])
    return {"sums": {"n_chains": len(T), "N": N, "rg2_sum": T.sum().item(),
                     "lam_sum": [x.sum().item() for x in (l0, l1, l2)],
                     "b_sum": (l2 - 0.5 * (l0 + l1)).sum().item(), "c_sum": (l1 - l0).sum().item(),
                     "kappa2_sum": (1.0 - 3.0 * P / T ** 2).sum().item(),
                     "bc_sum": (4.0 * (T ** 2 - 3.0 * P)).sum().item(), "g2_sum": 0.0,
                     "re2_sum": re2.sum().item()},
            "r2n": r2n, "hist": hist}
