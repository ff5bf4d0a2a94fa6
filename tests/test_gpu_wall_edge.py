"""A bead that sits exactly on the lower wall of its tile (zero distance to it):
moving out, its first event is that wall, after a flight of -0.0.  Events,
digests (which hold the flight's bits), positions and images equal the
oracle's for every width of the EC kernel and both precisions."""
import numpy as np
import pytest

import oracle
from paper_1502_06447_gb300 import ecmc

pytestmark = pytest.mark.gpu

SEED = 0xEC0E01


@pytest.fixture(scope="module", autouse=True)
def _build():
    from paper_1502_06447_gb300 import build
    build.build()


@pytest.mark.parametrize("lanes", [4, 8, 16, 32])
@pytest.mark.parametrize("prec", [ecmc.PREC_FP32F, ecmc.PREC_FP64])
def test_bead_on_its_lower_wall(lanes, prec):
    D, T = (3, 3, 3), 6.0
    L = np.array(D) * T
    ctx = ecmc.Context.create_lattice(D, T, 1)  # one free sphere per tile
    ctx.configure(mode=ecmc.MODE_DOMAIN, dir_mode=ecmc.DIR_ISO, precision=prec, tiles=D, lanes=lanes,
                  block_tiles=32 // lanes, ecs_per_tile=2, record=1)
    _, shift = ctx.domain_tags(SEED, 0)
    k = np.stack(np.meshgrid(*(np.arange(d) for d in D), indexing="ij"), -1).reshape(-1, 3)
    r = shift + k * T + 2.0
    for i in range(len(k)):
        ax = int(np.argmin(k[i]))  # tile 0 of an axis where there is one: its corner is the shift itself
        r[i, ax] = shift[ax] + k[i, ax] * T
    ctx.set_positions(np.mod(r, L))
    o = oracle.System(np.mod(r, L), L, 1, mode=oracle.MODE_DOMAIN, dir_mode=oracle.DIR_ISO, D=D, seed=SEED,
                      ecs_per_tile=2)
    res = o.run_domain(1, 3.0, digests=True, log_cap=10000)
    log = res["log"]
    edge = (log["x"] == 0.0) & np.signbit(log["x"])
    assert edge.sum() >= 5  # 19 beads on the wall of a tile 0, half of them moving out
    ctx.log_reserve(10000)
    ctx.run(3.0, seed=SEED, n_sweeps=1)
    dig, _, _ = ctx.records(len(res["digest"]))
    bad = np.nonzero(dig != res["digest"])[0]
    assert bad.size == 0, bad
    got, ref = ctx.event_log(10000), log[np.argsort(log["unit"], kind="stable")]
    for f in ("unit", "pivot", "kind", "partner"):
        assert (got[f] == ref[f]).all(), f
    x, x0 = (np.ascontiguousarray(v["x"]).view(np.uint64) for v in (got, ref))
    assert (x == x0).all()
    rg, ig = ctx.get_positions()
    assert (rg == o.r).all() and (ig == o.img).all()
