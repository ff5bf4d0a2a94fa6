"""Every form of the EC kernel at its own width.  Melts of few tiles run with
more lanes than asked for unless the tiles per block are given, so these runs
give them: 4, 8, 16 and 32 lanes per tile with the exhaustive evaluation,
swaps, springs, batches in both precisions, the push-off, a second pass for
tiles past the first one's capacities, and the bounds-checked build.  Digests,
positions and images equal the oracle's bit for bit."""
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle
from paper_1502_06447_gb300 import ecmc
from paper_1502_06447_gb300.configs import Melt, small_domain

from helpers import gpu_context, oracle_system
from test_gpu_batch import check_batch, ragged_specs
from test_gpu_parity import BLOCKS, RAGGED
from test_gpu_pushoff import pair

pytestmark = pytest.mark.gpu

P32, P64 = ecmc.PREC_FP32F, ecmc.PREC_FP64
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module", autouse=True)
def _build():
    from paper_1502_06447_gb300 import build
    build.build()


_ref = {}


def reference(m, **kw):
    key = (m.name, m.p_swap) + tuple(sorted(kw.items()))
    if key not in _ref:
        o = oracle_system(m, **kw)
        res = o.run_domain(m.sweeps, m.ell, digests=True)
        assert res["rc"] == 0
        _ref[key] = (o.r.copy(), o.img.copy(), res)
    return _ref[key]


def check(m, lanes, prec, ecs=1, k_spring=0.0, **kw):
    r, img, res = reference(m, ecs_per_tile=ecs, k_spring=k_spring)
    ctx = gpu_context(m, precision=prec, lanes=lanes, block_tiles=32 // lanes, ecs_per_tile=ecs,
                      k_spring=k_spring, **kw)
    ctx.run(m.ell, seed=m.seed, n_sweeps=m.sweeps)
    dig, lift, ev = ctx.records(len(res["digest"]))
    bad = np.nonzero(dig != res["digest"])[0]
    assert bad.size == 0, f"{bad.size} ECs differ, first {bad[:5]}"
    assert (lift == res["ec_lift"]).all() and (ev == res["ec_events"]).all()
    rg, ig = ctx.get_positions()
    assert (rg == r).all() and (ig == img).all()
    return ctx, res


@pytest.mark.parametrize("lanes", [4, 8, 16, 32])
@pytest.mark.parametrize("prec", [P32, P64])
@pytest.mark.parametrize("m", [small_domain(), RAGGED], ids=lambda m: m.name)
def test_domain(m, prec, lanes):
    check(m, lanes, prec, ecs=2)


@pytest.mark.parametrize("lanes,request_cap", [(4, 1), (8, 1), (16, 1), (32, 1), (4, 3), (8, 2), (16, 2)])
def test_exhaustive_evaluation(lanes, request_cap):
    ctx, _ = check(BLOCKS, lanes, P32, request_cap=request_cap)
    ob = ctx.observables()
    if request_cap == 1:
        assert ob["exhaustive"] > ob["events_total"] // 4


@pytest.mark.parametrize("lanes", [4, 8, 16, 32])
@pytest.mark.parametrize("prec", [P32, P64])
@pytest.mark.parametrize("p_swap,N", [(1.0, 2), (0.5, 1)])
def test_swaps(p_swap, N, prec, lanes):
    """Dimers and free spheres: accepted swaps."""
    m = small_domain(N=N, p_swap=p_swap, seed=0xEC00A4, ell=6.0)
    ctx, res = check(m, lanes, prec)
    obs = ctx.observables()
    assert obs["swap_tried"] == res["stats"]["swap_tried"] and obs["swap"] == res["stats"]["swap"] > 0


@pytest.mark.parametrize("lanes", [4, 8, 16, 32])
@pytest.mark.parametrize("prec", [P32, P64])
@pytest.mark.parametrize("k_spring", [1.0, 30.0])
def test_springs(k_spring, prec, lanes):
    check(small_domain(seed=0xEC00A7), lanes, prec, ecs=2, k_spring=k_spring)


@pytest.mark.parametrize("lanes", [4, 8, 16, 32])
@pytest.mark.parametrize("prec", [P32, P64])
def test_batch(prec, lanes):
    check_batch(ragged_specs(), lanes, prec, True, block_tiles=32 // lanes)


@pytest.mark.parametrize("lanes", [4, 8, 16])
def test_batch_exhaustive_and_swaps(lanes):
    check_batch(ragged_specs(), lanes, P32, True, sweeps=2, request_cap=1, p_swap=0.5,
                block_tiles=32 // lanes)


@pytest.mark.parametrize("lanes", [4, 8, 16])
@pytest.mark.parametrize("k_spring", [0.0, 30.0])
def test_pushoff(k_spring, lanes):
    D = (4, 3, 4)
    ctx, o = pair(0.40, 16, 16.0, seed=51, po_seed=0xEC0F2F, D=D, lanes=lanes, k_spring=k_spring)
    ctx.configure(mode=ecmc.MODE_DOMAIN, dir_mode=ecmc.DIR_ISO, precision=P64, tiles=D, lanes=lanes,
                  k_spring=k_spring, block_tiles=32 // lanes)
    n = ctx.pushoff(f0=0.5, stages=4, ell=2.0, seed=0xEC0F2F, max_sweeps=6000)
    rc, sweeps, _ = o.pushoff(0.5, 4, 2.0, 6000)
    assert rc == 0 and n == sweeps > 0
    r, img = ctx.get_positions()
    assert (r == o.r).all() and (img == o.img).all()


# 8,000 tiles of 3.6 sigma: more than stay resident with the full capacities
# (shared memory: at most 42 tiles of 4 or 8 lanes per SM, 24 of 16 lanes)
MANY = Melt("widths_8000", (68, 68, 68), 1.05, 8, ell=0.8, seed=0xEC0D12, mode="domain", dir_mode="iso",
            sweeps=1, D=(20, 20, 20))


@pytest.mark.parametrize("lanes", [4, 8, 16, 32])
@pytest.mark.parametrize("prec", [P32, P64])
@pytest.mark.parametrize("k_spring", [0.0, 30.0])
def test_second_pass(k_spring, prec, lanes):
    """A first pass at 0.8 of the mean content, at the lattice start: it leaves
    925 of the tiles to the second."""
    check(MANY, lanes, prec, k_spring=k_spring, tight_factor=0.8)


CHILD = r"""
import os, sys
sys.path.insert(0, os.path.join(ROOT, "tests"))
sys.path.insert(0, ROOT)
from paper_1502_06447_gb300 import build, ecmc
build.build()
assert os.path.basename(ecmc.LIB_PATH) == "libecmc_checked.so", ecmc.LIB_PATH
from paper_1502_06447_gb300.configs import small_domain
import test_gpu_widths as w
for lanes in (4, 8, 16):
    w.test_exhaustive_evaluation(lanes, 1)
    w.check(small_domain(seed=0xEC00A7), lanes, w.P32, ecs=2, k_spring=30.0)
    w.check(small_domain(N=1, p_swap=0.5, seed=0xEC00A4, ell=6.0), lanes, w.P64)
    w.test_pushoff(30.0, lanes)
    w.test_batch(w.P64, lanes)
print("checked ok")
"""


def test_checked_build():
    """No index out of range at 4, 8 and 16 lanes (a child process: the
    binding picks its library when it is first loaded)."""
    env = dict(os.environ, ECMC_CHECKED="1")
    p = subprocess.run([sys.executable, "-c", "ROOT = " + repr(ROOT) + "\n" + CHILD], env=env,
                       capture_output=True, text=True, timeout=1500)
    assert p.returncode == 0, (p.stdout[-3000:], p.stderr[-3000:])
    assert "checked ok" in p.stdout
