"""Calls that run out of device memory half way (the injected limit of
ECMC_ALLOC_LIMIT lets the first buffer of a group through and refuses a later
one): they return ENOMEM, launch nothing, and once memory is there again the
same context gives the oracle's events and the structure of a fresh one."""
import numpy as np
import pytest

from paper_1502_06447_gb300 import ecmc
from paper_1502_06447_gb300.configs import small_domain

from helpers import gpu_context, oracle_system

pytestmark = pytest.mark.gpu

ENOMEM = -2


@pytest.fixture(scope="module", autouse=True)
def _build():
    from paper_1502_06447_gb300 import build
    build.build()


def refused(monkeypatch, limit, call):
    with monkeypatch.context() as m:
        m.setenv("ECMC_ALLOC_LIMIT", str(limit))
        with pytest.raises(ecmc.EcmcError) as e:
            call()
    assert e.value.code == ENOMEM


def settings(m, **kw):
    return dict(dict(mode=ecmc.MODE_DOMAIN, dir_mode=ecmc.DIR_ISO, precision=ecmc.PREC_FP32F,
                     tiles=m.D, lanes=8, record=1), **kw)


def assert_runs_as_oracle(ctx, m, o, sweeps, sweep0=0):
    ctx.run(m.ell, seed=m.seed, n_sweeps=sweeps)
    res = o.run_domain(sweeps, m.ell, sweep0=sweep0, digests=True)
    dig, _, _ = ctx.records(len(res["digest"]))
    assert len(dig) == len(res["digest"]) and (dig == res["digest"]).all()
    r, img = ctx.get_positions()
    assert (r == o.r).all() and (img == o.img).all()


def test_cell_arrays_half_allocated(monkeypatch):
    """The counts fit the limit (4 B per cell), the starts (one more) do not."""
    m = small_domain()
    ctx, o = gpu_context(m, precision=ecmc.PREC_FP32F, lanes=8), oracle_system(m)
    assert_runs_as_oracle(ctx, m, o, 1)
    side = 1.5
    limit = 4 * int(np.prod([int(L / side) for L in m.L]))
    refused(monkeypatch, limit, lambda: ctx.configure(**settings(m, cell_side=side)))
    assert_runs_as_oracle(ctx, m, o, 1, sweep0=1)
    assert ctx.observables()["overlaps"] == 0


def test_structure_scratch_half_allocated(monkeypatch):
    """Chains of two: the positions along the chains take 24 B per bead, the
    records of the chains 52."""
    m = small_domain(N=2)
    ctx = gpu_context(m, precision=ecmc.PREC_FP32F, lanes=8)
    refused(monkeypatch, 24 * ctx.n, lambda: ctx.structure(dR=0.5, nbins=8))
    refused(monkeypatch, 24 * ctx.n, ctx.g1_reset)
    got, r2n, hist = ctx.structure(dR=0.5, nbins=8)
    ref, r2n0, hist0 = gpu_context(m, precision=ecmc.PREC_FP32F, lanes=8).structure(dR=0.5, nbins=8)
    assert got == ref and (r2n == r2n0).all() and (hist == hist0).all()


@pytest.mark.parametrize("kw,limit,code", [
    (dict(tiles=(4, 4, 2)), 0, -1),                      # the third axis is refused after two others
    (dict(tiles=(4, 4, 4), cell_side=0.5), 0, -1),
    (dict(tiles=(3, 4, 5), ecs_per_tile=2, block_tiles=3), 0, -1),
    (dict(tiles=(5, 5, 5)), 4 * 125 - 1, ENOMEM),        # the list of tiles for a second pass
    (dict(k_spring=30.0), 4 * 4096 - 1, ENOMEM),         # the springs' tags by bead
    (dict(tiles=(4, 4, 4), cell_side=1.5), 4 * 11 ** 3, ENOMEM),
])
def test_refused_settings_leave_those_in_force(kw, limit, code, monkeypatch):
    m = small_domain()
    ctx, o = gpu_context(m, precision=ecmc.PREC_FP32F, lanes=8), oracle_system(m)
    assert_runs_as_oracle(ctx, m, o, 1)
    with monkeypatch.context() as env:
        env.setenv("ECMC_ALLOC_LIMIT", str(limit))
        with pytest.raises(ecmc.EcmcError) as e:
            ctx.configure(**settings(m, **kw))
    assert e.value.code == code
    assert_runs_as_oracle(ctx, m, o, 2, sweep0=1)


BATCH = [dict(dims=(12, 12, 12), spacing=1.05, N=8), dict(dims=(10, 12, 14), spacing=1.12, N=10)]
SEED = 0xEC0B21


def batch_cells(side):
    return sum(int(np.prod([int(d * s["spacing"] / side) for d in s["dims"]])) for s in BATCH)


@pytest.mark.parametrize("kw,limit,code", [
    (dict(cell_side=1.5), 4 * batch_cells(1.5), ENOMEM),  # the counts fit, the starts do not
    (dict(tile_side=3.0), 4 * 124 - 1, ENOMEM),           # 4 x 4 x 4 + 3 x 4 x 5 tiles: the second pass's list
    (dict(request_cap=9, tile_side=3.0), 0, -1),
])
def test_refused_batch_settings_leave_those_in_force(kw, limit, code, monkeypatch):
    """A sweep captured before the refused call and replays after it, against
    a batch that never saw it."""
    out = []
    for refuse in (True, False):
        b = ecmc.Batch(BATCH, jitter=0.01, seed=SEED)
        b.configure(dir_mode=ecmc.DIR_ISO, precision=ecmc.PREC_FP32F, lanes=8)
        b.run(3.0, seed=SEED, n_sweeps=2, graph=True)
        if refuse:
            with monkeypatch.context() as env:
                env.setenv("ECMC_ALLOC_LIMIT", str(limit))
                with pytest.raises(ecmc.EcmcError) as e:
                    b.configure(dir_mode=ecmc.DIR_ISO, precision=ecmc.PREC_FP32F, lanes=8, **kw)
            assert e.value.code == code
        b.run(3.0, seed=SEED, n_sweeps=3, graph=True)
        out.append([b.get_positions(r) for r in range(len(BATCH))] + [b.stats()["events_total"]])
    for (r, img), (r0, img0) in zip(out[0][:-1], out[1][:-1]):
        assert (r == r0).all() and (img == img0).all()
    assert out[0][-1] == out[1][-1]
