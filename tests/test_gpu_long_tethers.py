"""Tethers several diameters long: a tile's tether halo holds many times the
beads that are staged.  Settings that are accepted run, with the oracle's
events."""
import pytest

from paper_1502_06447_gb300 import ecmc
from paper_1502_06447_gb300.configs import Melt

from helpers import gpu_context, oracle_system

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    from paper_1502_06447_gb300 import build
    build.build()


# capacities of 11,136 (the largest that fits as it is) and 11,680 beads per tile
@pytest.mark.parametrize("k,N", [(43, 43), (44, 11)])
@pytest.mark.parametrize("k_spring", [0.0, 3.0])
def test_staging_capacity_past_a_block(k, N, k_spring):
    m = Melt(f"long_{k}", (k, k, k), 1.05, N, ell=2.0, b_max=6.4, seed=0xEC0E11, mode="domain",
             dir_mode="iso", sweeps=2, D=(3, 3, 3))
    o = oracle_system(m, k_spring=k_spring)
    res = o.run_domain(m.sweeps, m.ell, digests=True)
    assert res["rc"] == 0
    ctx = gpu_context(m, precision=ecmc.PREC_FP32F, lanes=32, k_spring=k_spring)
    ctx.run(m.ell, seed=m.seed, n_sweeps=m.sweeps)
    dig, _, _ = ctx.records(len(res["digest"]))
    assert (dig == res["digest"]).all()
    r, img = ctx.get_positions()
    assert (r == o.r).all() and (img == o.img).all()
