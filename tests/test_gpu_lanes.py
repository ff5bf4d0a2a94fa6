"""Lane counts on a melt of 2,744 tiles with the tiles per block fixed (the
launch then gives no tile extra lanes), so that every instance of the EC
kernel runs at its own width with ragged last warps, and the first pass with
tight capacities defers tiles to the second.  Per-EC
digests, positions and images equal the oracle's bit for bit."""
import numpy as np
import pytest

from paper_1502_06447_gb300 import ecmc
from paper_1502_06447_gb300.configs import Melt

from helpers import gpu_context, oracle_system

pytestmark = pytest.mark.gpu

# 2,744 tiles; one axis two beads longer, so that tile counts are uneven
M = Melt("lanes_2744", (48, 48, 50), 1.05, 8, ell=1.0, seed=0xEC0D11, mode="domain", dir_mode="iso",
         sweeps=1, D=(14, 14, 14), p_swap=0.2)


@pytest.fixture(scope="module")
def reference():
    out = {}
    for k_spring in (0.0, 30.0):
        o = oracle_system(M, k_spring=k_spring, p_swap=0.0 if k_spring else M.p_swap)
        res = o.run_domain(M.sweeps, M.ell, digests=True)
        assert res["rc"] == 0
        out[k_spring] = (o.r.copy(), o.img.copy(), res["digest"])
    return out


@pytest.mark.parametrize("lanes", [4, 8, 16, 32])
@pytest.mark.parametrize("prec", [ecmc.PREC_FP32F, ecmc.PREC_FP64])
@pytest.mark.parametrize("k_spring", [0.0, 30.0])
def test_lanes_match_oracle_at_full_width(lanes, prec, k_spring, reference):
    r, img, digest = reference[k_spring]
    ctx = gpu_context(M, precision=prec, lanes=lanes, block_tiles=32 // lanes, tight_factor=0.8,
                      k_spring=k_spring,
                      p_swap=0.0 if k_spring else M.p_swap)
    ctx.run(M.ell, seed=M.seed, n_sweeps=M.sweeps)
    dig, _, _ = ctx.records(len(digest))
    bad = np.nonzero(dig != digest)[0]
    assert bad.size == 0, f"{bad.size} ECs differ, first {bad[:5]}"
    rg, ig = ctx.get_positions()
    assert (rg == r).all() and (ig == img).all()
