"""Cell pass at its edges: coordinates on and next to tile, joint and cell
boundaries (where FP32 cannot tell and the FP64 expressions decide), melts on
both sides of the size that takes the one-block pass, and the pair counts that
go through the cells.  Tags equal the oracle's; overlaps and contact shells
equal a direct count."""
import numpy as np
import pytest

import oracle
from paper_1502_06447_gb300 import ecmc

pytestmark = pytest.mark.gpu

SEED = 0xEC0ED6


def edge_positions(dims, a, D, w, shift, cell_side, rng):
    """Lattice of single spheres; one coordinate of each is moved to the nearest
    tile start, tile end, cell boundary or box edge and up to two ulps off it."""
    L = np.array(dims) * a
    r = (np.stack(np.meshgrid(*(np.arange(d) for d in dims), indexing="ij"), -1).reshape(-1, 3) + 0.5) * a
    T = L / np.array(D)
    cs = L / np.floor(L / cell_side)
    for i in range(len(r)):
        ax = rng.integers(3)
        x = r[i, ax]
        k = np.arange(-1, D[ax] + 2)
        edges = np.concatenate([shift[ax] + k * T[ax], shift[ax] + k * T[ax] + T[ax] - w,
                                np.arange(0, int(L[ax] / cs[ax]) + 2) * cs[ax], [0.0]])
        e = edges[np.argmin(np.abs(edges - x))]
        if abs(e - x) < 0.24 * (a - 1.0):
            for _ in range(rng.integers(3)):
                e = np.nextafter(e, rng.choice([-np.inf, np.inf]))
            r[i, ax] = e
    return np.mod(r, L)


@pytest.mark.parametrize("dims", [(12, 13, 14), (20, 20, 20), (21, 20, 20), (64, 12, 11)])
def test_tags_on_boundaries_match_oracle(dims):
    rng = np.random.default_rng(5)
    a, D, w, side = 1.9, (4, 5, 4), 1.2, 1.3
    L = np.array(dims) * a
    ctx = ecmc.Context.create_lattice(dims, a, 1, b_max=1.2, jitter=0.0, seed=SEED)
    ctx.configure(mode=ecmc.MODE_DOMAIN, dir_mode=ecmc.DIR_ISO, tiles=D, lanes=32, cell_side=side)
    for sweep in (0, 7):
        _, shift = ctx.domain_tags(SEED, sweep)
        r = edge_positions(dims, a, D, w, shift, side, rng)
        ctx.set_positions(r)
        tags, _ = ctx.domain_tags(SEED, sweep)
        o = oracle.System(r, L, 1, mode=oracle.MODE_DOMAIN, dir_mode=oracle.DIR_ISO, D=D, seed=SEED)
        ref, _ = o.domain_tags(sweep)
        assert (tags == ref).all(), np.nonzero(tags != ref)[0][:5]


@pytest.mark.parametrize("dims", [(4, 4, 5), (20, 20, 20), (21, 20, 20)])
def test_pair_counts_match_direct_count(dims):
    """Shells at contact through the cells (3 cells on an axis and more)."""
    rng = np.random.default_rng(6)
    a = 1.045
    L = np.array(dims) * a
    r = (np.stack(np.meshgrid(*(np.arange(d) for d in dims), indexing="ij"), -1).reshape(-1, 3) + 0.5) * a
    r = r + rng.uniform(-0.022, 0.022, r.shape)
    ctx = ecmc.Context.create_lattice(dims, a, 1, b_max=1.2, jitter=0.0, seed=SEED)
    ctx.set_positions(r)
    obs = ctx.observables()
    s1 = s2 = 0
    for i in range(len(r)):
        d = r[i + 1:] - r[i]
        d -= L * np.round(d / L)
        q = (d ** 2).sum(1)
        s1 += int(((q >= 1.0 - 1e-10) & (q < 1.02 * 1.02)).sum())
        s2 += int(((q >= 1.02 * 1.02) & (q < 1.04 * 1.04)).sum())
    assert obs["overlaps"] == 0
    assert tuple(obs["contact_pairs"]) == (s1, s2)


def test_pairs_just_beyond_the_outer_shell():
    """Squared distances next to the bound up to which FP32 leaves a pair to
    FP64 (outer shell + error of a square): beyond the shell, so none counts."""
    a, dims = 3.0, (12, 12, 24)
    L = np.array(dims) * a
    rng = np.random.default_rng(7)
    site = np.stack(np.meshgrid(*(np.arange(d) for d in (12, 12, 12)), indexing="ij"), -1).reshape(-1, 3)
    r0 = (site + 0.5) * np.array([3.0, 3.0, 6.0])
    s2 = 1.04 ** 2
    err = 16.0 * 1.04 * (L.max() + 1.04) / 2.0 ** 24 + 1e-6 * s2
    d2 = s2 + err * rng.uniform(0.5, 1.5, len(r0))
    v = rng.normal(size=r0.shape)
    v *= (np.sqrt(d2) / np.linalg.norm(v, axis=1))[:, None]
    ctx = ecmc.Context.create_lattice(dims, a, 1, b_max=1.2)
    ctx.set_positions(np.concatenate([r0 - 0.5 * v, r0 + 0.5 * v]))
    obs = ctx.observables()
    assert obs["overlaps"] == 0 and tuple(obs["contact_pairs"]) == (0, 0)
