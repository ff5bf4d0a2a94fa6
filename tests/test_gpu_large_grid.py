"""Cell pass on dilute melts with many cells: the pair counts on both sides of
the grid size from which the scan's tile sums are scanned by themselves, and
a pass whose time grows with the cells, not with their square."""
import time

import numpy as np
import pytest

from paper_1502_06447_gb300 import ecmc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    from paper_1502_06447_gb300 import build
    build.build()


@pytest.mark.parametrize("a", [33.5, 34.0])  # 510^3 and 518^3 cells: 32,386 and 33,934 tiles of 4,096
def test_pair_counts_on_large_grids(a):
    k = 16
    with ecmc.Context.create_lattice((k, k, k), a, 1) as ctx:
        rng = np.random.default_rng(3)
        r, _ = ctx.get_positions()
        r += rng.uniform(-0.4 * a, 0.4 * a, r.shape)
        near = rng.permutation(len(r))[:3000].reshape(-1, 2)  # 1,500 pairs at contact, the rest far apart
        v = rng.normal(size=(1500, 3))
        d = rng.choice([1.01, 1.03, 1.05], 1500)
        r[near[:, 1]] = r[near[:, 0]] + v * (d / np.linalg.norm(v, axis=1))[:, None]
        ctx.set_positions(np.mod(r, ctx.L))
        obs = ctx.observables()
    assert obs["overlaps"] == 0
    assert tuple(obs["contact_pairs"]) == ((d == 1.01).sum(), (d == 1.03).sum())


def test_pass_grows_with_the_cells():
    """761^3 and 1280^3 cells, 4.8 times as many: a linear pass takes 4.7 times
    as long, one whose blocks all add up the sums of the blocks before them
    some 10 times."""
    t = []
    for a in (50.0, 84.0):
        with ecmc.Context.create_lattice((16, 16, 16), a, 1) as ctx:
            ctx.observables()
            s = []
            for _ in range(8):
                t0 = time.perf_counter()
                ctx.observables()
                s.append(time.perf_counter() - t0)
            t.append(min(s))
    assert t[1] < 6.0 * t[0], t
