"""Resident grids of a few islands of another size than 32, which run in one
block with an island to a warp: the smallest, the largest and the first that
are cut into tiles instead, bit-exact with the oracle."""
import numpy as np
import pytest

from conftest import oracle_config
from paper_2404_10861_gb300 import inputs

pytestmark = pytest.mark.gpu
ONE, TILES = 2, 3    # hsga_stats.kernel


@pytest.fixture(scope="module")
def hb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2404_10861_gb300 import _build, binding
    _build.build()
    return binding


@pytest.mark.parametrize("rows,cols,n,kernel,kw", [
    (1, 1, 1, ONE, {}), (1, 1, 64, ONE, dict(tournament=5)), (1, 2, 33, ONE, {}),
    (2, 2, 31, ONE, dict(policy="none")), (2, 4, 17, ONE, dict(interval=2)), (2, 4, 17, TILES, dict(interval=3)),
    (2, 11, 31, ONE, dict(tournament=3)), (11, 2, 9, ONE, dict(policy="hybrid", bits=2)),
    (1, 22, 20, ONE, dict(policy="none", p_del=0.2)), (1, 23, 20, TILES, {}),
    (3, 4, 64, ONE, {}), (1, 12, 33, ONE, dict(tournament=7, p_del=0.2)),
    (1, 13, 33, TILES, {}), (3, 4, 40, TILES, dict(interval=0)), (1, 7, 40, ONE, dict(interval=0))])
def test_few_islands(hb, orc, rows, cols, n, kernel, kw):
    kw = dict(dict(rows=rows, cols=cols, n=n, tournament=2, policy="tilted", bits=1, p_ben=0.1,
                   seed=rows + cols), **kw)
    c = oracle_config(orc, kw)
    trait, surf = inputs.small_trait_population(c.agents, seed=1, levels=4)
    if kw["policy"] == "none":
        surf = np.zeros_like(surf)
    want = orc.run(c, trait, surf, G0=9, generations=40)[:2]
    for request in (hb.KERNEL_RESIDENT, hb.KERNEL_RESIDENT_GRID):
        with hb.Grid(kernel=request, **kw) as g:
            assert g.stats()["kernel"] == (kernel if request == hb.KERNEL_RESIDENT else TILES)
            g.set_population(trait, surf, 9)
            g.run(1)
            g.migrate()
            g.run(39)
            g.sync()
            got = g.population()
        if kw.get("interval", 1) == 1:      # an explicit migration is the generation's own
            assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
        with hb.Grid(kernel=request, **kw) as g:
            g.set_population(trait, surf, 9)
            g.run(40)
            g.sync()
            got = g.population()
        assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
