"""Resident kernels at the edges of their tiles: the smallest and largest
tiles of each variant, tiles cut off at the torus's last row and column, the
one-block limit and island sizes that do not fill a warp, each bit-exact with
the oracle's run of the same grid."""
import numpy as np
import pytest

from conftest import oracle_config
from paper_2404_10861_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2404_10861_gb300 import _build, binding
    _build.build()
    return binding


# Sides are chosen for tiles on 152 SMs; on another device they are still grids.
SHAPES = [
    dict(rows=1, cols=3), dict(rows=4, cols=6), dict(rows=5, cols=5),   # one block, then tiles
    dict(rows=8, cols=19), dict(rows=9, cols=17),                       # one island a tile, two
    dict(rows=2, cols=1976), dict(rows=54, cols=76),                    # 26 islands a tile, 27
    dict(rows=92, cols=76), dict(rows=47, cols=152),                    # 46, 47
    dict(rows=76, cols=128), dict(rows=95, cols=104),                   # 64, 65
    dict(rows=131, cols=149),                                           # tiles cut off both ways
    dict(rows=2, cols=4, n=20, tournament=3), dict(rows=15, cols=15, n=22),   # a warp an island
    dict(rows=7, cols=9, n=47, policy="hybrid", bits=2, interval=2), dict(rows=64, cols=64, n=31),
    dict(rows=1, cols=7, n=33), dict(rows=33, cols=62, n=64, policy="none"),
    dict(rows=3, cols=400, n=1), dict(rows=40, cols=61, n=31), dict(rows=70, cols=71, n=33),
    dict(rows=97, cols=101, n=17, tournament=3), dict(rows=64, cols=77, n=64, tournament=5),
    dict(rows=90, cols=93, policy="none", p_del=0.1), dict(rows=20, cols=31, policy="none"),
    dict(rows=60, cols=61, policy="hybrid", bits=2, p_del=0.3, tournament=7),
    dict(rows=101, cols=99, policy="steady", interval=2, tournament=5, p_del=0.33),
    dict(rows=16, cols=16, policy="stretched", interval=3, coarsen=2),
]


@pytest.mark.parametrize("case", range(len(SHAPES)))
def test_tiles_match_the_oracle(hb, orc, case):
    kw = dict(dict(n=32, tournament=2, policy="tilted", bits=1, p_ben=0.02, seed=50 + case),
              **SHAPES[case])
    c = oracle_config(orc, kw)
    trait, surf = inputs.small_trait_population(c.agents, seed=case, levels=5)
    if kw["policy"] == "none":
        surf = np.zeros_like(surf)
    G0 = 1021
    want = orc.run(c, trait, surf, G0=G0, generations=19)[:2]
    with hb.Grid(kernel=hb.KERNEL_RESIDENT, **kw) as g:
        g.set_population(trait, surf, G0)
        g.run(1)
        g.run(18)
        g.sync()
        got = g.population()
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])


@pytest.mark.parametrize("policy", ["none", "tilted"])
def test_records_are_never_torn(hb, policy):
    """Fast tiles of one island, whose records are read as they are written:
    repeated runs from random states against the streamed kernel."""
    kw = dict(rows=12, cols=12, n=32, tournament=1, policy=policy, bits=1, seed=3)
    with hb.Grid(kernel=hb.KERNEL_STREAMED, **kw) as a, \
            hb.Grid(kernel=hb.KERNEL_RESIDENT_GRID, **kw) as b:
        for rep in range(40):
            trait, surf = inputs.random_population(a.agents, seed=rep)
            if policy == "none":
                surf = np.zeros_like(surf)
            for g in (a, b):
                g.set_population(trait, surf, 7 * rep)
                g.run(23)
                g.sync()
            x, y = a.population(), b.population()
            assert np.array_equal(x[0], y[0]) and np.array_equal(x[1], y[1])


def test_tiles_of_two_sizes_from_two_threads(hb):
    """Each launch gets its own tile's shared memory, whatever another thread
    launches the same kernel with."""
    import threading
    shapes, failed = [(76, 128), (150, 200)], []

    def steps(rows, cols):
        try:
            with hb.Grid(kernel=hb.KERNEL_RESIDENT, rows=rows, cols=cols, n=32, tournament=2,
                         policy="tilted", bits=1, seed=1) as g:
                g.set_population(*inputs.random_population(g.agents, seed=1), 0)
                for _ in range(2000):
                    g.run(1)
                g.sync()
        except Exception as e:
            failed.append(e)

    threads = [threading.Thread(target=steps, args=s) for s in shapes]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed
