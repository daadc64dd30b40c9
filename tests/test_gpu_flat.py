"""Streamed generations of every shape that the 32-agent kernel does not serve
(other island sizes, binary32 fitness, wide surfaces), where the flat
numbering of a group's children can go wrong: groups cut off at the end of the
grid, island sizes around a warp, more groups than resident warps, and groups
that do not start on a 16-byte boundary.  Bit-exact with the oracle."""
import numpy as np
import pytest

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


CASES = [dict(rows=1, cols=c, n=n) for c in (1, 7, 9) for n in (1, 3, 31, 33, 64)]
CASES += [dict(rows=173, cols=197, n=n, tournament=t)        # more groups than warps
          for n, t in ((1, 2), (3, 3), (17, 2), (24, 2), (33, 1))]
CASES += [dict(rows=13, cols=17, n=n, words=k, policy=pol, bits=b, tournament=t)
          for n, k, pol, b, t in ((32, 4, "tilted", 1, 2), (19, 4, "hybrid", 4, 5),
                                  (32, 2, "steady", 16, 2), (5, 2, "hybrid", 2, 1))]
CASES += [dict(rows=13, cols=17, n=n, fitness="float", sigma=0.7, policy=pol, words=k, bits=b)
          for n, k, pol, b in ((32, 1, "tilted", 1), (7, 1, "none", 1), (32, 1, "hybrid", 2),
                               (31, 4, "stretched", 1))]
CASES += [dict(rows=181, cols=199, n=32, words=2, policy="tilted"),
          dict(rows=181, cols=199, n=32, fitness="float", sigma=1.0, tournament=5),
          dict(rows=11, cols=13, n=40, policy="hybrid", interval=2, coarsen=2),
          dict(rows=11, cols=13, n=50, policy="none", interval=0)]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_flat_generations_match_the_oracle(hb, orc, case):
    kw = dict(dict(tournament=2, policy="steady", bits=1, W=2, interval=1, p_ben=0.05, p_del=0.1,
                   seed=70 + case), **CASES[case])
    flt = kw.get("fitness") == "float"
    c = orc.Config(rows=kw["rows"], cols=kw["cols"], n=kw["n"], tournament=kw["tournament"],
                   policy=orc.POLICY_NAMES[kw["policy"]], bits=kw["bits"], W=kw["W"],
                   interval=kw["interval"], p_ben=kw["p_ben"], p_del=kw["p_del"],
                   seed=kw["seed"], coarsen=kw.get("coarsen", 1),
                   fitness=orc.FITNESS_FLOAT if flt else 0, sigma=kw.get("sigma", 1.0),
                   words=kw.get("words", 1))
    rng = np.random.default_rng(case)
    trait, _ = inputs.small_trait_population(c.agents, seed=case, levels=4)
    if flt:
        trait = rng.normal(size=c.agents).astype(np.float32).view(np.uint32)
    surf = rng.integers(0, 2**64 - 1, size=c.agents * kw.get("words", 1), dtype=np.uint64)
    if kw["policy"] == "none":
        surf[:] = 0
    want = orc.run(c, trait, surf, G0=60, generations=5)[:2]
    with hb.Grid(kernel=hb.KERNEL_STREAMED, **kw) as g:
        g.set_population(trait, surf, 60)
        g.run(5)
        g.sync()
        got = g.population()
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])


def test_planes_without_16_byte_alignment(hb, orc):
    """An allocator that returns 8-byte aligned memory: plain loads and stores
    take the place of bulk copies and 16-byte stores."""
    import ctypes
    import torch
    held = []

    def alloc(nbytes, stream, ctx):
        t = torch.empty(nbytes + 64, dtype=torch.uint8, device="cuda")
        held.append(t)
        return t.data_ptr() + 8

    cbs = (hb.ALLOC_FN(alloc), hb.FREE_FN(lambda *a: None))
    for kw in (dict(rows=9, cols=7, n=48, policy="tilted"),
               dict(rows=9, cols=7, n=32, policy="tilted", words=4)):
        kw = dict(kw, tournament=2, bits=1, p_ben=0.1, seed=5)
        c = orc.Config(rows=9, cols=7, n=kw["n"], tournament=2, policy=orc.TILTED, bits=1, W=2,
                       interval=1, p_ben=0.1, seed=5, words=kw.get("words", 1))
        trait, _ = inputs.small_trait_population(c.agents, seed=1, levels=4)
        surf = np.random.default_rng(2).integers(0, 2**64 - 1, dtype=np.uint64,
                                                 size=c.agents * kw.get("words", 1))
        want = orc.run(c, trait, surf, G0=3, generations=6)[:2]
        assert hb.lib().hsga_set_allocator(cbs[0], cbs[1], ctypes.c_void_p()) == 0
        try:
            g = hb.Grid(kernel=hb.KERNEL_STREAMED, **kw)
        finally:
            hb.use_default_allocator()
        with g:
            g.set_population(trait, surf, 3)
            g.run(6)
            g.sync()
            got = g.population()
        assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
