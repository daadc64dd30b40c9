"""Streamed runs whose launches work out the migration of later generations and
walk every other generation backwards: grids of at least two groups per warp
and grids beyond L2, island counts that no group size divides, one- and
two-wide torus sides, migration intervals, and runs cut into calls at which the
planning starts again.  Bit-exact with the oracle."""
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


CASES = [
    dict(rows=1, cols=3), dict(rows=7, cols=1, tournament=5), dict(rows=5, cols=6),  # groups of four
    dict(rows=41, cols=59, policy="hybrid", bits=2), dict(rows=64, cols=228, p_del=0.2),
    dict(rows=97, cols=151, policy="none", tournament=3),                  # one round of eight
    dict(rows=205, cols=191),                                              # groups of 32-agent islands
    dict(rows=2, cols=19501, interval=2, tournament=5, p_del=0.3),
    dict(rows=39003, cols=1, interval=3, policy="none", calls=(9,)),
    dict(rows=229, cols=173, policy="hybrid", bits=2, coarsen=2, calls=(5, 1)),
    dict(rows=331, cols=521, calls=(4,)),                                  # beyond L2
    dict(rows=331, cols=521, tournament=3, p_del=0.3, calls=(3,)),
    dict(rows=301, cols=260, n=17), dict(rows=1, cols=70001, n=1, interval=2),
    dict(rows=241, cols=202, n=33, tournament=3, p_del=0.2, calls=(4, 2)),
    dict(rows=223, cols=233, n=64, tournament=5, policy="none", calls=(4,)),
    dict(rows=251, cols=241, words=4, calls=(4, 1)),                       # beyond L2
    dict(rows=353, cols=347, words=2, calls=(3,)),
    dict(rows=443, cols=397, fitness="float", sigma=0.7, calls=(3,)),
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_planned_generations_match_the_oracle(hb, orc, case):
    kw = dict(dict(n=32, tournament=2, policy="tilted", bits=1, W=2, interval=1, p_ben=0.05,
                   seed=170 + case), **CASES[case])
    calls = kw.pop("calls", (1, 2, 5))
    flt, words = kw.get("fitness") == "float", kw.get("words", 1)
    c = orc.Config(rows=kw["rows"], cols=kw["cols"], n=kw["n"], tournament=kw["tournament"],
                   policy=orc.POLICY_NAMES[kw["policy"]], bits=kw["bits"], W=kw["W"],
                   interval=kw["interval"], p_ben=kw["p_ben"], p_del=kw.get("p_del", 0.0),
                   seed=kw["seed"], coarsen=kw.get("coarsen", 1),
                   fitness=orc.FITNESS_FLOAT if flt else 0, sigma=kw.get("sigma", 1.0),
                   words=words)
    rng = np.random.default_rng(case)
    trait, _ = inputs.small_trait_population(c.agents, seed=case, levels=4)
    if flt:
        trait = rng.normal(size=c.agents).astype(np.float32).view(np.uint32)
    surf = rng.integers(0, 2**64 - 1, size=c.agents * words, dtype=np.uint64)
    if kw["policy"] == "none":
        surf[:] = 0
    want = orc.run(c, trait, surf, G0=61, generations=sum(calls))[:2]
    with hb.Grid(kernel=hb.KERNEL_STREAMED, **kw) as g:
        g.set_population(trait, surf, 61)
        for n in calls:
            g.run(n)
        g.sync()
        got = g.population()
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])


def test_explicit_migration_before_a_planned_run(hb):
    """The migrant records share the moves' buffer."""
    kw = dict(rows=205, cols=191, n=32, tournament=2, policy="tilted", bits=1, p_ben=0.05, seed=9)
    got = []
    for explicit in (False, True):
        with hb.Grid(kernel=hb.KERNEL_STREAMED, **kw) as g:
            g.set_population(*inputs.random_population(g.agents, seed=4), 10)
            for _ in range(2):
                if explicit:
                    g.migrate()
                g.run(5)
            g.sync()
            got.append(g.population())
    assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])
