"""Calls of a few generations on grids that the library runs resident by its own
choice are streamed: runs cut into calls of every length around the limit, with
explicit migrations, samples and fossils between them, are bit-exact with the
oracle, and under capture nothing changes plane."""
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


@pytest.mark.parametrize("kw", [
    dict(rows=1, cols=1), dict(rows=4, cols=4, tournament=5), dict(rows=4, cols=4, n=17),
    dict(rows=9, cols=8, policy="none"), dict(rows=64, cols=64, policy="hybrid", bits=2),
    dict(rows=65, cols=66, n=48), dict(rows=30, cols=31, n=40, tournament=7),
    dict(rows=9, cols=9, tournament=9), dict(rows=100, cols=100, interval=2, coarsen=2),
    dict(rows=150, cols=160, p_del=0.2), dict(rows=170, cols=150, tournament=5),
    dict(rows=300, cols=290, n=1)])
def test_cut_runs(hb, orc, kw):
    kw = dict(dict(n=32, tournament=2, policy="tilted", bits=1, p_ben=0.1, seed=12), **kw)
    c = oracle_config(orc, kw)
    trait, surf = inputs.small_trait_population(c.agents, seed=1, levels=4)
    if kw["policy"] == "none":
        surf = np.zeros_like(surf)
    calls = (1, 2, 3, 4, 1, 5, 2, 1, 3, 6)
    with hb.Grid(**kw) as g:
        assert g.stats()["kernel"] != hb.KERNEL_STREAMED
        g.set_population(trait, surf, 30)
        launches = []
        for i, n in enumerate(calls):
            if i in (2, 4, 5) and kw.get("interval", 1) == 1:
                g.migrate()                  # the generation's own, ahead of its call
            before = g.stats()["kernel_launches"]
            g.run(n)
            launches.append(g.stats()["kernel_launches"] - before)
        g.sync()
        got = g.population()
    want = orc.run(c, trait, surf, G0=30, generations=sum(calls))[:2]
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
    blocks = (1 if c.tournament <= 2 else 1 + -(-(c.tournament - 2) // 4)) * (2 if c.n > 32 else 1)
    few = c.rows * c.cols < 64 or c.n > 32 or c.interval != 1
    most = 1 if blocks > 2 else 2 if few else 3 if blocks == 2 else 4
    assert launches == [n if n <= most else 1 for n in calls]


def test_short_calls_under_capture_work_in_place(hb, orc):
    import torch
    kw = dict(rows=16, cols=16, n=32, tournament=2, policy="tilted", bits=1, p_ben=0.1, seed=2)
    c = oracle_config(orc, kw)
    trait, surf = inputs.random_population(c.agents, seed=3)
    stream = torch.cuda.Stream()
    with hb.Grid(stream=stream.cuda_stream, **kw) as g:
        g.set_population(trait, surf, 7)
        g.run(1)
        g.sync()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.stream(stream):
            graph.capture_begin(capture_error_mode="thread_local")
            try:
                g.run(1)
                g.run(2)
            finally:
                graph.capture_end()
            graph.replay()
        g.run(3)
        g.sync()
        got = g.population()
    want = orc.run(c, trait, surf, G0=7, generations=7)[:2]
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
