"""Fossil sampling of more genomes than one block resolves needs scratch
memory, and a captured run keeps its address: it is the fossils' own, whatever
samples are taken between capture and launch."""
import ctypes

import numpy as np
import pytest

from conftest import oracle_config
from paper_2404_10861_gb300 import inputs

pytestmark = pytest.mark.gpu
KW = dict(rows=64, cols=64, n=32, tournament=2, policy="tilted", bits=1, p_ben=0.02, seed=8)
K, EVERY = 2000, 4          # above 1,024: drawn through scratch memory


@pytest.fixture(scope="module")
def hb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2404_10861_gb300 import _build, binding
    _build.build()
    return binding


def test_a_larger_sample_leaves_the_fossils_memory(hb):
    import torch
    live, freed = {}, []

    def alloc(nbytes, stream, ctx):
        t = torch.empty(nbytes + 256, dtype=torch.uint8, device="cuda")
        live[t.data_ptr()] = t
        return t.data_ptr()

    cbs = (hb.ALLOC_FN(alloc), hb.FREE_FN(lambda p, s, c: freed.append(p)))
    assert hb.lib().hsga_set_allocator(cbs[0], cbs[1], ctypes.c_void_p()) == 0
    try:
        g = hb.Grid(**KW)
    finally:
        hb.use_default_allocator()
    with g:
        before = set(live)
        hb.hsga_set_fossil_sampling(g.handle, EVERY, K, capacity=4 * K)
        fossils = set(live) - before
        assert len(fossils) == 3
        g.sample(4096)
        assert not fossils & set(freed)
        hb.hsga_set_fossil_sampling(g.handle, 0, 0, 0)
        assert fossils <= set(freed)


@pytest.mark.parametrize("kernel", [0, 1])
def test_captured_fossils_after_a_larger_sample(hb, orc, kernel):
    import torch
    stream = torch.cuda.Stream()
    c = oracle_config(orc, KW)
    trait, surf = inputs.random_population(c.agents, seed=2)
    with hb.Grid(stream=stream.cuda_stream, kernel=kernel, **KW) as g:
        hb.hsga_set_fossil_sampling(g.handle, EVERY, K, capacity=4 * K)
        g.set_population(trait, surf, 40)
        g.sync()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.stream(stream):
            graph.capture_begin(capture_error_mode="thread_local")
            try:
                g.run(2 * EVERY)
            finally:
                graph.capture_end()
        g.sample(4096)
        with torch.cuda.stream(stream):
            graph.replay()
        g.sync()
        words, where = hb.hsga_get_fossils(g.handle, 4 * K)
        got = g.population()
    assert len(words) == 2 * K
    t, s = trait, surf
    for i in range(2):
        t, s, _ = orc.run(c, t, s, G0=40 + EVERY * i, generations=EVERY)
        ow, owhere = orc.sample(c, t, s, 40 + EVERY * (i + 1), K)
        assert np.array_equal(words[i * K:(i + 1) * K], ow)
        assert np.array_equal(where[i * K:(i + 1) * K], owhere)
    assert np.array_equal(got[0], t) and np.array_equal(got[1], s)
