"""Device memory from allocator hooks that align to eight bytes only: whatever
the library reads or writes in 16-byte pieces starts on a 16-byte boundary all
the same, or is read and written otherwise.  Bit-exact with the oracle."""
import contextlib
import ctypes

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


@contextlib.contextmanager
def eight_byte_memory(hb):
    """Grids and batches made inside hold memory that starts 8 bytes past a
    16-byte boundary."""
    import torch
    held = []

    def alloc(nbytes, stream, ctx):
        held.append(torch.empty(nbytes + 64, dtype=torch.uint8, device="cuda"))
        return held[-1].data_ptr() + 8

    cbs = (hb.ALLOC_FN(alloc), hb.FREE_FN(lambda *a: None))
    assert hb.lib().hsga_set_allocator(cbs[0], cbs[1], ctypes.c_void_p()) == 0
    try:
        yield
    finally:
        hb.use_default_allocator()


def check(hb, orc, gens=6, migrate=False, **kw):
    kw = dict(dict(n=32, tournament=2, policy="tilted", bits=1, p_ben=0.1, seed=5), **kw)
    c = oracle_config(orc, kw)
    trait, surf = inputs.small_trait_population(c.agents, seed=1, levels=4)
    if kw["policy"] == "none":
        surf = np.zeros_like(surf)
    want = orc.run(c, trait, surf, G0=3, generations=gens)[:2]
    with eight_byte_memory(hb), hb.Grid(**kw) as g:
        g.set_population(trait, surf, 3)
        if migrate:
            g.migrate()
        g.run(gens)
        g.sync()
        got = g.population()
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])


# several tiles of the small, the general and the register kernel, and one block
@pytest.mark.parametrize("kw", [
    dict(rows=11, cols=12), dict(rows=11, cols=12, policy="none"), dict(rows=64, cols=66),
    dict(rows=95, cols=104), dict(rows=70, cols=71, n=9), dict(rows=9, cols=10, n=20),
    dict(rows=4, cols=4), dict(rows=11, cols=12, migrate=True)])
def test_resident_grids(hb, orc, kw):
    check(hb, orc, kernel=hb.KERNEL_RESIDENT, **kw)


@pytest.mark.parametrize("kw", [
    dict(rows=9, cols=7), dict(rows=9, cols=7, policy="none", tournament=5),
    dict(rows=181, cols=199, p_del=0.2), dict(rows=9, cols=7, policy="hybrid", bits=2)])
def test_streamed_grids_of_32_agents(hb, orc, kw):
    check(hb, orc, kernel=hb.KERNEL_STREAMED, **kw)


@pytest.mark.parametrize("k", [30, 1200])
def test_samples_and_fossils(hb, orc, k):
    kw = dict(rows=40, cols=41, n=32, tournament=2, policy="tilted", bits=1, p_ben=0.1, seed=6)
    c = oracle_config(orc, kw)
    t, s = orc.run(c, generations=8)[:2]
    want = orc.sample(c, t, s, 8, k)
    with eight_byte_memory(hb), hb.Grid(**kw) as g, hb.Batch() as b, \
            hb.Grid(**dict(kw, words=2)) as w:
        hb.hsga_set_fossil_sampling(g.handle, 4, k, 2 * k)
        g.run(8)
        rid = b.add(8, **kw)
        b.run(8)
        w.run(8)
        words, where = hb.hsga_get_fossils(g.handle, 2 * k)
        got = [g.sample(k), b.sample(rid, k), (words[k:], where[k:])]
        assert np.array_equal(w.sample(k)[1], want[1])
    for x, y in got:
        assert np.array_equal(x, want[0]) and np.array_equal(y, want[1])


def test_buffered_channels(hb):
    kw = dict(rows=9, cols=7, n=32, tournament=2, policy="tilted", bits=1, seed=7, mode="buffered")
    with eight_byte_memory(hb), hb.Grid(**kw) as g:
        g.run(40)
        g.sync()
        chan, _ = g.buffers()
    assert chan[:, :, 0].min() > 0 and chan[:, :, 2].max() <= 4
