"""A tick that gave up a bounded wait leaves islands behind and sets the batch's
error word; every call that hands results out reports it, and the batch does
not run on.  The word is set here from the host, in the allocation that holds
it beside the tick."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
KW = dict(rows=4, cols=4, n=32, tournament=2, policy="tilted", bits=1, seed=4)


@pytest.fixture(scope="module")
def hb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2404_10861_gb300 import _build, binding
    _build.build()
    return binding


@pytest.mark.parametrize("word,status", [(1, -5), (2, -4)])   # wait timeout, inconsistent state
@pytest.mark.parametrize("call", ["population", "sample", "sync"])
def test_a_ticks_error_reaches_the_caller(hb, call, word, status):
    import torch
    held = []

    def alloc(nbytes, stream, ctx):
        held.append(torch.zeros(nbytes + 256, dtype=torch.uint8, device="cuda"))
        return held[-1].data_ptr()

    cbs = (hb.ALLOC_FN(alloc), hb.FREE_FN(lambda *a: None))
    assert hb.lib().hsga_set_allocator(cbs[0], cbs[1], ctypes.c_void_p()) == 0
    try:
        b = hb.Batch()
    finally:
        hb.use_default_allocator()
    with b:
        assert len(held) == 1 and held[0].numel() == 8 + 256     # tick, error word
        rid = b.add(100, **KW)
        b.run(10)
        b.sync()
        b.population(rid)
        held[0].view(torch.int32)[1] = word
        torch.cuda.synchronize()
        calls = dict(population=lambda: b.population(rid), sample=lambda: b.sample(rid, 3),
                     sync=b.sync, run=lambda: b.run(10))
        for name in (call, "run", "population", "sample", "sync"):
            with pytest.raises(hb.HsgaError) as e:
                calls[name]()
            assert e.value.status == status, name
        assert b.info(rid)["generation"] == 10
