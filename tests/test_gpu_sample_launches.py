"""Kernels that a sample launches, as the counters report them: one up to 1,024
genomes, two above (and one more that gathers wide surfaces)."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2404_10861_gb300 import _build, binding
    _build.build()
    return binding


@pytest.mark.parametrize("k,kernels", [(1, 1), (1024, 1), (1025, 2), (1600, 2)])
def test_launches(hb, k, kernels):
    kw = dict(rows=40, cols=40, n=4, tournament=2, policy="tilted", bits=1, seed=1)
    with hb.Grid(**kw) as g, hb.Grid(**dict(kw, words=2)) as w, hb.Batch() as b:
        rid = b.add(4, **kw)
        b.run(4)
        for x, sample, more in ((g, g.sample, 0), (w, w.sample, 1),
                                (b, lambda m: b.sample(rid, m), 0)):
            before = x.stats()["kernel_launches"]
            sample(k)
            assert x.stats()["kernel_launches"] - before == kernels + more
        hb.hsga_set_fossil_sampling(g.handle, 8, k, k)
        before = g.stats()["kernel_launches"]
        g.run(8)
        assert g.stats()["kernel_launches"] - before == 1 + kernels
