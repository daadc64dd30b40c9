"""Tori of one row or column around the sizes at which tiles of one island end:
the resident kernel takes them all, bit-exact with the oracle."""
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


@pytest.mark.parametrize("rows,cols", [(1, 96), (1, 97), (1, 151), (1, 152), (1, 153), (120, 1),
                                       (2, 49), (97, 1)])
def test_one_row(hb, orc, rows, cols):
    import torch
    kw = dict(rows=rows, cols=cols, n=32, tournament=2, policy="tilted", bits=1, p_ben=0.1, seed=3)
    c = oracle_config(orc, kw)
    trait, surf = inputs.small_trait_population(c.agents, seed=1, levels=4)
    want = orc.run(c, trait, surf, G0=9, generations=20)[:2]
    with hb.Grid(kernel=hb.KERNEL_RESIDENT, **kw) as g:
        g.set_population(trait, surf, 9)
        g.run(20)
        g.sync()
        got = g.population()
    t = torch.from_numpy(trait.view(np.int32)).cuda()
    s = torch.from_numpy(surf.view(np.int64)).cuda()
    torch.cuda.synchronize()
    hb.hsga_run_generations_noalloc(hb.make_config(**kw), 9, 20, t, s)
    for x in (got, (t.cpu().numpy().view(np.uint32), s.cpu().numpy().view(np.uint64))):
        assert np.array_equal(x[0], want[0]) and np.array_equal(x[1], want[1])
