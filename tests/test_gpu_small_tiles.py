"""The resident kernel for tiles of up to 64 islands with two and with four
islands to a child warp and tournaments of other than two: draws of a second
block for every child, of more for tournaments above six, two fields and
deleterious mutations.  Tile sizes are those on 152 SMs, where the block count
tells that the case is on the instance that it is for.  Bit-exact with the
oracle."""
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


@pytest.mark.parametrize("rows,cols,tile", [(54, 76, 27), (92, 76, 46), (47, 152, 47), (76, 128, 64)])
@pytest.mark.parametrize("kw", [
    dict(tournament=5, policy="tilted", p_del=0.3), dict(tournament=5, policy="none"),
    dict(tournament=7, policy="hybrid", bits=2), dict(tournament=7, policy="none", p_del=0.2),
    dict(tournament=1, policy="steady", interval=2), dict(tournament=11, policy="stretched")])
def test_tournaments(hb, orc, rows, cols, tile, kw):
    import torch
    kw = dict(dict(rows=rows, cols=cols, n=32, bits=1, p_ben=0.05, seed=tile), **kw)
    c = oracle_config(orc, kw)
    trait, surf = inputs.small_trait_population(c.agents, seed=1, levels=5)
    if kw["policy"] == "none":
        surf = np.zeros_like(surf)
    want = orc.run(c, trait, surf, G0=30, generations=11)[:2]
    with hb.Grid(kernel=hb.KERNEL_RESIDENT, **kw) as g:
        if torch.cuda.get_device_properties(0).multi_processor_count == 152:
            assert rows * cols == tile * g.stats()["blocks"]
        g.set_population(trait, surf, 30)
        g.run(1)
        g.run(10)
        g.sync()
        got = g.population()
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
