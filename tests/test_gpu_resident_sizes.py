"""Resident grids of islands of another size than 32 on both sides of the limits
at which tiles of four islands give way to one large tile per SM, and of the
large tiles' group sizes, bit-exact with the oracle; the block count tells which
kernel took them."""
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


@pytest.mark.parametrize("rows,cols,n,small,kw", [
    (64, 64, 16, True, {}), (65, 66, 16, False, {}), (64, 76, 31, True, dict(tournament=5)),
    (68, 71, 17, True, dict(policy="none", tournament=3)), (70, 71, 31, False, {}),
    (70, 71, 25, False, dict(tournament=5, p_del=0.2)), (66, 66, 24, True, {}),
    (48, 64, 48, True, dict(policy="hybrid", bits=2)), (55, 56, 33, False, {}),
    (66, 66, 49, True, dict(tournament=5)), (70, 71, 64, False, dict(tournament=5)),
    (66, 66, 48, False, dict(policy="none", tournament=7)), (80, 80, 40, False, {}),
    (2, 2400, 20, True, dict(interval=2)), (1, 19, 48, True, {})])
def test_island_sizes(hb, orc, rows, cols, n, small, kw):
    import torch
    kw = dict(dict(rows=rows, cols=cols, n=n, tournament=2, policy="tilted", bits=1, p_ben=0.1,
                   seed=rows + cols), **kw)
    c = oracle_config(orc, kw)
    trait, surf = inputs.small_trait_population(c.agents, seed=1, levels=4)
    if kw["policy"] == "none":
        surf = np.zeros_like(surf)
    want = orc.run(c, trait, surf, G0=9, generations=12)[:2]
    with hb.Grid(kernel=hb.KERNEL_RESIDENT, **kw) as g:
        sms = torch.cuda.get_device_properties(0).multi_processor_count
        if sms == 152:          # the limits follow from the SMs
            assert (g.stats()["blocks"] == -(-rows * cols // 4)
                    or g.stats()["blocks"] > sms) == small
        g.set_population(trait, surf, 9)
        g.run(12)
        g.sync()
        got = g.population()
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
