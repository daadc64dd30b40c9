"""Streamed 32-agent grids of a few more islands than one round of groups of
eight takes go in groups of four: both sides of each limit on 152 SMs (other
devices run other groups, with the same results), bit-exact with the oracle."""
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


@pytest.mark.parametrize("rows,cols,kw", [
    (1, 19456, {}), (1, 19457, {}), (19459, 1, dict(policy="none")), (1, 24320, dict(tournament=5)),
    (1, 24321, dict(tournament=5, p_del=0.2)), (1, 29184, {}), (1, 29185, {}),
    (137, 213, dict(policy="hybrid", bits=2, interval=2)), (163, 179, dict(tournament=3))])
def test_groups_of_four(hb, orc, rows, cols, kw):
    kw = dict(dict(rows=rows, cols=cols, n=32, tournament=2, policy="tilted", bits=1, p_ben=0.1,
                   seed=rows + cols), **kw)
    c = oracle_config(orc, kw)
    trait, surf = inputs.small_trait_population(c.agents, seed=1, levels=4)
    if kw["policy"] == "none":
        surf = np.zeros_like(surf)
    want = orc.run(c, trait, surf, G0=9, generations=5)[:2]
    with hb.Grid(kernel=hb.KERNEL_STREAMED, **kw) as g:
        g.set_population(trait, surf, 9)
        g.run(5)
        g.sync()
        got = g.population()
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
