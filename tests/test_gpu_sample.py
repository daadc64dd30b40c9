"""End-state sampling around the sizes where the sampler changes form (one
block's table up to 1,024 draws, scratch memory above) and where every island
is drawn, so that long chains of swaps must be followed: equal to the
oracle's shuffle."""
import numpy as np
import pytest

from conftest import oracle_config

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2404_10861_gb300 import _build, binding
    _build.build()
    return binding


@pytest.mark.parametrize("rows,cols", [(1, 1), (25, 41), (50, 61)])
def test_samples_match_the_oracle(hb, orc, rows, cols):
    kw = dict(rows=rows, cols=cols, n=5, tournament=2, policy="tilted", bits=1, seed=rows)
    islands = rows * cols
    with hb.Grid(**kw) as g:
        for G in (1, 300):
            g.run(G - g.stats()["generation"])
            g.sync()
            t, s = g.population()
            for k in (1, 31, 32, 33, 1023, 1024, 1025, 2049, islands - 1, islands):
                if not 1 <= k <= islands:
                    continue
                w, where = g.sample(k)
                ow, owhere = orc.sample(oracle_config(orc, kw), t, s, G, k)
                assert np.array_equal(w, ow) and np.array_equal(where, owhere), (G, k)
