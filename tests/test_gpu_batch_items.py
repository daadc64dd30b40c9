"""Batches whose runs are cut into items of other than eight islands: islands of
odd, even and fourfold sizes, whose items start on 16-byte boundaries in
different steps, lists of every item size, and a large run whose end leaves the
others a list of smaller items.  Bit-exact with the oracle."""
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


def run(rows, cols, gens=30, **kw):
    return gens, dict(dict(rows=rows, cols=cols, n=32, tournament=2, policy="tilted", bits=1,
                           p_ben=0.1), **kw)


@pytest.mark.parametrize("runs", [
    [run(1, 1), run(1, 3, n=17), run(3, 3, n=18, tournament=5)],               # twos
    [run(63, 65, tournament=5), run(5, 7, n=19, policy="hybrid", bits=2)],
    [run(70, 71, n=18)], [run(70, 71, n=20, policy="none"), run(9, 9, n=33)],  # threes
    [run(100, 100, tournament=3, p_del=0.2)],                                  # fives
    [run(110, 120, n=17, interval=2)], [run(100, 121, n=34, policy="steady")],
    [run(100, 160, n=8)], [run(120, 135, n=64)],                               # sevens
    [run(150, 160, gens=14), run(31, 33, n=17, gens=40), run(40, 40, n=50, gens=23)]])
def test_items(hb, orc, runs):
    with hb.Batch() as b:
        ids = [b.add(gens, seed=5 + i, **kw) for i, (gens, kw) in enumerate(runs)]
        b.run(9)
        b.run(10**6)
        for rid, (gens, kw) in zip(ids, runs):
            want = orc.run(oracle_config(orc, dict(kw, seed=5 + rid)), generations=gens)[:2]
            got = b.population(rid)
            assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1]), rid
