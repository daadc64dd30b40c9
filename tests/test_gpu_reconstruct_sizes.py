"""Reconstruction at the sizes where its kernels change form: one block's sort
and tiles of keys, blocks of 1,024 lcps and their neighbours, more blocks than
one step of the scan over them, keys of two and four words.  Surfaces descend
from a few ancestors, so that intervals span many blocks.  The reference is
the lcp-interval tree of the sorted keys, built with a stack."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
G, W = 1000, 2


@pytest.fixture(scope="module")
def hb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2404_10861_gb300 import _build, binding
    _build.build()
    return binding


def lineage_surfaces(rng, k, words):
    """k surfaces: copies of a few ancestors with a handful of bits changed."""
    base = rng.integers(0, 2**64 - 1, size=(5, words), dtype=np.uint64)
    surf = base[rng.integers(0, 5, k)]
    for _ in range(4):
        pick = rng.random(k) < 0.4
        bit = rng.integers(0, 64 * words, k)
        flip = np.uint64(1) << (bit % 64).astype(np.uint64)
        rows = np.nonzero(pick)[0]
        surf[rows, bit[rows] // 64] ^= flip[rows]
    return surf


def reference(hb, surf, policy, bits, words):
    """{(time, first leaf, last leaf)} of the internal nodes, and the samples'
    retained fields in order of time."""
    S = 64 * words // bits
    when = hb.hsga_lookup(policy, S, W, G)
    order = [s for s in np.argsort(when, kind="stable") if when[s] >= 0]
    fields = np.stack([(surf[:, s * bits // 64] >> np.uint64(s * bits % 64)) &
                       np.uint64((1 << bits) - 1) for s in order], axis=1)
    rank = np.lexsort(fields.T[::-1])
    f = fields[rank]
    k = len(f)
    differ = f[1:] != f[:-1]
    lcp = np.where(differ.any(axis=1), differ.argmax(axis=1), len(order))
    nodes, stack = set(), [(0, 0)]                     # (value, first leaf)
    for p, l in enumerate(lcp.tolist() + [0]):
        first = p
        while stack[-1][0] > l:
            v, first = stack.pop()
            nodes.add((int(when[order[v - 1]]), first, p))
        if l > stack[-1][0]:
            stack.append((l, first))
    return nodes, fields


@pytest.mark.parametrize("k,words,policy,bits", [
    (1, 1, 1, 1), (2, 1, 1, 1), (33, 1, 1, 1), (1023, 1, 0, 1), (1024, 1, 1, 1), (1025, 1, 1, 2),
    (1026, 1, 2, 1), (2049, 1, 1, 1), (12288, 1, 1, 1), (12289, 1, 1, 1), (12289, 1, 0, 1),
    (5000, 2, 1, 1), (5000, 4, 0, 1), (9000, 4, 5, 4), (34000, 1, 1, 1), (270000, 1, 1, 1)])
def test_interval_tree(hb, k, words, policy, bits):
    rng = np.random.default_rng(k + words)
    surf = lineage_surfaces(rng, k, words)
    want, fields = reference(hb, surf, policy, bits, words)
    parent, time, leaf = hb.hsga_reconstruct(surf.reshape(-1), policy, bits, W, G, words=words)
    n = len(parent)
    assert sorted(leaf.tolist()) == list(range(n - k, n))
    # leaves in sorted order of their keys
    by_place = fields[np.argsort(leaf)]
    step = by_place[1:] != by_place[:-1]
    first = step.argmax(axis=1)
    rows = np.nonzero(step.any(axis=1))[0]
    assert (by_place[rows + 1, first[rows]] > by_place[rows, first[rows]]).all()
    # first and last leaf below every node
    lo, hi = np.full(n, n), np.full(n, -1)
    lo[n - k:] = hi[n - k:] = np.arange(k)
    node = np.arange(n - k, n)
    for _ in range(fields.shape[1] + 2):
        up = parent[node]
        live = up >= 0
        np.minimum.at(lo, up[live], lo[node[live]])
        np.maximum.at(hi, up[live], hi[node[live]])
        node = np.unique(up[live])
    got = {(int(time[v]), int(lo[v]), int(hi[v])) for v in range(1, n - k)}
    assert len(got) == n - k - 1 and got == want
    # every leaf hangs from the smallest interval around it
    size = {}
    for v in range(1, n - k):
        size[v] = hi[v] - lo[v]
    inside = np.zeros(k, dtype=np.int64)
    for v in sorted(size, key=lambda v: -size[v]):
        inside[lo[v]:hi[v] + 1] = v
    assert (parent[n - k:] == inside).all()
