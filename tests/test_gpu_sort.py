"""Sorting of pattern codes at the sizes where its forms meet: disjoint labeled paths, each its own
pattern, so a level has exactly as many quick patterns as paths -- around the block sort's 2048
records and the radix sort's tiles, and codes of more than 64 bits (8 vertices)."""
import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fsm():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2101_07690_gb300 import build, fsm as f
    build.build()
    f.load()
    return f


def _paths(count, k):
    """count disjoint paths of k vertices with distinct label sequences that are not reversals of
    each other (the last label is above the first)."""
    rng = np.random.default_rng(count + k)
    seen = set()
    while len(seen) < count:
        s = tuple(int(x) for x in rng.integers(0, 64, k))
        if s[0] < s[-1]:
            seen.add(s)
    lab = np.array(sorted(seen), np.int32)[rng.permutation(count)].reshape(-1)
    edges = [(k * p + i, k * p + i + 1) for p in range(count) for i in range(k - 1)]
    perm = rng.permutation(count * k)
    out = np.empty_like(lab)
    out[perm] = lab
    return gg.from_edges(count * k, perm[np.array(edges)], out, 64)


@pytest.mark.parametrize("count,k", [(1, 3), (2, 3), (33, 3), (2047, 3), (2048, 3), (2049, 3), (4096, 3), (4097, 3),
                                     (6145, 3), (2049, 5), (2100, 8)])
def test_every_path_is_one_pattern(fsm, count, k):
    g = _paths(count, k)
    exp = oracle.mine(g, k, 1)
    assert len(exp["support"]) == count
    G = fsm.Graph.from_graphgen(g)
    got = G.mine(k, 1)
    G.close()
    for key in ("labels", "adj", "support", "count"):
        assert np.array_equal(got[key], exp[key]), key
