"""Vertices without edges among the others: key positions without pieces, in long runs, and vertex counts
from 2^26 on, whose ranks no longer fit beside the labels in the neighbour lists."""
import numpy as np
import pytest

import graphgen as gg

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


def _padded(g, n, gap):
    """(row_ptr, col, labels) of g on n vertices: ids from `gap` on moved to the end, isolated vertices of
    every label between."""
    ids = np.arange(g.n)
    ids[gap:] += n - g.n
    deg = np.zeros(n, np.int64)
    deg[ids] = np.diff(g.row_ptr)
    row = np.zeros(n + 1, np.int32)
    row[1:] = np.cumsum(deg)
    labels = (np.arange(n) % g.num_labels).astype(np.int32)
    labels[ids] = g.labels
    return row, ids[g.col].astype(np.int32), labels


def _equal(a, b):
    assert len(a["support"]) > 0
    for key in ("labels", "adj", "support", "count"):
        assert np.array_equal(a[key], b[key]), key


@pytest.mark.parametrize("opts", [{}, {"launch": 1, "fused": 1}, {"join_quota": 3}], ids=["default", "one pass", "quota"])
def test_a_run_of_isolated_vertices_costs_no_more_in_the_middle(fsm, opts):
    """2^23 isolated vertices after the graph's, or between its two halves, where one chunk of pieces spans
    them all: the same result, in no more than four times the time (and 5 ms)."""
    g = gg.workload("cl100k", scale=0.02, cap=40)
    took, out = [], []
    for gap in (g.n, g.n // 2):
        G = fsm.Graph(*_padded(g, 1 << 23, gap), g.num_labels)
        for key, val in opts.items():
            G.set_option(key, val)
        G.mine(4, 20)
        out.append(G.mine(4, 20, stats=True))
        took.append(out[-1]["stats"]["time_ns"] / 1e6)
        G.close()
    if "join_quota" not in opts:   # what the quotas draw depends on the ids
        _equal(out[0], out[1])
    print("ms after, between:", took)
    assert took[1] <= 4 * took[0] + 5, took


def test_ranks_beside_the_lists_end_at_two_to_the_26(fsm):
    """On either side of 2^26 vertices, the same patterns, supports and counts: exact (two passes and one),
    vertex-induced and rate-sampled (ids as they are, so that the same edges are kept)."""
    g = gg.workload("cl3700k", scale=0.0002, cap=20)
    for mode in ("edge", "vertex"):
        ref = None
        for n in (g.n, 1 << 26):
            G = fsm.Graph(*_padded(g, n, g.n), g.num_labels, mode)
            got = []
            for k in (3, 4, 5):
                got.append(G.mine(k, 4))
            G.set_option("fused", 1)
            got.append(G.mine(5, 4))
            G.set_option("launch", 2)
            got.append(G.mine(4, 4))
            G.set_option("candidates", 1)
            got.append(G.mine(4, 4, sample_rate=0.5))
            G.close()
            if ref:
                for a, b in zip(got, ref):
                    _equal(a, b)
            ref = got
