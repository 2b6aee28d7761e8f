"""What a level costs does not hang on how its joins fall: few keys, hubs, rare pieces.  Times of a pass are
those of option profile, best of three, compared with the same enumeration in another dress."""
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


def _two_hubs(labels, degree=20000, n=30000):
    """Two vertices of that degree over a sparse rest."""
    rng = np.random.default_rng(1)
    pairs = np.concatenate([np.stack([np.full(degree, h), rng.choice(np.arange(2, n), degree, replace=False)], 1)
                            for h in (0, 1)] + [rng.integers(2, n, (n - 10000, 2))])
    pairs = np.unique(np.sort(pairs[pairs[:, 0] != pairs[:, 1]], 1), axis=0)
    ids = rng.permutation(n)
    return gg.from_edges(n, ids[pairs], rng.integers(0, labels, n).astype(np.int32), labels)


def _pass_ms(fsm, g, k, t, name, options=None):
    G = fsm.Graph.from_graphgen(g)
    for key, val in {**(options or {}), "profile": 1}.items():
        G.set_option(key, val)
    try:
        return min(G.mine(k, t, stats=True)["stats"][name] for _ in range(4)) / 1e6
    finally:
        G.close()


def test_few_keys_cost_no_more_than_many(fsm):
    """Size 3 on two hubs: 4e8 joins of some 100 quick patterns (4 labels) or of 100000 (64 labels)."""
    few, many = (_pass_ms(fsm, _two_hubs(labels), 3, 100, "count_ns_l1") for labels in (4, 64))
    assert few <= 1.5 * many, (few, many)


@pytest.mark.parametrize("name", ["count_ns_l1", "domain_ns_l1"])
def test_a_level_that_draws_nothing_costs_what_an_exact_one_does(fsm, name):
    """Join quotas draw nothing at size 3."""
    g = gg.workload("cl3700k", scale=0.1, cap=300)
    exact, quota = (_pass_ms(fsm, g, 3, 2000, name, o) for o in ({}, {"join_quota": 2}))
    assert quota <= 1.25 * exact, (exact, quota)


def test_matching_quota_alone_leaves_the_joins_exact(fsm):
    """With match_quota large enough to cut nothing and no join_quota: exact mining, in all three sizes."""
    g = gg.workload("cl3700k", scale=0.002, cap=40)
    G = fsm.Graph.from_graphgen(g)
    exact = [G.mine(k, 30) for k in (3, 4, 5)]
    G.set_option("match_quota", 1 << 32)
    for k, want in zip((3, 4, 5), exact):
        got = G.mine(k, 30)
        assert len(want["support"]) > 0
        for key in ("labels", "adj", "support", "count"):
            assert np.array_equal(got[key], want[key]), (k, key)
    G.close()


def test_a_hub_in_an_embedding_does_not_cost_its_list_per_batch(fsm):
    """Quota 2 joins the edges of two hubs of degree 20000: some 2e5 pieces, at most 5 ns each."""
    assert _pass_ms(fsm, _two_hubs(4), 4, 100, "count_ns_l2", {"join_quota": 2}) <= 1.0


def _sampled_ms(fsm, g, rate):
    G = fsm.Graph.from_graphgen(g)
    G.set_option("profile", 1)
    try:
        return min(G.mine(3, 2, sample_rate=rate, stats=True)["stats"]["count_ns_l1"] for _ in range(4)) / 1e6
    finally:
        G.close()


@pytest.mark.parametrize("rate", [1e-2, 1e-3, 1e-4])
def test_rare_pieces_cost_no_more_than_frequent_ones(fsm, rate):
    """A path of 200k vertices: 10000, 1000, 100 pieces among as many units take no more than twice the
    time of 100000."""
    n = 200000
    g = gg.from_edges(n, [(i, i + 1) for i in range(n - 1)], (np.arange(n) % 5).astype(np.int32), 5)
    assert _sampled_ms(fsm, g, rate) <= 2 * _sampled_ms(fsm, g, 0.1)


def test_sampled_results_do_not_depend_on_the_chunk(fsm):
    """The chunks of a sparse level (8 pieces) and given ones find the same joins."""
    g = gg.workload("cl3700k", scale=0.002, cap=20)
    out = []
    for opts in ({}, {"launch": 1}, {"chunk": 32}, {"chunk": 4096, "launch": 1}):
        G = fsm.Graph.from_graphgen(g)
        for key, val in {**opts, "candidates": 1}.items():
            G.set_option(key, val)
        out.append([G.mine(k, 20, sample_rate=p) for k, p in ((5, 0.001), (4, 0.01), (3, 0.01))])
        G.close()
    assert all(len(r["support"]) > 0 for r in out[0])
    for got in out[1:]:
        for a, b in zip(got, out[0]):
            for key in ("labels", "adj", "support", "count"):
                assert np.array_equal(a[key], b[key]), key


def test_a_table_that_overflows_is_left_at_once(fsm):
    """Size 3 of 45000 quick patterns from a table of 64 slots, grown to 2^18 in six steps: at most ten times
    the call that has its table from the start."""
    g = gg.workload("cl100k", scale=0.3, cap=300)
    took = []
    for cap in (1 << 20, 64):
        G = fsm.Graph.from_graphgen(g)
        G.set_option("qp_capacity", cap)
        r = [G.mine(3, 150, stats=True)["stats"] for _ in range(3)]
        G.close()
        assert r[0]["qp_grows"] == (0 if cap > 64 else 6)
        took.append(min(x["time_ns"] for x in r) / 1e6)
    assert took[1] <= 10 * took[0], took


def test_small_launches_take_chunks_that_pay(fsm):
    """Size 3 around hubs in batches of 1024 vertices, and per label: no more than 1.25 times what chunks of
    256 pieces take."""
    g = gg.workload("cl100k", scale=0.3, cap=300)
    for opts in ({"batch": 1024}, {"launch": 2}):
        took = []
        for chunk in (256, 0):
            G = fsm.Graph.from_graphgen(g)
            for key, val in {**opts, "chunk": chunk}.items():
                G.set_option(key, val)
            took.append(min(G.mine(3, 150, stats=True)["stats"]["time_ns"] for _ in range(4)) / 1e6)
            G.close()
        assert took[1] <= 1.25 * took[0], (opts, took)
