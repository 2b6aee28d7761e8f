"""The join kernel (stored sizes 1..5) at the sizes where it can go wrong, against the CPU oracle:
label bits up to 63, more distinct keys than a block's key table holds, chunks that cut a unit's
rows, batches around 16 units, hubs beyond one warp's Bloom filters, and every stored size."""
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


def _many_labels():
    """150 vertices, mean degree 5, 64 labels: label 63 in the masks' top bit, thousands of keys."""
    return gg.erdos_renyi(150, 5.0, seed=11, num_labels=64)


def _two_hubs():
    """Two hubs of degree about 300 sharing half their neighbours, on a sparse rest."""
    rng = np.random.default_rng(7)
    e = [(0, v) for v in range(2, 302)] + [(1, v) for v in range(152, 452)] + [(0, 1)]
    e += [tuple(int(x) for x in rng.choice(np.arange(2, 452), 2, replace=False)) for _ in range(60)]
    perm = rng.permutation(452)
    return gg.from_edges(452, [(perm[a], perm[b]) for a, b in e], rng.integers(0, 5, 452).astype(np.int32), 5)


def _dense():
    return gg.random_small(17, 0.5, 2, 4)


CASES = [("many labels", _many_labels, (3, 4, 5), 1), ("two hubs", _two_hubs, (3, 4), 3),
         ("dense", _dense, (3, 4, 5, 6), 2), ("sparse", lambda: gg.erdos_renyi(34, 2.4, seed=3, num_labels=2), (6, 7), 1)]


@pytest.mark.parametrize("mode", ["edge", "vertex"])
@pytest.mark.parametrize("case", CASES, ids=[c[0] for c in CASES])
def test_join_kernel_matches_oracle(fsm, case, mode):
    _, make, ks, t = case
    g = make()
    for k in ks:
        exp = oracle.mine(g, k, t, mode)
        for opts in ({}, {"chunk": 32, "fused": 1}, {"chunk": 65536, "launch": 1}, {"launch": 1, "fused": 1},
                     {"debug": 1, "launch": 2}):
            G = fsm.Graph.from_graphgen(g, mode)
            for key, val in opts.items():
                G.set_option(key, val)
            got = G.mine(k, t)
            G.close()
            for key in ("labels", "adj", "support", "count"):
                assert np.array_equal(got[key], exp[key]), (k, opts, key)


@pytest.mark.parametrize("opts", [{}, {"launch": 1}, {"join_quota": 3}], ids=["default", "persistent", "quota"])
@pytest.mark.parametrize("n,deg,k", [(700, 6.0, 4), (300, 5.0, 5), (200, 4.0, 7), (150, 4.0, 6), (40, 20.0, 4)])
@pytest.mark.parametrize("mode", ["edge", "vertex"])
def test_domain_bits_from_kept_joins(fsm, mode, n, deg, k, opts):
    """Levels of enough pieces keep their accepted joins in the count pass and set the domain bits from
    them.  Launches per pattern never do: the same result.  The dense graphs accept more joins a piece
    than there is room for, so their levels enumerate again."""
    g = gg.erdos_renyi(n, deg, seed=5, num_labels=3)
    out = []
    for o in (opts, {**opts, "launch": 2}):
        G = fsm.Graph.from_graphgen(g, mode)
        for key, val in o.items():
            G.set_option(key, val)
        out.append(G.mine(k, max(2, n // 40), stats=True))
        G.close()
    assert out[1]["stats"]["kept_levels"] == 0
    if n >= 300 and not opts.get("join_quota"):
        assert out[0]["stats"]["kept_levels"] > 0
    assert len(out[0]["support"]) > 0
    for key in ("labels", "adj", "support", "count"):
        assert np.array_equal(out[0][key], out[1][key]), key


@pytest.mark.parametrize("mode", ["edge", "vertex"])
@pytest.mark.parametrize("k,scale", [(5, 0.002), (4, 0.1), (3, 0.3)])
def test_one_pass_level_with_keys_its_sample_missed(fsm, k, scale, mode):
    """Levels large enough that the one-pass form samples their pieces first (more than 2^26): joins
    whose keys the sample missed are put aside and entered after the level.  Same result as the count
    and domain passes, also when the bitmap pool runs out on the way."""
    g = gg.workload("cl3700k", scale=scale, cap=20)
    t = max(2, g.n // 400)
    out = []
    for opts in ({"fused": 0}, {"fused": 1}, {"fused": 1, "launch": 1}, {"fused": 1, "fused_pool": 1 << 20}):
        G = fsm.Graph.from_graphgen(g, mode)
        for key, val in opts.items():
            G.set_option(key, val)
        out.append(G.mine(k, t, stats=True))
        G.close()
    assert out[0]["stats"]["pieces"] >> 26 and len(out[0]["support"]) > 0
    assert out[1]["stats"]["fused_fallbacks"] == 0 and out[1]["stats"]["fused_deferred"] > 0
    for got in out[1:]:
        for key in ("labels", "adj", "support", "count"):
            assert np.array_equal(got[key], out[0][key]), key
