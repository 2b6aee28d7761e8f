"""Calls that meet a limit on the way: every outcome is the result or the documented error."""
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


@pytest.mark.parametrize("opts", [{}, {"launch": 1}, {"launch": 2}], ids=["batches", "persistent", "per pattern"])
@pytest.mark.parametrize("k,scale,rate,hi", [(7, 0.003, 1.0, 40), (5, 0.02, 0.5, 30)], ids=["exact", "sampled"])
def test_a_time_limit_that_runs_out_in_any_pass_is_reported_as_one(fsm, k, scale, rate, hi, opts):
    """Limits from 1 ms on, so that each pass of each level is the one cut short: size 5 is counted, its
    domains filled and its embeddings stored on the way to size 7; a sampled level ends with its domains."""
    g = gg.workload("cl3700k", scale=scale, cap=20)
    G = fsm.Graph.from_graphgen(g)
    for key, val in {**opts, "candidates": 1}.items():
        G.set_option(key, val)
    stopped = 0
    try:
        for ms in range(1, hi):
            G.set_option("time_limit_ms", ms)
            try:
                G.mine(k, max(2, g.n // 185), sample_rate=rate)
            except fsm.FsmError as e:
                assert e.code == fsm.FSM_ETIMEOUT, (ms, e)
                stopped += 1
    finally:
        G.close()
    assert stopped > 0


def _refused_one_by_one(fsm, g, k, t, opts, most=60):
    """Results (or None for FSM_ENOMEM) of a mine whose n-th request for device memory is refused."""
    G = fsm.Graph.from_graphgen(g)
    for key, val in opts.items():
        G.set_option(key, val)
    try:
        G.mine(k, t)   # the handle's tables are made
        whole = G.mine(k, t, stats=True)
        out = []
        for n in range(1, most):
            G.set_option("refuse_alloc", n)
            try:
                out.append(G.mine(k, t, stats=True))
            except fsm.FsmError as e:
                assert e.code == fsm.FSM_ENOMEM, (n, e)
                out.append(None)
    finally:
        G.close()
    for got in out:
        if got:
            for key in ("labels", "adj", "support", "count"):
                assert np.array_equal(got[key], whole[key]), key
    return whole, out


@pytest.mark.parametrize("opts", [{}, {"launch": 1}, {"launch": 2}, {"profile": 1}],
                         ids=["batches", "persistent", "per pattern", "profiled"])
def test_the_one_pass_level_does_without_its_pool_and_its_buffer(fsm, opts):
    """Refused one or the other, the level is finished in two passes."""
    g = gg.workload("cl3700k", scale=0.001, cap=20)
    whole, out = _refused_one_by_one(fsm, g, 5, 20, {**opts, "fused": 1})
    assert whole["stats"]["fused_fallbacks"] == 0 and len(whole["support"]) > 0
    assert sum(1 for r in out if r and r["stats"]["fused_fallbacks"] == 1) == 2


def _device_memory_taken(body):
    """Bytes of device memory a fresh process holds after `body`, beyond those it held after loading."""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    code = ("import torch, numpy as np, graphgen as gg\nfrom paper_2101_07690_gb300 import fsm\n"
            "def free():\n    torch.cuda.synchronize()\n    return torch.cuda.mem_get_info()[0]\n" + body)
    r = subprocess.run([sys.executable, "-c", code], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    return int(r.stdout.split()[-1])


@pytest.mark.parametrize("launch,t,mib", [(0, 10 ** 6, 8), (1, 10 ** 6, 8), (2, 10 ** 6, 8), (0, 30, 64), (2, 30, 64)])
def test_a_small_one_pass_level_takes_little_memory(fsm, launch, t, mib):
    """Nothing frequent, hence no stored embeddings (two-pass mining of it first, so that only what the
    one-pass form adds is seen), and a thousand vertices: no buffer for joins that cannot be put aside."""
    body = ("G = fsm.Graph.from_graphgen(gg.workload('er1000'))\n"
            f"G.set_option('launch', {launch})\nG.mine(5, {t})\nf = free()\n"
            f"G.set_option('fused', 1)\nG.mine(5, {t})\nprint(f - free())\n")
    assert _device_memory_taken(body) <= mib << 20


@pytest.mark.parametrize("launch", [0, 1])
def test_a_level_gives_its_prefix_back(fsm, launch):
    """Size 3, which keeps no joins: the prefix of the level's units is the one allocation to give back, and
    every pass left makes its own."""
    whole, out = _refused_one_by_one(fsm, gg.workload("cl3700k", scale=0.001, cap=20), 3, 5, {"launch": launch})
    assert len(whole["support"]) > 0
    assert sum(r is not None and r["stats"]["kernel_launches"] > whole["stats"]["kernel_launches"] for r in out) >= 5


@pytest.mark.parametrize("launch", [0, 1])
def test_a_level_gives_its_kept_joins_back(fsm, launch):
    whole, out = _refused_one_by_one(fsm, gg.workload("cl3700k", scale=0.001, cap=20), 5, 20, {"launch": launch})
    assert whole["stats"]["kept_levels"] == 1
    assert sum(r is not None and r["stats"]["kept_levels"] == 0 for r in out) >= 2


def test_the_one_pass_level_falls_back_when_joins_put_aside_run_out(fsm):
    """A level larger than its sample (2^26 pieces) meets keys the sample missed; with room for 16 of their
    joins it is redone in two passes, and has put none aside."""
    g = gg.workload("cl3700k", scale=0.002, cap=20)
    out = []
    for defer in (0, 16):
        G = fsm.Graph.from_graphgen(g)
        G.set_option("fused", 1)
        G.set_option("fused_defer", defer)
        out.append(G.mine(5, g.n // 400, stats=True))
        G.close()
    assert out[0]["stats"]["fused_deferred"] > 16 and out[0]["stats"]["fused_fallbacks"] == 0
    assert out[1]["stats"]["fused_deferred"] == 0 and out[1]["stats"]["fused_fallbacks"] == 1
    for key in ("labels", "adj", "support", "count"):
        assert np.array_equal(out[0][key], out[1][key]), key


def test_a_pool_too_small_puts_nothing_aside(fsm):
    """Pools with room for the sample's patterns but not for those met later, too: joins were put aside, then
    the level was redone in two passes, and the statistics are those of the passes that count.  (How many
    words a call uses varies by what lanes that resolve one pattern together reserve twice.)"""
    g = gg.workload("cl3700k", scale=0.002, cap=20)
    G = fsm.Graph.from_graphgen(g)
    G.set_option("fused", 1)
    whole = G.mine(5, g.n // 400, stats=True)
    fell_back = 0
    for percent in (50, 90, 94, 96, 97, 98, 99):
        G.set_option("fused_pool", whole["stats"]["fused_pool_words"] * percent // 100)
        got = G.mine(5, g.n // 400, stats=True)
        if got["stats"]["fused_fallbacks"]:
            fell_back += 1
            assert got["stats"]["fused_deferred"] == 0, percent
        for key in ("labels", "adj", "support", "count"):
            assert np.array_equal(got[key], whole[key]), key
    G.close()
    assert fell_back > 0
