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
