"""The mining calls a user of this library makes, as measurable cases.

A case is one call (or one short session) through the public Python binding of the C ABI: exact
mining at the sizes and options the repository's workloads, tests and benchmark use, Section 5's
sampling quotas, rate-sampled mining with its features, and the support-prediction network.
Graphs are drawn on the device from the seed alone with the laws of the ``graphgen`` workloads
(Chung-Lu with capped expected degrees, or Erdos-Renyi; uniform or Zipf labels).

Graph laws, as in ``graphgen.WORKLOADS``:
    er1000    n = 1000, mean degree 6, 4 uniform labels
    ci3k      CiteSeer's shape: n = 3312, m = 4732, beta 2.5, 6 uniform labels, cap 99
    cl100k    MiCo's shape: n = 100k, m = 1.1M, beta 2.1, 29 Zipf(1.2) labels
    cl1100k   n = 1.1M, m = 3M, beta 2.0, 16 uniform labels
    cl3700k   n = 3.7M, m = 16.5M, beta 2.3, 37 Zipf(1.0) labels, cap 20 in the benchmark
"""
import ctypes
import math

import numpy as np
import torch

from paper_2101_07690_gb300 import fsm, learn

_LAWS = {
    "er1000": dict(n=1000, m=3000, beta=0.0, labels=4, zipf=0.0, cap=0.0),
    "ci3k": dict(n=3312, m=4732, beta=2.5, labels=6, zipf=0.0, cap=99.0),
    "cl100k": dict(n=100_000, m=1_100_000, beta=2.1, labels=29, zipf=1.2, cap=100.0),
    "cl1100k": dict(n=1_100_000, m=3_000_000, beta=2.0, labels=16, zipf=0.0, cap=16.0),
    "cl3700k": dict(n=3_700_000, m=16_500_000, beta=2.3, labels=37, zipf=1.0, cap=20.0),
}

_POINTERS = {np.dtype(a).char: ctypes.POINTER(b) for a, b in
             ((np.int32, ctypes.c_int32), (np.uint64, ctypes.c_uint64), (np.int64, ctypes.c_int64),
              (np.float32, ctypes.c_float))}


def _mine(name, law, scale, k, t, mode="edge", p=1.0, **options):
    spec = dict(_LAWS[law])
    spec["n"] = max(16, int(round(spec["n"] * scale)))
    spec["m"] = max(16, int(round(spec["m"] * scale)))
    case = {"kind": "mine", "law": law, **spec, "k": k, "t": t, "mode": mode, "p": p,
            "launch": 0, "fused": 0, "join_quota": 0, "candidates": 0, **options}
    if name:
        case["name"] = name
    return case


def listed():
    return [
        # The smallest call: size-3 patterns of a 1000-vertex graph, default options.  Launches,
        # synchronisations and host work, hardly any enumeration.
        _mine("er1000_k3", "er1000", 1.0, 3, 30),
        # A small graph with a low threshold: 370 vertices, size 5, over a hundred thousand
        # patterns; the benchmark's time-to-solution problem.  Key tables, canonicalisation and
        # sorting weigh as much as enumeration.
        _mine("cl370_k5", "cl3700k", 1e-4, 5, 2, fused=1),
        # The paper's 5-FSM on CiteSeer's shape at t = 0.001 n (Table 2), default options.
        _mine("citeseer_k5", "ci3k", 1.0, 5, 3),
        # The paper's 6-FSM on CiteSeer's shape at t = 0.01 n, at half its size: the even path
        # 2 -> 4 -> 6.
        _mine("citeseer_k6", "ci3k", 0.5, 6, 16, launch=1),
        # The paper's 4-FSM on MiCo's shape: hub key vertices with long lists, edges joined with
        # pieces (2 -> 4), one-pass last level.
        _mine("mico_k4", "cl100k", 1.0, 4, 300, launch=1, fused=1),
        # The benchmark's problem (exact size 5 at t/n = 0.0054, one-pass last level, persistent
        # launch) at 1/50 of its size.
        _mine("cl74k_k5", "cl3700k", 0.02, 5, 400, launch=1, fused=1),
        # The benchmark graph at full size up to size 3: the base levels and the size-3 level over
        # 3.7M vertices, where memory traffic counts.
        _mine("cl3700k_k3", "cl3700k", 1.0, 3, 20000, launch=1),
        # Vertex-induced mining of the same law, two-pass last level.
        _mine("cl37k_k5_vertex", "cl3700k", 0.01, 5, 200, mode="vertex", launch=1),
        # Section 5's ST 8 quotas at size 7 (levels 1 -> 3 -> 5 -> 7).
        _mine("cl4k_k7_st8", "cl3700k", 0.001, 7, 20, join_quota=8),
        # Rate-sampled size-5 mining that returns every candidate with its 32 features: what
        # training the support network collects (p = 0.05).
        _mine("cl11k_k5_sampled", "cl3700k", 0.003, 5, 60, p=0.05, candidates=1),
        # A session: a host graph of 1.1M vertices uploaded, validated, prepared, mined once at
        # size 3 and released.
        {"name": "cl1100k_session", "kind": "session", "law": "cl1100k", **_LAWS["cl1100k"], "k": 3, "t": 1000,
         "mode": "edge", "p": 1.0, "launch": 1, "fused": 0, "join_quota": 0, "candidates": 0},
        # The support network: standardisation, two epochs of minibatches of 256 and the
        # prediction of held-out rows, as the training harness runs them.
        {"name": "network_fit", "kind": "network", "rows": 20_000, "heldout": 100_000, "epochs": 2, "batch": 256},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["small", "citeseer", "mico", "cl_k5", "cl_k3", "cl_k4", "vertex", "quota", "sampled",
                       "session", "network"])
    fused, launch = rng.randint(0, 1), rng.randint(0, 1)
    if kind == "small":
        s = _log(rng, 0.2, 4.0)
        c = _mine(None, "er1000", s, rng.choice([2, 3, 4, 5]), 1, launch=launch, fused=fused,
                  mode=rng.choice(["edge", "vertex"]))
        c["t"] = max(2, int(c["n"] * rng.uniform(0.01, 0.05)))
        c["labels"] = rng.randint(2, 9)
    elif kind == "citeseer":
        k = rng.choice([3, 4, 5, 6])
        c = _mine(None, "ci3k", _log(rng, 0.2, 0.45 if k == 6 else 1.5), k, 1, launch=launch, fused=fused)
        c["t"] = max(3, int(c["n"] * (rng.uniform(0.01, 0.02) if k == 6 else rng.choice([0.001, 0.003, 0.005]))))
    elif kind == "mico":
        c = _mine(None, "cl100k", _log(rng, 0.05, 1.0), rng.choice([3, 4]), 1, launch=launch, fused=fused)
        c["t"] = max(4, int(c["n"] * rng.uniform(0.003, 0.01)))
        c["cap"] = float(rng.randint(40, 100))
    elif kind == "cl_k5":
        c = _mine(None, "cl3700k", _log(rng, 1e-4, 0.018), 5, 1, launch=launch, fused=fused)
        c["t"] = max(2, int(c["n"] * rng.uniform(0.0054, 0.02)))
    elif kind == "cl_k3":
        c = _mine(None, rng.choice(["cl3700k", "cl1100k"]), _log(rng, 0.02, 1.0), rng.choice([2, 3]), 1,
                  launch=launch, fused=fused)
        c["t"] = max(2, int(c["n"] * rng.uniform(0.0005, 0.0015 if c["law"] == "cl1100k" else 0.01)))
    elif kind == "cl_k4":
        c = _mine(None, "cl3700k", _log(rng, 0.005, 0.3), 4, 1, launch=launch, fused=fused)
        c["t"] = max(2, int(c["n"] * rng.uniform(0.0054, 0.02)))
    elif kind == "vertex":
        c = _mine(None, "cl3700k", _log(rng, 1e-4, 0.012), 5, 1, mode="vertex", launch=launch, fused=fused)
        c["t"] = max(2, int(c["n"] * rng.uniform(0.0054, 0.02)))
    elif kind == "quota":
        c = _mine(None, "cl3700k", _log(rng, 3e-4, 9e-4), rng.choice([5, 6, 7]), 1, join_quota=rng.randint(2, 8))
        c["t"] = max(3, int(c["n"] * rng.uniform(0.0054, 0.02)))
    elif kind == "sampled":
        c = _mine(None, "cl3700k", _log(rng, 3e-4, 3e-3), 5, 1, p=round(_log(rng, 0.02, 0.05), 4), candidates=1)
        c["t"] = max(2, int(c["n"] * rng.uniform(0.0054, 0.02)))
    elif kind == "session":
        c = _mine(None, "cl1100k", _log(rng, 0.01, 1.0), rng.choice([2, 3]), 1, launch=launch)
        c["kind"] = "session"
        c["t"] = max(2, int(c["n"] * rng.uniform(0.0005, 0.0015)))
    else:
        return {"kind": "network", "rows": int(_log(rng, 500, 19_000)), "heldout": int(_log(rng, 100, 99_000)),
                "epochs": rng.randint(1, 2), "batch": rng.choice([128, 200, 256, 300, 512])}
    if c["law"] != "er1000":
        c["n"] += rng.randint(0, 12)   # odd and ragged vertex counts
        c["m"] -= rng.randint(0, 12)
    return c


def _host_graph(case, seed):
    """row_ptr, col, labels (int32 host arrays) of the case's graph law, drawn on the device."""
    n, m = case["n"], case["m"]
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    if case["beta"] > 0.0:
        w = torch.arange(1, n + 1, dtype=torch.float64, device=dev) ** (-1.0 / (case["beta"] - 1.0))
        for _ in range(100):
            w *= 2.0 * m / w.sum()
            if float(w.max()) <= case["cap"] * (1 + 1e-12):
                break
            w = w.clamp(max=case["cap"])
        cdf = torch.cumsum(w, 0)
        cdf /= cdf[-1].clone()
    have = torch.zeros(0, dtype=torch.int64, device=dev)
    while have.numel() < m:
        r = torch.rand((2, int((m - have.numel()) * 1.15) + 1024), generator=gen, device=dev, dtype=torch.float64)
        e = torch.searchsorted(cdf, r, right=True).clamp(max=n - 1) if case["beta"] > 0.0 else (r * n).long()
        lo, hi = torch.minimum(e[0], e[1]), torch.maximum(e[0], e[1])
        have = torch.unique(torch.cat([have, (lo * n + hi)[lo != hi]]))
    have = have[torch.randperm(have.numel(), generator=gen, device=dev)[:m]]
    ids = torch.randperm(n, generator=gen, device=dev)
    u, v = ids[have // n], ids[have % n]
    key = torch.sort(torch.cat([u * n + v, v * n + u])).values
    row = torch.zeros(n + 1, dtype=torch.int64, device=dev)
    row[1:] = torch.cumsum(torch.bincount(key // n, minlength=n), 0)
    if case["zipf"] > 0.0:
        pw = torch.arange(1, case["labels"] + 1, dtype=torch.float64, device=dev) ** (-case["zipf"])
        lc = torch.cumsum(pw, 0)
        lab = torch.searchsorted(lc / lc[-1], torch.rand(n, generator=gen, device=dev, dtype=torch.float64), right=True)
        lab = lab.clamp(max=case["labels"] - 1)
    else:
        lab = torch.randint(0, case["labels"], (n,), generator=gen, device=dev)
    return tuple(x.to(torch.int32).cpu().numpy() for x in (row, key % n, lab))


def _options(G, case, seed):
    for key in ("launch", "fused", "join_quota", "candidates"):
        if case[key]:
            G.set_option(key, case[key])
    if case["join_quota"] or case["p"] < 1.0:
        G.set_option("seed", seed)


def _network_data(case, seed):
    """Feature rows with the columns' real ranges (log popcounts, log frequencies, mean log
    degrees, pattern scalars) and log supports that depend on them."""
    rng = np.random.default_rng(seed)
    n = case["rows"] + case["heldout"]
    X = np.empty((n, 32), np.float32)
    X[:, :8] = np.sort(rng.uniform(0.0, 9.0, (n, 8)), axis=1)
    X[:, 8:16] = rng.uniform(-4.5, -1.0, (n, 8))
    X[:, 16:24] = rng.uniform(1.5, 3.5, (n, 8))
    X[:, 24] = 5.0
    X[:, 25] = rng.integers(4, 9, n)
    X[:, 26] = np.log(0.05)
    X[:, 27] = X[:, 0] + rng.uniform(0.0, 3.0, n)
    X[:, 28] = np.log(0.0054)
    X[:, 29] = np.log(rng.choice([1.0, 2.0, 4.0, 6.0], n))
    X[:, 30] = X[:, 0] + 3.0
    X[:, 31] = np.log(11100.0)
    y = (0.8 * X[:, 30] + 0.4 * X[:, 8:16].mean(1) + rng.normal(0.0, 0.2, n)).astype(np.float32)
    r = case["rows"]
    return X[:r], y[:r], X[r:]


def prepare(case, seed):
    if case["kind"] == "network":
        X, y, H = _network_data(case, seed)
        return {"case": case, "seed": seed, "X": X, "y": y, "H": H}
    # the caller's result table, filled by every call; rows past the result are zero
    rows = 1 << (16 if case["k"] <= 3 else 17 if case["k"] == 4 else 18 if case["k"] <= 6 else 19)
    table = {"labels": np.zeros((rows, case["k"]), np.int32), "adj": np.zeros(rows, np.uint64),
             "support": np.zeros(rows, np.int64), "count": np.zeros(rows, np.int64), "exact": np.zeros(rows, np.int32)}
    if case["candidates"]:
        table["features"] = np.zeros((rows, 32), np.float32)
    graph = _host_graph(case, seed)
    state = {"case": case, "seed": seed, "graph": graph, "table": table, "filled": 0}
    if case["kind"] == "mine":
        state["G"] = fsm.Graph(*graph, case["labels"], case["mode"])
        _options(state["G"], case, seed)
    return state


def _mine_into_table(state, G):
    """One mining call and its whole result, copied by the C ABI into the caller's table."""
    case, table, lib = state["case"], state["table"], fsm.load()

    def at(name):
        return table[name].ctypes.data_as(_POINTERS[table[name].dtype.char])

    r = fsm.fsm_mine(G.handle, case["k"], case["t"], case["p"])
    try:
        n = fsm.fsm_result_count(r)
        if n > len(table["support"]):
            raise ValueError(f"{n} patterns are more than the result table holds")
        rc = lib.fsm_result_copy(r, at("labels"), at("adj"), at("support"), at("count"))
        rc = rc or lib.fsm_result_exact(r, at("exact"))
        if case["candidates"]:
            rc = rc or lib.fsm_result_features(r, at("features"))
        if rc != fsm.FSM_OK:
            raise fsm.FsmError(rc, fsm.fsm_last_error())
    finally:
        fsm.fsm_free_result(r)
    if n < state["filled"]:
        for column in table.values():
            column[n:state["filled"]] = 0
    state["filled"] = n
    return {"patterns": n, **table}


def run(state):
    case = state["case"]
    if case["kind"] == "network":
        m = learn.fit(state["X"], state["y"], epochs=case["epochs"], batch=case["batch"])
        try:
            return {"params": fsm.fsm_mlp_get_params(m), "predicted": fsm.fsm_mlp_predict(m, state["H"])}
        finally:
            fsm.fsm_mlp_free(m)
    if case["kind"] == "session":
        G = fsm.Graph(*state["graph"], case["labels"], case["mode"])
        try:
            _options(G, case, state["seed"])
            return _mine_into_table(state, G)
        finally:
            G.close()
    return _mine_into_table(state, state["G"])


def work(case):
    """One reading of the inputs, and the position updates (one per vertex of an embedding) of at
    least the expected number of k-vertex paths of a graph of this mean degree, each a size-k
    embedding to be counted and entered in its pattern's image sets."""
    if case["kind"] == "network":
        mac = 32 * 64 + 64 * 64 + 64
        return {"bytes": 132 * case["rows"] + 132 * case["heldout"] + 4 * fsm.MLP_NPARAM,
                "flops": 2 * mac * (3 * case["epochs"] * case["rows"] + case["heldout"])}
    n, m, k = case["n"], case["m"], case["k"]
    deg = 2.0 * m / n
    paths = m * deg ** (k - 2) * case["p"] if not case["join_quota"] else float(m)
    return {"bytes": 4 * (2 * n + 1 + 2 * m), "flops": int(k * paths)}


def _bf16(x):
    """Round-to-nearest-even to bfloat16, held in float64."""
    u = np.ascontiguousarray(x, np.float32).view(np.uint32).astype(np.uint64)
    u = (u + 0x7FFF + ((u >> np.uint64(16)) & np.uint64(1))) & np.uint64(0xFFFF0000)
    return u.astype(np.uint32).view(np.float32).astype(np.float64)


def _splitmix(state):
    state = (state + 0x9E3779B97F4A7C15) & 0xFFFFFFFFFFFFFFFF
    z = state
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & 0xFFFFFFFFFFFFFFFF
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & 0xFFFFFFFFFFFFFFFF
    return state, z ^ (z >> 31)


def exact(case, seed):
    """The network's training in 64 bits: He-uniform weights and shuffles from splitmix64 streams,
    float64 forward, backward and Adam with float32 master weights' bfloat16 copies in every
    product.  Mining returns whole numbers only (and, sampled, features whose reference is an
    enumeration of every sampled embedding), so it has no entry here."""
    if case["kind"] != "network":
        return None
    X, y, H = _network_data(case, seed)
    X64, y64, H64 = X.astype(np.float64), y.astype(np.float64), H.astype(np.float64)
    st, vals = 0, []
    for _ in range(32 * 64 + 64 * 64 + 64):
        st, z = _splitmix(st)
        vals.append(float(np.float32((z >> 11) / 9007199254740992.0)) * 2.0 - 1.0)
    vals = np.array(vals)
    a1, a2 = math.sqrt(6.0 / 32), math.sqrt(6.0 / 64)
    w = np.zeros(fsm.MLP_NPARAM)
    o = np.cumsum([0, 32 * 64, 64, 64 * 64, 64, 64, 1])
    w[o[0]:o[1]] = np.float32(a1) * vals[:2048]
    w[o[2]:o[3]] = np.float32(a2) * vals[2048:2048 + 4096]
    w[o[4]:o[5]] = np.float32(a2) * vals[2048 + 4096:]
    w = w.astype(np.float32).astype(np.float64)
    mu = X64.mean(0)
    sd = np.maximum(np.sqrt(((X64 - mu) ** 2).mean(0)), 1e-3)

    def views(p):
        q = _bf16(p)
        return (q[o[0]:o[1]].reshape(32, 64), p[o[1]:o[2]], q[o[2]:o[3]].reshape(64, 64), p[o[3]:o[4]],
                q[o[4]:o[5]], p[o[5]])

    def forward(p, x):
        W1, b1, W2, b2, w3, b3 = views(p)
        z1 = x @ W1 + b1
        z2 = np.maximum(z1, 0.0) @ W2 + b2
        return z1, z2, np.maximum(z2, 0.0) @ w3 + b3

    Xn, Hn = (X64 - mu) / sd, (H64 - mu) / sd
    n, lr, b1c, b2c, eps = len(y), 3e-3, 0.9, 0.999, 1e-8
    m1, m2, step, st = np.zeros_like(w), np.zeros_like(w), 0, 0
    order = list(range(n))
    for _ in range(case["epochs"]):
        for i in range(n - 1, 0, -1):
            st, z = _splitmix(st)
            j = z % (i + 1)
            order[i], order[j] = order[j], order[i]
        idx = np.array(order)
        for b0 in range(0, n, case["batch"]):
            r = idx[b0:b0 + case["batch"]]
            x = Xn[r]
            W1, _, W2, _, w3, _ = views(w)
            z1, z2, out = forward(w, x)
            dy = 2.0 * (out - y64[r]) / len(r)
            dz2 = np.where(z2 > 0, dy[:, None] * w3, 0.0)
            dz1 = np.where(z1 > 0, dz2 @ W2.T, 0.0)
            g = np.concatenate([(x.T @ dz1).ravel(), dz1.sum(0), (np.maximum(z1, 0).T @ dz2).ravel(), dz2.sum(0),
                                np.maximum(z2, 0).T @ dy, [dy.sum()]])
            step += 1
            m1 = b1c * m1 + (1 - b1c) * g
            m2 = b2c * m2 + (1 - b2c) * g * g
            w = w - lr * (m1 / (1 - b1c ** step)) / (np.sqrt(m2 / (1 - b2c ** step)) + eps)
    return {"params": w, "predicted": forward(w, Hn)[2]}
