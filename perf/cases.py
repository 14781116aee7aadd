"""What a user of this framework has it do, as cases that can be timed.

A case names one kind of call (`kind`), a graph family with its size, a
cascade model and the query.  `prepare` draws the graph on the GPU from the
seed and loads it; `run` makes one pass through the public entry points;
`exact` recomputes small selections with dense torch matrices.

Graph families: "er" (directed, uniform endpoints), "cl" (undirected
Chung-Lu power law, exponent 2.5, both arcs stored) and "rmat" (directed
R-MAT, 0.57/0.19/0.19/0.05, n a power of two).
"""

import math
import time

import numpy as np
import torch

from paper_1212_4779_gb300 import inputs, sg


def listed():
    return [
        # The smallest query in use: 2,000 nodes, ten rounds; latency of
        # dependent launches and short walks.
        dict(name="er2k_uic_select", kind="select", family="er", n=2000, m=10000, model="uic", p=0.1, R=100, k=10),
        # A NetHEPT-shaped collaboration network under both cascades of the
        # paper, 100 snapshots (a partial last word), 50 seeds.
        dict(name="cl15k_uic_select", kind="select", family="cl", n=15000, m=116000, model="uic", p=0.01, R=100, k=50),
        dict(name="cl15k_wic_select", kind="select", family="cl", n=15000, m=116000, model="wic", p=0.0, R=100, k=50),
        # The throughput query: a million-node social network, 256 snapshots.
        dict(name="rmat20_wic_select", kind="select", family="rmat", n=1 << 20, m=8388608, model="wic", p=0.0, R=256,
             k=50),
        # A uniform cascade with a giant component at a ragged size; the
        # caller keeps the gain vector and the coverage as well as the seeds.
        dict(name="cl97k_uic_state", kind="state", family="cl", n=97001, m=1164012, model="uic", p=0.05, R=200, k=33),
        # Ranking every node by its spread, no selection: initial gains only.
        dict(name="rmat18_wic_gains", kind="gains", family="rmat", n=1 << 18, m=2097152, model="wic", p=0.0, R=128,
             k=1),
        # The linear threshold model.
        dict(name="cl60k_lt_select", kind="select", family="cl", n=60000, m=480000, model="lt", p=0.0, R=128, k=50),
        # One coin per undirected edge on a NetPHY-shaped network.
        dict(name="cl37k_undirected_select", kind="select", family="cl", n=37154, m=463168, model="uic_undirected",
             p=0.05, R=100, k=50),
        # Judging a chosen seed set on 20,000 fresh snapshots.
        dict(name="rmat20_wic_spread", kind="spread", family="rmat", n=1 << 20, m=8388608, model="wic", p=0.0, R=20000,
             k=50),
        # The lazy-forward variant on the collaboration network.
        dict(name="cl15k_wic_celf", kind="celf", family="cl", n=15000, m=116000, model="wic", p=0.0, R=100, k=50),
        # Many queries of uneven size at once: a captured batch, replayed.
        dict(name="batch16_graph", kind="batch", queries=16, first=0, n_max=200000, k_max=100),
        # Requests that arrive together at a server over resident graphs.
        dict(name="served24", kind="served", queries=24, first=0, n_max=60000, k_max=100),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["select"] * 6 + ["state", "gains", "spread", "celf", "batch", "served"])
    if kind in ("batch", "served"):
        return dict(kind=kind, queries=rng.randrange(5, 17 if kind == "batch" else 25), first=rng.randrange(1, 240),
                    n_max=_log_int(rng, 5000, 200000 if kind == "batch" else 60000), k_max=rng.randrange(20, 101))
    family = rng.choice(["er", "cl", "cl", "rmat"])
    model = rng.choice(["uic", "wic", "wic"])
    if kind in ("select", "spread") and rng.random() < 0.4:
        model = rng.choice(["lt", "uic_undirected"])
        if model == "uic_undirected":
            family = "cl"
    if family == "rmat":
        n = 1 << rng.randrange(12, 20 if model != "lt" else 18)
        m = int(n * rng.uniform(4.0, 8.0))
    elif family == "er":
        n = _log_int(rng, 1000, 100000)
        m = int(n * rng.uniform(2.0, 8.0))
    else:
        n = _log_int(rng, 1000, 200000)
        m = 2 * int(n * rng.uniform(2.0, 10.0))
    p = 0.0
    if model.startswith("uic"):
        p = rng.choice([0.01, 0.02, 0.05] if family != "er" else [0.01, 0.05, 0.1])
    if kind == "celf":
        n, m = min(n, 16384), m * min(n, 16384) // n // 2 * 2
    R = rng.choice([64, 100, 128, 200, 256, rng.randrange(33, 257)])
    if kind == "spread":
        R = _log_int(rng, 1000, 20000)
    if model == "uic_undirected":
        R = min(R, 2000)
    return dict(kind=kind, family=family, n=n, m=m, model=model, p=p, R=R,
                k=1 if kind == "gains" else rng.randrange(10, 51))


# ------------------------------------------------------------------- graphs


def _distinct(draw_keys, count, gen):
    """`count` distinct sorted keys; draw_keys(b) gives about b candidates."""
    keys = torch.empty(0, dtype=torch.int64, device="cuda")
    while keys.numel() < count:
        b = max(1024, int(1.15 * (count - keys.numel())) + 1024)
        keys = torch.unique(torch.cat([keys, draw_keys(b)]))
    if keys.numel() > count:
        keep = torch.randperm(keys.numel(), generator=gen, device="cuda")[:count]
        keys = keys[keep].sort().values
    return keys


def _arcs(family, n, m, gen):
    """(source << 32 | destination) of m distinct arcs, sorted."""

    def rand(b):
        return torch.rand(b, generator=gen, device="cuda", dtype=torch.float64)

    if family == "er":
        def keys(b):
            u = torch.randint(0, n, (b,), generator=gen, device="cuda")
            v = torch.randint(0, n, (b,), generator=gen, device="cuda")
            return ((u << 32) | v)[u != v]

        return _distinct(keys, m, gen)
    if family == "rmat":
        scale = n.bit_length() - 1

        def keys(b):
            u = torch.zeros(b, dtype=torch.int64, device="cuda")
            v = torch.zeros(b, dtype=torch.int64, device="cuda")
            for _ in range(scale):
                x = rand(b)
                u = (u << 1) | (x >= 0.76).long()
                v = (v << 1) | (((x >= 0.57) & (x < 0.76)) | (x >= 0.95)).long()
            return ((u << 32) | v)[u != v]

        return _distinct(keys, m, gen)
    w = torch.arange(1, n + 1, dtype=torch.float64, device="cuda") ** (-1.0 / 1.5)
    cdf = torch.cumsum(w, 0)
    cdf /= cdf[-1].clone()

    def keys(b):
        u = torch.searchsorted(cdf, rand(b), right=True).clamp_(max=n - 1)
        v = torch.searchsorted(cdf, rand(b), right=True).clamp_(max=n - 1)
        return ((torch.minimum(u, v) << 32) | torch.maximum(u, v))[u != v]

    e = _distinct(keys, m // 2, gen)
    return torch.cat([e, (e << 32) | (e >> 32)]).sort().values


def _csr(n, keys):
    rp = torch.searchsorted(keys, torch.arange(n + 1, dtype=torch.int64, device="cuda") << 32)
    return rp, (keys & 0xFFFFFFFF).int()


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _graph(family, n, m, seed):
    return sg.Graph.from_csr(n, *_csr(n, _arcs(family, n, m, _gen(seed))))


def _top_degrees(g, k):
    """The k nodes of largest out-degree, lowest ids first on ties."""
    deg = np.diff(g.csr()[0])
    return np.ascontiguousarray(np.argsort(-deg, kind="stable")[:k].astype(np.int32))


def _hash_seed(seed):
    return (int(seed) * 0x9E3779B97F4A7C15 + 11) & (2**64 - 1)


# -------------------------------------------------------------------- cases


class _Many:
    """Graphs, workspaces, outputs and the batch or server over them."""

    def __init__(self, case, seed):
        self.batch = self.server = None
        self.graphs, self.spaces, self.items = [], [], []
        # recipes of the batched workload, capped in size; graphs and hash
        # seeds come from `seed`
        recipes = inputs.batch_queries(case["queries"], case["first"])
        if case["kind"] == "served":
            recipes = recipes[:8]
        for i, q in enumerate(recipes):
            n = min(q["n"], case["n_max"])
            m = 2 * int(round(n * q["mean_deg"] / 2))
            self.graphs.append(_graph("cl", n, m, int(seed) * 131 + i))
        for i, q in enumerate(recipes if case["kind"] == "batch" else range(case["queries"])):
            if case["kind"] == "served":
                r = np.random.Generator(np.random.PCG64([case["first"], i]))
                q = dict(recipes[i % len(recipes)], R=int(r.choice([100, 200])), k=int(r.integers(10, 101)))
            g = self.graphs[i % len(self.graphs)]
            k = min(q["k"], case["k_max"], g.n)
            hash_seed = _hash_seed(int(seed) * 131 + i)
            if case["kind"] == "batch":
                space = sg.sg_workspace_create(g.handle, q["R"], k)
                self.spaces.append(space)
                out = [torch.zeros(k, dtype=t, device="cuda") for t in (torch.int32, torch.int64)]
                self.items.append((g.handle, space, q["R"], k, q["model"], q["p"], hash_seed, *out))
            else:
                self.items.append((g.handle, q["R"], k, q["model"], q["p"], hash_seed))
        if case["kind"] == "batch":
            stream = torch.cuda.Stream()  # capture needs a stream of its own
            stream.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(stream):
                self.batch = sg.sg_batch_capture(self.items, concurrency=16)
            torch.cuda.current_stream().wait_stream(stream)
            self.seeds = [it[7] for it in self.items]
            self.gains = [it[8] for it in self.items]
        else:
            self.server = sg.sg_server_create(max_running=8, k_cap=128)

    def run(self):
        if self.batch is not None:
            sg.sg_batch_launch(self.batch)
            return {"seeds": self.seeds, "gains": self.gains}
        ids = [sg.sg_server_submit(self.server, *it) for it in self.items]
        done = {}
        while len(done) < len(ids):
            for i, rid in enumerate(ids):
                if i not in done:
                    ready, seeds, gains, _ = sg.sg_server_poll(self.server, rid, self.items[i][2])
                    if ready:
                        done[i] = (seeds, gains)
            time.sleep(0.0002)  # the poll interval of serve.run_served
        return {"seeds": [done[i][0] for i in range(len(ids))], "gains": [done[i][1] for i in range(len(ids))]}

    def __del__(self):
        try:
            torch.cuda.synchronize()
            if self.batch is not None:
                sg.sg_batch_free(self.batch)
            if self.server is not None:
                sg.sg_server_destroy(self.server)
            for w in self.spaces:
                sg.sg_workspace_free(w)
            for g in self.graphs:
                g.close()
        except Exception:  # noqa: BLE001 - the interpreter may be ending
            pass


def prepare(case, seed):
    if case["kind"] in ("batch", "served"):
        return _Many(case, seed)
    state = dict(case, g=_graph(case["family"], case["n"], case["m"], seed), hash_seed=_hash_seed(seed))
    if case["kind"] == "spread":
        state["S"] = _top_degrees(state["g"], case["k"])  # the degree heuristic's seed set
    return state


def run(state):
    if isinstance(state, _Many):
        return state.run()
    g, kind = state["g"], state["kind"]
    query = (state["R"], state["k"], state["model"], state["p"], state["hash_seed"])
    if kind == "select":
        res = g.select(*query)
        return {"seeds": res.seeds, "gains": res.gains}
    if kind == "state":
        res, s, cov = g.select_state(*query)
        return {"seeds": res.seeds, "gains": res.gains, "s": s, "cov": cov.view(np.int64)}
    if kind == "gains":
        s, edges = g.init_gains(state["R"], *query[2:])
        return {"s": s, "edges": edges}
    if kind == "spread":
        total, edges = g.spread(state["R"], *query[2:], state["S"])
        return {"total": total, "edges": edges}
    res, evaluations = g.select_celf(*query)
    return {"seeds": res.seeds, "gains": res.gains, "evaluations": evaluations}


def work(case):
    """Bytes: the graph read once and the outputs written once.  Operations:
    one coin (about 12 integer operations) per arc and snapshot, since the
    gains of all nodes depend on every arc; a spread needs the coins of its
    seeds' arcs at least."""
    if case["kind"] in ("batch", "served"):
        n, m, R = case["n_max"] * 0.19, case["n_max"] * 0.19 * 12, 150  # the recipes' means
        each = {"bytes": 4 * n + 4 * m + 12 * case["k_max"] / 2, "flops": 12 * m * R}
        graphs = case["queries"] if case["kind"] == "batch" else min(8, case["queries"])
        return {"bytes": graphs * each["bytes"], "flops": case["queries"] * each["flops"]}
    n, m, R, k = case["n"], case["m"], case["R"], case["k"]
    words = (R + 63) // 64
    out = {"state": 8 * n + 8 * n * words, "gains": 8 * n, "spread": 16}.get(case["kind"], 0) + 12 * k
    if case["kind"] == "spread":
        return {"bytes": 4 * n + 4 * m + out, "flops": 12 * R * k * m / n}
    return {"bytes": 4 * n + 4 * m + out, "flops": 12 * m * R}


# -------------------------------------------------------------------- exact


def _mul64(a, b):
    """a * b mod 2^64 on uint64 numpy arrays."""
    with np.errstate(over="ignore"):
        return a * np.uint64(b)


def _coin(base, r):
    """High 32 bits of splitmix64(base ^ (r << 40))."""
    with np.errstate(over="ignore"):
        z = (base ^ np.uint64(r << 40)) + np.uint64(0x9E3779B97F4A7C15)
        z = _mul64(z ^ (z >> np.uint64(30)), 0xBF58476D1CE4E5B9)
        z = _mul64(z ^ (z >> np.uint64(27)), 0x94D049BB133111EB)
        return (z ^ (z >> np.uint64(31))) >> np.uint64(32)


def exact(case, seed):
    """Greedy selection from dense reach matrices, for graphs of up to 2,500
    nodes under the uniform and weighted cascades."""
    if case["kind"] != "select" or case["n"] > 2500 or case["model"] not in ("uic", "wic"):
        return None
    n, R, k = case["n"], case["R"], case["k"]
    keys = _arcs(case["family"], n, case["m"], _gen(seed))
    src, dst = keys >> 32, keys & 0xFFFFFFFF
    e = np.arange(keys.numel(), dtype=np.uint64)
    if case["model"] == "uic":
        thr = np.full(e.size, int(math.floor(case["p"] * 2.0**32)), dtype=np.uint64)
    else:
        thr = np.uint64(2**32) // torch.bincount(dst, minlength=n)[dst].cpu().numpy().astype(np.uint64)
    reach = torch.zeros((R, n, n), dtype=torch.bool, device="cuda")
    for r in range(R):
        live = torch.from_numpy(_coin(np.uint64(_hash_seed(seed)) ^ e, r) < thr).cuda()
        a = torch.eye(n, device="cuda")
        a[src[live], dst[live]] = 1.0
        while True:
            b = ((a @ a) > 0).float()
            if torch.equal(a, b):
                break
            a = b
        reach[r] = a.bool()
    left = torch.ones((R, n), device="cuda")
    seeds, gains = [], []
    for _ in range(k):
        s = torch.zeros(n, dtype=torch.float64, device="cuda")
        for r in range(R):
            s += (reach[r].float() @ left[r]).double()
        if seeds:
            s[seeds] = -1.0
        v = int((s == s.max()).nonzero()[0])
        seeds.append(v)
        gains.append(int(s[v]))
        left[reach[:, v]] = 0.0
    return {"seeds": np.array(seeds, dtype=np.int32), "gains": np.array(gains, dtype=np.int64)}
