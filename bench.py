#!/usr/bin/env python3
"""Benchmark: StaticGreedyDU k-seed selection on one GB300.

One step = one full pass of the hot path on one query: initial gains over
R hash-defined snapshots, then k rounds of argmax + forward DU + reverse
DU (Algorithm 2 of Cheng et al., CIKM'13), with the graph resident in HBM.

Workload (default): directed R-MAT scale 20 (1,048,576 nodes, 8,388,608
arcs, (0.57, 0.19, 0.19, 0.05)), weighted cascade, R = 256 (4 x 64-snapshot
words), k = 50, hash seed 11; seeded synthetic graph.

Metric: snapshot-edges per second (GTEPS), with snapshot-edges the
implementation-independent count init + forward DU + reverse DU reported
by the library; ms_per_step is the k-seed select time.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

With --impl reference the CPU oracle (the plain StaticGreedyDU of oracle/)
is timed on the host cores on a bounded sample of the same workload;
--workload oracle_select times the oracle's whole selection at full R
(CPU only, about 40 s on 16 cores for the default query).
Under torchrun each rank runs an independent replica (the path has no
cross-GPU exchange); value is the sum over ranks.
"""

from __future__ import annotations

import argparse
import json
import os
import shutil
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

from paper_1212_4779_gb300 import inputs  # noqa: E402

METRIC = "GTEPS (snapshot-edges/s) of StaticGreedyDU k-seed selection"
UNIT = "GTEPS"

# Bytes that the cover kernel of a round cannot do without.  Per newly covered
# (node, snapshot): its node-list entry (8), its coverage word read and written
# (16) and its gain read and written (16).  Per range that loses gains: the
# in-arc that led to it (8), its way up (8), its join's record for the round (16),
# its range (8) and its task (4).
BYTES_PER_COVERED = 40
BYTES_PER_RANGE = 44
# ... and a closure walk: 16 bytes per visited join, 4 per scanned join arc
BYTES_PER_JOIN = 16
BYTES_PER_JOIN_ARC = 4


def _peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as f:
            d = json.load(f)
        return d, "measured"
    return {"hbm_gbs": 6800.0, "sm_max_mhz": 2070.0}, "fallback"


class ClockSampler:
    """nvidia-smi clock/throttle sampling during the timed region."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index):
        self.index = index
        self.proc = None
        self.lines = []
        self.thread = None

    def start(self):
        exe = shutil.which("nvidia-smi")
        if not exe:
            return
        self.proc = subprocess.Popen([exe, f"--id={self.index}", f"--query-gpu={self.FIELDS}",
                                      "--format=csv,noheader,nounits", "-lms", "100"],
                                     stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        self.thread = threading.Thread(target=self._read, daemon=True)
        self.thread.start()

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def stop(self):
        if not self.proc:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        self.thread.join(timeout=2)
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            parts = [x.strip() for x in ln.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                smax.append(float(parts[2]))
            except ValueError:
                continue
            for nm, v in zip(names, parts[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(nm)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples"]}
        return {"sm_mhz": float(np.median(sm)), "sm_max_mhz": float(max(smax)), "reasons": sorted(reasons),
                "samples": len(sm)}


def _recorded_traffic(kernel_src="paper_1212_4779_gb300/csrc/sg_snap_kernels.cuh",
                      summary="profiles/snap_cover_rmat20_traffic.md"):
    """DRAM bytes per launch (mean over the rounds) of the cover kernel from
    the committed ncu summary, or None when the kernel source has changed
    since that capture (its sha256 prefix is recorded in the summary)."""
    import hashlib

    here = os.path.dirname(os.path.abspath(__file__))
    try:
        text = open(os.path.join(here, summary)).read()
        digest = hashlib.sha256(open(os.path.join(here, kernel_src), "rb").read()).hexdigest()[:16]
    except OSError:
        return None
    rec = dict(line.split(": ", 1) for line in text.splitlines() if line.startswith(("kernel_source", "traffic_bytes")))
    if not rec.get("kernel_source", "").endswith(digest):
        return None
    try:
        return int(rec["traffic_bytes_per_launch"])
    except (KeyError, ValueError):
        return None


def _dist():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


def _barrier_and_max(x, ws):
    """Maximum of `x` over the ranks after a barrier (a CUDA tensor under
    NCCL, a host tensor under gloo)."""
    if ws <= 1:
        return x
    import torch
    import torch.distributed as dist

    dev = "cuda" if dist.get_backend() == "nccl" else "cpu"
    t = torch.tensor([x], dtype=torch.float64, device=dev)
    dist.barrier()
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def replica_throughput(local_ms_total, units_per_step, steps, ws):
    """Whole-job throughput of `ws` independent replicas, each running
    `steps` steps of `units_per_step` units: the units of all ranks divided
    by the slowest rank's time.  Returns (ms per step, units per second)."""
    total_ms = _barrier_and_max(float(local_ms_total), ws)
    ms_step = total_ms / steps
    return ms_step, units_per_step * ws / (ms_step / 1e3)


def _oracle_du(g, R, wl, cores):
    """One oracle StaticGreedyDU selection (Algorithm 2: initial gains, then k
    rounds of argmax, forward BFS and reverse BFS per snapshot) over
    snapshots 0..R-1.  Returns (seconds, snapshot-edges: init + forward +
    reverse counters)."""
    import oracle

    t0 = time.perf_counter()
    out = g.select(R, wl.k, wl.seed, mode=oracle.DU, nthreads=cores)
    return time.perf_counter() - t0, int(sum(int(x) for x in out["counters"]))


def cpu_baseline(wl, n, s, d, target_s=15.0, steps=1):
    """The oracle's whole selection -- the same phase mix as one GPU step:
    initial gains, then the k rounds of forward and reverse dynamic update,
    all three snapshot-edge counters -- on the same graph, k and hash seed,
    over the first R' of the R snapshots (R' sized to about target_s seconds
    per step).  The oracle runs its initial gains on all host cores and its
    rounds on one (it is plain sequential code there).  Returns (GTEPS per
    step, sample description, seconds per step, cores)."""
    import oracle

    cores = os.cpu_count() or 1
    g = oracle.Graph(n, s, d, wl.model, wl.p)
    t1, _ = _oracle_du(g, 1, wl, cores)  # calibration: one snapshot
    rs = int(max(1, min(wl.R, target_s // max(t1, 1e-3))))
    vals, secs = [], []
    for _ in range(steps):
        dt, edges = _oracle_du(g, rs, wl, cores)
        vals.append(edges / dt / 1e9)
        secs.append(dt)
    sample = (f"oracle StaticGreedyDU selection (initial gains + {wl.k} rounds of forward and reverse update; "
              f"init + forward + reverse snapshot-edges) on the same graph, k and hash seed over snapshots "
              f"0..{rs - 1} of {wl.R}: {float(np.mean(secs)):.2f} s per selection; initial gains on {cores} "
              f"threads, rounds sequential")
    return float(np.mean(vals)), sample, float(np.mean(secs)), cores, rs


def run_reference(args, wl):
    ws, rank, _ = _dist()
    if rank != 0:
        return 0
    n, s, d = wl.graph()
    # the oracle keeps no state between steps, so warm-up steps are not run;
    # each step is one oracle selection on a bounded snapshot sample, sized so
    # that all steps end within about two minutes
    per_step = max(1.0, min(args.ref_seconds, 120.0 / max(1, args.steps)))
    value, sample, secs, cores, rs = cpu_baseline(wl, n, s, d, target_s=per_step, steps=args.steps)
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": 1, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": secs * 1e3, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "int64", "data": "synthetic",
        "config": {"workload": wl_desc(wl), "l2": "n/a (CPU)", "snapshots_per_step": rs},
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores, "kind": "oracle", "sample": sample},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)
    return 0


def run_oracle_select(args, wl):
    """The oracle's whole k-seed selection of the workload, at full R, on
    the host cores: lazy forward evaluation (StaticGreedyCELF, which the
    pins prove equal to Algorithm 2; the oracle's Algorithm 2 route itself
    walks every (w, r, u) of the reverse update, about 2.2 T snapshot-edges
    here, out of reach), timed once per step.  The select time to compare
    with the GPU's ms_per_step."""
    import oracle

    n, s, d = wl.graph()
    cores = os.cpu_count() or 1
    g = oracle.Graph(n, s, d, wl.model, wl.p)
    times, out = [], None
    for _ in range(args.steps):
        t0 = time.perf_counter()
        out = g.select(wl.R, wl.k, wl.seed, mode=oracle.CELF, nthreads=cores)
        times.append(time.perf_counter() - t0)
    line = {"impl": "oracle", "metric": "k-seed select time, oracle StaticGreedyCELF (full R)",
            "value": float(np.mean(times)) * 1e3, "unit": "ms", "steps": args.steps, "higher_is_better": False,
            "config": {"workload": wl_desc(wl)}, "cores": cores, "celf_evaluations": int(out["evals"]),
            "init_and_forward_snapshot_edges": [int(x) for x in out["counters"][:2]]}
    print(json.dumps(line), flush=True)
    return 0


def wl_desc(wl):
    if wl.name.startswith("rmat"):
        scale = int(wl.name[4:])
        return (f"R-MAT scale {scale}, {8 << scale} arcs, (0.57,0.19,0.19,0.05), weighted cascade, R={wl.R}, "
                f"k={wl.k}, hash seed {wl.seed}")
    return f"{wl.name} {wl.model} p={wl.p} R={wl.R} k={wl.k} seed={wl.seed}"


def _gen_graph(q):
    return inputs.batch_graph(q)


def _batch_graphs(qs, workers=None):
    """The recipe graphs of `qs`, generated in a spawned process pool (before
    any CUDA call, so no worker inherits a CUDA context)."""
    import concurrent.futures as cf
    import multiprocessing as mp

    workers = workers or max(1, min(16, os.cpu_count() or 1))
    with cf.ProcessPoolExecutor(workers, mp_context=mp.get_context("spawn")) as ex:
        return list(ex.map(_gen_graph, qs, chunksize=4))


def run_batched(args):
    """Config 4: the 256 batched-recipe queries (Chung-Lu graphs, n
    log-uniform in [1e3, 2e5], mixed cascades, R in {64, 128, 256}, k in
    [10, 100]).  Times one query per launch in sequence, the same queries as
    one batch over concurrent streams, and the batch captured once as a CUDA
    graph and replayed with a single launch; checks that all three agree."""
    import torch

    import __graft_entry__

    __graft_entry__.build()
    from paper_1212_4779_gb300 import sg

    apply_knobs(sg, args)

    sg.sg_set_mask_cache(args.mask_cache)
    qs = inputs.batch_queries(args.queries)
    coo = _batch_graphs(qs)
    torch.cuda.set_device(0)
    graphs = [sg.Graph.from_coo(*c) for c in coo]
    del coo
    dev = torch.device("cuda", 0)
    outs = [(torch.zeros(q["k"], dtype=torch.int32, device=dev), torch.zeros(q["k"], dtype=torch.int64, device=dev))
            for q in qs]
    stream = torch.cuda.Stream()

    def serial():
        for q, g, (so, go) in zip(qs, graphs, outs):
            sg.sg_select(g.handle, q["R"], q["k"], q["model"], q["p"], q["seed"], so, go, stream=stream)

    serial()
    stream.synchronize()
    ref = [(so.cpu().numpy().copy(), go.cpu().numpy().copy()) for so, go in outs]
    t0 = time.perf_counter()
    for _ in range(args.steps):
        serial()
    stream.synchronize()
    t_serial = (time.perf_counter() - t0) / args.steps
    for g in graphs:  # the batch runs on workspaces of its own
        g.trim()
    torch.cuda.empty_cache()

    wss = [sg.sg_workspace_create(g.handle, q["R"], q["k"]) for q, g in zip(qs, graphs)]
    items = [(g.handle, w, q["R"], q["k"], q["model"], q["p"], q["seed"], so, go)
             for q, g, w, (so, go) in zip(qs, graphs, wss, outs)]
    sg.sg_select_batch(items, concurrency=args.concurrency, stream=stream)
    stream.synchronize()
    t0 = time.perf_counter()
    for _ in range(args.steps):
        sg.sg_select_batch(items, concurrency=args.concurrency, stream=stream)
    stream.synchronize()
    t_batch = (time.perf_counter() - t0) / args.steps
    ok_batch = all(np.array_equal(so.cpu().numpy(), a) and np.array_equal(go.cpu().numpy(), b)
                   for (so, go), (a, b) in zip(outs, ref))

    b = sg.sg_batch_capture(items, concurrency=args.concurrency, stream=stream)
    sg.sg_batch_launch(b, stream=stream)
    stream.synchronize()
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    ev0.record(stream)
    for _ in range(args.steps):
        sg.sg_batch_launch(b, stream=stream)
    ev1.record(stream)
    ev1.synchronize()
    t_graph = ev0.elapsed_time(ev1) / 1e3 / args.steps
    ok_graph = all(np.array_equal(so.cpu().numpy(), a) and np.array_equal(go.cpu().numpy(), b_)
                   for (so, go), (a, b_) in zip(outs, ref))
    sg.sg_batch_free(b)
    for w in wss:
        sg.sg_workspace_free(w)
    nq = len(qs)
    line = {"metric": "queries/s, batched StaticGreedy-DU (config 4)", "value": nq / t_graph, "unit": "queries/s",
            "n_gpus": 1, "steps": args.steps, "higher_is_better": True, "dtype": "int64", "data": "synthetic",
            "config": {"workload": f"{nq} batched-recipe queries (Chung-Lu, n log-uniform 1e3..2e5)",
                       "concurrency": args.concurrency},
            "one_query_per_launch_qps": nq / t_serial, "batch_streams_qps": nq / t_batch,
            "batch_graph_qps": nq / t_graph, "speedup_vs_serial": t_serial / t_graph,
            "results_equal_serial": bool(ok_batch and ok_graph)}
    print(json.dumps(line), flush=True)
    return 0


def batched_served_summary(sg, args):
    """Bounded versions of the batched and served workloads for the default
    line: the first `summary_queries` batched recipes (Chung-Lu, n
    log-uniform in [1e3, 2e5], mixed cascades, R in {64, 128, 256}, k in
    [10, 100]) one query per launch and as one captured CUDA graph; then a
    Poisson trace (`summary_requests` requests at `summary_rate`/s, R in
    {100, 200}, k in [10, 100]) against those resident graphs through the
    continuous-batching server and one query per launch.  Every result of
    the batch, the graph replay and the server equals the one-per-launch
    result."""
    import torch

    from paper_1212_4779_gb300 import serve

    qs = inputs.batch_queries(args.summary_queries)
    coo = _batch_graphs(qs)
    graphs = [sg.Graph.from_coo(*c) for c in coo]
    del coo
    dev = torch.device("cuda", torch.cuda.current_device())
    outs = [(torch.zeros(q["k"], dtype=torch.int32, device=dev), torch.zeros(q["k"], dtype=torch.int64, device=dev))
            for q in qs]
    stream = torch.cuda.Stream()
    t0 = time.perf_counter()
    for q, g, (so, go) in zip(qs, graphs, outs):
        sg.sg_select(g.handle, q["R"], q["k"], q["model"], q["p"], q["seed"], so, go, stream=stream)
    stream.synchronize()
    t_serial = time.perf_counter() - t0
    ref = [(so.cpu().numpy().copy(), go.cpu().numpy().copy()) for so, go in outs]
    for g in graphs:
        g.trim()
    wss = [sg.sg_workspace_create(g.handle, q["R"], q["k"]) for q, g in zip(qs, graphs)]
    items = [(g.handle, w, q["R"], q["k"], q["model"], q["p"], q["seed"], so, go)
             for q, g, w, (so, go) in zip(qs, graphs, wss, outs)]
    b = sg.sg_batch_capture(items, concurrency=args.concurrency, stream=stream)
    sg.sg_batch_launch(b, stream=stream)
    stream.synchronize()
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    reps = 2
    ev0.record(stream)
    for _ in range(reps):
        sg.sg_batch_launch(b, stream=stream)
    ev1.record(stream)
    ev1.synchronize()
    t_graph = ev0.elapsed_time(ev1) / 1e3 / reps
    same_batch = all(np.array_equal(so.cpu().numpy(), a) and np.array_equal(go.cpu().numpy(), b_)
                     for (so, go), (a, b_) in zip(outs, ref))
    sg.sg_batch_free(b)
    for w in wss:
        sg.sg_workspace_free(w)
    nq = len(qs)
    batched = {"queries": nq, "one_query_per_launch_qps": nq / t_serial, "batch_graph_qps": nq / t_graph,
               "speedup": t_serial / t_graph, "results_equal": bool(same_batch)}
    models = [(q["model"], q["p"]) for q in qs]
    trace = serve.poisson_trace(args.summary_requests, args.summary_rate, 5000, models)
    st_served, res_s = serve.run_served(graphs, trace, max_running=args.concurrency, k_cap=128)
    st_serial, res_1 = serve.run_serial(graphs, trace)
    same = all(np.array_equal(res_s[i][0], res_1[i][0]) and np.array_equal(res_s[i][1], res_1[i][1])
               for i in range(len(trace)))
    served = {"workload": f"Poisson {args.summary_rate}/s, {len(trace)} requests over the {nq} recipe graphs, "
                          f"R in {{100,200}}, k in [10,100]",
              "max_running": args.concurrency, "served": st_served, "one_query_per_launch": st_serial,
              "results_equal": bool(same)}
    for g in graphs:
        g.close()
    return batched, served


def run_served(args):
    """Config 5: Poisson arrivals against resident graphs -- a directed R-MAT
    (scale 22 by default, WIC) plus the first 64 batched-recipe graphs;
    per-request R in {100, 200}, k in [10, 100]; continuous batching through
    the library's server vs one query per launch in arrival order."""
    import torch

    import __graft_entry__

    __graft_entry__.build()
    from paper_1212_4779_gb300 import serve, sg

    apply_knobs(sg, args)

    sg.sg_set_mask_cache(args.mask_cache)
    qs = inputs.batch_queries(64)
    coo = _batch_graphs(qs)
    big = inputs.rmat(args.served_scale, 16 << args.served_scale, (0.57, 0.19, 0.19, 0.05), 105)
    torch.cuda.set_device(0)
    graphs = [sg.Graph.from_coo(*big)] + [sg.Graph.from_coo(*c) for c in coo]
    del coo, big
    models = [("wic", 0.0)] + [(q["model"], q["p"]) for q in qs]
    trace = serve.poisson_trace(args.requests, args.rate, 5000, models)
    st_served, res_s = serve.run_served(graphs, trace, max_running=args.concurrency, k_cap=128)
    st_serial, res_1 = serve.run_serial(graphs, trace)
    same = all(np.array_equal(res_s[i][0], res_1[i][0]) and np.array_equal(res_s[i][1], res_1[i][1])
               for i in range(len(trace)))
    line = {"metric": "served queries/s and latency, StaticGreedy-DU (config 5)", "value": st_served["qps"],
            "unit": "queries/s", "n_gpus": 1, "higher_is_better": True, "dtype": "int64", "data": "synthetic",
            "config": {"workload": f"Poisson {args.rate}/s, {args.requests} requests, R-MAT scale {args.served_scale} "
                                   f"(WIC) + 64 batched-recipe graphs, R in {{100,200}}, k in [10,100]",
                       "max_running": args.concurrency,
                       "requests_on_rmat": sum(1 for r in trace if r.graph == 0)},
            "served": st_served, "one_query_per_launch": st_serial, "results_equal": bool(same)}
    print(json.dumps(line), flush=True)
    return 0


def run_spread_bench(args):
    """Seed-set spread evaluation on fresh snapshots: the 50 seeds that
    StaticGreedy-DU selects on the R-MAT scale-20 weighted-cascade graph
    (R = 256, hash seed 11), rated on R = 20,000 new snapshots (hash seed
    20011, the Monte Carlo count of the paper's evaluation).  One step = one
    sg_spread call; GTEPS = snapshot-edges of the walk per second."""
    import torch

    import __graft_entry__

    __graft_entry__.build()
    from paper_1212_4779_gb300 import sg

    apply_knobs(sg, args)

    wl = inputs.workload("rmat20_wic")
    n, s, d = wl.graph()
    torch.cuda.set_device(0)
    g = sg.Graph.from_coo(n, s, d)
    S = g.select(wl.R, wl.k, wl.model, wl.p, wl.seed).seeds
    R_eval, seed_eval = args.spread_R, 20011
    W_eval = (R_eval + 63) // 64
    S_dev = torch.from_numpy(S).cuda()
    stream = torch.cuda.current_stream()
    for _ in range(args.warmup):
        sg.sg_spread(g.handle, R_eval, wl.model, wl.p, seed_eval, S_dev, stream=stream)
    sampler = ClockSampler(0)
    sampler.start()
    times, res = [], None
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    for _ in range(args.steps):
        ev0.record(stream)
        res = sg.sg_spread(g.handle, R_eval, wl.model, wl.p, seed_eval, S_dev, stream=stream)
        ev1.record(stream)
        ev1.synchronize()
        times.append(ev0.elapsed_time(ev1))
    clocks = sampler.stop()
    total, edges = res
    ms = float(np.mean(times))
    cpu = None
    if not args.no_cpu_baseline:
        import oracle

        o = oracle.Graph(n, s, d, wl.model, wl.p)
        cores = os.cpu_count() or 1
        t0 = time.perf_counter()
        _, e1 = o.spread(64, seed_eval, S, nthreads=cores, want_edges=True)
        t1 = time.perf_counter() - t0
        r_cpu = int(max(64, min(R_eval, 64 * round(args.ref_seconds / max(t1, 1e-3)))))
        t0 = time.perf_counter()
        _, e2 = o.spread(r_cpu, seed_eval, S, nthreads=cores, want_edges=True)
        t2 = time.perf_counter() - t0
        cpu = {"value": e2 / t2 / 1e9, "unit": UNIT, "cores": cores, "kind": "oracle",
               "sample": f"oracle spread of the same 50 seeds over {r_cpu} of the {R_eval} snapshots, {cores} threads"}
    line = {"metric": "GTEPS (snapshot-edges/s) of seed-set spread evaluation", "value": edges / (ms / 1e3) / 1e9,
            "unit": UNIT, "n_gpus": 1, "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms,
            "higher_is_better": True, "dtype": "int64", "data": "synthetic",
            "config": {"workload": f"spread of the 50 StaticGreedy-DU seeds of R-MAT scale 20 (weighted cascade) "
                                   f"on {R_eval} fresh snapshots (hash seed {seed_eval})",
                       "l2": "inputs larger than L2 (graph 100 MB + 2-4 GB of per-word state per launch)"},
            "spread_estimate": total / R_eval, "snapshot_edges_per_step": edges,
            "gpu_launches": args.steps * -(-W_eval // max(1, min(W_eval, (8 << 30) // (n * 24)))),
            "cpu_baseline": cpu, "clocks": clocks}
    print(json.dumps(line), flush=True)
    return 0


def run_celf_bench(args):
    """StaticGreedyCELF against StaticGreedyDU (Section 6 times both) on the
    R-MAT scale-20 weighted-cascade query (R = 256, k = 50, hash seed 11):
    the same seeds and gains, selected with lazy evaluation.  One step = one
    sg_select_celf call (host-driven: one GPU walk per evaluation)."""
    import torch

    import __graft_entry__

    __graft_entry__.build()
    from paper_1212_4779_gb300 import sg

    apply_knobs(sg, args)

    wl = inputs.workload(args.celf_workload)
    n, s, d = wl.graph()
    torch.cuda.set_device(0)
    g = sg.Graph.from_coo(n, s, d)
    stream = torch.cuda.current_stream()
    for _ in range(args.warmup):
        g.select_celf(wl.R, wl.k, wl.model, wl.p, wl.seed, stream=stream)
        g.select(wl.R, wl.k, wl.model, wl.p, wl.seed, stream=stream)
    torch.cuda.synchronize()
    t_celf, t_du, evals, same = [], [], 0, True
    for _ in range(args.steps):
        t0 = time.perf_counter()
        res, evals = g.select_celf(wl.R, wl.k, wl.model, wl.p, wl.seed, stream=stream)
        torch.cuda.synchronize()
        t_celf.append(time.perf_counter() - t0)
        t0 = time.perf_counter()
        du = g.select(wl.R, wl.k, wl.model, wl.p, wl.seed, stream=stream)
        torch.cuda.synchronize()
        t_du.append(time.perf_counter() - t0)
        same = same and bool(np.array_equal(res.seeds, du.seeds) and np.array_equal(res.gains, du.gains))
    line = {"metric": "k-seed select time, StaticGreedyCELF vs StaticGreedyDU", "value": float(np.mean(t_celf)) * 1e3,
            "unit": "ms", "n_gpus": 1, "steps": args.steps, "warmup": args.warmup, "higher_is_better": False,
            "dtype": "int64", "data": "synthetic", "config": {"workload": wl_desc(wl)},
            "du_ms": float(np.mean(t_du)) * 1e3, "celf_over_du": float(np.mean(t_celf) / np.mean(t_du)),
            "celf_evaluations": evals, "results_equal": same}
    print(json.dumps(line), flush=True)
    return 0


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="rmat20_wic")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--ref-seconds", type=float, default=15.0)
    ap.add_argument("--queries", type=int, default=256, help="batched: number of queries")
    ap.add_argument("--concurrency", type=int, default=16, help="batched/served: concurrent queries")
    ap.add_argument("--requests", type=int, default=512, help="served: trace length")
    ap.add_argument("--rate", type=float, default=200.0, help="served: arrivals per second")
    ap.add_argument("--served-scale", type=int, default=22, help="served: R-MAT scale of the large graph")
    ap.add_argument("--spread-R", type=int, default=20000, help="spread: snapshots of the evaluation")
    ap.add_argument("--celf-workload", default="rmat20_wic", help="celf: the query compared with the dynamic update")
    ap.add_argument("--oracle-workload", default="rmat20_wic", help="oracle_select: the query the oracle selects on")
    ap.add_argument("--mask-cache", type=int, default=0, choices=[0, 1],
                    help="1: evaluate every arc's coins once per query into the live-mask cache")
    ap.add_argument("--no-summary", action="store_true",
                    help="skip the bounded batched and served summary of the default line")
    ap.add_argument("--summary-queries", type=int, default=64, help="summary: batched recipes (and served graphs)")
    ap.add_argument("--summary-requests", type=int, default=256, help="summary: served trace length")
    ap.add_argument("--summary-rate", type=float, default=200.0, help="summary: served arrivals per second")
    ap.add_argument("--walk-groups", type=int, default=None, choices=[8, 16, 32, 64],
                    help="blocks per 64-snapshot word of the forward and landmark walks (library default if unset)")
    ap.add_argument("--direction", type=str, default=None,
                    help="MODE,DIVISOR of the walks' direction-optimising switch (library default if unset)")
    args = ap.parse_args()
    if args.workload == "batched" and args.impl == "ours":
        return run_batched(args)
    if args.workload == "served" and args.impl == "ours":
        return run_served(args)
    if args.workload == "spread" and args.impl == "ours":
        return run_spread_bench(args)
    if args.workload == "celf" and args.impl == "ours":
        return run_celf_bench(args)
    if args.workload == "oracle_select":
        return run_oracle_select(args, inputs.workload(args.oracle_workload))
    wl = inputs.workload(args.workload)
    if args.impl == "reference":
        return run_reference(args, wl)

    import torch

    ws, rank, local = _dist()
    if ws > 1:
        import torch.distributed as dist

        torch.cuda.set_device(local)
        dist.init_process_group("nccl")
    else:
        torch.cuda.set_device(0)
    import __graft_entry__

    __graft_entry__.build()
    from paper_1212_4779_gb300 import sg

    sg.sg_set_mask_cache(args.mask_cache)
    apply_knobs(sg, args)
    n, s, d = wl.graph()
    g = sg.Graph.from_coo(n, s, d)
    dev = torch.device("cuda", torch.cuda.current_device())
    stream = torch.cuda.current_stream()
    seeds = torch.zeros(wl.k, dtype=torch.int32, device=dev)
    gains = torch.zeros(wl.k, dtype=torch.int64, device=dev)
    flush = torch.empty(512 * 1024 * 1024 // 4, dtype=torch.int32, device=dev)  # 512 MB > 129 MB L2

    def step():
        return sg.sg_select(g.handle, wl.R, wl.k, wl.model, wl.p, wl.seed, seeds, gains, stream=stream, stats=True)

    for _ in range(args.warmup):
        flush.fill_(1)
        step()
    torch.cuda.synchronize()
    sampler = ClockSampler(torch.cuda.current_device())
    sampler.start()
    if ws > 1:
        torch.distributed.barrier()
    torch.cuda.synchronize()
    t_steps, t_walk, t_fwd, t_lose, edges, launches, st_last = [], [], [], [], [], 0, None
    ev0 = torch.cuda.Event(enable_timing=True)
    ev1 = torch.cuda.Event(enable_timing=True)
    for _ in range(args.steps):
        flush.fill_(1)  # evict the graph from L2 between timed steps
        ev0.record(stream)
        st = step()
        ev1.record(stream)
        ev1.synchronize()
        t_steps.append(ev0.elapsed_time(ev1))
        t_walk.append(st["ms_init_tier1"])
        t_fwd.append(st["ms_fwd"])
        t_lose.append(st["ms_rounds"] - st["ms_fwd"])
        edges.append(st["init_edges"] + st["fwd_edges"] + st["rev_edges"])
        launches += st["kernel_launches"]
        st_last = st
    torch.cuda.synchronize()
    clocks = sampler.stop()
    edges_step = float(np.mean(edges))
    ms_step, value = replica_throughput(np.sum(t_steps), edges_step, args.steps, ws)
    value /= 1e9

    peaks, src = _peaks()
    roofline, walks = cover_roofline(wl, st_last, float(np.mean(t_fwd)), peaks, src), None
    if roofline:
        walks = {"initial gains": walk_view(st_last, 0, 0, float(np.mean(t_walk))),
                 "rounds": walk_view(st_last, 1, 2, float(np.mean(t_lose)))}

    e2e = None
    if not args.no_e2e:
        e2e = measure_e2e(sg, wl, n, s, d, args, stream)

    batched = served = None
    if not args.no_summary and ws == 1:
        g.trim()
        batched, served = batched_served_summary(sg, args)

    cpu = None
    if not args.no_cpu_baseline and ws == 1 and rank == 0:
        v, sample, _t, cores, _rs = cpu_baseline(wl, n, s, d, target_s=args.ref_seconds)
        cpu = {"value": v, "unit": UNIT, "cores": cores, "kind": "oracle", "sample": sample,
               "phases": "initial gains + forward + reverse (the GPU step's phase mix)"}

    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": ws, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": ms_step, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "int64", "data": "synthetic",
        "config": {"workload": wl_desc(wl), "n": n, "m": int(g.m), "R": wl.R, "k": wl.k,
                   "l2": "512 MB buffer written between timed steps", "parallelism": f"replicas x{ws}",
                   "mask_cache": bool(st_last["mask_cache"]),
                   "walk_groups": args.walk_groups or "library default",
                   "direction": args.direction or "library default"},
        "snapshot_edges_per_step": edges_step,
        "phase_ms": {k: round(st_last[k], 3) for k in ("ms_index", "ms_landmarks", "ms_init_tier1", "ms_init_tier2",
                                                      "ms_init_tier3", "ms_init", "ms_fwd", "ms_rounds", "ms_total")},
        "tiers": {k: st_last[k] for k in ("init_tier2_tasks", "init_tier3_tasks", "rev_tier2_tasks",
                                          "rev_tier3_tasks", "rev_tasks", "du_entries")},
        "edges": {k: st_last[k] for k in ("init_edges", "fwd_edges", "rev_edges")},
        "gteps_by_phase": phase_rates(st_last),
        "work": {"keys": st_last["work_keys"], "elems": st_last["work_elems"]},
        "gpu_launches": launches,
        "roofline": roofline,
        "closure_walks": walks,
        "cpu_baseline": cpu,
        "e2e": e2e,
        "clocks": clocks,
        "peaks_source": src,
        "batched": batched,
        "served": served,
    }
    if rank == 0:
        print(json.dumps(line), flush=True)
    g.close()
    if ws > 1:
        torch.distributed.destroy_process_group()
    return 0


def cover_roofline(wl, st, fwd_ms, peaks, src):
    """The dominant kernel, snap_cover_kernel: its bytes over the rounds against
    the copy bandwidth.  Its time includes the rounds' argmax (a few
    microseconds each).  None where a knob on the command line sent the query to
    the tiered engines."""
    if st["init_tier2_tasks"] or st["init_tier3_tasks"] or fwd_ms <= 0:
        return None
    need = st["du_entries"] * BYTES_PER_COVERED + st["rev_tasks"] * BYTES_PER_RANGE
    peak = float(peaks.get("hbm_gbs", 6800.0))
    achieved = need / (fwd_ms / 1e3) / 1e9
    return {"bound": "hbm", "kernel": "snap_cover_kernel (one launch a round, with the argmax)",
            "achieved": achieved, "peak": peak, "unit": "GB/s", "frac": achieved / peak,
            "traffic": _recorded_traffic() if wl.name == "rmat20" else None,
            "traffic_source": "profiles/snap_cover_rmat20_traffic.md (full-size ncu capture)",
            "peak_source": f"MEASURED_PEAKS.json hbm_gbs ({src})",
            "kernel_ms": fwd_ms / wl.k, "launches": wl.k, "algorithmic_bytes_per_launch": need / wl.k,
            "bytes_per_covered_pair": BYTES_PER_COVERED, "bytes_per_range": BYTES_PER_RANGE}


def walk_view(st, phase, col, ms):
    """Joins visited and join arcs scanned by one phase's closure walks; most
    of their bytes come from L2, their visited bits from shared memory."""
    joins, arcs = st["work_keys"][phase][col], st["work_elems"][phase][col]
    need = joins * BYTES_PER_JOIN + arcs * BYTES_PER_JOIN_ARC
    return {"ms": ms, "joins": joins, "arcs": arcs, "algorithmic_bytes": need,
            "gb_per_s": need / (ms / 1e3) / 1e9 if ms > 0 else None}


def apply_knobs(sg, args):
    """Library tuning knobs named on the command line (none changes a result)."""
    if args.walk_groups:
        sg.sg_set_walk_groups(args.walk_groups)
    if args.direction:
        mode, div = (int(x) for x in args.direction.split(","))
        sg.sg_set_direction(mode, div)


def phase_rates(st):
    """Snapshot-edges per second of each phase, and elements actually
    expanded per second.  The reverse counter is the implementation-
    independent sum over every (w, r) the dynamic update removes and every u
    reaching w of indeg(u) (the paper's per-node reverse BFS); the library
    settles most of it without walking (|N_r| comes off every ancestor of v*
    at once, the others lose a closure's sizes), so the reverse and total
    rates are nominal, while `elements_per_s` counts the join arcs that the
    walks really scanned."""
    ms_init = st["ms_init"]
    ms_fwd = st["ms_fwd"]
    ms_rev = max(1e-6, st["ms_rounds"] - ms_fwd)
    elems = sum(sum(row) for row in st["work_elems"])
    return {"init": st["init_edges"] / (ms_init / 1e3) / 1e9 if ms_init > 0 else None,
            "forward_and_argmax": st["fwd_edges"] / (ms_fwd / 1e3) / 1e9 if ms_fwd > 0 else None,
            "reverse_nominal": st["rev_edges"] / (ms_rev / 1e3) / 1e9,
            "elements_per_s": elems / (st["ms_total"] / 1e3) if st["ms_total"] > 0 else None,
            "elements_expanded": elems,
            "note": "reverse counter nominal: most of it is credited without traversal"}


def measure_e2e(sg, wl, n, s, d, args, stream):
    """End to end through the C ABI with host buffers: every step uploads
    the graph from pinned host memory (sg_load_graph, CSR), selects, and
    reads the seeds and gains back into pinned host memory."""
    import torch

    order = np.lexsort((d, s))
    ss, dd = s[order], d[order]
    rp = np.zeros(n + 1, dtype=np.int64)
    np.add.at(rp, ss.astype(np.int64) + 1, 1)
    rp = np.cumsum(rp)
    rp_h = torch.from_numpy(rp).pin_memory()
    col_h = torch.from_numpy(np.ascontiguousarray(dd, dtype=np.int32)).pin_memory()
    seeds_h = torch.zeros(wl.k, dtype=torch.int32).pin_memory()
    gains_h = torch.zeros(wl.k, dtype=torch.int64).pin_memory()
    edges = None

    def one():
        nonlocal edges
        h = sg.sg_load_graph(n, col_h.numel(), rp_h, col_h, stream=stream)
        st = sg.sg_select(h, wl.R, wl.k, wl.model, wl.p, wl.seed, seeds_h, gains_h, stream=stream, stats=True)
        stream.synchronize()
        sg.sg_free_graph(h)
        edges = st["init_edges"] + st["fwd_edges"] + st["rev_edges"]

    for _ in range(max(1, min(2, args.warmup))):
        one()
    steps = max(1, min(args.steps, 3))
    t0 = time.perf_counter()
    for _ in range(steps):
        one()
    dt = (time.perf_counter() - t0) / steps
    return {"value": edges / dt / 1e9, "unit": UNIT, "ms_per_step": dt * 1e3,
            "h2d_bytes_per_step": int(rp_h.numel() * 8 + col_h.numel() * 4),
            "d2h_bytes_per_step": int(wl.k * (4 + 8))}


if __name__ == "__main__":
    sys.exit(main())
