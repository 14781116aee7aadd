"""Device memory that runs short or is shared: allocations refused for a while,
scratch that does not fit, and a server whose requests take different routes.
Results stay the oracle's; integers, so the tolerance is zero."""

import time

import numpy as np
import pytest

import oracle
from paper_1212_4779_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sg():
    import __graft_entry__

    __graft_entry__.build()
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1212_4779_gb300 import sg as _sg

    return _sg


class _Hooks:
    """Allocator hooks that ask `refuse(bytes)` before every allocation."""

    def __init__(self, sg, refuse):
        self.sg, self.refuse, self.held, self.refused = sg, refuse, {}, []

    def __enter__(self):
        import torch

        def alloc(nbytes, stream):
            if self.refuse(nbytes):
                self.refused.append(nbytes)
                return None
            t = torch.empty(max(1, nbytes), dtype=torch.uint8, device="cuda")
            self.held[t.data_ptr()] = t
            return t.data_ptr()

        def release(ptr, nbytes, stream):
            torch.cuda.synchronize()
            self.held.pop(ptr, None)

        self.sg.sg_set_allocator(alloc, release)
        return self

    def __exit__(self, *exc):
        self.sg.sg_set_allocator(None, None)

    def largest(self):
        return max((t.numel() for t in self.held.values()), default=0)


BIG = 128 << 20  # the compact graphs below take more, every array of the engines less


def _same(res, ref):
    assert np.array_equal(res.seeds, ref["seeds"]) and np.array_equal(res.gains, ref["gains"])


def test_a_refused_allocation_is_asked_for_again(sg):
    """One refusal sends a query to the engines; once there is room again, one
    of the next few takes the compact graphs.  While there is none, they are
    asked for now and then only."""
    n, s, d = inputs.er_directed(2000, 20000, 6)
    ref = oracle.Graph(n, s, d, "uic", 0.5).select(200, 4, 9, mode=oracle.COVER)
    short = [True]
    with _Hooks(sg, lambda b: short[0] and b > BIG) as h:
        with sg.Graph.from_coo(n, s, d) as g:
            _same(g.select(200, 4, "uic", 0.5, 9), ref)
            assert len(h.refused) == 1 and h.largest() < BIG
            short[0] = False
            for _ in range(5):
                _same(g.select(200, 4, "uic", 0.5, 9), ref)
            assert h.largest() > BIG
        short[0] = True
        with sg.Graph.from_coo(n, s, d) as g:
            del h.refused[:]
            for _ in range(40):
                _same(g.select(200, 4, "uic", 0.5, 9), ref)
            assert 2 <= len(h.refused) <= 6


@pytest.mark.parametrize("times", [1, 3, 5])
def test_lazy_evaluation_with_little_scratch(sg, times):
    """Scratch of the evaluations refused: fewer candidates a launch, and with
    none left the engines."""
    n, s, d = inputs.chung_lu_undirected(2000, 8000, 2.5, 8.0, 2)
    ref = oracle.Graph(n, s, d, "wic").select(100, 12, 5, mode=oracle.CELF)
    left = [0]

    def refuse(nbytes):
        if nbytes > BIG:
            left[0] = times  # the arena was given; the next requests are the scratch
            return False
        if left[0] and nbytes > 1 << 19:
            left[0] -= 1
            return True
        return False

    with _Hooks(sg, refuse) as h:
        with sg.Graph.from_coo(n, s, d) as g:
            res, evals = g.select_celf(100, 12, "wic", 0.0, 5)
            _same(res, ref)
            assert evals == ref["evals"]
            assert len(h.refused) == times and left[0] == 0
            assert (h.largest() > BIG) == (times < 5)
            _same(g.select(100, 12, "wic", 0.0, 5), ref)


def _serve(sg, sv, requests, together):
    """Results of the requests, all submitted at once or one after another."""
    out, ids = [], []
    end = time.time() + 120

    def wait(rid, k):
        while time.time() < end:
            done, seeds, gains, _ = sg.sg_server_poll(sv, rid, k)
            if done:
                return sg.Selection(seeds, gains, None)
            time.sleep(0.002)
        raise AssertionError("the server did not answer")

    for q in requests:
        ids.append((sg.sg_server_submit(sv, *q), q[2]))
        if not together:
            out.append(wait(*ids.pop()))
    return out + [wait(*i) for i in ids]


@pytest.fixture(scope="module")
def mixed():
    """A symmetric graph, requests of three routes on it, their results."""
    n, s, d = inputs.symmetric(*inputs.er_directed(20000, 60000, 3))
    cases = [("uic_undirected", 0.05, 2000, 6), ("wic", 0.0, 32, 6), ("uic", 0.1, 64, 6)]
    refs = {}
    for model, p, R, k in cases:
        mode = oracle.COVER if model == "uic_undirected" else oracle.DU
        refs[model] = oracle.Graph(n, s, d, model, p).select(R, k, 13, mode=mode)
    return (n, s, d), cases, refs


@pytest.mark.parametrize("together", [False, True])
def test_server_memory_over_mixed_routes(sg, mixed, together):
    """Undirected, compact and dense requests on one graph: what they hold
    together stays within the budget, in every order."""
    import torch

    (n, s, d), cases, refs = mixed
    budget = 800 << 20
    g = sg.Graph.from_coo(n, s, d)
    # what stays with the graph after its first undirected query
    g.select(1, 1, "uic_undirected", 0.05, 13)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    sv = sg.sg_server_create(3, budget, 64)
    try:
        order = [cases[i] for i in (0, 1, 2, 1, 0, 2, 0, 1)]
        got = _serve(sg, sv, [(g.handle, R, k, model, p, 13) for model, p, R, k in order], together)
        for (model, *_), res in zip(order, got):
            _same(res, refs[model])
        torch.cuda.synchronize()
        assert free - torch.cuda.mem_get_info()[0] <= budget + (96 << 20)
    finally:
        sg.sg_server_destroy(sv)
        g.close()


def test_workspace_bytes_cover_the_workspace(sg):
    """sg_workspace_bytes is no less than what sg_workspace_create takes, and
    leaves out compact graphs of a size that is never built (64 GiB)."""
    n, s, d = inputs.er_directed(3000, 12000, 4)
    with _Hooks(sg, lambda b: False) as h:
        with sg.Graph.from_coo(n, s, d) as g:
            for R in (1, 64, 200, 1000):
                before = sum(t.numel() for t in h.held.values())
                ws = sg.sg_workspace_create(g.handle, R, 10)
                assert sum(t.numel() for t in h.held.values()) - before <= sg.sg_workspace_bytes(g.handle, R, 10)
                sg.sg_workspace_free(ws)
            # 190 bytes per place, 3,000 places a snapshot: past 64 GiB from R = 120,000 on
            small, large = (sg.sg_workspace_bytes(g.handle, R, 10) for R in (64 * 1500, 64 * 3000))
            assert small < 64 << 30 and large < 64 << 30
