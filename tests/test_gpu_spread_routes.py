"""Seed-set spread on both sides of the line between its two walks (snapshot by
snapshot, 64 at a time), and the time of many snapshots of a small graph."""

import time

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


@pytest.mark.parametrize("model,p", [("uic", 0.3), ("uic", 0.0), ("wic", 0.0)])
def test_both_sides_of_the_line(sg, model, p):
    """n = 100: the line lies at R = 8000."""
    n, s, d = inputs.random_small(100, 400, 3)
    o = oracle.Graph(n, s, d, model, p)
    with sg.Graph.from_coo(n, s, d) as g:
        for R in (7999, 8000, 8001, 8065):
            for S in ([7], [0, 3, 3, 99]):
                assert g.spread(R, model, p, 5, S) == o.spread(R, 5, S, want_edges=True)


def test_many_snapshots_of_a_small_graph(sg):
    """400,000 snapshots of 200 nodes: 4.5 ms one at a time, 1.5 ms in words."""
    n, s, d = inputs.er_directed(200, 1000, 3)
    with sg.Graph.from_coo(n, s, d) as g:
        best = 1e9
        for _ in range(5):
            t = time.perf_counter()
            g.spread(400000, "wic", 0.0, 5, list(range(10)))
            best = min(best, time.perf_counter() - t)
    assert best < 0.003, best
