"""Joins with many in-arcs (a hub under a uniform cascade): the initial gains
at the lengths from which warps share such a join's arcs, and the time they
take.  Integers, so the tolerance is zero."""

import time

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sg():
    import __graft_entry__

    __graft_entry__.build()
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1212_4779_gb300 import sg as _sg

    return _sg


def _hub(leaves, mids, hubs=1):
    """`hubs` times: `leaves` nodes over one, which with a second node is over
    `mids` joins."""
    s, d, at = [], [], 0
    for _ in range(hubs):
        h, x = at + leaves, at + leaves + 1
        m = np.arange(mids) + x + 1
        s += [np.arange(leaves) + at, np.full(mids, h), np.full(mids, x)]
        d += [np.full(leaves, h), m, m]
        at = x + 1 + mids
    return at, np.concatenate(s).astype(np.int32), np.concatenate(d).astype(np.int32)


@pytest.mark.parametrize("leaves,hubs,p,R", [(64, 3, 1.0, 2), (65, 3, 1.0, 65), (2048, 1, 1.0, 3), (2049, 2, 1.0, 1),
                                             (70, 1100, 1.0, 1), (9000, 2, 0.7, 65)])
def test_gains_of_hubs(sg, leaves, hubs, p, R):
    n, s, d = _hub(leaves, 6, hubs)
    ref = oracle.Graph(n, s, d, "uic", p).select(R, 3, 8, mode=oracle.DU, want_init=True)
    with sg.Graph.from_coo(n, s, d) as g:
        gains, edges = g.init_gains(R, "uic", p, 8)
        assert np.array_equal(gains, ref["s_init"]) and edges == int(ref["counters"][0])
        res = g.select(R, 3, "uic", p, 8)
        assert np.array_equal(res.seeds, ref["seeds"]) and np.array_equal(res.gains, ref["gains"])


def test_a_large_hub_takes_no_thread_of_its_own(sg):
    """400,000 in-arcs of one join in each of 64 snapshots: 70 ms where one
    thread sums them, 5 ms where the block does."""
    n, s, d = _hub(400000, 64)
    with sg.Graph.from_coo(n, s, d) as g:
        best = 1e9
        for _ in range(4):
            t = time.perf_counter()
            g.init_gains(64, "uic", 1.0, 8)
            best = min(best, time.perf_counter() - t)
    assert best < 0.03, best
