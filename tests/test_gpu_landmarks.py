"""Landmarks of the compact snapshot graphs: the arcs that walks scan over large
strongly connected components, and the exact results.  Integers, so the
tolerance is zero."""

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


def _check(sg, graph, p, R, k):
    """Exact against the oracle; the work counters of a selection."""
    n, s, d = graph
    ref = oracle.Graph(n, s, d, "uic", p).select(R, k, 11, mode=oracle.DU, want_init=True)
    with sg.Graph.from_coo(n, s, d) as g:
        gains, edges = g.init_gains(R, "uic", p, 11)
        res = g.select(R, k, "uic", p, 11, stats=True)
        celf, _ = g.select_celf(R, k, "uic", p, 11)
    assert np.array_equal(gains, ref["s_init"]) and edges == int(ref["counters"][0])
    for r in (res, celf):
        assert np.array_equal(r.seeds, ref["seeds"]) and np.array_equal(r.gains, ref["gains"])
    got = [res.stats["init_edges"], res.stats["fwd_edges"], res.stats["rev_edges"]]
    assert got == [int(x) for x in ref["counters"]]
    return res.stats["work_elems"]


def _component_under_sources(n, m, sources, leaves):
    """A random digraph of n nodes, `sources` nodes over one of them each, and
    one more with `leaves` leaves of its own, which is the first seed."""
    _, s, d = inputs.er_directed(n, m, 5)
    r = np.random.default_rng(1)
    top = n + sources
    s = np.concatenate([s, np.arange(n, top), [top], np.full(leaves, top)])
    d = np.concatenate([d, r.integers(0, n, sources), [3], np.arange(top + 1, top + 1 + leaves)])
    return top + 1 + leaves, s.astype(np.int32), d.astype(np.int32)


@pytest.mark.parametrize("p,R", [(1.0, 2), (0.9, 65)])
def test_a_round_over_a_component(sg, p, R):
    """The first seed lies above a component of 2000 nodes that 1500 others
    reach at nodes of their own: their walks start from what the component
    reaches (16,000 arcs a walk otherwise, 24 M a snapshot)."""
    work = _check(sg, _component_under_sources(2000, 16000, 1500, 1800), p, R, 4)
    assert sum(work[1]) < 1000000 * R, work


def _components(count, n, m):
    """`count` random digraphs of n nodes, each below a node of its own."""
    s, d = [], []
    for c in range(count):
        _, a, b = inputs.er_directed(n, m, 20 + c)
        at = c * (n + 1)
        s += [a + at, [at + n]]
        d += [b + at, [at + c % n]]
    return count * (n + 1), np.concatenate(s).astype(np.int32), np.concatenate(d).astype(np.int32)


@pytest.mark.parametrize("count,n,p,R,bound", [
    (1, 700, 1.0, 2, 2000), (2, 700, 1.0, 65, 4000), (3, 1200, 0.9, 64, 100000),
    (32, 600, 1.0, 1, 200000), (34, 600, 1.0, 3, 14000000),  # more than there are landmarks: two walk in full
    (5, 400, 1.0, 3, 20000000),                              # components below the size that calls for another
])
def test_gains_over_several_components(sg, count, n, p, R, bound):
    """Every large component has a landmark: a node's walk starts from what the
    landmark reaches (8 n arcs for each of the n nodes otherwise)."""
    work = _check(sg, _components(count, n, 8 * n), p, R, 3)
    assert sum(work[0]) < bound * R, work
