"""Compact snapshot graphs (the default route of selections, gains, CELF) and
what goes with them, at the sizes where they can go wrong: against the oracle,
and against the tiered engines, which take every query once a knob is off its
default.  All outputs are integers, so the tolerance is zero."""

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


def _arcs(n, pairs):
    a = np.array(pairs, dtype=np.int32).reshape(-1, 2)
    return n, a[:, 0].copy(), a[:, 1].copy()


def _ring(n, chords=()):
    return _arcs(n, [(i, (i + 1) % n) for i in range(n)] + list(chords))


def _cycles_with_tails():
    """Rings of 2 to 9 nodes, none with a join, each under a path; every second
    one also feeds a node of the next."""
    pairs, at = [], 0
    for c in range(2, 10):
        ring = [at + i for i in range(c)]
        pairs += [(ring[i], ring[(i + 1) % c]) for i in range(c)]
        pairs += [(ring[c // 2], at + c), (at + c, at + c + 1)]
        if c % 2 == 0:
            pairs.append((at + c + 1, at + c + 2 + 1))
        at += c + 2
    return _arcs(at + 2, pairs)


def _two_over(mids, sinks):
    """Two nodes over `mids` joins, each over one of `sinks` nodes."""
    m = np.arange(2, mids + 2, dtype=np.int32)
    s, d = [np.zeros(mids, np.int32), np.ones(mids, np.int32)], [m, m]
    if sinks:
        s.append(m)
        d.append((mids + 2 + np.arange(mids) % sinks).astype(np.int32))
    return mids + 2 + sinks, np.concatenate(s), np.concatenate(d)


def _hubs(hubs, deg):
    """A root over `hubs` nodes, each over `deg` others in turn."""
    n = 1 + hubs + 700
    pairs = [(0, 1 + h) for h in range(hubs)]
    pairs += [(1 + h, 1 + hubs + (7 * h + i) % 700) for h in range(hubs) for i in range(deg - h % 3)]
    return _arcs(n, pairs)


CASES = {
    # tile edges of nodes (256) and words of snapshots (64)
    "n255": (lambda: inputs.random_small(255, 900, 1), "uic", 0.3, 1, 5),
    "n256": (lambda: inputs.random_small(256, 900, 2), "uic", 0.3, 63, 5),
    "n257": (lambda: inputs.random_small(257, 900, 3, loops_and_dups=True), "uic", 0.3, 64, 5),
    "wic65": (lambda: inputs.chung_lu_undirected(800, 3000, 2.5, 7.0, 2), "wic", 0.0, 65, 30),
    "lt130": (lambda: inputs.chung_lu_undirected(800, 3000, 2.5, 7.0, 2), "lt", 0.0, 130, 30),
    # no live arc, every arc live, more seeds than gains
    "none": (lambda: inputs.er_directed(300, 900, 4), "uic", 0.0, 70, 8),
    "all": (lambda: inputs.er_directed(300, 900, 4), "uic", 1.0, 3, 300),
    # one-parent cycles, alone, under paths and with chords
    "ring": (lambda: _ring(300), "uic", 1.0, 2, 4),
    "ring_cut": (lambda: _ring(300), "uic", 0.99, 66, 10),
    "chords": (lambda: _ring(300, [(i, (i * 7) % 300) for i in range(0, 300, 11)]), "uic", 0.9, 70, 10),
    "cycles": (_cycles_with_tails, "uic", 1.0, 2, 12),
    "cycles_cut": (_cycles_with_tails, "uic", 0.8, 129, 12),
    # closures past the queues of a walk (128 + 8192) and the rounds' landmark
    # (512 newly covered joins)
    "giant": (lambda: inputs.er_directed(3000, 24000, 5), "uic", 0.5, 3, 8),
    "wide": (lambda: _two_over(10000, 100), "uic", 1.0, 2, 5),
    "wide_cut": (lambda: _two_over(10000, 100), "uic", 0.97, 2, 5),
    # more joins than visited bits fit into shared memory
    "bits": (lambda: _two_over(900000, 0), "uic", 1.0, 1, 2),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_snapshot_graphs_match_oracle_and_tiers(sg, name):
    make, model, p, R, k = CASES[name]
    n, s, d = make()
    o = oracle.Graph(n, s, d, model, p)
    ref = o.select(R, k, 21, mode=oracle.DU, want_init=True)
    cnt = [int(x) for x in ref["counters"]]
    with sg.Graph.from_coo(n, s, d) as g:
        def run():
            gains, ed = g.init_gains(R, model, p, 21)
            plain = g.select(R, k, model, p, 21)
            full = g.select(R, k, model, p, 21, stats=True)
            _, left, cov = g.select_state(R, k, model, p, 21)
            celf, evals = g.select_celf(R, k, model, p, 21)
            assert full.stats["status_flags"] == 0
            edges = [full.stats["init_edges"], full.stats["fwd_edges"], full.stats["rev_edges"]]
            return dict(s_init=gains, ed=ed, seeds=plain.seeds, gains=plain.gains, seeds2=full.seeds,
                        gains2=full.gains, edges=edges, left=left, cov=cov, cseeds=celf.seeds, cgains=celf.gains,
                        evals=evals)

        got = run()
        assert np.array_equal(got["s_init"], ref["s_init"]) and got["ed"] == cnt[0] and got["edges"] == cnt
        for key in ("seeds", "seeds2", "cseeds"):
            assert np.array_equal(got[key], ref["seeds"]), key
        for key in ("gains", "gains2", "cgains"):
            assert np.array_equal(got[key], ref["gains"]), key
        sg.sg_set_walk_groups(32)  # the tiered engines
        try:
            want = run()
        finally:
            sg.sg_set_walk_groups(64)
        for key in want:
            assert np.array_equal(got[key], want[key]), key


@pytest.mark.parametrize("hubs,deg,p,R", [(1, 512, 1.0, 1), (3, 513, 0.5, 65), (140, 514, 0.4, 3), (9, 66, 0.9, 63)])
def test_spread_of_long_rows(sg, hubs, deg, p, R):
    """Rows at the lengths from which a warp reads them straight (64) and the
    block shares them (512), more of the latter than are remembered (128)."""
    n, s, d = _hubs(hubs, deg)
    o = oracle.Graph(n, s, d, "uic", p)
    with sg.Graph.from_coo(n, s, d) as g:
        for S in ([0], [n - 1, 0, 0, 31, 32], list(range(n))):
            assert g.spread(R, "uic", p, 3, S) == o.spread(R, 3, S, want_edges=True)


@pytest.mark.parametrize("n,R,k,p", [(255, 1, 1, 0.5), (257, 511, 6, 0.2), (256, 512, 6, 0.2), (300, 515, 300, 0.15),
                                     (40, 1030, 12, 1.0)])
def test_undirected_rounds(sg, n, R, k, p):
    """Rounds over more snapshots than one pass takes (512), to the last node."""
    n, s, d = inputs.symmetric(*inputs.random_small(n, 2 * n, 8))
    o = oracle.Graph(n, s, d, "uic_undirected", p)
    ref = o.select(R, k, 4, mode=oracle.COVER, want_init=True)
    with sg.Graph.from_coo(n, s, d) as g:
        res = g.select(R, k, "uic_undirected", p, 4, stats=True)
        assert np.array_equal(res.seeds, ref["seeds"]) and np.array_equal(res.gains, ref["gains"])
        assert [res.stats["init_edges"], res.stats["fwd_edges"]] == [int(x) for x in ref["counters"][:2]]
        assert np.array_equal(g.init_gains(R, "uic_undirected", p, 4)[0], ref["s_init"])


@pytest.mark.parametrize("p,R", [(1.0, 256), (0.5, 200)])
def test_dense_cascades_that_do_not_fit(sg, p, R):
    """Compact graphs that the allocator, or a server's budget, has no room for
    leave the query to the tiered engines, whose arrays do not grow with the
    live arcs: in a selection, in a captured batch and in a server."""
    import time

    import torch

    n, s, d = inputs.er_directed(2000, 20000, 6)
    ref = oracle.Graph(n, s, d, "uic", p).select(R, 4, 9, mode=oracle.COVER)
    held, refused = {}, []

    def alloc(nbytes, stream):
        if nbytes > 128 << 20:
            refused.append(nbytes)
            return None
        t = torch.empty(max(1, nbytes), dtype=torch.uint8, device="cuda")
        held[t.data_ptr()] = t
        return t.data_ptr()

    def release(ptr, nbytes, stream):
        torch.cuda.synchronize()
        held.pop(ptr, None)

    sg.sg_set_allocator(alloc, release)
    try:
        g = sg.Graph.from_coo(n, s, d)
        got = [g.select(R, 4, "uic", p, 9), g.select(R, 4, "uic", p, 9), g.select_celf(R, 4, "uic", p, 9)[0]]
        ws = sg.sg_workspace_create(g.handle, 64, 4)
        so = torch.zeros(4, dtype=torch.int32, device="cuda")
        go = torch.zeros(4, dtype=torch.int64, device="cuda")
        stream = torch.cuda.Stream()
        b = sg.sg_batch_capture([(g.handle, ws, R, 4, "uic", p, 9, so, go)], 1, stream)
        sg.sg_batch_launch(b, stream)
        stream.synchronize()
        got.append(sg.Selection(so.cpu().numpy(), go.cpu().numpy(), None))
        sg.sg_batch_free(b)
        sg.sg_workspace_free(ws)
        assert len(refused) == 2  # asked for once by each workspace
        g.close()
    finally:
        sg.sg_set_allocator(None, None)
    g = sg.Graph.from_coo(n, s, d)
    sv = sg.sg_server_create(2, sg.sg_workspace_bytes(g.handle, R, 128), 128)
    try:
        ids = [sg.sg_server_submit(sv, g.handle, R, 4, "uic", p, 9) for _ in range(3)]
        end = time.time() + 60
        while ids and time.time() < end:
            done, seeds, gains, _ = sg.sg_server_poll(sv, ids[0], 4)
            if not done:
                time.sleep(0.01)
                continue
            got.append(sg.Selection(seeds, gains, None))
            ids.pop(0)
        assert not ids
    finally:
        sg.sg_server_destroy(sv)
    g.close()
    for res in got:
        assert np.array_equal(res.seeds, ref["seeds"]) and np.array_equal(res.gains, ref["gains"])
