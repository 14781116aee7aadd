"""The tuning cache: lines of builds without the default route's compact
graphs, and results measured while those had no room, are not returned."""

import pytest

from paper_1212_4779_gb300 import inputs

pytestmark = pytest.mark.gpu

LINE = ('{"key": "n=%d m=%d dmax=%d model=%d p=%.6f W=%d", "walk_groups": 32, "direction_mode": 1, '
        '"direction_div": 4, "tier1_keys": 64, "tier2_keys": 2048, "landmarks": 8, "scc": 1, "forward_lists": 1, '
        '"word_major": 1, "tier1_direct": 16, "ms": 0.001}\n')


@pytest.fixture(scope="module")
def sg():
    import __graft_entry__

    __graft_entry__.build()
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1212_4779_gb300 import sg as _sg

    return _sg


def test_lines_without_a_route_are_not_returned(sg, tmp_path):
    n, s, d = inputs.er_directed(500, 2500, 3)
    path = tmp_path / "tuning.jsonl"
    with sg.Graph.from_coo(n, s, d) as g:
        rp, col = g.csr()
        path.write_text(LINE % (n, col.size, int((rp[1:] - rp[:-1]).max()), 0, 0.1, 2))
        t, ms = sg.sg_autotune(g.handle, 100, 5, "uic", 0.1, 3, cache_path=str(path))
        assert ms > 0.01  # timed, not read
        assert len(path.read_text().splitlines()) == 2
        t2, ms2 = sg.sg_autotune(g.handle, 100, 5, "uic", 0.1, 3, cache_path=str(path))
        assert t2.as_dict() == t.as_dict() and abs(ms2 - ms) < 1e-2
        assert len(path.read_text().splitlines()) == 2


def test_results_without_room_are_not_kept(sg, tmp_path):
    import torch

    n, s, d = inputs.er_directed(2000, 20000, 6)
    path = tmp_path / "tuning.jsonl"
    held = {}

    def alloc(nbytes, stream):
        if nbytes > 128 << 20:
            return None
        t = torch.empty(max(1, nbytes), dtype=torch.uint8, device="cuda")
        held[t.data_ptr()] = t
        return t.data_ptr()

    def release(ptr, nbytes, stream):
        torch.cuda.synchronize()
        held.pop(ptr, None)

    sg.sg_set_allocator(alloc, release)
    try:
        with sg.Graph.from_coo(n, s, d) as g:
            _, ms = sg.sg_autotune(g.handle, 200, 2, "uic", 0.5, 3, cache_path=str(path))
            assert ms > 0 and (not path.exists() or path.read_text() == "")
    finally:
        sg.sg_set_allocator(None, None)
    with sg.Graph.from_coo(n, s, d) as g:
        sg.sg_autotune(g.handle, 200, 2, "uic", 0.5, 3, cache_path=str(path))
    assert len(path.read_text().splitlines()) == 1
