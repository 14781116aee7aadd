"""Entry points called from several host threads at once, each with a graph of
its own: every call must succeed and return what it returns alone."""

import threading

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


@pytest.mark.parametrize("model,p", [("uic", 0.5), ("wic", 0.0)])
def test_spread_of_a_small_and_a_large_graph(sg, model, p):
    """A launch's shared memory grows with its graph: 16 bytes of visited bits
    on three of the threads, 150 KB on the other."""
    n, s, d = inputs.er_directed(100, 400, 1)
    want = [oracle.Graph(n, s, d, model, p).spread(3, 7, [0, 5], want_edges=True)]
    big = 1200000
    s2, d2 = (s.astype(np.int64) * 11999).astype(np.int32), (d.astype(np.int64) * 11999).astype(np.int32)
    want.append(oracle.Graph(big, s2, d2, model, p).spread(3, 7, [0, 5 * 11999], want_edges=True))
    failed = []
    with sg.Graph.from_coo(n, s, d) as small, sg.Graph.from_coo(big, s2, d2) as large:
        def work(g, S, ref):
            import torch

            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                for _ in range(3000):
                    try:
                        if g.spread(3, model, p, 7, S) != ref:
                            failed.append("result")
                    except sg.SGError as e:
                        failed.append(str(e))

        ts = [threading.Thread(target=work, args=a)
              for a in [(small, [0, 5], want[0])] * 3 + [(large, [0, 5 * 11999], want[1])]]
        for t in ts:
            t.start()
        for t in ts:
            t.join()
    assert not failed, (len(failed), failed[:3])
