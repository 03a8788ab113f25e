"""A graph built on a stream that is held up does not hold up work on other streams."""
import ctypes
import threading

import numpy as np
import pytest

from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_1906_03420_gb300 as p
    p.load()
    torch.cuda.init()
    return p


def test_a_build_on_a_stream_that_waits_leaves_others_alone(pkg):
    """A host function keeps one stream waiting while a thread builds a graph of 2^20 edges there (large enough to copy its
    edges beside the sorts).  Replays of a prepared batch, whose results are released on the library's own stream and whose
    next results take the same memory, go on meanwhile."""
    import torch
    n = 1100
    a, b = np.triu_indices(n, 1)                      # 604,450 pairs: two copies of the graph side by side make 2^20
    a, b = np.concatenate([a, a + n])[: 1 << 20], np.concatenate([b, b + n])[: 1 << 20]
    big = H.G(np.zeros(2 * n, np.int32), a.astype(np.int32), b.astype(np.int32), np.zeros(1 << 20, np.int32))
    s, t = np.triu_indices(40, 1)
    G = pkg.Graph(np.zeros(40, np.int32), s.astype(np.int32), t.astype(np.int32), np.zeros(s.size, np.int32))
    path = H.query(3, [(0, 1), (1, 2)], [0, 0, 0], [0, 0])
    batch = pkg.PreparedBatch(G, [path] * 4, mem_budget=2 << 30)

    def replay():
        res = batch.run()
        counts = [r.count for r in res]
        for r in res:
            r.close()
        return counts

    want = [40 * 39 * 38] * 4
    assert replay() == want
    cudart = ctypes.CDLL("libcudart.so.13")
    free, stop = threading.Event(), threading.Event()
    hold = ctypes.CFUNCTYPE(None, ctypes.c_void_p)(lambda _: free.wait(60) and None)
    stream, made, got = torch.cuda.Stream(), [], []
    started = threading.Event()

    def build():
        started.set()
        made.append(pkg.Graph(big.vlab, big.src, big.dst, big.elab, stream=stream))

    def replays():
        while not stop.is_set() and len(got) < 20:
            got.append(replay())

    assert cudart.cudaLaunchHostFunc(ctypes.c_void_p(stream.cuda_stream), hold, None) == 0
    builder, other = threading.Thread(target=build), threading.Thread(target=replays)
    builder.start()
    started.wait()
    builder.join(0.5)                                 # it has come to its first wait
    assert builder.is_alive()
    other.start()
    other.join(10)
    went_on = not other.is_alive()
    held_up = builder.is_alive()
    stop.set()
    free.set()
    builder.join(60)
    other.join(60)
    assert held_up and went_on and got == [want] * 20
    assert made[0].info().m == 1 << 20
    made[0].close()
    batch.close()
    G.close()
