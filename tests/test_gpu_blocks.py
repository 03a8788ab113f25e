"""Arena blocks kept between calls, on the device: threads on streams of their own that share them, a query that is redone
with larger arenas, results that outlive their graph, and giving them back.  Whole numbers, equal to the counts alone."""
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


def complete(n):
    """All pairs of n vertices, one label."""
    a, b = np.triu_indices(n, 1)
    return H.G(np.zeros(n, np.int32), a.astype(np.int32), b.astype(np.int32), np.zeros(a.size, np.int32))


PATH = H.query(3, [(0, 1), (1, 2)], [0, 0, 0], [0, 0])


def test_threads_share_blocks_while_one_query_outgrows_its_first_arena(pkg):
    """1000 * 999 * 998 rows of three columns (12 GB) pass the first arena's table region (5.7 GB), so that query gives its
    blocks back and starts again with larger ones, while two other threads take and give back blocks of the first size."""
    import torch
    big, small = complete(1000), complete(60)
    GB, GS = pkg.Graph(big.vlab, big.src, big.dst, big.elab), pkg.Graph(small.vlab, small.src, small.dst, small.elab)
    want = {1000: 1000 * 999 * 998, 60: 60 * 59 * 58}
    wrong = []

    def work(G, n, times):
        stream = torch.cuda.Stream()
        for _ in range(times):
            r = G.query(PATH, stream=stream)
            rows = 1000 if n == 1000 else r.count
            got = torch.empty((rows, 3), dtype=torch.int32, device="cuda")
            r.copy_to(got.data_ptr(), rows)
            ok = (got >= 0).all() & (got < n).all() & (got[:, 0] != got[:, 1]).all() & (got[:, 1] != got[:, 2]).all() \
                & (got[:, 0] != got[:, 2]).all()
            distinct = torch.unique(got, dim=0).shape[0]
            if r.count != want[n] or not bool(ok) or distinct != rows:
                wrong.append((n, r.count, bool(ok), distinct))
            r.close()

    threads = [threading.Thread(target=work, args=a) for a in [(GB, 1000, 3), (GS, 60, 40), (GS, 60, 40)]]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong
    GB.close()
    GS.close()


def test_result_outlives_its_graph(pkg):
    g = complete(60)
    G = pkg.Graph(g.vlab, g.src, g.dst, g.elab)
    r = G.query(PATH)
    G.close()
    rows = r.rows()
    assert rows.shape == (60 * 59 * 58, 3) and np.unique(rows, axis=0).shape == rows.shape
    r.close()
    G = pkg.Graph(g.vlab, g.src, g.dst, g.elab)
    assert G.query(PATH).count == 60 * 59 * 58
    G.close()


def test_trim_gives_back_what_is_kept_and_only_that(pkg):
    g = complete(60)
    G = pkg.Graph(g.vlab, g.src, g.dst, g.elab)
    pkg.memory_trim()
    held = G.query(PATH, mem_budget=1 << 30)
    assert pkg.memory_trim() >= 600 << 20             # two of the three blocks of a third of the budget each
    assert pkg.memory_trim() == 0
    assert held.rows().shape[0] == 60 * 59 * 58       # the third is the result's
    held.close()
    assert pkg.memory_trim() >= 300 << 20
    assert G.query(PATH, mem_budget=1 << 30, count_only=True).count == 60 * 59 * 58
    G.close()
    assert pkg.memory_trim() == 0                     # nothing is kept without a graph


def test_a_query_does_not_wait_for_another_streams_work(pkg):
    """A result goes back while a host function holds up its stream. A query of the same size on another stream goes on."""
    import ctypes
    import torch
    g = complete(60)
    G = pkg.Graph(g.vlab, g.src, g.dst, g.elab)
    held_up, other = torch.cuda.Stream(), torch.cuda.Stream()
    pkg.memory_trim()
    results = [G.query(PATH, stream=held_up, mem_budget=1 << 30) for _ in range(3)]
    pkg.memory_trim()                                 # nothing is kept but what these give back
    free, began, count = threading.Event(), threading.Event(), []
    hold = ctypes.CFUNCTYPE(None, ctypes.c_void_p)(lambda _: (began.set(), free.wait(60)) and None)
    assert ctypes.CDLL("libcudart.so.13").cudaLaunchHostFunc(ctypes.c_void_p(held_up.cuda_stream), hold, None) == 0
    began.wait(10)
    for r in results:
        r.close()
    t = threading.Thread(target=lambda: count.append(G.query(PATH, stream=other, mem_budget=1 << 30, count_only=True).count))
    t.start()
    t.join(10)
    went_on = not t.is_alive()
    free.set()
    t.join(60)
    assert went_on and count == [60 * 59 * 58]
    torch.cuda.synchronize()
    G.close()
