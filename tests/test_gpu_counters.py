"""The byte counters of gsi_stats against counts made by hand from the graph."""
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


def stats_of(pkg, G, q, **kw):
    st = pkg.c_stats()
    n = G.query(q, stats=st, **kw).count
    return n, st


def test_filter_bytes_are_the_words_that_the_query_uses(pkg):
    """Ids and used signature words of each label's group (whole warps), and the bitmaps: labels that share words of the query
    vertices read them once."""
    n = 1000
    edges = [(i, i + 1) for i in range(n - 1)]
    vlab = [i % 3 for i in range(n)]
    g = H.graph(n, edges, vlab=vlab, elab=[i % 2 for i in range(n - 1)])
    G = pkg.Graph(g.vlab, g.src, g.dst, g.elab)
    for k in (2, 3, 5):
        q = H.query(k, [(i, i + 1) for i in range(k - 1)], [i % 3 for i in range(k)], [i % 2 for i in range(k - 1)])
        sig = pkg.query_signatures(q)
        want = k * ((n + 31) // 32) * 4
        for label in set(q.vlab.tolist()):
            words = np.bitwise_or.reduce(sig[q.vlab == label], axis=0)[1:]
            size = int((g.vlab == label).sum())
            want += (size + 31) // 32 * 32 * 4 * (1 + int(np.count_nonzero(words)))
        _, st = stats_of(pkg, G, q)
        assert st.filter_bytes == want
        res = G.batch([q] * 40, stats=(bst := pkg.c_stats()))
        assert len(res) == 40
        assert bst.filter_bytes == want + 39 * k * ((n + 31) // 32) * 4


def test_a_hub_list_that_rows_share_is_counted_once(pkg):
    """A hub (label 0) with 50 arms (label 1) and 3,000 leaves (label 2).  Counting arm - hub - leaf, the last step has 50 rows
    that meet the hub's list of 3,000 leaves, which is read once: a row's list entry and its memo entry, not 50 lists."""
    arms, leaves = 50, 3000
    n = 1 + arms + leaves
    g = H.graph(n, [(0, i) for i in range(1, n)], vlab=[0] + [1] * arms + [2] * leaves, elab=[0] * (n - 1))
    G = pkg.Graph(g.vlab, g.src, g.dst, g.elab)
    q = H.query(3, [(0, 1), (1, 2)], [1, 0, 2], [0, 0])
    count, st = stats_of(pkg, G, q, count_only=True, order=[0, 1, 2])
    assert count == arms * leaves and st.join_items == arms + arms * leaves
    # step 1: each arm's row of one column, its list located (16) and its one candidate with its bitmap word (8), and the row
    # of two columns that it leaves; step 2: each row and the memo entry (8), at least one list located (at most one by each
    # row, as the rows meet the hub together), and the leaves with their bitmap words once
    least = arms * (4 + 16 + 8 + 8) + arms * (8 + 8) + 16 + 8 * leaves
    assert least <= st.join_bytes <= least + (arms - 1) * 16


def test_entries_that_the_memo_keeps_are_counted_without_their_bitmap_words(pkg):
    """Rows that meet a short list again read the memo entry (8) and the entries that it keeps (4 each); only a CTA's first
    rows can meet it for the first time, with its place (16) and a bitmap word beside each entry (8)."""
    arms, leaves = 1_000_000, 8
    n = 1 + arms + leaves
    vlab = np.concatenate([[0], np.full(arms, 1), np.full(leaves, 2)]).astype(np.int32)
    G = pkg.Graph(vlab, np.zeros(n - 1, np.int32), np.arange(1, n, dtype=np.int32), np.zeros(n - 1, np.int32))
    q = H.query(3, [(0, 1), (1, 2)], [1, 0, 2], [0, 0])
    count, st = stats_of(pkg, G, q, order=[0, 1, 2])
    assert count == arms * leaves
    written = arms * 8 + count * 12
    first = arms * (4 + 16 + 8)                       # step 1: no vertex twice, one candidate each
    again, new = 8 + 8 + 4 * leaves, 8 + 16 + 8 * leaves
    least = written + first + arms * again
    assert least <= st.join_bytes <= least + 608 * 512 * (new - again)
