"""Tables of as many rows as the row pass deals in turn, one row fewer and more, and so many that the rest is dealt on
demand: every row is joined once."""
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


ROUND = 152 * 4 * 512                                 # rows of one round of full batches


@pytest.mark.parametrize("rows", [2 * ROUND - 1, 2 * ROUND, 2 * ROUND + 1, 3 * ROUND + 1, 4 * ROUND, 7 * ROUND + 13])
def test_every_row_of_a_table_past_the_dealt_rounds_is_joined_once(pkg, rows):
    """`rows` vertices of label 0 with one to three neighbours of label 1: the first step's table has a row for each, its
    result is the list of the edges, and the second step's pairs of neighbours are d (d - 1) to a vertex."""
    right = 5003
    deg = 1 + np.arange(rows) % 3
    a = np.repeat(np.arange(rows), deg).astype(np.int32)
    b = (rows + (a.astype(np.int64) * 7 + np.arange(a.size) - np.repeat(np.cumsum(deg) - deg, deg)) % right).astype(np.int32)
    vlab = np.concatenate([np.zeros(rows), np.ones(right)]).astype(np.int32)
    G = pkg.Graph(vlab, a, b, np.zeros(a.size, np.int32))
    q = H.query(2, [(0, 1)], [0, 1], [0])
    r = G.query(q, order=[0, 1])
    got = r.rows()
    r.close()
    key = np.sort(got[:, 0].astype(np.int64) * (1 << 32) + got[:, 1])
    assert np.array_equal(key, np.sort(a.astype(np.int64) * (1 << 32) + b))
    q = H.query(3, [(0, 1), (0, 2)], [0, 1, 1], [0, 0])
    want = int((deg * (deg - 1)).sum())
    r = G.query(q, order=[0, 1, 2])
    got = r.rows()
    assert r.count == want and got.shape[0] == want
    assert np.array_equal(np.bincount(got[:, 0], minlength=rows), deg * (deg - 1))
    assert (got[:, 1] != got[:, 2]).all()
    r.close()
    assert G.query(q, order=[0, 1, 2], count_only=True).count == want
    G.close()
