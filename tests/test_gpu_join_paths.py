"""The join's size rules at their edges, each against the CPU oracle: label directories of long lists, and the paths that
a step's tables take.  Whole numbers throughout, so the row sets are equal."""
import numpy as np
import pytest

import oracle
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


def same_rows(pkg, G, g, q, **kw):
    want = oracle.enumerate_rows(oracle.OracleGraph(g.vlab, g.src, g.dst, g.elab), q)
    r = G.query(q, **kw)
    assert r.count == want.shape[0]
    assert np.array_equal(oracle.sort_rows(r.rows()), want)
    assert G.query(q, count_only=True, **kw).count == want.shape[0]
    return want.shape[0]


@pytest.mark.parametrize("n_labels", [1, 3, 40])
@pytest.mark.parametrize("extra", [-1, 0, 1, 50])
def test_lists_around_the_directory_length(pkg, n_labels, extra):
    """Hubs whose lists are one short of, at and past 2 (labels + 1) entries, the length from which a directory is kept;
    labels with no neighbour at the start, in the middle and at the end of a list."""
    deg = 2 * (n_labels + 2) + extra                  # labels: n_labels of the leaves and one of the hubs
    n = 2 + 2 * deg
    edges = [(0, 2 + i) for i in range(deg)] + [(1, 2 + deg + i) for i in range(deg)]
    lab = [n_labels, n_labels] + [(i * 7) % n_labels for i in range(deg)] + [0 if i % 2 else n_labels - 1 for i in range(deg)]
    g = H.graph(n, edges, vlab=lab, elab=[0] * len(edges))
    assert np.unique(g.vlab).shape[0] == n_labels + 1 or extra < 0
    G = pkg.Graph(g.vlab, g.src, g.dst, g.elab)
    for r in {0, n_labels // 2, n_labels - 1}:
        q = H.query(2, [(0, 1)], [n_labels, r], [0])
        assert same_rows(pkg, G, g, q, order=[0, 1]) == int((g.vlab[2:] == r).sum())
        q = H.query(3, [(0, 1), (0, 2)], [n_labels, r, 0], [0, 0])
        same_rows(pkg, G, g, q, order=[0, 1, 2])
