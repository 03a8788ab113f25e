"""The two forms of the filter kernel, a query's and a batch's, beside the oracle: query vertices that use every word of a
signature, several to a label, and labels with few and with many vertices."""
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


@pytest.mark.parametrize("n_vlabels,n_elabels", [(1, 1), (3, 40), (40, 3)])
def test_batch_and_single_filter_agree_with_the_oracle(pkg, n_vlabels, n_elabels):
    n, rng = 2048, np.random.default_rng(91)
    v = np.repeat(np.arange(n), 6)                    # a circulant graph of degree 12: stars have few embeddings
    w = (v + np.tile([1, 2, 3, 5, 8, 13], n)) % n
    g = H.G(rng.integers(0, n_vlabels, n).astype(np.int32), np.minimum(v, w).astype(np.int32), np.maximum(v, w).astype(np.int32),
            rng.integers(0, n_elabels, 6 * n).astype(np.int32))
    most = 4 if n_vlabels * n_elabels == 1 else 9
    G = pkg.Graph(g.vlab, g.src, g.dst, g.elab)
    qs, words = [], set()
    for i in range(60):                               # a vertex and some of its neighbours: a star
        v = int(rng.integers(0, n))
        e = np.nonzero((g.src == v) | (g.dst == v))[0][: 1 + i % most]
        other = np.where(g.src[e] == v, g.dst[e], g.src[e])
        q = H.query(1 + e.size, [(0, j + 1) for j in range(e.size)], [g.vlab[v]] + g.vlab[other].tolist(), g.elab[e])
        qs.append(q)
        words |= set(np.nonzero(np.bitwise_or.reduce(pkg.query_signatures(q), axis=0))[0].tolist())
    if n_vlabels * n_elabels >= 120:
        assert words >= set(range(1, 16))             # each of the 15 words is someone's
    O = oracle.OracleGraph(g.vlab, g.src, g.dst, g.elab)
    for q in qs:
        member, want = oracle.filter_sets(O, q)
        bm, counts = G.filter(q)
        assert np.array_equal(counts, want)
        bits = np.unpackbits(bm.view(np.uint8), axis=1, bitorder="little")[:, :n]
        assert np.array_equal(bits.astype(bool), member)
    # a batch of more than 32 query vertices takes the other form: a candidate that it drops is missing from the counts
    for q, r in zip(qs, G.batch(qs, count_only=True)):
        assert r.count == oracle.count(O, q)[0]
    # one-vertex queries have their candidate sets as their results
    ones = [H.query(1, [], [int(x)]) for x in np.unique(g.vlab)] * 40
    for q, r in zip(ones, G.batch(ones)):
        assert r.count == int((g.vlab == q.vlab[0]).sum())
    G.close()
