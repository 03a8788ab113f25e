"""The graph build where its passes change: label ranges and counts that need none, one or several sort digits, entries at
the ends of sort tiles and warps, and repeated pairs of labels, against numpy."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _expect(vlab, src, dst, elab):
    """off, ci, cl and the label frequencies as plain numpy sorts them."""
    n, L = len(vlab), int(elab.max()) + 1 if len(elab) else 1
    uniq, rank = np.unique(vlab, return_inverse=True)
    v, w, l = np.concatenate([src, dst]), np.concatenate([dst, src]), np.concatenate([elab, elab])
    order = np.lexsort((w, rank[w], l, v))
    off = np.concatenate([[0], np.cumsum(np.bincount(v.astype(np.int64) * L + l, minlength=n * L))])
    return off, w[order], rank[w][order], np.bincount(elab, minlength=L)


def _edges(rng, n, m):
    """m distinct pairs, in random order and direction."""
    e = np.unique(rng.integers(0, n, (3 * m + 16, 2)), axis=0)
    e = e[e[:, 0] < e[:, 1]]
    e = e[rng.permutation(len(e))[:m]]
    flip = rng.random(len(e)) < 0.5
    e[flip] = e[flip][:, ::-1]
    return e[:, 0].astype(np.int32), e[:, 1].astype(np.int32)


# vertices, edges, edge labels, and the vertex labels: one value; a few; a range of several digits, with negative ones
@pytest.mark.parametrize("n,m,L,labels", [
    (2, 1, 1, "one"), (33, 31, 3, "few"), (1000, 4095, 1, "few"), (1000, 4096, 8, "one"), (1001, 4097, 5, "wide"),
    (3000, 8191, 2, "wide"), (40_000, 70_001, 7, "few"), (70_000, 50_000, 1500, "few"), (66_000, 3000, 4, "many"),
])
def test_build_against_numpy(n, m, L, labels):
    import oracle
    import paper_1906_03420_gb300 as pkg

    rng = np.random.default_rng(n + m)
    vlab = {"one": lambda: np.full(n, 7), "few": lambda: rng.integers(0, 5, n),
            "wide": lambda: rng.choice([-2**31, -5, 0, 3, 2**20, 2**31 - 1], n),
            "many": lambda: rng.permutation(np.arange(n) % 65_000)}[labels]().astype(np.int32)
    src, dst = _edges(rng, n, m)
    elab = rng.integers(0, L, len(src)).astype(np.int32)
    elab[0] = L - 1
    g = pkg.Graph(vlab, src, dst, elab)
    off, ci, cl, freq = _expect(vlab, src, dst, elab)
    a = g.export()
    assert np.array_equal(a[0].astype(np.int64), off)
    assert np.array_equal(a[1], ci) and np.array_equal(a[2], cl)
    assert np.array_equal(g.label_freq(), freq.astype(np.uint64))
    assert np.array_equal(a[3].T, oracle.data_signatures(oracle.OracleGraph(vlab, src, dst, elab)))
    g.close()


def test_hub_pairs_and_repeats():
    """A star of one pair (both state bits from one run), and a pair given twice under two labels (refused)."""
    import paper_1906_03420_gb300 as pkg

    n = 9000
    vlab = np.zeros(n, np.int32)
    src, dst = np.zeros(n - 1, np.int32), np.arange(1, n, dtype=np.int32)
    g = pkg.Graph(vlab, src, dst, np.zeros(n - 1, np.int32))
    sig = g.export()[3]
    bits = [bin(int(x)).count("1") for x in np.bitwise_or.reduce(sig[1:, :2], axis=0)]
    assert bits == [2, 1]
    g.close()
    with pytest.raises(pkg.GsiError):
        pkg.Graph(vlab, np.r_[src, 5].astype(np.int32), np.r_[dst, 0].astype(np.int32), np.r_[np.zeros(n - 1), 3].astype(np.int32))
