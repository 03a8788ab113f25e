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
    G = pkg.Graph(g.vlab, g.src, g.dst, g.elab)
    for r in {0, n_labels // 2, n_labels - 1}:
        q = H.query(2, [(0, 1)], [n_labels, r], [0])
        assert same_rows(pkg, G, g, q, order=[0, 1]) == int((g.vlab[2:] == r).sum())
        q = H.query(3, [(0, 1), (0, 2)], [n_labels, r, 0], [0, 0])
        same_rows(pkg, G, g, q, order=[0, 1, 2])


@pytest.mark.parametrize("degrees", [[16], [17], [1, 15, 16, 17, 18, 31, 63, 64, 65], [255, 256, 257, 17, 300, 2, 400]])
def test_long_rows_around_the_tile_edges(pkg, degrees):
    """Rows with as many candidates as the short rows' limit, the tile's slots and a warp's share, one more and one less;
    every (hub, leaf) row of the second step is a long one again."""
    edges, n = [], len(degrees)
    for h, d in enumerate(degrees):
        edges += [(h, n + i) for i in range(d)]
        n += d
    g = H.graph(n, edges, vlab=[0] * len(degrees) + [1] * (n - len(degrees)), elab=[0] * len(edges))
    G = pkg.Graph(g.vlab, g.src, g.dst, g.elab)
    q = H.query(3, [(0, 1), (0, 2)], [0, 1, 1], [0, 0])
    for order in ([0, 1, 2], [1, 0, 2]):
        assert same_rows(pkg, G, g, q, order=order) == sum(d * (d - 1) for d in degrees)
    assert G.query(q, semantics=pkg.GSI_HOMOMORPHISM, count_only=True).count == sum(d * d for d in degrees)
    r = G.query(q, row_cap=33)
    assert r.count == sum(d * (d - 1) for d in degrees) and r.rows(33).shape[0] == min(33, r.count)


@pytest.mark.parametrize("n", [40, 130])
def test_long_rows_with_several_lists(pkg, n):
    """Dense graph: the closing steps have two and three linking edges and more than 16 candidates each."""
    g = H.random_graph(np.random.default_rng(n), n, 0.55, 1, 1)
    G = pkg.Graph(g.vlab, g.src, g.dst, g.elab)
    same_rows(pkg, G, g, H.clique_query(3))
    if n < 100:
        same_rows(pkg, G, g, H.clique_query(4))
        same_rows(pkg, G, g, H.query(4, [(0, 1), (1, 2), (2, 3), (3, 0)]))


@pytest.mark.parametrize("k", [9, 31, 32])
def test_long_rows_of_many_columns(pkg, k):
    """A chain of k - 1 vertices that ends in a hub with 40 leaves: the widest rows a long step can have."""
    edges = [(i, i + 1) for i in range(k - 2)] + [(k - 2, k - 1 + i) for i in range(40)]
    g = H.graph(k - 1 + 40, edges, vlab=list(range(k - 1)) + [99] * 40, elab=[0] * len(edges))
    G = pkg.Graph(g.vlab, g.src, g.dst, g.elab)
    q = H.query(k, [(i, i + 1) for i in range(k - 1)], list(range(k - 1)) + [99], [0] * (k - 1))
    assert same_rows(pkg, G, g, q, order=list(range(k))) == 40
    assert same_rows(pkg, G, g, q) == 40


@pytest.mark.parametrize("rows", [1, 7, 8, 9, 607, 608 * 8, 608 * 8 + 1, 608 * 512 + 3])
def test_tables_that_fill_some_or_all_of_the_grid(pkg, rows):
    """One edge per row, so that the second table has `rows` rows: a batch of 8 rows, several, and full batches."""
    n = 3 * rows
    edges = [(i, rows + i) for i in range(rows)] + [(rows + i, 2 * rows + i) for i in range(rows)]
    lab = [0] * rows + [1] * rows + [2] * rows
    G = pkg.Graph(lab, [a for a, _ in edges], [b for _, b in edges], [0] * len(edges))
    q = H.query(3, [(0, 1), (1, 2)], [0, 1, 2], [0, 0])
    r = G.query(q)
    got = r.rows()
    got = got[np.argsort(got[:, 0])]
    want = np.arange(rows, dtype=np.int32)[:, None] + np.array([0, rows, 2 * rows], np.int32)
    assert r.count == rows and np.array_equal(got, want)


@pytest.mark.parametrize("t,d,rows,shift", [(1, 1, 63, 0), (1, 1, 5000, 1), (2, 2, 64, 3), (3, 3, 4097, 0), (6, 5, 9001, 1),
                                            (31, 7, 700, 2), (4, 2, 40_000, 0)])
def test_step_in_one_launch_against_the_scan_path(pkg, t, d, rows, shift):
    """A step over the caller's table, with fewer and with more rows than vertices (with and without a memo), more lists than
    the memo has, buffers off a 16-byte boundary, and out_cap short, exact and zero: the allocation-free call still
    takes the scan and the slot tiles."""
    import torch
    rng = np.random.default_rng(1000 * t + d)
    g = H.random_graph(rng, 220, 0.45, 2, 2)
    G = pkg.Graph(g.vlab, g.src, g.dst, g.elab)
    flat = torch.zeros(shift + rows * t, dtype=torch.int32, device="cuda")
    flat[shift:] = torch.from_numpy(rng.integers(0, 220, rows * t).astype(np.int32)).cuda()
    ptr = flat.data_ptr() + 4 * shift
    cand = torch.from_numpy(rng.integers(-2**31, 2**31, 7).astype(np.int32)).cuda()
    cols, labs = sorted(rng.choice(t, d, replace=False).tolist()), rng.integers(0, 2, d).tolist()
    full = G.join_step_noalloc(ptr, rows, t, cand.data_ptr(), 1, cols, labs, 0, 0)
    assert G.join_step(ptr, rows, t, cand.data_ptr(), 1, cols, labs, 0, 0) == full

    def out_of(call, cap):
        out = torch.full((shift + cap * (t + 1) + 1,), -7, dtype=torch.int32, device="cuda")
        assert call(ptr, rows, t, cand.data_ptr(), 1, cols, labs, out.data_ptr() + 4 * shift, cap) == full
        torch.cuda.synchronize()
        assert int(out[-1]) == -7                     # nothing past the last row
        return out[shift:-1].cpu().numpy().reshape(cap, t + 1)

    want = oracle.sort_rows(out_of(G.join_step_noalloc, full))
    assert np.array_equal(oracle.sort_rows(out_of(G.join_step, full)), want)
    short = out_of(G.join_step, full // 2)
    have = {r.tobytes() for r in np.ascontiguousarray(want)}
    assert all(r.tobytes() in have for r in np.ascontiguousarray(short))
