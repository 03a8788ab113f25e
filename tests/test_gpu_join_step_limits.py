"""gsi_join_step at the limits of its arguments and of its one-launch path: whole numbers, equal to the allocation-free
call and, where it is small, to the oracle."""
import numpy as np
import pytest

import oracle
import synth
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


@pytest.fixture(scope="module")
def step(pkg):
    """A graph with hubs, and a function that makes a step's arguments for tables of t columns and d linking edges."""
    import torch
    s, d = synth.rmat(78, 12, 30_000)
    n = 1 << 12
    g = H.G(synth.labels_zipf(78, 1, n, 6, 1.1), s, d, synth.labels_uniform(78, 2, 30_000, 3))
    G = pkg.Graph(g.vlab, g.src, g.dst, g.elab)
    rng = np.random.default_rng(78)

    def make(R, t, links):
        M = rng.integers(0, n, (R, t)).astype(np.int32)
        member = rng.random(n) < 0.7
        bits = np.packbits(np.pad(member, (0, -n % 32)), bitorder="little").view(np.int32)
        return (torch.from_numpy(M).cuda(), torch.from_numpy(bits.copy()).cuda(), list(range(links)),
                [j % 3 for j in range(links)])

    return G, make


def run(fn, args, room, cap):
    """The call's count and the rows it wrote into a buffer of `room` rows, called with `cap` as its size."""
    import torch
    M, cand, cols, labs = args
    out = torch.full((room, M.shape[1] + 1), -1, dtype=torch.int32, device="cuda")
    n = fn(M.data_ptr(), M.shape[0], M.shape[1], cand.data_ptr(), 0, cols, labs, out.data_ptr(), cap)
    torch.cuda.synchronize()
    return n, out.cpu().numpy()


@pytest.mark.parametrize("t", [1, 3, 7])
@pytest.mark.parametrize("cap", [1 << 61, 1 << 62, (1 << 62) + 1, 1 << 63, (1 << 64) - 1])
def test_a_row_limit_past_every_buffer_writes_all_rows(step, t, cap):
    """The row limit times the row size passes 2^64 (at 2^62 rows of 4 columns it is 0 modulo 2^64): every row is written."""
    G, make = step
    args = make(2000, t, min(t, 2))
    n, none = run(G.join_step_noalloc, args, 1, 0)
    assert n > 0
    want, rows = run(G.join_step_noalloc, args, n, n)
    got, out = run(G.join_step, args, n, cap)
    assert got == want == n
    assert np.array_equal(oracle.sort_rows(out), oracle.sort_rows(rows))


@pytest.mark.parametrize("rows,t,links", [(1, 1, 1), (2000, 1, 1), (2000, 3, 2), (2000, 7, 7), (400_003, 2, 2)])
@pytest.mark.parametrize("counted", [False, True])
def test_a_barrier_that_gave_up_leaves_the_step_to_the_scan(step, rows, t, links, counted):
    """The cooperative launch finds its barrier given up; the call still returns every row, or their number."""
    G, make = step
    args = make(rows, t, links)
    n, _ = run(G.join_step_noalloc, args, 1, 0)
    cap = 0 if counted else n
    want, rows_want = run(G.join_step_noalloc, args, max(n, 1), cap)
    got, out = run(G.selftest_join_step, args, max(n, 1), cap)
    assert got == want == n
    assert np.array_equal(oracle.sort_rows(out), oracle.sort_rows(rows_want))
    got, out = run(G.join_step, args, max(n, 1), cap)
    assert got == n and np.array_equal(oracle.sort_rows(out), oracle.sort_rows(rows_want))
