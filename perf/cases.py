"""What this library is timed on: its public entry points over the range of graphs and queries it is used with.

A case is a labelled data graph (R-MAT or Erdos-Renyi), random-walk queries drawn from it, and one way of asking them: a
single query, a batch, a prepared batch, a server, an edge-isomorphism query, or one of the step-level calls (filter, join
step, graph build).  Graphs and queries are made on the GPU from the seed alone.  As in the paper's setup (Sec. VIII-A) a
query is a walk's visited vertices with the walk's edges (sparse) or with more edges among them, up to 2k (dense); a walk
whose labelled spanning tree has more homomorphisms than the case's bound is not taken, which stands in for a time limit.

The order of a result's rows is unspecified, so a pass gathers the rows of all its queries in one table of the caller's, in
the order of a hash of each row.  The table has room for `cap` rows (a query with more than its share is not taken) and
holds -1 where no row is.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1906_03420_gb300 as gsi

_COMMON = dict(graph="rmat", n=1 << 20, m=16_000_000, nvl=64, nel=8, queries=1, k_lo=6, k_hi=12, dense=1, bound=1e6,
               rare=0, cap=0, count_only=False, hom=False, split=False, budget_mb=0, rows=0, t=0, links=1, noalloc=False, host=False)


def _case(kind, **kw):
    return {"kind": kind, **_COMMON, **kw}


def listed():
    return [
        # One small lookup on a small graph, its rows on the host (a service's smallest call): launches and latency are what
        # it costs.
        _case("query", name="tiny_query", graph="er", n=1000, m=5000, nvl=4, nel=4, k_lo=4, k_hi=4, bound=1e5,
              cap=4096, host=True),
        # The candidate sets of one query alone, on the host: index lookups before a search.
        _case("filter", name="filter_k10", k_lo=10, k_hi=10, bound=1e300),
        # Single queries with their rows, one after another: the everyday use on a social-network-like graph.
        _case("query", name="rows_medium", queries=4, bound=3e7, cap=1 << 21),
        # Large counting queries, sparse and dense in turn: motif counting, the heaviest tables on the same graph.
        _case("query", name="count_medium", queries=8, dense=2, bound=1e8, count_only=True),
        # A graph four times larger with twice the labels: lists and tables far outside of L2.
        _case("query", name="count_large", n=1 << 22, m=64_000_000, nvl=128, queries=4, k_lo=8, k_hi=14, dense=2,
              bound=1e9, count_only=True),
        # Homomorphisms (Sec. VII-A) on a ragged graph: pattern matching as graph databases ask for it.
        _case("query", name="hom_ragged", graph="rmat", n=300_007, m=3_000_001, nvl=20, nel=5, queries=4, k_lo=3, k_hi=7,
              dense=2, bound=2e6, cap=1 << 20, hom=True),
        # One join step on a table that the caller holds (a plugin of another engine), two linking edges or more.
        _case("step", name="step_3m", rows=3_000_017, t=4, k_lo=5, k_hi=5, bound=3e7, links=2),
        # A batch of small requests with all their rows, planned and run in one call.
        _case("batch", name="batch_rows", queries=96, k_lo=4, k_hi=16, dense=2, bound=1e5, rare=8, cap=1 << 20,
              budget_mb=24576),
        # A prepared batch replayed: the same patterns counted again and again (monitoring).
        _case("replay", name="replay_768", queries=768, k_lo=4, k_hi=16, dense=2, bound=1e6, rare=8, count_only=True,
              budget_mb=24576),
        # A burst of requests to the server, each one's rows read back.
        _case("serve", name="serve_burst", queries=200, k_lo=4, k_hi=16, dense=2, bound=1e5, rare=8, cap=1 << 20,
              budget_mb=16384),
        # Edge isomorphism through the line graph of a low-degree graph (road networks, molecules).
        _case("edge", name="edge_er", graph="er", n=1 << 17, m=500_000, nvl=4, nel=2, queries=4, k_lo=4, k_hi=6, dense=2,
              bound=1e5, cap=1 << 19),
        # Loading a graph: what every user pays first.
        _case("build", name="build_16m"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["query", "query", "query", "filter", "step", "batch", "replay", "serve", "edge", "build"])
    if kind == "edge":
        n = _log(rng, 1 << 12, 1 << 17)
        c = _case(kind, graph="er", n=n, m=int(n * rng.uniform(2.0, 3.8)), nvl=rng.randint(3, 8), nel=rng.randint(1, 4),
                  queries=rng.randint(1, 4), k_lo=3, k_hi=rng.randint(4, 6), dense=rng.randint(0, 2),
                  bound=float(_log(rng, 1e3, 1e5)), cap=1 << 19)
        return c
    n = _log(rng, 1 << 12, 1 << 20)
    c = _case(kind, graph=rng.choice(["rmat", "rmat", "rmat", "er"]), n=n, m=int(n * rng.uniform(4.0, 15.0)) | 1,
              nvl=_log(rng, 16, 128), nel=rng.randint(3, 12), dense=rng.randint(0, 2))
    c["k_lo"] = rng.randint(3, 8)
    c["k_hi"] = min(16, c["k_lo"] + rng.randint(0, 6))
    if kind == "query":
        c["queries"] = rng.randint(1, 6)
        c["count_only"] = rng.random() < 0.5
        c["hom"] = rng.random() < 0.2
        c["bound"] = float(_log(rng, 1e4, 5e7 if c["count_only"] else 3e6))
        c["cap"] = 0 if c["count_only"] else 1 << 20
        if rng.random() < 0.2:                        # a small memory budget: the splitting driver
            c["split"], c["bound"], c["budget_mb"] = True, float(_log(rng, 1e4, 3e6)), _log(rng, 64, 1024)
    elif kind == "filter":
        c["bound"] = 1e300
    elif kind == "step":
        c["t"] = rng.randint(1, 8)
        c["k_lo"] = c["k_hi"] = c["t"] + 1
        c["noalloc"] = rng.random() < 0.3
        c["rows"] = _log(rng, 1000, 1_000_000 if c["noalloc"] else 3_000_000)
        c["links"] = rng.randint(1, 2) if c["t"] > 1 else 1
    elif kind in ("batch", "serve", "replay"):
        c["queries"] = _log(rng, 16, {"batch": 96, "serve": 200, "replay": 512}[kind])
        c["rare"] = min(8, c["nvl"] // 4)
        c["count_only"] = kind == "replay"
        c["cap"] = 0 if c["count_only"] else 1 << 20
        c["bound"] = float(_log(rng, 1e3, 1e6 if kind == "replay" else 1e5))
        c["budget_mb"] = rng.choice([8192, 16384])
    return c


# ------------------------------------------------------------------ graphs
def _draw_pairs(c, count, gen):
    """`count` pairs of vertex ids (before the permutation), as int64 tensors."""
    n, dev = c["n"], "cuda"
    if c["graph"] == "er":
        return (torch.randint(0, n, (count,), generator=gen, device=dev), torch.randint(0, n, (count,), generator=gen, device=dev))
    a = torch.zeros(count, dtype=torch.int64, device=dev)
    b = torch.zeros(count, dtype=torch.int64, device=dev)
    for _ in range(max(1, (n - 1).bit_length())):     # one quadrant of (.57, .19, .19, .05) per level
        r = torch.rand(count, generator=gen, device=dev)
        a = a * 2 + (r >= 0.76)
        b = b * 2 + (((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
    return a % n, b % n


def _graph(c, gen):
    """(vlab, src, dst, elab) on the device: m distinct undirected edges in random order, ids permuted."""
    n, m, dev = c["n"], c["m"], "cuda"
    perm = torch.randperm(n, generator=gen, device=dev)
    keys = torch.zeros(0, dtype=torch.int64, device=dev)
    while keys.numel() < m:
        a, b = _draw_pairs(c, int((m - keys.numel()) * 1.3) + 64, gen)
        a, b = perm[a], perm[b]
        k = (torch.minimum(a, b) * n + torch.maximum(a, b))[a != b]
        keys = torch.unique(torch.cat([keys, k]))
    keys = keys[torch.randperm(keys.numel(), generator=gen, device=dev)[:m]]
    if c["graph"] == "er":
        vlab = torch.randint(0, c["nvl"], (n,), generator=gen, device=dev)
    else:                                             # Zipf(1.1) vertex labels
        w = torch.arange(1, c["nvl"] + 1, dtype=torch.float64, device=dev) ** -1.1
        vlab = torch.searchsorted(torch.cumsum(w / w.sum(), 0), torch.rand(n, generator=gen, device=dev, dtype=torch.float64))
        vlab = vlab.clamp(max=c["nvl"] - 1)
    elab = torch.randint(0, c["nel"], (m,), generator=gen, device=dev)
    return vlab, keys // n, keys % n, elab


def _host(x):
    return x.to(torch.int32).cpu().numpy()


# ----------------------------------------------------------------- queries
class _Walks:
    """Random-walk queries of a graph, each with the homomorphism count of its walk tree."""

    def __init__(self, c, g, gen):
        self.c, self.gen = c, gen
        vlab, src, dst, elab = g
        self.vlab, self.n, self.nvl = vlab, c["n"], c["nvl"]
        s, d, l = torch.cat([src, dst]), torch.cat([dst, src]), torch.cat([elab, elab])
        bucket = (l * self.nvl + vlab[s]) * self.nvl + vlab[d]
        order = torch.argsort(bucket, stable=True)
        self.bs, self.bd = s[order], d[order]
        cnt = torch.bincount(bucket, minlength=c["nel"] * self.nvl * self.nvl)
        self.boff = [0] + torch.cumsum(cnt, 0).tolist()
        if c["rare"]:                                 # walks among rare labels only
            keep = (vlab[s] >= c["rare"]) & (vlab[d] >= c["rare"])
            s, d, l = s[keep], d[keep], l[keep]
        self.key, order = torch.sort(s * self.n + d)
        self.d, self.l = d[order], l[order]
        deg = torch.bincount(s, minlength=self.n)
        self.off = torch.cat([torch.zeros(1, dtype=torch.int64, device="cuda"), torch.cumsum(deg, 0)])
        self.deg, self.starts = deg, torch.nonzero(deg)[:, 0]

    def walk(self, count, steps):
        cur = self.starts[torch.randint(0, self.starts.numel(), (count,), generator=self.gen, device="cuda")]
        at, lab = [cur], []
        for _ in range(steps):
            p = self.off[cur] + (torch.rand(count, generator=self.gen, device="cuda", dtype=torch.float64) * self.deg[cur]).long()
            cur = self.d[p]
            at.append(cur)
            lab.append(self.l[p])
        at = torch.stack(at, 1)
        return at.cpu().numpy(), torch.stack(lab, 1).cpu().numpy(), self.vlab[at].cpu().numpy()

    def bound(self, vl, tree):
        x = {}
        for p, ch, l in reversed(tree):
            b = (l * self.nvl + vl[p]) * self.nvl + vl[ch]
            es, ed = self.bs[self.boff[b]:self.boff[b + 1]], self.bd[self.boff[b]:self.boff[b + 1]]
            w = x.pop(ch)[ed] if ch in x else torch.ones(es.numel(), dtype=torch.float64, device="cuda")
            y = torch.zeros(self.n, dtype=torch.float64, device="cuda").index_add_(0, es, w)
            x[p] = x[p] * y if p in x else y
        return float(x[0].sum())

    def induced(self, verts):
        """Edges among `verts` as (i, j, label), i < j."""
        v = torch.tensor(verts, device="cuda")
        i, j = torch.triu_indices(len(verts), len(verts), 1, device="cuda")
        k = v[i] * self.n + v[j]
        p = torch.searchsorted(self.key, k).clamp(max=self.key.numel() - 1)
        hit = self.key[p] == k
        return list(zip(i[hit].tolist(), j[hit].tolist(), self.l[p][hit].tolist()))

    def queries(self, sizes, dense, fits):
        """One query per wanted size that `fits`; a size that no walk reaches within the bound in 300 tries shrinks by one."""
        got, tries, k, pool, at = [], 0, None, None, 0
        while len(got) < len(sizes):
            if pool is None or at == pool[0].shape[0]:
                pool, at = self.walk(max(256, 2 * len(sizes)), 96), 0
            if k is None:
                k, tries = sizes[len(got)], 0
            path, lab, vl = pool[0][at], pool[1][at], pool[2][at]
            at += 1
            tries += 1
            if tries > 300 and k > 2:
                k, tries = k - 1, 0
            seen, verts, vls, edges, tree = {int(path[0]): 0}, [int(path[0])], [int(vl[0])], {}, []
            for a, b, l, x in zip(path[:-1].tolist(), path[1:].tolist(), lab.tolist(), vl[1:].tolist()):
                if len(verts) == k:
                    break
                if b not in seen:
                    seen[b] = len(verts)
                    verts.append(b)
                    vls.append(x)
                    tree.append((seen[a], seen[b], l))
                edges[(min(seen[a], seen[b]), max(seen[a], seen[b]))] = l
            if len(verts) < k or len(edges) > 2 * k or (self.bound(vls, tree) > self.c["bound"] and k > 2):
                continue
            if self.c["kind"] == "step" and k > 2 and self.bound(vls[:-1], tree[:-1]) > self.c["bound"]:
                continue
            if dense[len(got)]:
                for i, j, l in self.induced(verts):
                    if len(edges) >= 2 * k:
                        break
                    edges.setdefault((i, j), l)
            e = sorted(edges)
            q = gsi.QueryArrays(np.array(vls, np.int32), np.array([a for a, _ in e], np.int32),
                                np.array([b for _, b in e], np.int32), np.array([edges[x] for x in e], np.int32))
            if fits(q, tries):
                got.append(q)
                k = None
        return got


def _sizes(c):
    return [c["k_lo"] + (7919 * i) % (c["k_hi"] - c["k_lo"] + 1) for i in range(c["queries"])]


def _queries(c, g, gen, graph):
    """The case's queries; where rows are asked for, none has more than its share of the caller's table."""
    most = c["cap"] // c["queries"]
    o = dict(semantics=gsi.GSI_HOMOMORPHISM) if c["hom"] else {}
    dense = [c["dense"] == 1 or (c["dense"] == 2 and i % 2 == 1) for i in range(c["queries"])]

    def fits(q, tries):
        if c["kind"] == "step":                       # a table of its own rows, not of a few repeated
            linked = int((q.dst == q.k - 1).sum()) >= c["links"]
            return tries > 200 or (linked and 16 * graph.query(_inner(q), count_only=True).count >= c["rows"])
        if not most:
            return True
        n = graph.query(q, count_only=True, **o).count
        return n <= most and (c["kind"] != "query" or tries > 60 or 64 * n >= most)     # a search that finds something

    return _Walks(c, g, gen).queries(_sizes(c), dense, fits)


def _inner(q):
    """The query without its last vertex (connected, as vertices are in the order of the walk)."""
    t = q.k - 1
    e = q.dst < t
    return gsi.QueryArrays(q.vlab[:t].copy(), q.src[e].copy(), q.dst[e].copy(), q.elab[e].copy())


# ------------------------------------------------------------------- cases
def prepare(case, seed):
    c = case
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    g = _graph(c, gen)
    arrays = [_host(x) for x in g]
    s = {"case": c}
    if c["kind"] == "build":
        s["arrays"] = arrays
        return s
    G = s["graph"] = gsi.EdgeGraph(*arrays) if c["kind"] == "edge" else gsi.Graph(*arrays)
    qs = s["queries"] = _queries(c, g, gen, G)
    del g
    if c["cap"]:
        s["table"] = _table(c["cap"], 1 + (2 * c["k_hi"] if c["kind"] == "edge" else c["k_hi"]))
    if c["kind"] == "replay":
        s["batch"] = gsi.PreparedBatch(G, qs, count_only=c["count_only"], mem_budget=c["budget_mb"] << 20)
    elif c["kind"] == "serve":
        s["server"] = gsi.Server(G, mem_budget=c["budget_mb"] << 20)
    elif c["kind"] == "step":
        _prepare_step(s, G, qs[0])
    return s


def _table(rows, cols):
    return torch.full((rows, cols), -1, dtype=torch.int32, device="cuda")


def _prepare_step(s, G, q):
    """The table of the query without its last vertex, the last vertex's candidates and its linking edges."""
    c, t = s["case"], q.k - 1
    link = [(int(a), int(l)) for a, b, l in zip(q.src, q.dst, q.elab) if b == t]
    r = G.query(_inner(q))
    M = torch.empty((r.count, t), dtype=torch.int32, device="cuda")
    r.copy_to(M.data_ptr(), M.shape[0])
    M = M[torch.argsort(_key(M))]
    M = M[torch.arange(c["rows"], device="cuda") % M.shape[0]].contiguous()
    bm, _ = G.filter(q)
    s["cand"] = torch.from_numpy(bm[t].view(np.int32)).cuda()
    s["ulabel"], s["cols"], s["labs"] = int(q.vlab[t]), [a for a, _ in link], [l for _, l in link]
    torch.cuda.synchronize()
    cap = max(64, c["rows"] // 2)
    while True:                                       # the caller's buffer: a row for every two of the table
        n = G.join_step(M.data_ptr(), M.shape[0], t, s["cand"].data_ptr(), s["ulabel"], s["cols"], s["labs"], 0, 0)
        if n <= cap or M.shape[0] == 1:
            break
        M = M[: (M.shape[0] + 1) // 2].contiguous()
        torch.cuda.synchronize()
    s["M"], s["step"] = M, G.join_step_noalloc if c["noalloc"] else G.join_step
    s["out"], s["table"] = _table(cap, t + 1), _table(cap, c["t"] + 1)


def _splitmix(i):
    z = (0x9E3779B97F4A7C15 * (i + 1)) & (2 ** 64 - 1)
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & (2 ** 64 - 1)
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & (2 ** 64 - 1)
    return (z ^ (z >> 31)) | 1


_MULT = torch.tensor([m - 2 ** 64 if m >= 2 ** 63 else m for m in map(_splitmix, range(40))])
_mult = {}


def _key(rows):
    """A 64-bit hash of each row."""
    k = rows.shape[1]
    if k not in _mult:
        _mult[k] = _MULT[:k].to(rows.device)
    return (rows * _mult[k]).sum(1)


def _gather(s, results, counts):
    """The rows of all results in the caller's table: the result's number, then the row (-1 past its end), in the order of
    the rows' hashes."""
    table = s["table"]
    cols, total = table.shape[1] - 1, int(counts.sum())
    ks = np.array([r.k for r in results])
    start = np.cumsum(counts * ks) - counts * ks      # where each result's rows begin
    flat = torch.empty(total * int(ks.max()), dtype=torch.int32, device="cuda")
    for r, n, a in zip(results, counts, start):
        if n:
            r.copy_to_async(flat.data_ptr() + 4 * int(a), int(n))
    meta = torch.from_numpy(np.stack([counts, ks, start - (np.cumsum(counts) - counts) * ks])).cuda()
    ids = torch.repeat_interleave(meta[0], output_size=total)
    k, base = meta[1][ids], meta[2][ids]
    col = torch.arange(cols, device="cuda")
    at = (base + torch.arange(total, device="cuda") * k)[:, None] + col
    rows = torch.where(col < k[:, None], flat[at.clamp_(max=flat.numel() - 1)], -1)
    order = torch.argsort(_key(rows) + ids * (_splitmix(50) % 2 ** 40))
    table[:total, 0] = ids[order]
    table[:total, 1:] = rows[order]
    return table


class _View:
    """A graph's device array as torch sees it."""

    def __init__(self, ptr, n, kind):
        self.__cuda_array_interface__ = {"shape": (n,), "typestr": kind, "data": (ptr, False), "version": 3}


def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind in ("query", "edge"):
        o = {}
        if kind == "query":
            o = dict(count_only=c["count_only"], mem_budget=c["budget_mb"] << 20, host_driven=c["split"],
                     semantics=gsi.GSI_HOMOMORPHISM if c["hom"] else gsi.GSI_ISOMORPHISM)
        res = [s["graph"].query(q, **o) for q in s["queries"]]
        if c["host"]:
            rows = res[0].rows()
            out = np.full((c["cap"], c["k_hi"]), -1, np.int32)
            out[: rows.shape[0], : rows.shape[1]] = rows[np.lexsort(rows.T)]
            return rows.shape[0], out
    elif kind == "filter":
        return s["graph"].filter(s["queries"][0])
    elif kind == "step":
        n = s["step"](s["M"].data_ptr(), s["M"].shape[0], s["M"].shape[1], s["cand"].data_ptr(), s["ulabel"], s["cols"],
                      s["labs"], s["out"].data_ptr(), s["out"].shape[0])
        rows = s["out"][:n]
        s["table"][:n, : rows.shape[1]] = rows[torch.argsort(_key(rows))]
        return n, s["table"]
    elif kind == "build":
        G = s["graph"] = None                         # the graph of the last pass goes first
        G = s["graph"] = gsi.Graph(*s["arrays"])
        i = G.info()
        return (torch.as_tensor(_View(i.off, i.n * i.n_elabels + 1, "<i4"), device="cuda"),
                torch.as_tensor(_View(i.ci, 2 * i.m, "<i4"), device="cuda"),
                torch.as_tensor(_View(i.cl, 2 * i.m, "<i2"), device="cuda"),
                torch.as_tensor(_View(i.sig, 16 * i.n, "<i4"), device="cuda"), G.label_freq())
    elif kind == "batch":
        res = s["graph"].batch(s["queries"], mem_budget=c["budget_mb"] << 20, count_only=c["count_only"])
    elif kind == "replay":
        res = s["batch"].run()
    else:
        tickets = [s["server"].submit(q) for q in s["queries"]]
        res = [s["server"].poll(t)[0] for t in tickets]
    counts = np.array([r.count for r in res], np.int64)
    return counts if c["count_only"] else (counts, _gather(s, res, counts))


def work(case):
    """Bytes of one pass.  A search reads the signatures of its query vertices' labels and writes their candidate bitmaps,
    then reads for each match the list entry that completes it (4 bytes) and, where rows are asked for, writes the row.
    The number of matches is taken as a typical share of the bound."""
    c = case
    n, m, k = c["n"], c["m"], (c["k_lo"] + c["k_hi"]) / 2
    if c["kind"] == "build":
        return {"bytes": 12 * m + 4 * n + 4 * n * c["nel"] + 12 * m + 64 * n, "flops": 0}
    if c["kind"] == "step":
        out = c["rows"]                               # about one survivor for each row
        return {"bytes": c["rows"] * (4 * c["t"] + 8 + 4) + n / 8 + out * 4 * (c["t"] + 1), "flops": 0}
    nv = m if c["kind"] == "edge" else n
    nvl = c["nel"] * c["nvl"] * (c["nvl"] + 1) / 2 if c["kind"] == "edge" else c["nvl"]
    calls = 1 if c["kind"] in ("batch", "replay", "serve") else c["queries"]      # signatures: once a call
    bits = calls * 64 * nv * min(1.0, c["queries"] / calls * k / nvl) + c["queries"] * k * nv / 8
    if c["kind"] == "filter":
        return {"bytes": bits, "flops": 0}
    found = c["bound"] * 0.1
    return {"bytes": bits + c["queries"] * found * (4 if c["count_only"] else 4 + 4 * k), "flops": 0}
