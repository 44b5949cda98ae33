"""The library's work as its users call it, case by case, at the sizes it is used at.

A case is a dict of plain values. `kind` says which entry points a pass goes through:

  decompose  a new graph arrives as a CSR (device tensors, or host arrays with "host"): nd_load_csr,
             optionally nd_orient, nd_decompose(r, s), nd_graph_free. Core numbers and rounds come back.
  count      the same with nd_count: s-clique counts per r-clique.
  noalloc    nd_kcore_noalloc: k-core of a resident CSR by a caller whose pool owns the memory.
  hierarchy  nd_hierarchy on a graph that was decomposed before (the handle and the core numbers are
             kept, as a program that explores nuclei keeps them).
  batch      nd_batch_run: many small graphs with mixed (r, s), host CSRs in, host core numbers out.
  serve      a burst of requests to a running server: nd_submit each, nd_server_drain, nd_poll each.

Graphs (`graph`), all made on the GPU from the seed alone, with as many edges as the case says, whatever
the seed (so the results of r <= 2 have one size; longer results go to a buffer with room, filled with
-1 past their end):

  chung_lu   power-law expected degrees, average `deg`, exponent `gamma`, largest expected degree `wmax`
             (0: the square root of their sum); `planted` disjoint communities of 20-60 vertices at edge
             density 0.7 on top.
  rmat       0.9 `deg` edges per vertex, quadrants a, b = c, d = 1 - a - 2 b; ids from n up are dropped.
"""
import itertools
import math

import numpy as np
import torch

import paper_2111_10980_gb300 as nd

DEVICE = "cuda:0"


# ---- the cases ---------------------------------------------------------------------------

def _chung_lu(n, deg, gamma, wmax=0, planted=0):
    return {"graph": "chung_lu", "n": n, "deg": deg, "gamma": gamma, "wmax": wmax, "planted": planted}


def _rmat(n, deg, a=0.57, b=0.19):
    return {"graph": "rmat", "n": n, "deg": deg, "a": a, "b": b}


def listed():
    return [
        # an ego network or one small community, on its own: latency is everything
        dict(_chung_lu(2000, 20.0, 2.1, 200), name="truss_small", kind="decompose", r=2, s=3),
        # k-core inside a training loop whose allocator owns the GPU
        dict(_chung_lu(100_003, 12.0, 2.3), name="core_noalloc", kind="noalloc", r=1, s=2),
        # trusses of a graph that a host program holds in its own memory, results back to the host
        dict(_chung_lu(200_001, 24.0, 2.2), name="truss_host", kind="decompose", r=2, s=3, host=True),
        # trusses of a large skewed graph: the (2,3) half of the benchmark
        dict(_rmat(1 << 20, 16), name="truss_rmat", kind="decompose", r=2, s=3),
        # (3,4) nuclei of a large skewed graph: the (3,4) half of the benchmark, two scales down
        dict(_rmat(1 << 18, 16), name="nucleus34_rmat", kind="decompose", r=3, s=4),
        # (3,4) nuclei of a sparse graph with planted communities, its CSR checked on the way in
        dict(_chung_lu(1_000_003, 30.0, 2.3, 0, 500), name="nucleus34_comm", kind="decompose", r=3, s=4, validate=True),
        # (2,4) nuclei of the same family with 64-bit tallies
        dict(_chung_lu(500_009, 30.0, 2.3, 0, 500), name="nucleus24_comm", kind="decompose", r=2, s=4, width=8),
        # larger cliques on a graph of low skew, oriented by degeneracy
        dict(_rmat(40_000, 32, 0.5, 0.1), name="nucleus45_flat", kind="decompose", r=4, s=5, degeneracy=True),
        # motif features of every edge of a skewed graph
        dict(_rmat(50_001, 16), name="count24_rmat", kind="count", r=2, s=4),
        # the tree of nested dense subgraphs, after the decomposition
        dict(_rmat(1 << 16, 16), name="hierarchy23_rmat", kind="hierarchy", r=2, s=3),
        # many small graphs of a data set at once
        {"name": "batch_mixed", "kind": "batch", "graph": "chung_lu", "graphs": 512, "nmin": 50, "nmax": 5000, "rs": "12,23,34"},
        # a burst of requests to a server, each a graph of its own
        {"name": "serve_burst", "kind": "serve", "graph": "chung_lu", "graphs": 64, "nmin": 30, "nmax": 10_000, "rs": "23,34,24"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the kind, then sizes spread over the range of that kind's uses."""
    kind = rng.choice(("truss", "truss", "nucleus34", "nucleus34", "nucleus24", "core", "noalloc", "larger", "count", "hierarchy", "batch", "serve"))
    flat = rng.random() < 0.5
    if kind == "truss":
        g = _chung_lu(_log(rng, 500, 1_000_000), rng.uniform(8, 40), rng.uniform(2.1, 2.6)) if flat else _rmat(_log(rng, 1000, 1 << 20), rng.choice((8, 16)))
        return dict(g, kind="decompose", r=2, s=3, host=rng.random() < 0.3, validate=rng.random() < 0.3)
    if kind == "nucleus34":
        g = _chung_lu(_log(rng, 500, 1_000_000), rng.uniform(8, 40), rng.uniform(2.2, 2.6), 0, rng.choice((0, 10))) if flat else _rmat(_log(rng, 1000, 1 << 18), rng.choice((8, 16)))
        return dict(g, kind="decompose", r=3, s=4, host=rng.random() < 0.3, width=rng.choice((0, 8)))
    if kind == "nucleus24":
        g = _chung_lu(_log(rng, 500, 500_000), rng.uniform(8, 30), rng.uniform(2.3, 2.6), 0, rng.choice((0, 10))) if flat else _rmat(_log(rng, 500, 1 << 14), rng.choice((8, 16)))
        return dict(g, kind="decompose", r=2, s=4, width=rng.choice((0, 8)))
    if kind == "core":
        g = _chung_lu(_log(rng, 500, 1_000_000), rng.uniform(8, 40), rng.uniform(2.1, 2.6)) if flat else _rmat(_log(rng, 1000, 1 << 20), rng.choice((8, 16)))
        return dict(g, kind="decompose", r=1, s=2)
    if kind == "noalloc":
        g = _chung_lu(_log(rng, 300, 262_144), rng.uniform(8, 40), rng.uniform(2.1, 2.6)) if flat else _rmat(_log(rng, 300, 262_144), rng.choice((8, 16)))
        return dict(g, kind="noalloc", r=1, s=2)
    if kind == "larger":
        r, s = rng.choice(((1, 3), (3, 5), (4, 5)))
        return dict(_rmat(_log(rng, 500, 40_000), rng.choice((8, 16, 32)), 0.5, 0.1), kind="decompose", r=r, s=s, degeneracy=rng.random() < 0.5)
    if kind == "count":
        r, s = rng.choice(((2, 3), (3, 4), (2, 4), (1, 3)))
        g = _chung_lu(_log(rng, 500, 200_000), rng.uniform(8, 30), rng.uniform(2.2, 2.6)) if flat else _rmat(_log(rng, 500, 50_001), rng.choice((8, 16)))
        return dict(g, kind="count", r=r, s=s)
    if kind == "hierarchy":
        r, s = rng.choice(((1, 2), (2, 3)))
        g = _chung_lu(_log(rng, 500, 100_000), rng.uniform(8, 30), rng.uniform(2.2, 2.6)) if flat else _rmat(_log(rng, 500, 1 << 16), 16)
        return dict(g, kind="hierarchy", r=r, s=s)
    if kind == "batch":
        lo = _log(rng, 20, 200)
        return {"kind": "batch", "graph": "chung_lu", "graphs": _log(rng, 8, 512), "nmin": lo, "nmax": _log(rng, 2 * lo, 5000), "rs": rng.choice(("12,23,34", "23", "34", "23,34,24"))}
    return {"kind": "serve", "graph": "chung_lu", "graphs": _log(rng, 8, 128), "nmin": 30, "nmax": _log(rng, 300, 10_000), "rs": "23,34,24"}


# ---- graphs ------------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(int(seed))
    return g


def _keys(n, u, v):
    """Each undirected edge's key, once, without loops."""
    keep = u != v
    u, v = u[keep], v[keep]
    return torch.unique(torch.minimum(u, v) * n + torch.maximum(u, v))


def _csr(n, key):
    """rowptr int64[n+1], col int32[2m] of the simple undirected graph with these edge keys."""
    u, v = key // n, key % n
    key = torch.sort(torch.cat([key, v * n + u]))[0]
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device=DEVICE)
    rowptr[1:] = torch.cumsum(torch.bincount(key // n, minlength=n), 0)
    return rowptr, (key % n).to(torch.int32)


def _weights(n, deg, gamma, wmax):
    """Expected degrees w_0 (i0 / (i + i0))^(1 / (gamma - 1)), i < n, with mean deg and w_0 = wmax."""
    wmax = min(wmax or math.sqrt(n * deg), n - 1.0)
    i = torch.arange(n, dtype=torch.float64, device=DEVICE)
    beta = 1.0 / (gamma - 1.0)
    lo, hi = math.log(1e-6), math.log(1e12)
    for _ in range(50):
        mid = 0.5 * (lo + hi)
        i0 = math.exp(mid)
        if float((wmax * (i0 / (i + i0)) ** beta).mean()) < deg:
            lo = mid
        else:
            hi = mid
    return wmax * (i0 / (i + i0)) ** beta


def _planted(n, k, g):
    """Edges of k disjoint communities of 20..60 vertices placed at random."""
    side = 60
    size = torch.randint(20, side + 1, (k,), generator=g, device=DEVICE)
    at = torch.randperm(n, generator=g, device=DEVICE)[: k * side].reshape(k, side)
    a, b = torch.triu_indices(side, side, 1, device=DEVICE)
    take = (b[None, :] < size[:, None]) & (torch.rand((k, a.numel()), generator=g, device=DEVICE) < 0.7)
    return at[:, a][take], at[:, b][take]


def _edges(case):
    """Undirected edges of a case's graph."""
    n, deg = case["n"], case["deg"]
    m = int(0.9 * n * deg) if case["graph"] == "rmat" else int(n * deg / 2) + 570 * case["planted"]
    return max(1, min(m, n * (n - 1) // 8))


def _rmat_pairs(case, g, count):
    n, a, b = case["n"], case["a"], case["b"]
    u = torch.zeros(count, dtype=torch.int64, device=DEVICE)
    v = torch.zeros_like(u)
    for _ in range(max(1, (n - 1).bit_length())):
        x = torch.rand(count, generator=g, device=DEVICE)
        right, down = ((x >= a) & (x < a + b)) | (x >= a + 2 * b), x >= a + b
        u, v = 2 * u + down, 2 * v + right
    keep = (u < n) & (v < n)
    return u[keep], v[keep]


def _graph(case, seed):
    g, n, m = _gen(seed), case["n"], _edges(case)
    key = torch.empty(0, dtype=torch.int64, device=DEVICE)
    if case["graph"] == "chung_lu":
        w = _weights(n, case["deg"], case["gamma"], case["wmax"])
        cum = torch.cumsum(w / w.sum(), 0)
        if case["planted"]:
            key = _keys(n, *_planted(n, case["planted"], g))
    while key.numel() < m:
        count = int(1.12 * (m - key.numel())) + 1000
        if case["graph"] == "rmat":
            u, v = _rmat_pairs(case, g, count)
        else:
            x = torch.rand(2 * count, generator=g, device=DEVICE, dtype=torch.float64)
            ends = torch.searchsorted(cum, x).clamp_(max=n - 1)
            u, v = ends[:count], ends[count:]
        key = torch.unique(torch.cat([key, _keys(n, u, v)]))
    csr = _csr(n, key[torch.randperm(key.numel(), generator=g, device=DEVICE)[:m]])
    torch.cuda.synchronize()  # the library works on a stream of its own
    return csr


def _many(case, seed):
    """The graphs of a batch or a burst: sizes n (log-uniform for a burst) and average degrees U[8, 40],
    Chung-Lu with exponent 2.2, and each one's (r, s), all three the case's; the edges are the seed's. One
    disjoint union on the GPU, then cut up."""
    k, lo, hi = case["graphs"], case["nmin"], case["nmax"]
    rng = np.random.RandomState((31 * k + 17 * lo + hi) % (1 << 31))
    if case["kind"] == "serve":
        sizes = np.exp(rng.uniform(math.log(lo), math.log(hi), k)).astype(np.int64)
    else:
        sizes = rng.randint(lo, hi + 1, k)
    deg = rng.uniform(8, 40, k)
    rs = [tuple(int(c) for c in x) for x in case["rs"].split(",")]
    rs = [rs[i] for i in rng.randint(0, len(rs), k)]
    off = np.concatenate([[0], np.cumsum(sizes)])
    n = int(off[-1])
    which = torch.repeat_interleave(torch.arange(k, device=DEVICE), torch.tensor(sizes, device=DEVICE))
    i = torch.arange(n, device=DEVICE) - torch.tensor(off[:-1], device=DEVICE)[which]
    # a largest expected degree of about the square root of their sum, as of a graph on its own
    w = ((i + 0.02 * torch.tensor(sizes, device=DEVICE)[which] + 1).double()) ** (-1 / 1.2)
    total = torch.zeros(k, dtype=torch.float64, device=DEVICE).index_add_(0, which, w)
    cum = torch.cumsum(w / total[which], 0)
    edges = np.maximum(1, (sizes * np.minimum(deg, sizes / 4) / 2).astype(np.int64))
    owner = torch.repeat_interleave(torch.arange(k, device=DEVICE), torch.tensor(edges, device=DEVICE))
    lo_t, hi_t = torch.tensor(off[:-1], device=DEVICE)[owner], torch.tensor(off[1:] - 1, device=DEVICE)[owner]
    g = _gen(seed)

    def end():
        x = owner + torch.rand(owner.numel(), generator=g, device=DEVICE, dtype=torch.float64)
        return torch.minimum(torch.maximum(torch.searchsorted(cum, x), lo_t), hi_t)

    rowptr, col = (x.cpu().numpy() for x in _csr(n, _keys(n, end(), end())))
    out = []
    for j in range(k):
        a, b = off[j], off[j + 1]
        p, q = rowptr[a], rowptr[b]
        out.append((np.ascontiguousarray(rowptr[a:b + 1] - p), np.ascontiguousarray(col[p:q] - np.int32(a)), *rs[j]))
    return out


# ---- what a program keeps, and a pass ----------------------------------------------------

_kept = {}


def _ctx():
    """One context for the process, as a program keeps it."""
    if "ctx" not in _kept:
        _kept["ctx"] = nd.nd_ctx_create(0)
    return _kept["ctx"]


def _server():
    if "server" not in _kept:
        _kept["server"] = nd.nd_server_create(_ctx(), workers=4, max_batch=256)
    return _kept["server"]


def _room(case, count):
    """Room for a result whose length the seed decides: half as much again as one of its graphs needs."""
    key = tuple(sorted((k, v) for k, v in case.items() if k != "name"))
    if key not in _kept:
        _kept[key] = count(0) * 3 // 2 + 4096
    return _kept[key]


class _State:
    graph = None

    def __init__(self, case):
        self.case = case

    def __del__(self):
        if self.graph is not None:
            nd.nd_graph_free(self.graph)


def prepare(case, seed):
    st = _State(case)
    kind = case["kind"]
    if kind in ("batch", "serve"):
        # each result's place in one host buffer, sized by a first run as a caller sizes it
        st.graphs = _many(case, seed)
        n_r = nd.nd_batch_run(_ctx(), st.graphs)[1]
        room = _room(case, lambda other: sum(nd.nd_batch_run(_ctx(), _many(case, other))[1]))
        at = np.concatenate([[0], np.cumsum(n_r)])
        if at[-1] > room:
            raise ValueError("no room for %d results in %d" % (at[-1], room))
        st.out = np.full(room, -1, np.int32)
        st.outs = [st.out[at[j]:at[j + 1]] if n_r[j] else np.zeros(1, np.int32) for j in range(len(n_r))]
        return st
    st.rowptr, st.col = _graph(case, seed)
    r, s = case["r"], case["s"]
    if kind == "noalloc":
        st.core = torch.empty(case["n"], dtype=torch.int32, device=DEVICE)
        return st
    if kind == "hierarchy":
        st.graph = nd.nd_load_csr(_ctx(), st.rowptr, st.col)
        st.core = torch.from_numpy(nd.nd_decompose(st.graph, r, s)[0]).to(DEVICE)
        return st

    def number(rowptr, col):
        if r <= 2:
            return case["n"] if r == 1 else col.numel() // 2
        g = nd.nd_load_csr(_ctx(), rowptr, col)
        got = len(nd.nd_rcliques(g, r)) if r == 4 else nd.nd_count(g, r, s)[1]
        nd.nd_graph_free(g)
        return got

    n_r = number(st.rowptr, st.col)
    room = n_r if r <= 2 else _room(case, lambda other: number(*_graph(case, other)))
    if n_r > room:
        raise ValueError("no room for %d results in %d" % (n_r, room))
    if case.get("host"):
        st.rowptr, st.col = st.rowptr.cpu().numpy(), st.col.cpu().numpy()
        st.core, st.round = np.full(room, -1, np.int32), np.full(room, -1, np.int32)
    elif kind == "count":
        st.counts = torch.full((room,), -1, dtype=torch.int64, device=DEVICE)
    else:
        st.core, st.round = (torch.full((room,), -1, dtype=torch.int32, device=DEVICE) for _ in range(2))
    torch.cuda.synchronize()
    return st


def run(st):
    case, kind = st.case, st.case["kind"]
    if kind == "batch":
        _, n_r, status, _ = nd.nd_batch_run(_ctx(), st.graphs, st.outs)
        return {"core": st.out, "n_r": np.array(n_r), "status": np.array(status)}
    if kind == "serve":
        sv = _server()
        tickets = [nd.nd_submit(sv, *g, o) for g, o in zip(st.graphs, st.outs)]
        nd.nd_server_drain(sv)
        got = [nd.nd_poll(sv, t) for t in tickets]
        return {"core": st.out, "n_r": np.array([d["n_r"] for _, d in got]), "status": np.array([rc for rc, _ in got])}
    if kind == "noalloc":
        return nd.nd_kcore_noalloc(st.rowptr, st.col, st.core)
    r, s = case["r"], case["s"]
    if kind == "hierarchy":
        comp, level, up, nodes = nd.nd_hierarchy(st.graph, r, s, st.core)
        return {"comp": comp, "parent_level": level, "parent_comp": up, "nodes": nodes}
    g = nd.nd_load_csr(_ctx(), st.rowptr, st.col, nd.ND_VALIDATE if case.get("validate") else 0)
    if case.get("degeneracy"):
        nd.nd_orient(g, nd.ND_ORIENT_DEGENERACY)
    if kind == "count":
        counts, n_r, n_s = nd.nd_count(g, r, s, out=st.counts)
        out = {"counts": counts, "n_r": n_r, "n_s": n_s}
    else:
        core, rounds, stats = nd.nd_decompose(g, r, s, case.get("width", 0), st.core, st.round)
        out = {"core": core, "round": rounds, "n_s": stats["n_s"], "rho": stats["rho"], "max_core": stats["max_core"]}
    nd.nd_graph_free(g)
    return out


# ---- what a pass cannot do without, and what it has to give ------------------------------

def _cliques(case):
    """Rough numbers of vertices, edges, triangles, 4- and 5-cliques of a case's graphs."""
    if case["kind"] in ("batch", "serve"):
        k, lo, hi = case["graphs"], case["nmin"], case["nmax"]
        n = k * ((hi - lo) / math.log(hi / lo) if case["kind"] == "serve" else (lo + hi) / 2)
        m = n * 11
        return n, m, 2.5 * m, 5 * m, 8 * m
    n, deg, m = case["n"], case["deg"], _edges(case)
    if case["graph"] == "rmat" and case["a"] > 0.55:
        t = m * 27 * (n / (1 << 20)) ** 0.17 * (deg / 16) ** 2
        return n, m, t, t * 40 * (n / (1 << 20)) ** 0.31 * (deg / 16), t * 900
    if case["graph"] == "rmat":
        t = m * 2.1 * (deg / 64) ** 2 * (n / (1 << 17)) ** -0.2
        return n, m, t, 0.5 * t * (deg / 64), 0.2 * t * (deg / 64) ** 2
    c = 570.0 * case["planted"]
    return n, m, 0.5 * (m - c) + 8.0 * c, 0.2 * (m - c) + 52.0 * c, 0.1 * (m - c) + 260.0 * c


def work(case):
    """Bytes: the CSR in, the results out. Operations: one decrement (or addition) for each r-clique of
    each s-clique, which no way of counting or peeling can do without."""
    counts = _cliques(case)
    n, m = counts[0], counts[1]
    csr = 8 * (n + 1) + 8 * m
    if case["kind"] in ("batch", "serve"):
        rs = [tuple(int(c) for c in x) for x in case["rs"].split(",")]
        ops = sum(math.comb(s, r) * counts[s - 1] for r, s in rs) / len(rs)
        return {"bytes": csr + 4 * sum(counts[r - 1] for r, _ in rs) / len(rs), "flops": ops}
    r, s = case["r"], case["s"]
    ops = math.comb(s, r) * counts[min(s, 5) - 1]
    out = {"decompose": 8, "count": 8, "noalloc": 4, "hierarchy": 16}[case["kind"]] * counts[r - 1]
    return {"bytes": csr + out, "flops": ops}


def tolerance(case):
    return "exact"  # whole numbers: counts, core numbers, rounds, ids


# ---- the same from the definition, in plain torch ----------------------------------------

def _all_cliques(n, rowptr, col, size, most):
    """All cliques of `size` vertices, each an ascending row, rows in lexicographic order; None if any
    level has more than `most` candidates."""
    src = torch.repeat_interleave(torch.arange(n, device=DEVICE), rowptr.diff())
    dst = col.long()
    deg = rowptr.diff()
    lower = (deg[src] < deg[dst]) | ((deg[src] == deg[dst]) & (src < dst))
    u, v = src[lower], dst[lower]  # oriented from lower to higher degree, rows still ascending
    if size == 1:
        return torch.arange(n, device=DEVICE)[:, None]
    keys = u * n + v
    start = torch.zeros(n + 1, dtype=torch.int64, device=DEVICE)
    start[1:] = torch.cumsum(torch.bincount(u, minlength=n), 0)
    rows = torch.stack([u, v], 1)
    for _ in range(size - 2):
        d = start.diff()[rows[:, -1]]
        total = int(d.sum())
        if total > most:
            return None
        which = torch.repeat_interleave(torch.arange(rows.shape[0], device=DEVICE), d)
        k = torch.arange(total, device=DEVICE) - torch.repeat_interleave(torch.cumsum(d, 0) - d, d)
        w = v[start[rows[which, -1]] + k]
        ok = torch.ones_like(w, dtype=torch.bool)
        for j in range(rows.shape[1] - 1):
            key = rows[which, j] * n + w
            at = torch.searchsorted(keys, key).clamp_(max=max(keys.numel() - 1, 0))
            ok &= keys[at] == key
        rows = torch.cat([rows[which[ok]], w[ok, None]], 1)
    rows = torch.sort(rows, 1)[0]
    for j in range(size - 1, -1, -1):
        rows = rows[torch.sort(rows[:, j], stable=True)[1]]
    return rows


def _ids(cliques, r, n, subset):
    """Place of each row of `subset` (ascending r-tuples) among the sorted r-cliques."""
    if r == 1:
        return subset[:, 0]
    at, have = None, None
    for j in range(r):
        a, b = subset[:, j], cliques[:, j]
        at, have = (a, b) if at is None else (at * n + a, have * n + b)
        if j < r - 1 and j > 0:  # compress, so that keys stay small
            vals = torch.unique(have)
            at, have = torch.searchsorted(vals, at), torch.searchsorted(vals, have)
    return torch.searchsorted(have, at)


def _incidence(n, rowptr, col, r, s, most):
    small = _all_cliques(n, rowptr, col, r, most)
    large = None if small is None else _all_cliques(n, rowptr, col, s, most)
    if large is None or large.shape[0] * math.comb(s, r) > most:
        return None
    if not large.shape[0]:
        return small, torch.zeros((0, math.comb(s, r)), dtype=torch.int64, device=DEVICE)
    return small, torch.stack([_ids(small, r, n, large[:, list(c)]) for c in itertools.combinations(range(s), r)], 1)


def _peel(n_r, inc):
    """Core number and round of every r-clique by the definition of a round: k rises to the smallest
    count left, every r-clique with a count of at most k goes at once, with the s-cliques it is in."""
    cnt = torch.bincount(inc.reshape(-1), minlength=n_r)
    core = torch.zeros(n_r, dtype=torch.int32, device=DEVICE)
    rnd = torch.full((n_r,), -1, dtype=torch.int32, device=DEVICE)
    left, k, t = n_r, 0, 0
    while left:
        k = max(k, int(cnt[rnd < 0].min()))
        take = (rnd < 0) & (cnt <= k)
        core[take], rnd[take] = k, t
        gone = take[inc].any(1)
        cnt -= torch.bincount(inc[gone].reshape(-1), minlength=n_r)
        inc = inc[~gone]
        left -= int(take.sum())
        t += 1
        if t > 5000:
            return None
    return core, rnd, t, k


MOST = 20_000_000


def exact(case, seed):
    kind = case["kind"]
    if kind in ("hierarchy", "serve", "batch") or work(case)["flops"] > MOST:
        return None
    rowptr, col = _graph(case, seed)
    r, s, n = case["r"], case["s"], case["n"]
    got = _incidence(n, rowptr, col, r, s, MOST)
    if got is None:
        return None
    small, inc = got
    n_r = small.shape[0]
    room = n_r if r <= 2 else _kept.get(tuple(sorted((k, v) for k, v in case.items() if k != "name")), n_r)

    def padded(x):
        return torch.nn.functional.pad(x, (0, room - n_r), value=-1)

    if kind == "count":
        return {"counts": padded(torch.bincount(inc.reshape(-1), minlength=n_r)), "n_r": n_r, "n_s": inc.shape[0]}
    peeled = _peel(n_r, inc)
    if peeled is None:
        return None
    core, rnd, rho, k = peeled
    if kind == "noalloc":
        return core
    return {"core": padded(core), "round": padded(rnd), "n_s": inc.shape[0], "rho": rho, "max_core": k}
