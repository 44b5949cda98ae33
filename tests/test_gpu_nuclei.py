"""Connected nuclei (Section 2, footnote): the components, through s-cliques whose r-subsets all
have core >= c, of the r-cliques with core >= c. The library's labels (smallest id of each
component, -1 outside) and component counts are compared with the oracle's sequential union-find
element by element, at every level of each decomposition, for every supported (r,s), on host and
device pointers, including disjoint unions (components that must stay apart) and graphs with hubs.
The core arrays given to both sides are the oracle's."""
import math

import numpy as np
import pytest

import graphgen as gg
import oracle as orc

pytestmark = pytest.mark.gpu

RS = [(1, 2), (1, 3), (1, 4), (2, 3), (2, 4), (2, 5), (3, 4), (3, 5), (3, 6), (4, 5), (4, 6)]


@pytest.fixture(scope="module")
def nd():
    import paper_2111_10980_gb300 as nd

    nd.lib()
    return nd


@pytest.fixture(scope="module")
def ctx(nd):
    c = nd.nd_ctx_create(0)
    yield c
    nd.nd_ctx_destroy(c)


def levels_of(core, cap=12):
    """0, every distinct core value (capped to `cap` of them, spread evenly) and max + 1."""
    vals = np.unique(core) if core.size else np.zeros(0, np.int64)
    if vals.size > cap:
        vals = vals[np.linspace(0, vals.size - 1, cap).astype(np.int64)]
    top = int(core.max()) + 1 if core.size else 1
    return sorted({0, top, *[int(v) for v in vals]})


def check(nd, ctx, g, r, s, device=False, cap=12):
    core = orc.decompose(g, r, s).core.astype(np.int32)
    G = nd.nd_load_csr(ctx, g.rowptr, g.col, flags=nd.ND_VALIDATE)
    try:
        for c in levels_of(core, cap):
            want, nw = orc.nuclei(g, r, s, core, c)
            if device:
                import torch

                got, ng = nd.nd_nuclei(G, r, s, torch.from_numpy(core).cuda(), c)
                got = got.cpu().numpy()
            else:
                got, ng = nd.nd_nuclei(G, r, s, core, c)
            assert ng == nw, (r, s, c, ng, nw)
            np.testing.assert_array_equal(got, want, err_msg=f"(r,s)=({r},{s}) level {c}")
    finally:
        nd.nd_graph_free(G)


@pytest.mark.parametrize("r,s", RS)
def test_small_graphs(nd, ctx, r, s):
    check(nd, ctx, gg.fig1(), r, s)
    check(nd, ctx, gg.disjoint_union(gg.complete(7), gg.fig1(), gg.complete(s), gg.complete(s + 2)), r, s)
    for seed in range(6):
        check(nd, ctx, gg.gnp(10 + 4 * seed, [0.3, 0.5, 0.7][seed % 3], 9100 + seed), r, s)


@pytest.mark.parametrize("r,s", RS)
def test_power_law_and_communities(nd, ctx, r, s):
    check(nd, ctx, gg.with_planted(gg.chung_lu(1200, 5.0, 2.3, seed=9201), 10, 8, 20, 0.7, seed=9202), r, s)
    if s - r == 1:
        check(nd, ctx, gg.rmat(11, 8, seed=9203), r, s, device=True)
    elif s - r == 2:
        check(nd, ctx, gg.rmat(9, 8, seed=9204), r, s, device=True)


@pytest.mark.parametrize("r,s,scale,ef", [(1, 2, 14, 16), (2, 3, 14, 8), (2, 4, 12, 8), (3, 4, 12, 8)])
def test_larger_graphs(nd, ctx, r, s, scale, ef):
    # 10^4 to 10^5 r-cliques; hubs whose r-cliques list long neighbourhoods
    check(nd, ctx, gg.rmat(scale, ef, seed=9301), r, s, device=True, cap=6)
    check(nd, ctx, gg.hubs_over_sparse(n_common=4000, hubs=4, p_hub=0.9, avg_deg=4.0, seed=9302), r, s)


def test_empty_and_edgeless(nd, ctx):
    for g in (gg.complete(1), gg.gnp(30, 0.0, 1)):
        for r, s in [(1, 2), (2, 3), (3, 4)]:
            check(nd, ctx, g, r, s)


def test_bad_arguments(nd, ctx):
    g = gg.fig1()
    G = nd.nd_load_csr(ctx, g.rowptr, g.col)
    try:
        core = np.zeros(g.n, np.int32)
        with pytest.raises(nd.NdError):
            nd.nd_nuclei(G, 4, 7, core, 0)
        with pytest.raises(ValueError):
            import torch

            nd.nd_nuclei(G, 1, 2, core, 0, out=torch.zeros(g.n, dtype=torch.int32, device="cuda"))
    finally:
        nd.nd_graph_free(G)


def check_hierarchy(nd, ctx, g, r, s, device=False):
    core = orc.decompose(g, r, s).core.astype(np.int32)
    want = orc.hierarchy(g, r, s, core)
    G = nd.nd_load_csr(ctx, g.rowptr, g.col, flags=nd.ND_VALIDATE)
    try:
        if device:
            import torch

            got = nd.nd_hierarchy(G, r, s, torch.from_numpy(core).cuda())
            got = [x.cpu().numpy() for x in got[:3]] + [got[3]]
        else:
            got = nd.nd_hierarchy(G, r, s, core)
        for name, a, b in zip(("comp", "parent_level", "parent_comp"), got[:3], want):
            np.testing.assert_array_equal(a, b, err_msg=f"(r,s)=({r},{s}) {name}")
        nodes = {(int(c), int(x)) for c, x in zip(core, want[0])}
        assert got[3] == len(nodes)
    finally:
        nd.nd_graph_free(G)


@pytest.mark.parametrize("r,s", RS)
def test_hierarchy_small_graphs(nd, ctx, r, s):
    check_hierarchy(nd, ctx, gg.fig1(), r, s)
    check_hierarchy(nd, ctx, gg.disjoint_union(gg.complete(7), gg.fig1(), gg.complete(s), gg.complete(s + 2)), r, s)
    for seed in range(4):
        check_hierarchy(nd, ctx, gg.gnp(10 + 4 * seed, [0.3, 0.5, 0.7][seed % 3], 9400 + seed), r, s, device=seed % 2 == 1)


@pytest.mark.parametrize("r,s", [(1, 2), (2, 3), (2, 4), (3, 4)])
def test_hierarchy_power_law_and_hubs(nd, ctx, r, s):
    check_hierarchy(nd, ctx, gg.with_planted(gg.chung_lu(1200, 5.0, 2.3, seed=9501), 10, 8, 20, 0.7, seed=9502), r, s)
    check_hierarchy(nd, ctx, gg.hubs_over_sparse(n_common=1500, hubs=3, p_hub=0.9, avg_deg=4.0, seed=9503), r, s,
                    device=True)
    if s - r == 1:
        check_hierarchy(nd, ctx, gg.rmat(11, 8, seed=9504), r, s)


def test_hierarchy_empty_and_bad_core(nd, ctx):
    g = gg.gnp(30, 0.0, 1)
    check_hierarchy(nd, ctx, g, 2, 3)  # no edges: nothing to build
    check_hierarchy(nd, ctx, g, 1, 2)  # isolated vertices: one root node each
    G = nd.nd_load_csr(ctx, g.rowptr, g.col)
    try:
        with pytest.raises(nd.NdError):
            nd.nd_hierarchy(G, 1, 2, np.full(g.n, -1, np.int32))
        with pytest.raises(nd.NdError):
            nd.nd_hierarchy(G, 4, 7, np.zeros(g.n, np.int32))
    finally:
        nd.nd_graph_free(G)


class _Hooks:
    """Allocator hooks that note every size and refuse those of `refuse` bytes and more."""

    def __init__(self, nd):
        self.alloc, self.free = nd.torch_allocator_hooks(0)
        self.refuse, self.sizes = 1 << 60, []

    def take(self, nbytes, stream):
        self.sizes.append(nbytes)
        return 0 if nbytes >= self.refuse else self.alloc(nbytes, stream)

    def largest(self, refuse, call):
        """(result of call, the largest size it asked for) with this limit."""
        self.refuse, self.sizes = refuse, []
        try:
            return call(), max(self.sizes, default=0)
        finally:
            self.refuse = 1 << 60


def _lists(r, s, n_s):
    """Bytes of the rows of the incidence lists."""
    return 4 * ((math.comb(s, r) + 3) // 4 * 4) * n_s


@pytest.mark.parametrize("r,s,scale,ef", [(1, 3, 13, 16), (2, 3, 14, 16), (2, 4, 12, 8), (3, 4, 14, 16), (3, 5, 11, 8), (3, 6, 9, 8), (4, 6, 9, 8)])
def test_with_lists_and_by_listing(nd, r, s, scale, ef):
    """Large enough for the incidence lists to be built, and without the memory for them: the same nuclei at
    the lowest, a middle and the top level, and the same hierarchy."""
    import torch

    g = gg.rmat(scale, ef, seed=9601)
    ctx = nd.nd_ctx_create(0, stream=torch.cuda.Stream())
    hooks = _Hooks(nd)
    nd.nd_ctx_set_allocator(ctx, hooks.take, hooks.free)
    G = nd.nd_load_csr(ctx, g.rowptr, g.col)
    try:
        core, _, st = nd.nd_decompose(G, r, s, want_round=False)
        rows = _lists(r, s, st["n_s"])
        assert rows > 4 * core.size
        dcore = torch.from_numpy(core).cuda()
        for level in (0, int(np.median(core)), int(core.max())):
            (want, n), most = hooks.largest(1 << 60, lambda: nd.nd_nuclei(G, r, s, dcore, level))
            assert level or most >= rows
            (got, k), most = hooks.largest(rows, lambda: nd.nd_nuclei(G, r, s, dcore, level))
            assert level or most >= rows
            assert k == n and torch.equal(got, want)
        want, most = hooks.largest(1 << 60, lambda: nd.nd_hierarchy(G, r, s, dcore))
        assert most >= rows
        got, _ = hooks.largest(rows, lambda: nd.nd_hierarchy(G, r, s, dcore))
        assert got[3] == want[3] and all(torch.equal(a, b) for a, b in zip(got[:3], want[:3]))
    finally:
        nd.nd_graph_free(G)
        nd.nd_ctx_destroy(ctx)


@pytest.mark.parametrize("r,s", [(1, 4), (2, 3), (2, 4), (2, 5), (3, 4), (3, 5), (4, 5)])
def test_a_level_of_few_r_cliques_is_listed(nd, r, s):
    """The nuclei of a level that only one K_25 of a larger graph reaches take no room for the lists of the
    whole graph."""
    import torch

    g = gg.with_planted(gg.chung_lu(40_000, 12.0, 2.3, seed=9701), 1, 25, 25, 1.0, seed=9702)
    ctx = nd.nd_ctx_create(0, stream=torch.cuda.Stream())
    hooks = _Hooks(nd)
    nd.nd_ctx_set_allocator(ctx, hooks.take, hooks.free)
    G = nd.nd_load_csr(ctx, g.rowptr, g.col)
    try:
        core, _, st = nd.nd_decompose(G, r, s, want_round=False)
        top = int(core.max())
        assert np.count_nonzero(core == top) == math.comb(25, r)
        got, most = hooks.largest(1 << 60, lambda: nd.nd_nuclei(G, r, s, core, top))
        want = orc.nuclei(g, r, s, core, top)
        assert got[1] == want[1] == 1 and np.array_equal(got[0], want[0])
        assert most <= 4 * core.size + 256
    finally:
        nd.nd_graph_free(G)
        nd.nd_ctx_destroy(ctx)


def test_lists_that_cannot_fit_are_not_counted_for(nd):
    """K_100 as (3,4), whose lists (125 MB) are over the context's budget: the hierarchy allocates neither counts'
    directory nor anything else as large."""
    import torch

    g = gg.complete(100)
    ctx = nd.nd_ctx_create(0, stream=torch.cuda.Stream(), mem_budget=100 << 20)
    hooks = _Hooks(nd)
    nd.nd_ctx_set_allocator(ctx, hooks.take, hooks.free)
    G = nd.nd_load_csr(ctx, g.rowptr, g.col)
    try:
        core = np.full(len(nd.nd_rcliques(G, 3)), 97, np.int32)
        got, most = hooks.largest(1 << 60, lambda: nd.nd_hierarchy(G, 3, 4, core))
        assert got[3] == 1 and not got[0].any() and np.all(got[1] == -1) and np.all(got[2] == -1)
        assert most <= 4 * core.size + 256
    finally:
        nd.nd_graph_free(G)
        nd.nd_ctx_destroy(ctx)


@pytest.mark.parametrize("r,s", [(1, 3), (2, 3), (1, 4), (2, 4), (2, 5), (3, 4), (3, 5), (3, 6), (4, 6)])
def test_a_budget_on_either_side_of_the_lists(nd, r, s):
    """The hierarchy under budgets that leave half and twice the bytes of the lists, on a graph where the bound on the
    counts does not settle which: read from the lists in one case, listed in the other, and the same."""
    import torch

    g = gg.rmat(13 if s < 5 else 10, 8, seed=9801)

    def run(budget, core):
        """The hierarchy (and the cores, if there are none yet), whether lists were built, bytes held by graph and index."""
        ctx = nd.nd_ctx_create(0, stream=torch.cuda.Stream(), mem_budget=budget)
        hooks = _Hooks(nd)
        nd.nd_ctx_set_allocator(ctx, hooks.take, hooks.free)
        G = nd.nd_load_csr(ctx, g.rowptr, g.col)
        try:
            n_s = nd.nd_count(G, r, s)[2]
            if core is None:
                core = torch.from_numpy(nd.nd_decompose(G, r, s, want_round=False)[0]).cuda()
            held = nd.nd_ctx_bytes_in_use(ctx)
            got, most = hooks.largest(1 << 60, lambda: nd.nd_hierarchy(G, r, s, core))
            return core, n_s, held, most >= _lists(r, s, n_s), got
        finally:
            nd.nd_graph_free(G)
            nd.nd_ctx_destroy(ctx)

    core, n_s, held, built, want = run(0, None)
    assert built
    n_r = core.numel()
    lists = _lists(r, s, n_s) + 4 * math.comb(s, r) * n_s + 16 * n_r
    others = held + 14 * 4 * n_r + (1 << 16)  # the hierarchy's arrays of one int32 for each r-clique, and the counts
    for budget, expect in ((others + lists // 2, False), (others + 2 * lists, True)):
        *_, built, got = run(budget, core)
        assert got[3] == want[3] and all(torch.equal(a, b) for a, b in zip(got[:3], want[:3]))
        # the (3,4) count's directory is larger than its lists here and may take the room of twice them
        assert built == expect or (r, s) == (3, 4)
