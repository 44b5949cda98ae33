"""Sizes at which the kernels change their way: closed forms on cliques whose edges have 127, 128 and
129 common neighbours (lists gathered and ordered up to 128, merged out of the rows beyond; the 4-cliques of
an edge staged up to 128 common out-neighbours, walked beyond), next to a hub whose row runs over many
segments of the edge index, long runs of empty rows before, between and after, and graphs too small to fill
a warp."""
import itertools
import math

import numpy as np
import pytest

import graphgen as gg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nd():
    import paper_2111_10980_gb300 as nd

    nd.lib()
    return nd


def _graph(cliques, leaves, gap):
    """Cliques of these sizes, then a star with that many leaves, with `gap` isolated vertices around each."""
    us, vs, first, at = [], [], [], gap
    for n in cliques:
        iu, ju = np.triu_indices(n, 1)
        us.append(iu + at)
        vs.append(ju + at)
        first.append(at)
        at += n + gap
    us.append(np.full(leaves, at + leaves // 2))  # the hub in the middle of its leaves' ids
    vs.append(at + np.delete(np.arange(leaves + 1), leaves // 2))
    n = at + leaves + 1 + gap
    return gg.csr_from_edges(n, np.concatenate(us).astype(np.int32), np.concatenate(vs).astype(np.int32)), first


@pytest.mark.parametrize("cliques,leaves,gap,limit", [((129, 130, 131), 5000, 300, None), ((2, 3, 4, 5), 1, 0, None), ((33, 34), 70, 40, None),
                                                      ((129, 130, 131), 60_000, 300, None), ((129, 130, 131), 60_000, 300, 14 << 20)])
def test_cliques_and_a_hub(nd, cliques, leaves, gap, limit):
    """With incidence lists ((2,3), and (2,4) where so many edges without s-cliques make the counts skewed), and where
    an allocator refuses their large buffers without."""
    import torch

    g, first = _graph(cliques, leaves, gap)
    alloc, free = nd.torch_allocator_hooks(0)
    large = []

    def hook(nbytes, stream):
        if nbytes >= 14 << 20:
            large.append(nbytes)
            if limit is not None:
                return 0
        return alloc(nbytes, stream)

    ctx = nd.nd_ctx_create(0, stream=torch.cuda.Stream())
    nd.nd_ctx_set_allocator(ctx, hook, free)
    G = nd.nd_load_csr(ctx, g.rowptr, g.col, flags=nd.ND_VALIDATE)
    try:
        edges = nd.nd_rcliques(G, 2)
        assert np.array_equal(edges, g.edges())
        tri = nd.nd_rcliques(G, 3)
        want = [np.array(list(itertools.combinations(range(n), 3)), np.int32).reshape(-1, 3) + a
                for n, a in zip(cliques, first)]
        assert np.array_equal(tri, np.concatenate(want))
        for r, s, cl in ((2, 3, edges), (2, 4, edges), (3, 4, tri)):
            large.clear()
            core, rnd, st = nd.nd_decompose(G, r, s)
            assert bool(large) or r == 3 or leaves < 60_000
            counts, _, n_s = nd.nd_count(G, r, s)
            # every r-clique of K_n lies in C(n - r, s - r) of its s-cliques, and all of them go at once
            expect = np.zeros(len(cl), np.int64)
            for n, a in zip(cliques, first):
                expect[(cl[:, 0] >= a) & (cl[:, -1] < a + n)] = math.comb(max(n - r, 0), s - r)
            assert np.array_equal(core, expect) and np.array_equal(counts, expect), (r, s)
            assert st["rho"] == len(np.unique(expect)) and st["listed"] == n_s == st["n_s"]
            assert np.array_equal(rnd, np.searchsorted(np.unique(expect), expect))
    finally:
        nd.nd_graph_free(G)
        nd.nd_ctx_destroy(ctx)


def _hooked(nd, refuse):
    """A context whose allocations are noted in a list, and refused where refuse(nbytes)."""
    import torch

    alloc, free = nd.torch_allocator_hooks(0)
    sizes = []

    def take(nbytes, stream):
        sizes.append(nbytes)
        return 0 if refuse(nbytes) else alloc(nbytes, stream)

    ctx = nd.nd_ctx_create(0, stream=torch.cuda.Stream())
    nd.nd_ctx_set_allocator(ctx, take, free)
    return ctx, sizes


def _scratch(n3):
    """Bytes that gathering the short lists of n3 triangles takes."""
    return (36 * n3 + 255) // 256 * 256


@pytest.mark.parametrize("leaves", [0, 1200])
def test_short_lists_of_long_rows_are_gathered(nd, leaves):
    """K_129, K_130 and K_131 (lists of 127, 128 and 129), alone and with so many leaves at every vertex of the first
    two that their rows are not worth merging."""
    cliques, us, vs, first, at = (129, 130, 131), [], [], [], 0
    for n in cliques:
        iu, ju = np.triu_indices(n, 1)
        us.append(iu + at)
        vs.append(ju + at)
        first.append(at)
        at += n
    hung = at + np.arange(259 * leaves)
    us.append(np.repeat(np.arange(259), leaves))
    vs.append(hung)
    g = gg.csr_from_edges(at + hung.size, np.concatenate(us).astype(np.int32), np.concatenate(vs).astype(np.int32))
    n3 = sum(math.comb(n, 3) for n in cliques)
    ctx, sizes = _hooked(nd, lambda nbytes: False)
    G = nd.nd_load_csr(ctx, g.rowptr, g.col, flags=nd.ND_VALIDATE)
    try:
        tri = nd.nd_rcliques(G, 3)
        assert (_scratch(n3) in sizes) == (leaves > 0)
        want = [np.array(list(itertools.combinations(range(n), 3)), np.int32) + a for n, a in zip(cliques, first)]
        assert np.array_equal(tri, np.concatenate(want))
        core, rnd, st = nd.nd_decompose(G, 3, 4)
        assert np.array_equal(core, np.repeat([n - 3 for n in cliques], [math.comb(n, 3) for n in cliques]))
        assert np.array_equal(rnd, core - 126) and st["listed"] == sum(math.comb(n, 4) for n in cliques)
    finally:
        nd.nd_graph_free(G)
        nd.nd_ctx_destroy(ctx)


@pytest.mark.parametrize("n", [1, 31, 4097, 60_000, 400_000])
def test_the_triangle_index_gathered_and_merged(nd, n):
    """The same index, seen through the triangles, the 4-cliques' counts and the (3,4) and (4,5) results, whether
    the short lists are gathered or, refused the scratch, merged out of the rows; from one edge per warp and step of
    the list kernels to 32."""
    g = gg.chung_lu(n, min(24.0, n / 4), 2.2, seed=9901)
    got, scratch = [], None
    for refused in (False, True):
        ctx, sizes = _hooked(nd, lambda nbytes: refused and nbytes == scratch)
        G = nd.nd_load_csr(ctx, g.rowptr, g.col, flags=nd.ND_VALIDATE)
        try:
            tri = nd.nd_rcliques(G, 3)
            scratch = _scratch(len(tri)) if len(tri) >= 1 << 16 else None  # fewer triangles are not gathered
            assert scratch is None or scratch in sizes
            got.append([tri, nd.nd_count(G, 3, 4)[0], *nd.nd_decompose(G, 3, 4)[:2], nd.nd_decompose(G, 4, 5)[0]])
        finally:
            nd.nd_graph_free(G)
            nd.nd_ctx_destroy(ctx)
    for a, b in zip(*got):
        assert np.array_equal(a, b)
