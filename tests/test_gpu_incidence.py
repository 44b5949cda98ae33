"""Peeling from incidence lists against peeling by listing the s-cliques again.

The lists are an accelerator that a context without the memory for them does without: an allocator
that refuses the large buffers sends the same decomposition down the other path. Both have to
give the oracle's cores, rounds and statistics, for every row length C(s,r) (3 to 20) and its padding.
"""
import math

import numpy as np
import pytest

import graphgen as gg
import oracle as orc
from test_gpu_parity import assert_parity

pytestmark = pytest.mark.gpu

RS = [(1, 3), (1, 4), (2, 3), (2, 4), (2, 5), (3, 4), (3, 5), (3, 6), (4, 5), (4, 6)]


@pytest.fixture(scope="module")
def nd():
    import paper_2111_10980_gb300 as nd

    nd.lib()
    return nd


@pytest.mark.parametrize("r,s", RS)
def test_with_and_without_room_for_the_lists(nd, r, s):
    import torch

    # dense communities over a sparse graph, so that the rows are the largest buffer (next to the stages
    # of the heavy edges when (2,4) lists its s-cliques again)
    g = gg.with_planted(gg.chung_lu(1200, 6.0, 2.3, seed=91), 30 if r == 2 and s < 5 else 12, 14, 20, 0.85, seed=92)
    rows = 4 * ((math.comb(s, r) + 3) // 4 * 4) * orc.decompose(g, r, s).n_s
    alloc, free = nd.torch_allocator_hooks(0)
    for limit in (None, rows):
        refused = []

        def hook(nbytes, stream):
            if limit is not None and nbytes >= limit:
                refused.append(nbytes)
                return 0
            return alloc(nbytes, stream)

        ctx = nd.nd_ctx_create(0, stream=torch.cuda.Stream())
        nd.nd_ctx_set_allocator(ctx, hook, free)
        try:
            for flags in (0, nd.ND_CONTRACT_ALWAYS, nd.ND_CONTRACT_OFF, nd.ND_PEEL_LOOP_GRAPH, nd.ND_NO_GRAPH):
                assert_parity(nd, ctx, g, r, s, flags=flags)
        finally:
            nd.nd_ctx_destroy(ctx)
        assert bool(refused) == (limit is not None)


@pytest.mark.parametrize("r,s", RS)
def test_no_s_clique(nd, r, s):
    g = gg.path(50)
    ctx = nd.nd_ctx_create(0)
    try:
        G = nd.nd_load_csr(ctx, g.rowptr, g.col)
        core, rnd, st = nd.nd_decompose(G, r, s)
        nd.nd_graph_free(G)
        assert st["n_s"] == 0 and not np.any(core) and st["rho"] == (1 if st["n_r"] else 0)
    finally:
        nd.nd_ctx_destroy(ctx)


@pytest.mark.parametrize("r,s", [(2, 3), (2, 4), (3, 5)])
def test_the_memory_of_a_run_without_lists_is_enough(nd, r, s):
    """A decomposition succeeds in exactly the bytes it needs without lists, wherever a run that tries
    them first runs out."""
    import torch

    g = gg.with_planted(gg.chung_lu(1200, 6.0, 2.3, seed=91), 30 if (r, s) == (2, 4) else 12, 14, 20, 0.85, seed=92)
    want = orc.decompose(g, r, s)
    rows = 4 * ((math.comb(s, r) + 3) // 4 * 4) * want.n_s
    alloc, free = nd.torch_allocator_hooks(0)
    held = {"now": 0, "peak": 0}

    def run(refuse, cap):
        held.update(now=0, peak=0)

        def take(nbytes, stream):
            if refuse and nbytes >= rows or held["now"] + nbytes > cap:
                return 0
            held["now"] += nbytes
            held["peak"] = max(held["peak"], held["now"])
            return alloc(nbytes, stream)

        def give(p, nbytes, stream):
            held["now"] -= nbytes
            free(p, nbytes, stream)

        ctx = nd.nd_ctx_create(0, stream=torch.cuda.Stream())
        nd.nd_ctx_set_allocator(ctx, take, give)
        try:
            G = nd.nd_load_csr(ctx, g.rowptr, g.col)
            core, rnd, st = nd.nd_decompose(G, r, s)
            nd.nd_graph_free(G)
        finally:
            nd.nd_ctx_destroy(ctx)
        assert np.array_equal(core, want.core) and np.array_equal(rnd, want.round) and st["listed"] == want.n_s
        return held["peak"]

    alone = run(True, 1 << 40)
    for extra in (0, rows // 2, rows, 2 * rows):
        run(False, alone + extra)


def test_a_peel_without_room_next_to_its_lists_has_its_directory(nd):
    """K_60 and K_5 as (3,4): when the peel's buffers are refused next to the incidence lists, the peel without them
    finds the hash directory that it looks up, which had made room for the lists."""
    import torch

    g = gg.disjoint_union(gg.complete(60), gg.complete(5))
    n_s = math.comb(60, 4) + 5
    want = np.repeat([57, 2], [math.comb(60, 3), 10])
    table = 16 * math.comb(60, 2) << 7  # 58 entries in 128 slots for every edge of K_60
    alloc, free = nd.torch_allocator_hooks(0)
    sizes, full, refused, arm = [], [False], [], False

    def take(nbytes, stream):
        if full[0]:
            refused.append(nbytes)
            return 0
        sizes.append(nbytes)
        return alloc(nbytes, stream)

    def give(p, nbytes, stream):
        if arm:
            full[0] = (full[0] or nbytes == table) and not refused  # from when the directory goes until the lists do
        free(p, nbytes, stream)

    ctx = nd.nd_ctx_create(0, stream=torch.cuda.Stream())
    nd.nd_ctx_set_allocator(ctx, take, give)
    G = nd.nd_load_csr(ctx, g.rowptr, g.col)
    try:
        nd.nd_rcliques(G, 3)
        for arm, tables in ((False, 1), (True, 2)):
            sizes.clear()
            core, rnd, st = nd.nd_decompose(G, 3, 4)
            assert np.array_equal(core, want) and np.array_equal(rnd, want > 2) and st["rho"] == 2 and st["listed"] == n_s
            assert max(sizes) >= 4 * 4 * n_s and sizes.count(table) == tables and bool(refused) == arm
    finally:
        arm = False
        nd.nd_graph_free(G)
        nd.nd_ctx_destroy(ctx)


@pytest.mark.parametrize("r,s,n,other,lists", [(1, 3, 100, 0, False), (2, 3, 60, 0, False), (2, 4, 60, 0, False), (3, 4, 60, 0, False),
                                               (2, 5, 20, 0, True), (1, 3, 100, 5, True), (2, 3, 60, 5, True), (2, 4, 60, 5, True),
                                               (3, 4, 60, 5, True), (2, 4, 125, 5, False), (3, 4, 110, 5, False)])
def test_lists_only_where_the_rounds_outweigh_them(nd, r, s, n, other, lists):
    """Cliques, alone (equal counts: one round) and next to a smaller one (two rounds, however many s-cliques):
    no lists where every (r,s) with an Update of its own is sooner without, and the closed form either way."""
    import torch

    g = gg.disjoint_union(gg.complete(n), gg.complete(other)) if other else gg.complete(n)
    want = np.repeat([math.comb(n - r, s - r), math.comb(max(other - r, 0), s - r)], [math.comb(n, r), math.comb(other, r)])
    n_s = math.comb(n, s) + math.comb(other, s)
    alloc, free = nd.torch_allocator_hooks(0)
    sizes = []

    def take(nbytes, stream):
        sizes.append(nbytes)
        return alloc(nbytes, stream)

    ctx = nd.nd_ctx_create(0, stream=torch.cuda.Stream())
    nd.nd_ctx_set_allocator(ctx, take, free)
    try:
        G = nd.nd_load_csr(ctx, g.rowptr, g.col)
        nd.nd_count(G, r, s)
        sizes.clear()
        core, rnd, st = nd.nd_decompose(G, r, s)
        nd.nd_graph_free(G)
    finally:
        nd.nd_ctx_destroy(ctx)
    assert np.array_equal(core, want) and np.array_equal(rnd, want == want[0] if other else 0 * want)
    assert st["n_s"] == st["listed"] == n_s and st["rho"] == (2 if other else 1)
    rows = 4 * ((math.comb(s, r) + 3) // 4 * 4) * n_s
    assert (max(sizes) >= rows) == lists, sizes
