"""Failure paths, triggered without faulting or hanging the GPU.

* Round cap: a context limited to 2 peeling rounds gives ND_ETIMEOUT on a graph that needs more,
  in every launch mode of the peeling loop; the same context then decomposes correctly.
* Bounded grid-barrier wait: with ND_LIMIT_DROP_BLOCK the last block of the persistent peel
  kernel leaves before its first barrier, so the other blocks wait for an arrival that never
  comes; each wait is bounded (here 50 ms), every block leaves, and the call returns
  ND_ETIMEOUT within about a second. The context stays usable and the next decomposition
  matches the oracle.
* Count overflow: with a width-4 count limit below the graph's largest count, width 4 gives
  ND_EOVERFLOW, while width 8 (and the automatic choice) give the oracle's result.
* Malformed graphs loaded without ND_VALIDATE: refused before an entry is used as an index.
"""
import time

import numpy as np
import pytest

import graphgen as gg
import oracle as orc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nd():
    import paper_2111_10980_gb300 as nd

    nd.lib()
    return nd


def _decompose(nd, ctx, g, r, s, **kw):
    G = nd.nd_load_csr(ctx, g.rowptr, g.col)
    try:
        return nd.nd_decompose(G, r, s, **kw)
    finally:
        nd.nd_graph_free(G)


def test_round_cap_gives_etimeout(nd):
    g = gg.rmat(11, 16, 0.57, 0.19, 0.19, seed=61)
    want = orc.decompose(g, 2, 3)
    assert want.rho > 2
    ctx = nd.nd_ctx_create(0)
    try:
        nd.nd_ctx_set_limits(ctx, max_rounds=2)
        for flags in (nd.ND_PEEL_PERSISTENT, nd.ND_PEEL_LOOP_GRAPH, nd.ND_NO_GRAPH):
            with pytest.raises(nd.NdError) as ei:
                _decompose(nd, ctx, g, 2, 3, flags=flags)
            assert ei.value.code == nd.ND_ETIMEOUT, flags
            assert "round cap" in str(ei.value)
        # a cap above rho changes nothing
        nd.nd_ctx_set_limits(ctx, max_rounds=want.rho)
        core, rnd, st = _decompose(nd, ctx, g, 2, 3)
        assert np.array_equal(core, want.core) and st["rho"] == want.rho
        nd.nd_ctx_set_limits(ctx)
        core, rnd, _ = _decompose(nd, ctx, g, 2, 3)
        assert np.array_equal(core, want.core) and np.array_equal(rnd, want.round)
    finally:
        nd.nd_ctx_destroy(ctx)


@pytest.mark.parametrize("r,s", [(2, 3), (3, 4)])
def test_bounded_barrier_wait_gives_etimeout(nd, r, s):
    g = gg.chung_lu(3000, 20.0, 2.2, seed=62)
    want = orc.decompose(g, r, s)
    ctx = nd.nd_ctx_create(0)
    try:
        nd.nd_ctx_set_limits(ctx, barrier_timeout_ns=50_000_000, flags=nd.ND_LIMIT_DROP_BLOCK)
        t0 = time.perf_counter()
        with pytest.raises(nd.NdError) as ei:
            _decompose(nd, ctx, g, r, s, flags=nd.ND_PEEL_PERSISTENT)
        dt = time.perf_counter() - t0
        assert ei.value.code == nd.ND_ETIMEOUT
        assert "barrier" in str(ei.value)
        assert dt < 10.0, dt
        # the context is still usable: the next decompositions match the oracle
        nd.nd_ctx_set_limits(ctx)
        for flags in (nd.ND_PEEL_PERSISTENT, 0):
            core, rnd, st = _decompose(nd, ctx, g, r, s, flags=flags)
            assert np.array_equal(core, want.core) and np.array_equal(rnd, want.round)
            assert st["listed"] == want.n_s
    finally:
        nd.nd_ctx_destroy(ctx)


def test_width4_count_overflow_gives_eoverflow(nd):
    g = gg.complete(10)  # every triangle lies in 7 4-cliques, every edge in 8 triangles
    ctx = nd.nd_ctx_create(0)
    try:
        nd.nd_ctx_set_limits(ctx, count_limit=6)
        G = nd.nd_load_csr(ctx, g.rowptr, g.col)
        try:
            for fn in (lambda: nd.nd_count(G, 3, 4, count_width=4), lambda: nd.nd_decompose(G, 3, 4, count_width=4)):
                with pytest.raises(nd.NdError) as ei:
                    fn()
                assert ei.value.code == nd.ND_EOVERFLOW
            counts, _, _ = nd.nd_count(G, 3, 4, count_width=8)
            assert np.all(counts == 7)
            for width in (0, 8):
                core, _, st = nd.nd_decompose(G, 3, 4, count_width=width)
                assert np.all(core == 7) and st["count_width"] == 8
            # (2,3): counts of 8 also exceed the limit; (1,2) degrees of 9 too
            with pytest.raises(nd.NdError) as ei:
                nd.nd_decompose(G, 2, 3, count_width=4)
            assert ei.value.code == nd.ND_EOVERFLOW
        finally:
            nd.nd_graph_free(G)
        nd.nd_ctx_set_limits(ctx, count_limit=7)
        core, _, st = _decompose(nd, ctx, g, 3, 4, count_width=4)
        assert np.all(core == 7) and st["count_width"] == 4
    finally:
        nd.nd_ctx_destroy(ctx)


def test_limits_reject_bad_arguments(nd):
    ctx = nd.nd_ctx_create(0)
    try:
        with pytest.raises(nd.NdError) as ei:
            nd.nd_ctx_set_limits(ctx, max_rounds=-1)
        assert ei.value.code == nd.ND_EINVAL
        with pytest.raises(nd.NdError) as ei:
            nd.nd_ctx_set_limits(ctx, flags=0x100)
        assert ei.value.code == nd.ND_EINVAL
    finally:
        nd.nd_ctx_destroy(ctx)


@pytest.mark.parametrize("bad_id", [-1, -(1 << 31), 60, (1 << 31) - 1])
@pytest.mark.parametrize("where", ["first", "last", "all"])
def test_ids_out_of_range_are_refused_without_validate(nd, bad_id, where):
    """A CSR with ids that are no vertices is refused with ND_EINVAL before any row is looked up by one of
    them, whether or not its upper and lower entries still balance."""
    g = gg.chung_lu(60, 6.0, 2.3, seed=62)
    col = g.col.copy()
    col[{"first": 0, "last": -1, "all": slice(None)}[where]] = bad_id
    ctx = nd.nd_ctx_create(0)
    try:
        G = nd.nd_load_csr(ctx, g.rowptr, col)
        with pytest.raises(nd.NdError) as ei:
            nd.nd_decompose(G, 2, 3)
        assert ei.value.code == nd.ND_EINVAL
        nd.nd_graph_free(G)
        core, rnd, _ = _decompose(nd, ctx, g, 2, 3)
        assert np.array_equal(core, orc.decompose(g, 2, 3).core)
    finally:
        nd.nd_ctx_destroy(ctx)


def _csr(n, rows):
    """CSR of these rows as they are: {vertex: entries}."""
    rowptr = np.zeros(n + 1, np.int64)
    for u, row in rows.items():
        rowptr[u + 1] = len(row)
    return np.cumsum(rowptr), np.concatenate([np.asarray(rows.get(u, ()), np.int32) for u in range(n)]).astype(np.int32)


def _clique_rows(k):
    return {u: [v for v in range(k) if v != u] for u in range(k)}


def _refused(nd, ctx, n, rows, call):
    G = nd.nd_load_csr(ctx, *_csr(n, rows))
    try:
        with pytest.raises(nd.NdError) as ei:
            call(G)
        assert ei.value.code == nd.ND_EINVAL
    finally:
        nd.nd_graph_free(G)


@pytest.mark.parametrize("k", [4, 40, 130, 131])
def test_a_duplicate_edge_of_a_triangle_is_refused_by_the_triangle_index(nd, k):
    """An edge that its two rows hold twice, in cliques whose edges have up to 128 common neighbours (lists
    ordered by counting) and more (lists merged out of the rows); so are rows out of order."""
    ctx = nd.nd_ctx_create(0)
    try:
        for u, v in ((0, 1), (0, k - 1), (k - 2, k - 1)):
            rows = _clique_rows(k)
            rows[u] = sorted(rows[u] + [v])
            rows[v] = sorted(rows[v] + [u])
            _refused(nd, ctx, k, rows, lambda G: nd.nd_rcliques(G, 3))
            for r, s in ((3, 4), (3, 5), (4, 5)):
                _refused(nd, ctx, k, rows, lambda G: nd.nd_decompose(G, r, s))
        rows = _clique_rows(k)
        rows[0] = rows[0][:-2] + rows[0][:-3:-1]
        _refused(nd, ctx, k, rows, lambda G: nd.nd_count(G, 3, 4))
    finally:
        nd.nd_ctx_destroy(ctx)


def test_entries_without_or_with_too_many_reverses_are_refused(nd):
    """As many upper as lower entries, and every lower entry has a reverse, but not every upper one: a
    duplicate lower entry makes up the number."""
    ctx = nd.nd_ctx_create(0)
    try:
        # 0-1 twice in row 0, once in row 1; 8-9 the other way round, so that the totals agree. Vertex 1 and vertex 8
        # have the larger degree, so both sides of the orientation take the doubled row
        rows = {0: [1, 1], 1: [0, 2, 3, 4], 2: [1], 3: [1], 4: [1], 5: [8], 6: [8], 7: [8], 8: [5, 6, 7, 9], 9: [8, 8]}
        _refused(nd, ctx, 10, rows, lambda G: nd.nd_orient(G, nd.ND_ORIENT_DEGREE))
        # vertex 0 lists 3, which does not list 0; 5 lists 4 twice and has the smaller degree of the two, so that
        # the orientation takes as many edges as there should be
        rows = {0: [1, 2, 3], 1: [0, 2, 3], 2: [0, 1, 3], 3: [1, 2], 4: [5, 6, 7], 5: [4, 4], 6: [4], 7: [4]}
        _refused(nd, ctx, 8, rows, lambda G: nd.nd_rcliques(G, 3))
    finally:
        nd.nd_ctx_destroy(ctx)


def test_a_duplicate_edge_outside_triangles_is_accepted(nd):
    """The triangles and their cores are those of the graph without the duplicate."""
    k, ctx = 6, nd.nd_ctx_create(0)
    try:
        got = []
        for times in (1, 2):
            rows = _clique_rows(k)
            rows[k - 1] = rows[k - 1] + [k] * times
            rows[k] = [k - 1] * times
            G = nd.nd_load_csr(ctx, *_csr(k + 1, rows))
            got.append([nd.nd_rcliques(G, 3)] + [nd.nd_decompose(G, 3, s)[0] for s in (4, 5)])
            nd.nd_graph_free(G)
        for a, b in zip(*got):
            assert np.array_equal(a, b)
        assert np.array_equal(got[0][1], np.full(20, k - 3))
    finally:
        nd.nd_ctx_destroy(ctx)


def test_another_orientation_without_memory_leaves_the_graph_usable(nd):
    """nd_orient to another mode, refused each of its allocations in turn: ND_ENOMEM, and the next call on the
    graph orients it again."""
    import torch

    g = gg.chung_lu(300, 10.0, 2.2, seed=63)
    want = orc.decompose(g, 2, 3)
    alloc, free = nd.torch_allocator_hooks(0)
    left = [None]

    def take(nbytes, stream):
        if left[0] is not None:
            left[0] -= 1
            if left[0] < 0:
                return 0
        return alloc(nbytes, stream)

    ctx = nd.nd_ctx_create(0, stream=torch.cuda.Stream())
    nd.nd_ctx_set_allocator(ctx, take, free)
    G = nd.nd_load_csr(ctx, g.rowptr, g.col)
    refused = 0
    try:
        for i in range(200):
            nd.nd_orient(G, nd.ND_ORIENT_DEGREE)
            left[0] = i
            try:
                nd.nd_orient(G, nd.ND_ORIENT_DEGENERACY)
                break
            except nd.NdError as e:
                assert e.code == nd.ND_ENOMEM
                refused += 1
            finally:
                left[0] = None
            core, rnd, st = nd.nd_decompose(G, 2, 3)
            assert np.array_equal(core, want.core) and np.array_equal(rnd, want.round)
        assert 5 < refused < 199
    finally:
        nd.nd_graph_free(G)
        nd.nd_ctx_destroy(ctx)
