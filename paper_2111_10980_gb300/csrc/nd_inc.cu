// Incidence lists for the peel: every s-clique once, as the ids of its r-subsets, and for every r-clique
// the numbers of the s-cliques it lies in (PeelView::inc_*). Update then reads lists instead of
// listing the s-cliques of each peeled r-clique again (Algorithm 2, Update), which for one r-clique is
// a chain of up to twenty-five dependent accesses and for all of them C(s,r) listings of each s-clique.
//
// The lists take (stride + C(s,r)) * 4 bytes for each s-clique, 16 for each r-clique (offsets, and cursors while
// they are filled) and a few spare rows (nd_inc_rows); they are built from the counts (their
// lengths) in one more listing. Rows come in listing order, so the members of neighbouring rows
// lie close together; the order inside an r-clique's list is that of the atomics and has no meaning.
//
// Measured, count and peel with the lists' building, before and after: (2,4) on a Chung-Lu graph of
// 500,009 vertices with 500 communities (8.4 M 4-cliques, 1,968 rounds) 87 -> 36 ms; (4,5) on a flat R-MAT
// graph of 40,000 vertices, degeneracy order and all, 15.4 -> 12.1 ms; (3,4) on a Chung-Lu graph of a million
// vertices (17 M 4-cliques) 64.0 -> 61.7 ms; (2,3) on R-MAT scale 20 (374 M triangles, 2,107 rounds) 208 ->
// 144 ms, the fill 34 ms of it.
#include "nd_common.cuh"
#include "nd_gen.cuh"
#include "nd_quad24.cuh"
#include "nd_tri.cuh"

namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ int64_t gwarp() { return ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; }
__device__ __forceinline__ int64_t nwarps() { return ((int64_t)gridDim.x * blockDim.x) >> 5; }

int blocks_for_warps(int64_t items) {
    int64_t want = (items + kThreads / 32 - 1) / (kThreads / 32), cap = (int64_t)nd_sm_count() * 16;
    if (want < 1) want = 1;
    return (int)(want < cap ? want : cap);
}

// A warp's run of rows: F.run at a time, or what it needs if that is more, from one counter (a counter update for
// every handful of matches is what the first form of k_inc_tri waited for: 130 ms for the 374 M triangles of
// R-MAT scale 20).
struct IncRun {
    unsigned at = 0, left = 0, used = 0;
};

// row and list places of one s-clique
template <int C>
__device__ __forceinline__ void inc_write(const IncFill& F, unsigned S, const int32_t* id) {
    if (S >= F.rows) {
        F.status[2] = 1;
        return;
    }
    unsigned long long at[C];
#pragma unroll
    for (int i = 0; i < C; ++i) at[i] = atomicAdd(&F.cursor[id[i]], 1ull);
    constexpr int kStride = (C + 3) / 4 * 4;
    int4* row = reinterpret_cast<int4*>(F.row + (int64_t)S * kStride);
#pragma unroll
    for (int i = 0; i < kStride; i += 4)
        row[i / 4] = make_int4(id[i], i + 1 < C ? id[i + 1] : -1, i + 2 < C ? id[i + 2] : -1, i + 3 < C ? id[i + 3] : -1);
#pragma unroll
    for (int i = 0; i < C; ++i) {
        if ((int64_t)at[i] < F.entries)
            F.list[at[i]] = S;
        else
            F.status[2] = 1;
    }
}

// The s-cliques of the lanes with hit set, members id[0..C). The whole warp calls it.
template <int C>
__device__ __forceinline__ void inc_put(const IncFill& F, IncRun& run, bool hit, const int32_t* id) {
    const unsigned full = 0xffffffffu, mask = __ballot_sync(full, hit);
    const unsigned n = __popc(mask), rank = __popc(mask & nd_lanemask_lt());
    unsigned next = 0;
    const unsigned more = n > run.left ? n - run.left : 0, take = more > F.run ? more : F.run;
    if (more) {
        if ((threadIdx.x & 31) == 0) next = atomicAdd(&F.status[0], take);
        next = __shfl_sync(full, next, 0);
    }
    const unsigned S = rank < run.left ? run.at + rank : next + (rank - run.left);
    if (more) {
        run.at = next + more;
        run.left = take - more;
    } else {
        run.at += n;
        run.left -= n;
    }
    run.used += n;
    if (hit) inc_write<C>(F, S, id);
}

__device__ __forceinline__ void inc_done(const IncFill& F, const IncRun& run) {
    if ((threadIdx.x & 31) == 0 && run.used) atomicAdd(&F.status[1], run.used);
}

// The same from lanes that come as they find them: a row each from the counter
template <int C>
__device__ __forceinline__ void inc_put_any(const IncFill& F, const int32_t* id) {
    const unsigned mask = __activemask();
    const int lane = threadIdx.x & 31, leader = __ffs(mask) - 1;
    unsigned base = 0;
    if (lane == leader) {
        base = atomicAdd(&F.status[0], (unsigned)__popc(mask));
        atomicAdd(&F.status[1], (unsigned)__popc(mask));
    }
    inc_write<C>(F, __shfl_sync(mask, base, leader) + __popc(mask & nd_lanemask_lt()), id);
}

// (1,3), (2,3): every triangle of DG
template <int R_>
struct PutTri {
    IncFill F;
    const int32_t* eid;
    IncRun run;
    __device__ void begin(int) const {}
    __device__ void tri(bool hit, int, int32_t e, int32_t px, int32_t py, bool, int32_t u, int32_t v, int32_t w) {
        int32_t id[3] = {u, v, w};
        if (R_ == 2 && hit) {
            id[0] = e;
            id[1] = eid[px];
            id[2] = eid[py];
        }
        inc_put<3>(F, run, hit, id);
    }
    __device__ void end(int, int32_t, int32_t, int32_t) const {}
};

template <int R_>
__global__ void __launch_bounds__(kTriThreads) k_inc_tri(GraphView g, int tile, IncFill F) {
    PutTri<R_> sink{F, g.dg_eid, IncRun{}};
    tri_list(g, tile, sink);
    inc_done(F, sink.run);
}

struct Put24 {
    IncFill F;
    IncRun run;
    static constexpr bool kTally = false;
    __device__ void clique(bool hit, const int32_t (&e)[6]) { inc_put<6>(F, run, hit, e); }
};

__global__ void __launch_bounds__(kQuadThreads) k_inc24(GraphView g, IncFill F) {
    Put24 sink{F, IncRun{}};
    quad24_list(g, sink);
    inc_done(F, sink.run);
}

// (3,4): every 4-clique from its lowest triangle (a < b < c): the vertices w > c of the shortest of the
// triangle's three lists that the other two hold as well; each entry names its triangle
__device__ __forceinline__ bool inc_look(const GraphView& g, int32_t e, int64_t b, int64_t n, int32_t w, int32_t& id) {
    if (g.htab && nd_hashed(n)) {
        int32_t rnd;
        return nd_hash_find(g.htab + g.hoff[e], nd_hash_bits(n), w, id, rnd);
    }
    const int64_t i = nd_find(g.et_w + b, n, w);
    if (i < 0) return false;
    id = g.et_t[b + i];
    return true;
}

__global__ void k_inc34(GraphView g, IncFill F) {
    int lane = threadIdx.x & 31;
    IncRun run;
    for (int64_t t = gwarp(); t < g.n3; t += nwarps()) {
        int32_t e[3];
        int64_t b[3], n[3];
        int d = 0;
#pragma unroll
        for (int x = 0; x < 3; ++x) {
            e[x] = g.tri_e[3 * t + x];
            b[x] = g.et_rp[e[x]];
            n[x] = g.et_rp[e[x] + 1] - b[x];
        }
        if (n[1] < n[0]) d = 1;
        if (n[2] < (d ? n[1] : n[0])) d = 2;
        const int32_t c = g.ev[e[1]];  // edges (ab, ac, bc): the largest vertex is ac's upper end
        const int64_t bd = d == 0 ? b[0] : d == 1 ? b[1] : b[2], nd = d == 0 ? n[0] : d == 1 ? n[1] : n[2];
        const int32_t e1 = d == 0 ? e[1] : e[0], e2 = d == 2 ? e[1] : e[2];
        const int64_t b1 = d == 0 ? b[1] : b[0], n1 = d == 0 ? n[1] : n[0];
        const int64_t b2 = d == 2 ? b[1] : b[2], n2 = d == 2 ? n[1] : n[2];
        for (int64_t j0 = nd_lower_bound(g.et_w + bd, nd, c + 1); j0 < nd; j0 += 32) {
            const int64_t j = j0 + lane;
            int32_t id[4] = {(int32_t)t, 0, 0, 0};
            bool hit = false;
            if (j < nd) {
                const int32_t w = g.et_w[bd + j];
                id[1] = g.et_t[bd + j];
                hit = inc_look(g, e1, b1, n1, w, id[2]) && inc_look(g, e2, b2, n2, w, id[3]);
            }
            inc_put<4>(F, run, hit, id);
        }
    }
    inc_done(F, run);
}

// Any other (r,s): every s-clique from the r-clique of its r lowest vertices, the others above them
template <int R_, int S_, int C = gen_binom(S_, R_)>
__global__ void k_inc_gen(GraphView g, int64_t n_r, IncFill F) {
    constexpr int K = S_ - R_;
    int lane = threadIdx.x & 31;
    for (int64_t id = gwarp(); id < n_r; id += nwarps()) {
        int32_t v[4];
        gen_verts<R_>(g, id, v);
        const int32_t* list = nullptr;
        int64_t len = 0;
        gen_drive<R_>(g, id, v, list, len);
        const int32_t top = v[R_ - 1];
        for (int64_t j = nd_lower_bound(list, len, top + 1) + lane; j < len; j += 32)
            gen_cand<R_, S_>(g, v, list[j], [&](const int32_t* Cv) {
                if (K > 1 && Cv[1] < top) return;
                if (K > 2 && Cv[2] < top) return;
                int32_t Sv[S_], o[C];
                gen_merge<R_, S_>(v, Cv, Sv);
                o[0] = (int32_t)id;
                if (!gen_others<R_, S_>(g, v, Sv, o + 1)) {
                    F.status[2] = 1;
                    return;
                }
                inc_put_any<C>(F, o);
            });
    }
}

}  // namespace

int nd_inc_stride(int r, int s) {
    int c = 1;
    for (int i = 1; i <= r; ++i) c = c * (s - r + i) / i;
    return (c + 3) / 4 * 4;
}

// the work items of a fill kernel, one per warp at a time
static int64_t inc_items(int r, int s, int64_t n_r, int64_t m) {
    const int tile = tri_tile(m);
    return s == 3 ? (m + tile - 1) / tile : r == 2 && s == 4 ? m : n_r;
}

// A run is an eighth of a warp's share of the s-cliques, and at least 32 where there is room for that. Every warp
// that finds an s-clique leaves less than a run unused: at most an eighth more rows, or 31 per warp. In runs
// of 1 (`tight`) no row is left.
int64_t nd_inc_rows(int r, int s, int64_t n_r, int64_t m, int64_t n_s, bool tight, unsigned* run) {
    const int64_t warps = (int64_t)blocks_for_warps(inc_items(r, s, n_r, m)) * (kThreads / 32);
    const int64_t share = n_s / (8 * warps);
    *run = (unsigned)(tight ? 1 : share < 32 ? 32 : share > 1024 ? 1024 : share);
    return n_s + (warps < n_s ? warps : n_s) * (*run - 1);
}

void nd_inc_fill(const GraphView& g, int r, int s, int64_t n_r, const IncFill& F, cudaStream_t st) {
    if (n_r <= 0) return;
    const int blk = blocks_for_warps(inc_items(r, s, n_r, g.m)), tile = tri_tile(g.m);
    static_assert(kTriThreads == kThreads && kQuadThreads == kThreads, "nd_inc_rows counts the warps");
    if (r == 1 && s == 3) {
        ND_K(k_inc_tri<1><<<blk, kTriThreads, 0, st>>>(g, tile, F));
    } else if (r == 2 && s == 3) {
        ND_K(k_inc_tri<2><<<blk, kTriThreads, 0, st>>>(g, tile, F));
    } else if (r == 2 && s == 4) {
        ND_K(k_inc24<<<blk, kQuadThreads, 0, st>>>(g, F));
    } else if (r == 3 && s == 4) {
        ND_K(k_inc34<<<blk, kThreads, 0, st>>>(g, F));
    } else if (r == 1 && s == 4) {
        ND_K(k_inc_gen<1, 4><<<blk, kThreads, 0, st>>>(g, n_r, F));
    } else if (r == 2 && s == 5) {
        ND_K(k_inc_gen<2, 5><<<blk, kThreads, 0, st>>>(g, n_r, F));
    } else if (r == 3 && s == 5) {
        ND_K(k_inc_gen<3, 5><<<blk, kThreads, 0, st>>>(g, n_r, F));
    } else if (r == 3 && s == 6) {
        ND_K(k_inc_gen<3, 6><<<blk, kThreads, 0, st>>>(g, n_r, F));
    } else if (r == 4 && s == 5) {
        ND_K(k_inc_gen<4, 5><<<blk, kThreads, 0, st>>>(g, n_r, F));
    } else if (r == 4 && s == 6) {
        ND_K(k_inc_gen<4, 6><<<blk, kThreads, 0, st>>>(g, n_r, F));
    }
}
