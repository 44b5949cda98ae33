// s-clique counts per r-clique: Algorithm 2's Count-Func over every s-clique listed once by
// Algorithm 1 (rec-list-cliques) on the oriented graph DG.
//
// Two kernel shapes, one per kind of (r,s):
//   * (1,2) reads the degrees; (3,4): count[R] = |I(R)|, the 4-cliques containing R being R plus one
//     vertex of I(R) = ∩_{v in R} N(v). One warp per triangle intersects the two shortest lists by merge
//     path (or probes / bisects the longer one when it is much longer); the result is written
//     once, with no atomics. The lists are the per-edge common-neighbour tables L(e) of the triangle
//     index (|L(e)| is the edge's triangle support, far shorter than the vertex degrees).
//   * (1,3), (2,3), (2,4): the s-cliques are listed once each over DG (Algorithm 1: I' = I ∩ N_DG(v) at each
//     level) and add 1 to each of their C(s,r) r-subsets (Count-Func), with one aggregated atomic for an
//     r-subset shared by a whole level: triangles 32 DG edges to a warp, 4-cliques one warp per
//     lowest DG edge, the pairs of its last level spread over the lanes.
#include "nd_common.cuh"
#include "nd_gen.cuh"
#include "nd_quad24.cuh"
#include "nd_tri.cuh"

namespace {

constexpr int kThreads = 256;
constexpr int kWarpsPerBlock = kThreads / 32;

int blocks_for_warps(int64_t items) {
    int64_t want = (items + kWarpsPerBlock - 1) / kWarpsPerBlock;
    int64_t cap = (int64_t)nd_sm_count() * 16;
    if (want < 1) want = 1;
    return (int)(want < cap ? want : cap);
}

__device__ __forceinline__ int64_t gwarp() { return ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; }
__device__ __forceinline__ int64_t nwarps() { return ((int64_t)gridDim.x * blockDim.x) >> 5; }

__device__ __forceinline__ int warp_sum(int v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

template <typename CT>
__global__ void k_count12(GraphView g, CT* __restrict__ cnt) {
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < g.n; v += (int64_t)gridDim.x * blockDim.x)
        cnt[v] = (CT)(g.rp[v + 1] - g.rp[v]);
}

// (2,3) and (1,3): nd_tri.cuh lists the triangles of DG; each adds 1 to its edges or vertices. What the
// triangles of one DG edge share is kept in shared memory and added once.
template <typename CT, int R_>
struct CountTri {
    CT* cnt;
    const int32_t* eid;
    unsigned* own;  // the warp's triangles per edge
    __device__ void begin(int slot) const {
        own[slot] = 0;
        __syncwarp();
    }
    __device__ void tri(bool hit, int slot, int32_t, int32_t px, int32_t py, bool, int32_t, int32_t, int32_t w) const {
        if (!hit) return;
        atomicAdd(&own[slot], 1u);
        if (R_ == 1) {
            nd_atomic_add(&cnt[w], 1);
        } else {
            nd_atomic_add(&cnt[eid[px]], 1);
            nd_atomic_add(&cnt[eid[py]], 1);
        }
    }
    __device__ void end(int slot, int32_t e, int32_t u, int32_t v) const {
        const unsigned c = own[slot];
        if (!c) return;
        if (R_ == 1) {
            nd_atomic_add(&cnt[u], c);
            nd_atomic_add(&cnt[v], c);
        } else {
            nd_atomic_add(&cnt[e], c);
        }
    }
};

template <typename CT, int R_>
__global__ void __launch_bounds__(kTriThreads) k_count_tri(GraphView g, int tile, CT* __restrict__ cnt) {
    __shared__ unsigned s_own[kTriThreads];
    CountTri<CT, R_> sink{cnt, g.dg_eid, s_own + (threadIdx.x & ~31u)};
    tri_list(g, tile, sink);
}

// count[t] = |L(ab) ∩ L(ac) ∩ L(bc)|. Any two of the lists already intersect to the common
// neighbourhood of the triangle (L(ab) ∩ L(ac) = N(a) ∩ N(b) ∩ N(c)), so the two shortest suffice.
template <typename CT>
__global__ void k_count34(GraphView g, CT* __restrict__ cnt) {
    int lane = threadIdx.x & 31;
    for (int64_t t = gwarp(); t < g.n3; t += nwarps()) {
        int32_t e0 = g.tri_e[3 * t], e1 = g.tri_e[3 * t + 1], e2 = g.tri_e[3 * t + 2];
        int64_t b0 = g.et_rp[e0], n0 = g.et_rp[e0 + 1] - b0;
        int64_t b1 = g.et_rp[e1], n1 = g.et_rp[e1 + 1] - b1;
        int64_t b2 = g.et_rp[e2], n2 = g.et_rp[e2 + 1] - b2;
        // the two shortest lists: (b0, n0) drives, (b1, n1) is searched
        if (n1 < n0) {
            int64_t tb = b0, tn = n0;
            int32_t te = e0;
            b0 = b1, n0 = n1, e0 = e1, b1 = tb, n1 = tn, e1 = te;
        }
        if (n2 < n0) {
            int64_t tb = b0, tn = n0;
            int32_t te = e0;
            b0 = b2, n0 = n2, e0 = e2, b2 = tb, n2 = tn, e2 = te;
        }
        if (n2 < n1) b1 = b2, n1 = n2, e1 = e2;
        // the longer list is probed in the hash directory once it is more than about twice the
        // shorter (measured on R-MAT scale 20: the merge pays only below that; 1x, 4x and never
        // measured slower); without a table, the merge up to 8x and bisection beyond
        int c = 0;
        const bool probe = g.htab && nd_hashed(n1) && n1 > 2 * n0 + 64;
        if (!probe && nd_prefer_merge(n0, n1)) {
            c = nd_merge_count(g.et_w + b0, (int)n0, g.et_w + b1, (int)n1);
        } else if (probe) {
            // the long list has a hash directory: one probe instead of a bisection
            const NdHashSlot* tab = g.htab + g.hoff[e1];
            int k = nd_hash_bits(n1);
            int32_t id, rnd;
            for (int64_t i = lane; i < n0; i += 32) c += nd_hash_find(tab, k, g.et_w[b0 + i], id, rnd) ? 1 : 0;
        } else {
            for (int64_t i = lane; i < n0; i += 32) c += nd_find(g.et_w + b1, n1, g.et_w[b0 + i]) >= 0 ? 1 : 0;
        }
        c = warp_sum(c);
        if (lane == 0) cnt[t] = (CT)c;
    }
}

// (2,4): nd_quad24.cuh lists the 4-cliques; each adds 1 to its six edges
template <typename CT>
struct Count24 {
    CT* cnt;
    static constexpr bool kTally = true;
    __device__ void pair(int32_t e_wx) const { nd_atomic_add(&cnt[e_wx], 1); }
    __device__ void add(int32_t e, int64_t c) const { nd_atomic_add(&cnt[e], c); }
    __device__ void clique(bool hit, const int32_t (&e)[6]) const {
        if (!hit) return;
#pragma unroll
        for (int i = 1; i < 6; ++i) nd_atomic_add(&cnt[e[i]], 1);
    }
};

template <typename CT>
__global__ void __launch_bounds__(kQuadThreads) k_count24_flat(GraphView g, CT* __restrict__ cnt) {
    Count24<CT> sink{cnt};
    quad24_list(g, sink);
}

// Any other supported (r,s) ((1,4), (2,5), (3,5), (3,6), (4,5), (4,6)): one warp per r-clique R counts the
// s-cliques containing it, listing the (s-r)-cliques of R's common neighbourhood from the entries
// of its driving list (nd_gen.cuh); written once, no atomics.
template <typename CT, int R_, int S_>
__global__ void k_count_gen(GraphView g, CT* __restrict__ cnt, int64_t n_r) {
    int lane = threadIdx.x & 31;
    for (int64_t id = gwarp(); id < n_r; id += nwarps()) {
        int32_t v[4];
        gen_verts<R_>(g, id, v);
        const int32_t* list = nullptr;
        int64_t len = 0;
        gen_drive<R_>(g, id, v, list, len);
        unsigned long long c = 0;
        for (int64_t j = lane; j < len; j += 32) gen_cand<R_, S_>(g, v, list[j], [&](const int32_t*) { ++c; });
        for (int o = 16; o > 0; o >>= 1) c += __shfl_down_sync(0xffffffffu, c, o);
        if (lane == 0) cnt[id] = (CT)c;
    }
}

// Estimates of the number of s-cliques, from a part of the graph: *out += those of one tile of DG edges in
// `every` (triangles), of one DG edge in `every` (4-cliques), of one r-clique in `every` (any (r,s), each s-clique
// from C(s,r) of them)
__device__ __forceinline__ void add_total(unsigned long long c, unsigned long long* out) {
    for (int o = 16; o > 0; o >>= 1) c += __shfl_down_sync(0xffffffffu, c, o);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(out, c);
}

struct TotalTri {
    unsigned long long n = 0;
    __device__ void begin(int) const {}
    __device__ void tri(bool hit, int, int32_t, int32_t, int32_t, bool, int32_t, int32_t, int32_t) { n += hit; }
    __device__ void end(int, int32_t, int32_t, int32_t) const {}
};

__global__ void __launch_bounds__(kTriThreads) k_sample_tri(GraphView g, int tile, int64_t every, unsigned long long* out) {
    TotalTri sink;
    tri_list(g, tile, sink, every);
    add_total(sink.n, out);
}

struct Total24 {
    unsigned long long n = 0;
    static constexpr bool kTally = false;
    __device__ void clique(bool hit, const int32_t (&)[6]) { n += hit; }
};

__global__ void __launch_bounds__(kQuadThreads) k_sample24(GraphView g, int64_t every, unsigned long long* out) {
    Total24 sink;
    quad24_list(g, sink, every);
    add_total(sink.n, out);
}

template <int R_, int S_>
__global__ void k_sample_gen(GraphView g, int64_t n_r, int64_t every, unsigned long long* out) {
    const int lane = threadIdx.x & 31;
    unsigned long long c = 0;
    for (int64_t id = gwarp() * every; id < n_r; id += nwarps() * every) {
        int32_t v[4];
        gen_verts<R_>(g, id, v);
        const int32_t* list = nullptr;
        int64_t len = 0;
        gen_drive<R_>(g, id, v, list, len);
        for (int64_t j = lane; j < len; j += 32) gen_cand<R_, S_>(g, v, list[j], [&](const int32_t*) { ++c; });
    }
    add_total(c, out);
}

template <typename CT>
__global__ void k_zero(CT* p, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        p[i] = 0;
}

}  // namespace

template <typename CT>
void nd_count_launch(const GraphView& g, int r, int s, CT* cnt, int64_t n_r, cudaStream_t st) {
    if (n_r <= 0) return;
    int blk = blocks_for_warps(n_r);
    const int tile = tri_tile(g.m);
    if (r == 1 && s == 2) {
        ND_K(k_count12<CT><<<blk, kThreads, 0, st>>>(g, cnt));
    } else if (r == 2 && s == 3) {
        ND_K(k_zero<CT><<<blk, kThreads, 0, st>>>(cnt, n_r));
        ND_K(k_count_tri<CT, 2><<<blocks_for_warps((g.m + tile - 1) / tile), kTriThreads, 0, st>>>(g, tile, cnt));
    } else if (r == 3 && s == 4) {
        ND_K(k_count34<CT><<<blk, kThreads, 0, st>>>(g, cnt));
    } else if (r == 1 && s == 3) {
        ND_K(k_zero<CT><<<blk, kThreads, 0, st>>>(cnt, n_r));
        ND_K(k_count_tri<CT, 1><<<blocks_for_warps((g.m + tile - 1) / tile), kTriThreads, 0, st>>>(g, tile, cnt));
    } else if (r == 2 && s == 4) {
        ND_K(k_zero<CT><<<blk, kThreads, 0, st>>>(cnt, n_r));
        ND_K(k_count24_flat<CT><<<blocks_for_warps(g.m), kQuadThreads, 0, st>>>(g, cnt));
    } else if (r == 1 && s == 4) {
        ND_K(k_count_gen<CT, 1, 4><<<blk, kThreads, 0, st>>>(g, cnt, n_r));
    } else if (r == 2 && s == 5) {
        ND_K(k_count_gen<CT, 2, 5><<<blk, kThreads, 0, st>>>(g, cnt, n_r));
    } else if (r == 3 && s == 5) {
        ND_K(k_count_gen<CT, 3, 5><<<blk, kThreads, 0, st>>>(g, cnt, n_r));
    } else if (r == 3 && s == 6) {
        ND_K(k_count_gen<CT, 3, 6><<<blk, kThreads, 0, st>>>(g, cnt, n_r));
    } else if (r == 4 && s == 5) {
        ND_K(k_count_gen<CT, 4, 5><<<blk, kThreads, 0, st>>>(g, cnt, n_r));
    } else if (r == 4 && s == 6) {
        ND_K(k_count_gen<CT, 4, 6><<<blk, kThreads, 0, st>>>(g, cnt, n_r));
    }
}

// a sixty-fourth of a large graph, and at least 16,384 DG edges or r-cliques (1,024 tiles of 32 edges)
int64_t nd_sample_cliques(const GraphView& g, int r, int s, int64_t n_r, unsigned long long* out, cudaStream_t st) {
    const int tile = tri_tile(g.m);
    const int64_t items = s == 3 ? (g.m + tile - 1) / tile : s == 4 ? g.m : n_r;
    const int64_t part = items >> (s == 3 ? 10 : 14), every = part < 1 ? 1 : part > 64 ? 64 : part;
    const int blk = blocks_for_warps((items + every - 1) / every);
    if (s == 3)
        ND_K(k_sample_tri<<<blk, kTriThreads, 0, st>>>(g, tile, every, out));
    else if (s == 4)
        ND_K(k_sample24<<<blk, kQuadThreads, 0, st>>>(g, every, out));
    else if (r == 2)
        ND_K(k_sample_gen<2, 5><<<blk, kThreads, 0, st>>>(g, n_r, every, out));
    else if (r == 3 && s == 5)
        ND_K(k_sample_gen<3, 5><<<blk, kThreads, 0, st>>>(g, n_r, every, out));
    else if (r == 3)
        ND_K(k_sample_gen<3, 6><<<blk, kThreads, 0, st>>>(g, n_r, every, out));
    else if (s == 5)
        ND_K(k_sample_gen<4, 5><<<blk, kThreads, 0, st>>>(g, n_r, every, out));
    else
        ND_K(k_sample_gen<4, 6><<<blk, kThreads, 0, st>>>(g, n_r, every, out));
    return every;
}

template void nd_count_launch<int32_t>(const GraphView&, int, int, int32_t*, int64_t, cudaStream_t);
template void nd_count_launch<int64_t>(const GraphView&, int, int, int64_t*, int64_t, cudaStream_t);
