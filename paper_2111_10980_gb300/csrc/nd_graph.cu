// Graph structure kernels: CSR validation, the canonical edge index (r = 2), the oriented
// graph DG (Section 3, O(alpha)-orientation; Algorithm 2, line "Orient") and the triangle
// index (r = 3; Sections 5.1-5.3: the per-edge last-level tables of the two-level T laid out
// contiguously with a prefix sum, and the inverse map from a triangle id to its edges).
//
// Layout choices for the GPU:
//   * vertex ids are never relabelled; DG's out-lists are order-preserving filters of the
//     sorted CSR rows, so every list stays sorted by vertex id and intersections of undirected
//     and oriented lists need no re-sort (the paper's relabelling, Section 5.4, is replaced by
//     this);
//   * the canonical edge id of (a<b) is its rank in CSR order, so per-edge outputs need no
//     permutation;
//   * L(a,b) stores every common neighbour w of a and b (all three edges of a triangle list
//     it), together with the triangle's canonical id; a triangle (a<b<c) gets id
//     tbase[e(a,b)] + rank of c among the entries of L(a,b) greater than b.
#include "nd_common.cuh"
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

int blocks_for_threads(int64_t items) {
    int64_t want = (items + kThreads - 1) / kThreads;
    int64_t cap = (int64_t)nd_sm_count() * 16;
    if (want < 1) want = 1;
    return (int)(want < cap ? want : cap);
}

__device__ __forceinline__ int64_t gwarp() { return ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; }
__device__ __forceinline__ int64_t nwarps() { return ((int64_t)gridDim.x * blockDim.x) >> 5; }

// err bits: 1 row pointers not monotone, 2 id out of range, 4 row not strictly ascending,
// 8 self-loop, 16 missing reverse entry
__global__ void k_validate(const int64_t* __restrict__ rp, const int32_t* __restrict__ col, int32_t n, int64_t nnz,
                           int* err) {
    int lane = threadIdx.x & 31;
    for (int64_t u = gwarp(); u < n; u += nwarps()) {
        int64_t b = rp[u], e = rp[u + 1];
        if (e < b || b < 0 || e > nnz) {
            if (lane == 0) atomicOr(err, 1);
            continue;
        }
        for (int64_t p = b + lane; p < e; p += 32) {
            int32_t v = col[p];
            if (v < 0 || v >= n) {
                atomicOr(err, 2);
                continue;
            }
            if (p > b && col[p - 1] >= v) atomicOr(err, 4);
            if (v == u) atomicOr(err, 8);
            int64_t vb = rp[v], ve = rp[v + 1];
            if (ve < vb || vb < 0 || ve > nnz || nd_find(col + vb, ve - vb, (int32_t)u) < 0) atomicOr(err, 16);
        }
    }
}

__global__ void k_split(const int64_t* __restrict__ rp, const int32_t* __restrict__ col, int32_t n,
                        int64_t* __restrict__ split, int64_t* __restrict__ updeg) {
    for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n; u += (int64_t)gridDim.x * blockDim.x) {
        int64_t b = rp[u], e = rp[u + 1];
        int64_t s = b + nd_lower_bound(col + b, e - b, (int32_t)u + 1);
        split[u] = s;
        updeg[u] = e - s;
    }
}

// The passes over CSR entries give every warp a segment of consecutive ones, whatever rows they belong to:
// with a warp per row, one hub of a skewed graph kept the pass going for as long as the rest together
// took (R-MAT scale 20: the three passes 14.3 -> 1.3 ms). Segments of 1,024 entries, and shorter ones, down to a
// step of 32, where the graph has too few entries to give every resident warp as many (2,000 vertices: 0.24 ->
// 0.11 ms for the whole orientation, 0.10 with rows).
int64_t seg_len(int64_t nnz) {
    const int64_t steps = nnz / (32 * (int64_t)nd_sm_count() * 64);
    return 32 * (steps < 1 ? 1 : steps > 32 ? 32 : steps);
}

// the last row at or after u0 that begins at or before entry p (rp[u0] <= p < rp[n]): p's row
__device__ __forceinline__ int64_t row_of(const int64_t* __restrict__ rp, int64_t n, int64_t u0, int64_t p) {
    int64_t lo = u0, step = 1;
    while (lo + step < n && __ldg(rp + lo + step) <= p) {
        lo += step;
        step <<= 1;
    }
    int64_t hi = lo + step < n ? lo + step : n;  // rp[hi] > p
    while (hi - lo > 1) {
        const int64_t mid = (lo + hi) >> 1;
        if (__ldg(rp + mid) <= p)
            lo = mid;
        else
            hi = mid;
    }
    return lo;
}

// A CSR entry whose reverse entry is missing, a self-loop or an id that is no vertex sets bit 0 of *err and
// gets edge id 0, so that no later kernel indexes outside the edge arrays; no row is looked up by such an id.
// An entry equal to the one before it in its row sets bit 1, one below it bit 2 (without either, and with as many
// upper as lower entries, the graph is simple); what depends on that is nd_api.cu's to refuse.
__global__ void k_pos2e(GraphView g, int64_t nnz, int64_t seg, int32_t* __restrict__ pos2e, int32_t* __restrict__ eu,
                        int32_t* __restrict__ ev, int* err) {
    const int lane = threadIdx.x & 31;
    for (int64_t s0 = gwarp() * seg; s0 < nnz; s0 += nwarps() * seg) {
        const int64_t s1 = s0 + seg < nnz ? s0 + seg : nnz;
        int64_t u0 = row_of(g.rp, g.n, 0, s0);
        for (int64_t p0 = s0; p0 < s1; p0 += 32) {
            const int64_t p = p0 + lane;
            int64_t u = u0;
            if (p < s1) {
                const int32_t v = g.col[p], prev = p > 0 ? g.col[p - 1] : -1;
                u = row_of(g.rp, g.n, u0, p);
                if (prev >= v && p > g.rp[u]) atomicOr(err, prev == v ? 2 : 4);
                int64_t id;
                if ((uint32_t)v >= (uint32_t)g.n) {
                    atomicOr(err, 1);
                    id = 0;
                } else if (v > u) {
                    id = g.ebase[u] + (p - g.split[u]);
                    if (id >= 0 && id < g.m) {
                        eu[id] = (int32_t)u;
                        ev[id] = v;
                    } else {  // more upper than lower entries
                        atomicOr(err, 1);
                        id = 0;
                    }
                } else {
                    // u is in the upper part of v's row
                    const int64_t vs = g.split[v], ve = g.rp[v + 1];
                    const int64_t q = vs + nd_lower_bound(g.col + vs, ve - vs, (int32_t)u);
                    if (v == u || q >= ve || g.col[q] != (int32_t)u) {
                        atomicOr(err, 1);
                        id = 0;
                    } else {
                        id = g.ebase[v] + (q - vs);
                    }
                }
                pos2e[p] = (int32_t)id;
            }
            u0 = __shfl_sync(0xffffffffu, u, 31);
        }
    }
}

__device__ __forceinline__ bool key_less(const int64_t* rp, const int32_t* key_hi, int32_t a, int32_t b) {
    int64_t ka = key_hi ? (int64_t)key_hi[a] : rp[a + 1] - rp[a];
    int64_t kb = key_hi ? (int64_t)key_hi[b] : rp[b + 1] - rp[b];
    return ka < kb || (ka == kb && a < b);
}

// Out-degrees (outdeg zeroed by the caller), and of every segment how many entries of its last row are
// taken: what the fill needs to place a row that runs over several segments.
__global__ void k_dg_count(GraphView g, int64_t nnz, int64_t seg, const int32_t* __restrict__ key_hi, int64_t* __restrict__ outdeg,
                           int32_t* __restrict__ tail) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    for (int64_t s0 = gwarp() * seg; s0 < nnz; s0 += nwarps() * seg) {
        const int64_t s1 = s0 + seg < nnz ? s0 + seg : nnz;
        int64_t u0 = row_of(g.rp, g.n, 0, s0);
        unsigned run = 0;  // taken so far in row u0, not yet added
        for (int64_t p0 = s0; p0 < s1; p0 += 32) {
            const int64_t p = p0 + lane;
            int64_t u = g.n;
            bool take = false;
            if (p < s1) {
                u = row_of(g.rp, g.n, u0, p);
                take = key_less(g.rp, key_hi, (int32_t)u, g.col[p]);
            }
            const unsigned taken = __ballot_sync(full, take), same = __match_any_sync(full, u);
            const int last = (int)(s1 - p0 < 32 ? s1 - p0 : 32) - 1;
            const int64_t u1 = __shfl_sync(full, u, last);  // the step's last row, whose count is carried on
            unsigned c = __popc(taken & same);
            if (!__any_sync(full, u == u0)) {  // row u0 ended with the last step
                if (lane == 0 && run) atomicAdd((unsigned long long*)&outdeg[u0], (unsigned long long)run);
                run = 0;
            }
            if (u == u0) c += run;
            const bool first = lane == __ffs(same) - 1;
            if (first && p < s1 && u != u1 && c) atomicAdd((unsigned long long*)&outdeg[u], (unsigned long long)c);
            run = __shfl_sync(full, c, last);
            u0 = u1;
        }
        if (lane == 0) {
            tail[s0 / seg] = (int32_t)run;
            if (run) atomicAdd((unsigned long long*)&outdeg[u0], (unsigned long long)run);
        }
    }
}

__global__ void k_dg_fill(GraphView g, int64_t nnz, int64_t seg, const int32_t* __restrict__ key_hi,
                          const int64_t* __restrict__ dg_rp, const int32_t* __restrict__ tail,
                          int32_t* __restrict__ dg_col, int32_t* __restrict__ dg_eid) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    for (int64_t s0 = gwarp() * seg; s0 < nnz; s0 += nwarps() * seg) {
        const int64_t s1 = s0 + seg < nnz ? s0 + seg : nnz;
        int64_t u0 = row_of(g.rp, g.n, 0, s0);
        // taken before this segment in the row it begins in: that row is the last one of every earlier
        // segment that it touches
        unsigned long long prior = 0;
        for (int64_t t = g.rp[u0] / seg + lane; t < s0 / seg; t += 32) prior += (unsigned)tail[t];
        for (int o = 16; o > 0; o >>= 1) prior += __shfl_xor_sync(full, prior, o);
        int64_t at = dg_rp[u0] + (int64_t)prior;  // place of the next taken entry of row u0
        for (int64_t p0 = s0; p0 < s1; p0 += 32) {
            const int64_t p = p0 + lane;
            int64_t u = g.n;
            bool take = false;
            int32_t v = 0;
            if (p < s1) {
                u = row_of(g.rp, g.n, u0, p);
                v = g.col[p];
                take = key_less(g.rp, key_hi, (int32_t)u, v);
            }
            const unsigned taken = __ballot_sync(full, take), same = __match_any_sync(full, u);
            const int64_t base = u == u0 ? at : (p < s1 ? dg_rp[u] : 0);
            if (take) {
                const int64_t to = base + __popc(taken & same & nd_lanemask_lt());
                dg_col[to] = v;
                dg_eid[to] = g.pos2e[p];
            }
            const int last = (int)(s1 - p0 < 32 ? s1 - p0 : 32) - 1;
            at = __shfl_sync(full, base + __popc(taken & same), last);
            u0 = __shfl_sync(full, u, last);
        }
    }
}

// sigma[e] = |N(a) ∩ N(b)|, up[e] = |{w in N(a) ∩ N(b) : w > b}| for canonical edge e = (a,b): each triangle,
// met once over DG, adds 1 to sigma of its edges and to up of the one without its largest vertex.
// The numbers of u -> v itself are kept in shared memory and added once.
struct SupportSink {
    int32_t* sigma;
    int32_t* up;
    const int32_t* eid;
    unsigned* own;  // per slot: triangles, then those with u -> v lowest
    __device__ void begin(int slot) const {
        own[slot] = 0;
        own[slot + 32] = 0;
        __syncwarp();
    }
    __device__ void tri(bool hit, int slot, int32_t, int32_t px, int32_t py, bool of_u, int32_t u, int32_t v,
                        int32_t w) const {
        if (!hit) return;
        const int32_t ex = eid[px], ey = eid[py];
        atomicAdd(&own[slot], 1u);
        atomicAdd(&sigma[ex], 1);
        atomicAdd(&sigma[ey], 1);
        if (w > u && w > v)
            atomicAdd(&own[slot + 32], 1u);
        else
            atomicAdd(&up[(u > v) == of_u ? ey : ex], 1);  // the edge without the larger of u and v
    }
    __device__ void end(int slot, int32_t e, int32_t, int32_t) const {
        if (own[slot]) atomicAdd(&sigma[e], (int)own[slot]);
        if (own[slot + 32]) atomicAdd(&up[e], (int)own[slot + 32]);
    }
};

__global__ void __launch_bounds__(kTriThreads) k_edge_support(GraphView g, int tile, int32_t* __restrict__ sigma,
                                                              int32_t* __restrict__ up) {
    __shared__ unsigned s_own[2 * kTriThreads];
    SupportSink sink{sigma, up, g.dg_eid, s_own + 2 * (threadIdx.x & ~31u)};
    tri_list(g, tile, sink);
}

// Whether a CSR with duplicate entries has the triangle lists of a simple graph: *err is set if a duplicate's
// edge lies in a triangle (two entries of a list would be equal, and k_edge_order would give both the same
// place, leaving the next one unwritten), or if an upper entry has no reverse (the rows would hold triangles
// that DG does not).
__global__ void k_dup_check(GraphView g, int64_t nnz, int64_t seg, const int32_t* __restrict__ sigma, int* err) {
    const int lane = threadIdx.x & 31;
    for (int64_t s0 = gwarp() * seg; s0 < nnz; s0 += nwarps() * seg) {
        const int64_t s1 = s0 + seg < nnz ? s0 + seg : nnz;
        for (int64_t p = s0 + lane; p < s1; p += 32) {
            const int64_t u = row_of(g.rp, g.n, 0, p);
            const int32_t v = g.col[p];
            if (p > g.rp[u] && g.col[p - 1] == v && (sigma[g.pos2e[p - 1]] || sigma[g.pos2e[p]])) atomicOr(err, 1);
            if (v > u && nd_find(g.col + g.rp[v], g.split[v] - g.rp[v], (int32_t)u) < 0) atomicOr(err, 1);
        }
    }
}

// The three kernels that write the lists give every warp a tile of up to 32 edges at a time, fewer where there would
// not be four tiles for every resident warp. A tile's edges lie 1,024 apart, because the edges of a hub, whose
// rows and lists are the longest, are neighbours, and a warp takes long lists one after another: with 32
// consecutive edges the index of R-MAT 2^12 took 0.94 ms and of R-MAT 2^18 with 0.9 M edges 4.0, now 0.30 and 1.8
// (one edge per warp 0.28 and 2.4); of a Chung-Lu graph with 15 M edges 12.7, now 9.2 (27.9). They lie no further
// apart, so that neighbouring warps stay in the same part of a large graph: 1,365 graphs in one, 41 M edges, 21 ms
// with consecutive edges, 23 so, 30 with m / 32 in between.
constexpr int64_t kTileSpan = 1024;  // tiles
struct EdgeTile {
    int64_t first, apart;
    __device__ __forceinline__ EdgeTile(int64_t m, int64_t k, int64_t tiles, int tile) {
        const int64_t span = k / kTileSpan * kTileSpan;
        apart = tiles - span < kTileSpan ? (m - span * tile + tile - 1) / tile : kTileSpan;
        first = span * tile + (k - span);
    }
    __device__ __forceinline__ int64_t edge(int lane) const { return first + lane * apart; }
};

// Lists of up to kShortList entries are not intersected out of the two rows, which are far longer, but
// gathered: a second listing of the triangles over DG appends every triangle to the short lists among
// its three (k_edge_gather, in no order), and k_edge_order puts each list in order by counting for every
// entry the smaller ones. That pays where the rows of these edges hold more than some 40 entries for each
// triangle (nd_gather_pays). Index with / without, in ms: Chung-Lu, a million vertices (518 entries) 9.4 / 16.7, 200,001
// vertices (343) 1.3 / 2.0; flat R-MAT of 40,000 vertices (131) 0.95 / 1.21; R-MAT 2^20 (49) 230 / 243, 2^15 (33) 2.41 /
// 2.33, 2^12 (27) 0.34 / 0.29; G(3000, 0.1) (60) 1.77 / 1.75, G(1500, 0.2) (30) 1.37 / 1.11; under 65,536 triangles or
// 32,768 edges launches are all that counts: 2,000 vertices 0.135 / 0.124.
constexpr int kShortList = 128;

// *rows += the row entries that merging (or, 16 for each that is bisected, searching) the rows of the edges with short
// lists would look at, estimated from 32 edges of every 32 * every
__global__ void k_row_work(GraphView g, const int32_t* __restrict__ sigma, int64_t every, unsigned long long* rows) {
    const int lane = threadIdx.x & 31;
    unsigned long long c = 0;
    for (int64_t e = gwarp() * 32 * every + lane; e < g.m; e += nwarps() * 32 * every) {
        const int32_t n = sigma[e];
        if (n == 0 || n > kShortList) continue;
        const int32_t a = g.eu[e], b = g.ev[e];
        const int64_t da = g.rp[a + 1] - g.rp[a], db = g.rp[b + 1] - g.rp[b], lo = da < db ? da : db, hi = da < db ? db : da;
        c += nd_prefer_merge(lo, hi) ? lo + hi : 16 * lo;
    }
    for (int o = 16; o > 0; o >>= 1) c += __shfl_down_sync(0xffffffffu, c, o);
    if (lane == 0 && c) atomicAdd(rows, c * every);
}

struct GatherSink {
    const int64_t* et_rp;
    const int32_t* sigma;
    const int32_t* eid;
    int32_t* cursor;
    int32_t *w_in, *p_in, *q_in;  // per entry: the vertex; the edge to et_t (see k_edge_fill); of an upper entry, bc
    __device__ void begin(int) const {}
    __device__ void put(int32_t e, int32_t w, int32_t p, int32_t q) const {
        if (sigma[e] > kShortList) return;
        const int64_t at = et_rp[e] + atomicAdd(&cursor[e], 1);
        w_in[at] = w;
        p_in[at] = p;
        q_in[at] = q;
    }
    __device__ void tri(bool hit, int, int32_t e, int32_t px, int32_t py, bool of_u, int32_t u, int32_t v,
                        int32_t w) const {
        if (!hit) return;
        const int32_t ex = eid[px], ey = eid[py];
        // vertices ascending, each with the edge across from it
        int32_t a = u, b = v, c = w, ea = of_u ? ey : ex, eb = of_u ? ex : ey, ec = e;
        auto order = [](int32_t& x, int32_t& y, int32_t& p, int32_t& q) {
            if (x > y) {
                int32_t t = x;
                x = y, y = t;
                t = p;
                p = q, q = t;
            }
        };
        order(a, b, ea, eb);
        order(b, c, eb, ec);
        order(a, b, ea, eb);
        put(ec, c, eb, ea);  // L(ab): the edges ac and bc
        put(eb, b, ec, 0);   // L(ac), L(bc): the lowest edge ab
        put(ea, a, ec, 0);
    }
    __device__ void end(int, int32_t, int32_t, int32_t) const {}
};

__global__ void __launch_bounds__(kTriThreads) k_edge_gather(GraphView g, int tile, GatherSink sink) {
    tri_list(g, tile, sink);
}

// One lane per entry of the short lists of a tile of edges at a time; the place of an entry is the number of
// smaller ones in its list (no two are alike). Writes what k_edge_fill writes.
__global__ void k_edge_order(GraphView g, const int64_t* __restrict__ et_rp, const int64_t* __restrict__ tbase,
                             const int32_t* __restrict__ w_in, const int32_t* __restrict__ p_in,
                             const int32_t* __restrict__ q_in, int32_t* __restrict__ et_w, int32_t* __restrict__ et_t,
                             int32_t* __restrict__ tri_e, int32_t* __restrict__ tri_pos, int tile) {
    const int lane = threadIdx.x & 31;
    const unsigned full = 0xffffffffu;
    const int64_t tiles = (g.m + tile - 1) / tile;
    for (int64_t k = gwarp(); k < tiles; k += nwarps()) {
        const EdgeTile T(g.m, k, tiles, tile);
        const int64_t e = lane < tile ? T.edge(lane) : g.m;
        int64_t lo = 0, tb = 0;
        int32_t n = 0, low = 0;
        if (e < g.m) {
            lo = et_rp[e];
            const int64_t len = et_rp[e + 1] - lo;
            if (len && len <= kShortList) {
                n = (int32_t)len;
                tb = tbase[e];
                low = n - (int32_t)(tbase[e + 1] - tb);
            }
        }
        int32_t inc = n;
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(full, inc, o);
            if (lane >= o) inc += y;
        }
        const int32_t total = __shfl_sync(full, inc, 31), before = inc - n;
        for (int32_t p0 = 0; p0 < total; p0 += 32) {
            const int32_t p = p0 + lane;
            int own = 0;  // the last lane with before <= p: the one whose entry it is
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                if (__shfl_sync(full, before, own + o) <= p) own += o;
            const int64_t b = __shfl_sync(full, lo, own), otb = __shfl_sync(full, tb, own);
            const int32_t k = p - __shfl_sync(full, before, own), on = __shfl_sync(full, n, own);
            const int32_t olow = __shfl_sync(full, low, own);
            if (p >= total) continue;
            const int32_t w = w_in[b + k];
            int32_t at = 0;
#pragma unroll 4
            for (int32_t i = 0; i < on; ++i) at += w_in[b + i] < w;
            et_w[b + at] = w;
            if (at >= olow) {
                const int64_t tid = otb + (at - olow);
                et_t[b + at] = (int32_t)tid;
                tri_e[3 * tid + 0] = (int32_t)T.edge(own);
                tri_e[3 * tid + 1] = p_in[b + k];
                tri_e[3 * tid + 2] = q_in[b + k];
                tri_pos[3 * tid + 0] = at;
            } else {
                et_t[b + at] = p_in[b + k];
            }
        }
    }
}

// Writes L(a,b) in ascending w with, per entry: the canonical triangle id when w > b, else
// (temporarily) the id of edge (a,w); and the edges of every triangle whose lowest edge is e. Lists of up to
// `above` entries are left out (k_edge_gather and k_edge_order write them; 0 without room for that). Edges
// without triangles, most of them in a sparse graph, cost a lane a look and not a warp an intersection
// (Chung-Lu, a million vertices, 15 M edges: 13.2 ms here of 16.3 before).
__global__ void k_edge_fill(GraphView g, const int64_t* __restrict__ et_rp, const int64_t* __restrict__ tbase,
                            int32_t* __restrict__ et_w, int32_t* __restrict__ et_t, int32_t* __restrict__ tri_e,
                            int32_t* __restrict__ tri_pos, int64_t above, int tile) {
    const int lane = threadIdx.x & 31;
    const unsigned full = 0xffffffffu;
    const int64_t tiles = (g.m + tile - 1) / tile;
    for (int64_t k = gwarp(); k < tiles; k += nwarps()) {
        const EdgeTile T(g.m, k, tiles, tile);
        // each lane looks one edge over and sets it up; those with triangles are then taken one after another
        const int64_t el = lane < tile ? T.edge(lane) : g.m;
        int32_t la = 0, lb = 0;
        int64_t lab = 0, lae = 0, lbb = 0, lbe = 0, lout = 0, lsig = 0, ltb = 0, lup = 0;
        if (el < g.m) {
            lout = et_rp[el];
            lsig = et_rp[el + 1] - lout;
            if (lsig <= above) lsig = 0;
            if (lsig) {
                la = g.eu[el], lb = g.ev[el];
                lab = g.rp[la], lae = g.rp[la + 1], lbb = g.rp[lb], lbe = g.rp[lb + 1];
                ltb = tbase[el], lup = tbase[el + 1] - ltb;
            }
        }
        for (unsigned todo = __ballot_sync(full, lsig != 0); todo; todo &= todo - 1) {
            const int src = __ffs(todo) - 1;
            const int64_t e = T.edge(src);
            const int32_t b = __shfl_sync(full, lb, src);
            const int64_t ab = __shfl_sync(full, lab, src), ae = __shfl_sync(full, lae, src);
            const int64_t bb = __shfl_sync(full, lbb, src), be = __shfl_sync(full, lbe, src);
            const int64_t out = __shfl_sync(full, lout, src), sig = __shfl_sync(full, lsig, src);
            const int64_t tb = __shfl_sync(full, ltb, src), split_e = sig - __shfl_sync(full, lup, src);
            const bool a_drives = (ae - ab) <= (be - bb);
            const int64_t xb = a_drives ? ab : bb, xe = a_drives ? ae : be;
            const int64_t yb = a_drives ? bb : ab, ye = a_drives ? be : ae;
            // writes common element w, found at driver position p and other-list position q, as entry
            // `local` of L(a,b)
            auto put = [&](int64_t local, int64_t p, int64_t q, int32_t w) {
                int64_t pa = a_drives ? p : q;  // position of w in N(a)
                int64_t pb = a_drives ? q : p;  // position of w in N(b)
                int32_t e_aw = g.pos2e[pa], e_bw = g.pos2e[pb];
                et_w[out + local] = w;
                if (w > b) {
                    int64_t tid = tb + (local - split_e);
                    et_t[out + local] = (int32_t)tid;
                    tri_e[3 * tid + 0] = (int32_t)e;
                    tri_e[3 * tid + 1] = e_aw;
                    tri_e[3 * tid + 2] = e_bw;
                    tri_pos[3 * tid + 0] = (int32_t)local;
                } else {
                    et_t[out + local] = e_aw;
                }
            };
            if (nd_prefer_merge(xe - xb, ye - yb)) {
                // merge path: count this lane's matches, place them after the lower lanes' (exclusive
                // scan), then walk the run again and write them
                const int32_t *X = g.col + xb, *Y = g.col + yb;
                const int nx = (int)(xe - xb), ny = (int)(ye - yb);
                const NdMergeRun run = nd_merge_run(X, nx, Y, ny);
                int cnt = 0;
                nd_merge_walk(X, nx, Y, ny, run, [&](int, int, int32_t) { ++cnt; });
                int inc = cnt;
                for (int o = 1; o < 32; o <<= 1) {
                    int y = __shfl_up_sync(0xffffffffu, inc, o);
                    if (lane >= o) inc += y;
                }
                int64_t local = inc - cnt;
                nd_merge_walk(X, nx, Y, ny, run, [&](int i, int j, int32_t w) { put(local++, xb + i, yb + j, w); });
            } else {
                int64_t pos = 0;
                for (int64_t p0 = xb; p0 < xe; p0 += 32) {
                    int64_t p = p0 + lane;
                    int64_t q = -1;
                    if (p < xe) q = nd_find(g.col + yb, ye - yb, g.col[p]);
                    unsigned m = __ballot_sync(0xffffffffu, q >= 0);
                    if (q >= 0) put(pos + __popc(m & nd_lanemask_lt()), p, yb + q, g.col[p]);
                    pos += __popc(m);
                }
            }
        }
    }
}

// For entries of L(a,b) with w < b, the triangle {a,w,b} has b as its largest vertex, so its
// lowest edge is (a,w) (or (w,a)); its id is tbase[e'] + rank of b among the upper entries of L(e').
// The entry is the triangle's (a,c) entry when a < w, its (b,c) entry when w < a (slots 1, 2).
// A warp takes the lower entries of a tile of edges together, 32 at a time.
__global__ void k_edge_fill_tid(GraphView g, int32_t* __restrict__ et_t, int32_t* __restrict__ tri_pos, int tile) {
    const int lane = threadIdx.x & 31;
    const unsigned full = 0xffffffffu;
    const int64_t tiles = (g.m + tile - 1) / tile;
    for (int64_t k = gwarp(); k < tiles; k += nwarps()) {
        const EdgeTile T(g.m, k, tiles, tile);
        const int64_t e = lane < tile ? T.edge(lane) : g.m;
        int64_t lo = 0, low = 0;
        int32_t a = 0, b = 0;
        if (e < g.m) {
            lo = g.et_rp[e];
            low = g.et_rp[e + 1] - lo - (g.tbase[e + 1] - g.tbase[e]);
            if (low) {
                a = g.eu[e];
                b = g.ev[e];
            }
        }
        int64_t inc = low;
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t y = __shfl_up_sync(full, inc, o);
            if (lane >= o) inc += y;
        }
        const int64_t total = __shfl_sync(full, inc, 31), before = inc - low;
        for (int64_t p0 = 0; p0 < total; p0 += 32) {
            const int64_t p = p0 + lane;
            int own = 0;  // the last lane with before <= p: the one whose entry it is
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                if (__shfl_sync(full, before, own + o) <= p) own += o;
            const int64_t k = p - __shfl_sync(full, before, own), j = __shfl_sync(full, lo, own) + k;
            const int32_t oa = __shfl_sync(full, a, own), ob = __shfl_sync(full, b, own);
            if (p >= total) continue;
            const int32_t e2 = et_t[j], w = g.et_w[j];
            const int64_t l2 = g.et_rp[e2], h2 = g.et_rp[e2 + 1], t2 = g.tbase[e2];
            const int64_t s2 = (h2 - l2) - (g.tbase[e2 + 1] - t2);
            const int64_t at = nd_lower_bound(g.et_w + l2 + s2, h2 - l2 - s2, ob), tid = t2 + at;
            et_t[j] = (int32_t)tid;
            tri_pos[3 * tid + (w > oa ? 1 : 2)] = (int32_t)k;
        }
    }
}

__global__ void k_tri_tuples(GraphView g, int32_t* __restrict__ out) {
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < g.n3; t += (int64_t)gridDim.x * blockDim.x) {
        int32_t e = g.tri_e[3 * t], e1 = g.tri_e[3 * t + 1];
        out[3 * t] = g.eu[e];
        out[3 * t + 1] = g.ev[e];
        out[3 * t + 2] = g.ev[e1];
    }
}

// 4-clique index (the paper's T one level deeper, Section 5.1): the children of triangle
// t = (a<b<c) are the vertices d > c adjacent to a, b and c, ascending. Any two of the triangle's
// edge lists intersect to its common neighbourhood (L(ab) ∩ L(bc) = N(a) ∩ N(b) ∩ N(c)), so a
// warp walks the part above c of the shortest list and searches the second shortest; matches are
// compacted in order with a ballot (count pass, then fill pass at qbase[t]).
template <bool kFill>
__device__ __forceinline__ int64_t quad_children(const GraphView& g, int64_t t, int32_t* out) {
    int lane = threadIdx.x & 31;
    int32_t e[3] = {g.tri_e[3 * t], g.tri_e[3 * t + 1], g.tri_e[3 * t + 2]};
    int32_t c = g.ev[e[1]];  // edges (ab, ac, bc): the largest vertex is ac's upper end
    int64_t b[3], n[3];
    for (int k = 0; k < 3; ++k) {
        b[k] = g.et_rp[e[k]];
        n[k] = g.et_rp[e[k] + 1] - b[k];
    }
    int i0 = 0, i1 = 1;
    if (n[1] < n[0]) i0 = 1, i1 = 0;
    if (n[2] < n[i0]) i1 = i0, i0 = 2;
    else if (n[2] < n[i1]) i1 = 2;
    const int32_t* xs = g.et_w + b[i0];
    const int32_t* ys = g.et_w + b[i1];
    int64_t xlo = nd_lower_bound(xs, n[i0], c + 1), ylo = nd_lower_bound(ys, n[i1], c + 1);
    int64_t pos = 0;
    for (int64_t p0 = xlo; p0 < n[i0]; p0 += 32) {
        int64_t p = p0 + lane;
        bool hit = p < n[i0] && nd_find(ys + ylo, n[i1] - ylo, xs[p]) >= 0;
        unsigned m = __ballot_sync(0xffffffffu, hit);
        if (kFill && hit) out[pos + __popc(m & nd_lanemask_lt())] = xs[p];
        pos += __popc(m);
    }
    return pos;
}

__global__ void k_quad_count(GraphView g, int64_t* __restrict__ qcnt) {
    for (int64_t t = gwarp(); t < g.n3; t += nwarps()) {
        int64_t k = quad_children<false>(g, t, nullptr);
        if ((threadIdx.x & 31) == 0) qcnt[t] = k;
    }
}

__global__ void k_quad_fill(GraphView g, const int64_t* __restrict__ qbase, int32_t* __restrict__ qval) {
    for (int64_t t = gwarp(); t < g.n3; t += nwarps()) quad_children<true>(g, t, qval + qbase[t]);
}

// the inverse map of the 4-clique index: 4-clique q -> (a, b, c, d), one warp per triangle
__global__ void k_quad_tuples(GraphView g, int32_t* __restrict__ out) {
    int lane = threadIdx.x & 31;
    for (int64_t t = gwarp(); t < g.n3; t += nwarps()) {
        int32_t e = g.tri_e[3 * t], e1 = g.tri_e[3 * t + 1];
        int32_t a = g.eu[e], b = g.ev[e], c = g.ev[e1];
        for (int64_t q = g.qbase[t] + lane; q < g.qbase[t + 1]; q += 32) {
            out[4 * q] = a;
            out[4 * q + 1] = b;
            out[4 * q + 2] = c;
            out[4 * q + 3] = g.qval[q];
        }
    }
}

__global__ void k_edge_tuples(GraphView g, int32_t* __restrict__ out) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < g.m; e += (int64_t)gridDim.x * blockDim.x) {
        out[2 * e] = g.eu[e];
        out[2 * e + 1] = g.ev[e];
    }
}

// max over edges (u,v) of min(deg u, deg v): a bound on |N(u) ∩ N(v)| for every edge
__global__ void k_max_edge_mindeg(GraphView g, unsigned long long* __restrict__ out) {
    unsigned long long best = 0;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < g.m; e += (int64_t)gridDim.x * blockDim.x) {
        int32_t u = g.eu[e], v = g.ev[e];
        int64_t du = g.rp[u + 1] - g.rp[u], dv = g.rp[v + 1] - g.rp[v];
        unsigned long long d = (unsigned long long)(du < dv ? du : dv);
        best = d > best ? d : best;
    }
    for (int o = 16; o > 0; o >>= 1) {
        unsigned long long y = __shfl_xor_sync(0xffffffffu, best, o);
        best = y > best ? y : best;
    }
    if ((threadIdx.x & 31) == 0 && best) atomicMax(out, best);
}

__global__ void k_tri_hash_sizes(GraphView g, int64_t* __restrict__ slots) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < g.m; e += (int64_t)gridDim.x * blockDim.x) {
        int64_t n = g.et_rp[e + 1] - g.et_rp[e];
        slots[e] = nd_hashed(n) ? ((int64_t)1 << nd_hash_bits(n)) : 0;
    }
}

// Filling one list's table: each entry claims a free slot by compare-and-swap on its (w, id) pair,
// its round is set to unpeeled and the slot is recorded for its triangle (hpos). A free slot is
// all ones. The triangle's edges are (xy, xz, yz) for x < y < z: e = (a, c) is xy when w > c, xz
// when a < w < c, yz when w < a.
__device__ __forceinline__ int hash_which(int32_t w, int32_t a, int32_t c) { return w > c ? 0 : (w > a ? 1 : 2); }

// Tables of at most 2^kHashSmemBits slots are built in shared memory, (w, id) pairs only, by one
// block per list, and written out whole and coalesced (free slots included), so the directory
// needs no clearing and the compare-and-swaps stay on chip. Each block collects the lists of
// 256 consecutive edges that qualify and then fills them one after another.
constexpr int kHashSmemBits = 13;  // 8,192 slots: 64 KiB of (w, id) pairs
constexpr int kHashBlock = 256;

__global__ void __launch_bounds__(kHashBlock) k_tri_hash_fill_smem(GraphView g, const int64_t* __restrict__ hoff,
                                                                    NdHashSlot* __restrict__ tab,
                                                                    int32_t* __restrict__ hpos) {
    extern __shared__ unsigned long long s_tab[];
    __shared__ int64_t s_list[kHashBlock];
    __shared__ int s_cnt;
    for (int64_t base = (int64_t)blockIdx.x * kHashBlock; base < g.m; base += (int64_t)gridDim.x * kHashBlock) {
        if (threadIdx.x == 0) s_cnt = 0;
        __syncthreads();
        const int64_t e0 = base + threadIdx.x;
        if (e0 < g.m) {
            int64_t n = g.et_rp[e0 + 1] - g.et_rp[e0];
            if (nd_hashed(n) && nd_hash_bits(n) <= kHashSmemBits) s_list[atomicAdd(&s_cnt, 1)] = e0;
        }
        __syncthreads();
        const int cnt = s_cnt;
        for (int q = 0; q < cnt; ++q) {
            const int64_t e = s_list[q];
            const int64_t b = g.et_rp[e], n = g.et_rp[e + 1] - b;
            const int k = nd_hash_bits(n);
            const uint32_t S = 1u << k, mask = S - 1u;
            for (uint32_t i = threadIdx.x; i < S; i += kHashBlock) s_tab[i] = ~0ull;
            __syncthreads();
            const int32_t a = g.eu[e], c = g.ev[e];
            for (int64_t p = threadIdx.x; p < n; p += kHashBlock) {
                const int32_t w = g.et_w[b + p], id = g.et_t[b + p];
                const unsigned long long key = ((unsigned long long)(uint32_t)id << 32) | (uint32_t)w;
                uint32_t sl = nd_hash_slot(w, k);
                for (uint32_t probes = 0; probes <= mask; ++probes) {
                    if (atomicCAS(&s_tab[sl], ~0ull, key) == ~0ull) {
                        hpos[3 * (int64_t)id + hash_which(w, a, c)] = (int32_t)sl;
                        break;
                    }
                    sl = (sl + 1) & mask;
                }
            }
            __syncthreads();
            int4* out = reinterpret_cast<int4*>(tab + hoff[e]);
            for (uint32_t i = threadIdx.x; i < S; i += kHashBlock) {
                const unsigned long long v = s_tab[i];
                out[i] = v == ~0ull ? make_int4(-1, -1, -1, -1)
                                    : make_int4((int32_t)(uint32_t)v, (int32_t)(v >> 32), ND_UNPEELED, -1);
            }
            __syncthreads();
        }
    }
}

// Larger tables: one warp per list clears its table, then claims slots in global memory.
__global__ void k_tri_hash_fill(GraphView g, const int64_t* __restrict__ hoff, NdHashSlot* __restrict__ tab,
                                int32_t* __restrict__ hpos) {
    int lane = threadIdx.x & 31;
    for (int64_t e = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; e < g.m;
         e += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        int64_t b = g.et_rp[e], n = g.et_rp[e + 1] - b;
        if (!nd_hashed(n)) continue;
        int k = nd_hash_bits(n);
        if (k <= kHashSmemBits) continue;
        uint32_t mask = (1u << k) - 1u;
        NdHashSlot* t = tab + hoff[e];
        int4* t4 = reinterpret_cast<int4*>(t);
        for (uint32_t i = lane; i <= mask; i += 32) t4[i] = make_int4(-1, -1, -1, -1);
        __syncwarp();
        const int32_t a = g.eu[e], c = g.ev[e];  // e = (a, c), a < c
        for (int64_t p = lane; p < n; p += 32) {
            int32_t w = g.et_w[b + p], id = g.et_t[b + p];
            unsigned long long key = ((unsigned long long)(uint32_t)id << 32) | (uint32_t)w;  // little endian: w first
            uint32_t s = nd_hash_slot(w, k);
            for (uint32_t probes = 0; probes <= mask; ++probes) {
                unsigned long long* half = reinterpret_cast<unsigned long long*>(t + s);
                if (atomicCAS(half, 0xffffffffffffffffull, key) == 0xffffffffffffffffull) {
                    t[s].rnd = ND_UNPEELED;
                    hpos[3 * (int64_t)id + hash_which(w, a, c)] = (int32_t)s;
                    break;
                }
                s = (s + 1) & mask;
            }
        }
    }
}

}  // namespace

void nd_tri_hash_sizes(const GraphView& g, int64_t* slots, cudaStream_t st) {
    if (g.m <= 0) return;
    ND_K(k_tri_hash_sizes<<<blocks_for_threads(g.m), kThreads, 0, st>>>(g, slots));
}

void nd_tri_hash_fill(const GraphView& g, const int64_t* hoff, NdHashSlot* tab, int32_t* hpos, cudaStream_t st) {
    if (g.m <= 0) return;
    const int smem = (int)sizeof(unsigned long long) << kHashSmemBits;
    cudaFuncSetAttribute(k_tri_hash_fill_smem, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    int64_t want = (g.m + kHashBlock - 1) / kHashBlock, cap = (int64_t)nd_sm_count() * 3;
    int blocks = (int)(want < cap ? (want > 0 ? want : 1) : cap);
    ND_K(k_tri_hash_fill_smem<<<blocks, kHashBlock, smem, st>>>(g, hoff, tab, hpos));
    ND_K(k_tri_hash_fill<<<blocks_for_warps(g.m), kThreads, 0, st>>>(g, hoff, tab, hpos));
}

void nd_max_edge_mindeg(const GraphView& g, unsigned long long* out, cudaStream_t st) {
    if (g.m <= 0) return;
    ND_K(k_max_edge_mindeg<<<blocks_for_threads(g.m), kThreads, 0, st>>>(g, out));
}

void nd_validate_csr(const int64_t* rp, const int32_t* col, int32_t n, int64_t nnz, int* err, cudaStream_t st) {
    if (n <= 0) return;
    ND_K(k_validate<<<blocks_for_warps(n), kThreads, 0, st>>>(rp, col, n, nnz, err));
}

void nd_build_split(const int64_t* rp, const int32_t* col, int32_t n, int64_t* split, int64_t* updeg,
                    cudaStream_t st) {
    if (n <= 0) return;
    ND_K(k_split<<<blocks_for_threads(n), kThreads, 0, st>>>(rp, col, n, split, updeg));
}

static int blocks_for_segments(int64_t nnz) { return blocks_for_warps((nnz + seg_len(nnz) - 1) / seg_len(nnz)); }

int64_t nd_dg_segments(int64_t m) { return (2 * m + seg_len(2 * m) - 1) / seg_len(2 * m); }

void nd_build_pos2e(const GraphView& g, int32_t* pos2e, int32_t* eu, int32_t* ev, int* err, cudaStream_t st) {
    if (g.m <= 0) return;
    ND_K(k_pos2e<<<blocks_for_segments(2 * g.m), kThreads, 0, st>>>(g, 2 * g.m, seg_len(2 * g.m), pos2e, eu, ev,
                                                                                    err));
}

void nd_dg_count(const GraphView& g, const int32_t* key_hi, int64_t* outdeg, int32_t* tail, cudaStream_t st) {
    if (g.m <= 0) return;
    ND_K(k_dg_count<<<blocks_for_segments(2 * g.m), kThreads, 0, st>>>(g, 2 * g.m, seg_len(2 * g.m), key_hi, outdeg,
                                                                                       tail));
}

void nd_dg_fill(const GraphView& g, const int32_t* key_hi, int64_t* dg_rp, const int32_t* tail, int32_t* dg_col,
                int32_t* dg_eid, cudaStream_t st) {
    if (g.m <= 0) return;
    ND_K(k_dg_fill<<<blocks_for_segments(2 * g.m), kThreads, 0, st>>>(g, 2 * g.m, seg_len(2 * g.m), key_hi, dg_rp,
                                                                                      tail, dg_col, dg_eid));
}

void nd_edge_support(const GraphView& g, int32_t* sigma, int32_t* up, cudaStream_t st) {
    if (g.m <= 0) return;
    const int tile = tri_tile(g.m);
    ND_K(k_edge_support<<<blocks_for_warps((g.m + tile - 1) / tile), kTriThreads, 0, st>>>(g, tile, sigma, up));
}

void nd_dup_check(const GraphView& g, const int32_t* sigma, int* err, cudaStream_t st) {
    if (g.m <= 0) return;
    ND_K(k_dup_check<<<blocks_for_segments(2 * g.m), kThreads, 0, st>>>(g, 2 * g.m, seg_len(2 * g.m), sigma, err));
}

void nd_row_work(const GraphView& g, const int32_t* sigma, unsigned long long* rows, cudaStream_t st) {
    if (g.m <= 0) return;
    const int64_t every = g.m >= 1 << 20 ? 16 : 1;
    ND_K(k_row_work<<<blocks_for_threads(g.m / every), kThreads, 0, st>>>(g, sigma, every, rows));
}

bool nd_gather_pays(int64_t n3, unsigned long long rows) { return n3 >= 1 << 16 && rows > 40 * (unsigned long long)n3; }

static int index_tile(int64_t m) {
    const int64_t t = m / ((int64_t)nd_sm_count() * 256);
    return (int)(t < 1 ? 1 : t > 32 ? 32 : t);
}

void nd_edge_fill(const GraphView& g, int64_t* et_rp, int64_t* tbase, int32_t* et_w, int32_t* et_t, int32_t* tri_e,
                  int32_t* tri_pos, const int32_t* sigma, int32_t* cursor, int32_t* entries, cudaStream_t st) {
    if (g.m <= 0) return;
    const int64_t nent = 3 * g.n3;
    const int edges = index_tile(g.m), blk = blocks_for_warps((g.m + edges - 1) / edges);
    if (cursor) {
        const int tile = tri_tile(g.m);
        GatherSink sink{et_rp, sigma, g.dg_eid, cursor, entries, entries + nent, entries + 2 * nent};
        ND_K(k_edge_gather<<<blocks_for_warps((g.m + tile - 1) / tile), kTriThreads, 0, st>>>(g, tile, sink));
        ND_K(k_edge_order<<<blk, kThreads, 0, st>>>(g, et_rp, tbase, entries, entries + nent, entries + 2 * nent, et_w, et_t,
                                                    tri_e, tri_pos, edges));
    }
    ND_K(k_edge_fill<<<blk, kThreads, 0, st>>>(g, et_rp, tbase, et_w, et_t, tri_e, tri_pos, cursor ? kShortList : 0, edges));
}

void nd_edge_fill_tid(const GraphView& g, int32_t* et_t, int32_t* tri_pos, cudaStream_t st) {
    if (g.m <= 0) return;
    const int edges = index_tile(g.m);
    ND_K(k_edge_fill_tid<<<blocks_for_warps((g.m + edges - 1) / edges), kThreads, 0, st>>>(g, et_t, tri_pos, edges));
}


void nd_tri_tuples(const GraphView& g, int32_t* out, cudaStream_t st) {
    if (g.n3 <= 0) return;
    ND_K(k_tri_tuples<<<blocks_for_threads(g.n3), kThreads, 0, st>>>(g, out));
}

void nd_edge_tuples(const GraphView& g, int32_t* out, cudaStream_t st) {
    if (g.m <= 0) return;
    ND_K(k_edge_tuples<<<blocks_for_threads(g.m), kThreads, 0, st>>>(g, out));
}

void nd_quad_count(const GraphView& g, int64_t* qcnt, cudaStream_t st) {
    if (g.n3 <= 0) return;
    ND_K(k_quad_count<<<blocks_for_warps(g.n3), kThreads, 0, st>>>(g, qcnt));
}

void nd_quad_fill(const GraphView& g, const int64_t* qbase, int32_t* qval, cudaStream_t st) {
    if (g.n3 <= 0) return;
    ND_K(k_quad_fill<<<blocks_for_warps(g.n3), kThreads, 0, st>>>(g, qbase, qval));
}

void nd_quad_tuples(const GraphView& g, int32_t* out, cudaStream_t st) {
    if (g.n3 <= 0) return;
    ND_K(k_quad_tuples<<<blocks_for_warps(g.n3), kThreads, 0, st>>>(g, out));
}
