// The triangles of the oriented graph, each once, with the ids of their vertices and edges: counted by
// nd_count.cu, put into incidence lists by nd_inc.cu.
#pragma once

#include "nd_common.cuh"

constexpr int kTriThreads = 256;

// Edges per warp and step: 32, and fewer where the graph has too few edges to give every resident warp as
// many (a graph of 534 vertices and 7,700 edges at 32: 240 warps, each with a thousand candidates in a row,
// 36 us for a count that takes 8 us with one edge each).
inline int tri_tile(int64_t m) {
    const int64_t warps = (int64_t)nd_sm_count() * 64;
    const int64_t t = (m + warps - 1) / warps;
    return (int)(t < 1 ? 1 : t > 32 ? 32 : t);
}

// A warp takes `tile` DG edges u -> v at a time. Each lane sets one up: the shorter of N_DG(u) and N_DG(v)
// drives and the longer is searched. The warp numbers the candidates of all its edges by a prefix sum and
// takes 32 at a time, whatever edges they belong to, so that the many edges with two or three
// candidates fill its lanes as well as the few with thousands. The whole warp calls sink.tri() with each
// lane's candidate: whether it is a triangle, the slot of u -> v among the edges, its edge, the DG
// positions of the other two edges (the first is u's if of_u), and the vertices. sink.end() is called once per edge by the lane
// that set it up.
//
// Bound by the bisections' loads (L1 and L2) and, past them, by the sinks' atomics. Against one warp per edge
// merging the two undirected rows, which meets each triangle three times: (2,3) counts of R-MAT scale 20
// 42 -> 16.5 ms, of a Chung-Lu graph with 2.4 M edges 1.10 -> 0.33 ms.
// With `every` > 1 only one tile of edges in that many is taken, for an estimate.
template <typename Sink>
__device__ __forceinline__ void tri_list(const GraphView& g, int tile, Sink& sink, int64_t every = 1) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5, apart = tile * every;
    for (int64_t j0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * apart; j0 < g.m; j0 += nwarps * apart) {
        const int64_t j = lane < tile ? j0 + lane : g.m;
        int32_t u = 0, v = 0, e = 0, xb = 0, xn = 0, yb = 0, yn = 0;  // DG positions are below m < 2^31
        int32_t of_u = 0;
        if (j < g.m) {
            e = g.dg_eid[j];
            v = g.dg_col[j];
            const int32_t a = g.eu[e];
            u = a == v ? g.ev[e] : a;
            const int32_t ub = (int32_t)g.dg_rp[u], un = (int32_t)g.dg_rp[u + 1] - ub;
            const int32_t vb = (int32_t)g.dg_rp[v], vn = (int32_t)g.dg_rp[v + 1] - vb;
            const bool u_drives = un <= vn;
            of_u = u_drives;
            xb = u_drives ? ub : vb, xn = u_drives ? un : vn;
            yb = u_drives ? vb : ub, yn = u_drives ? vn : un;
        }
        sink.begin(lane);
        int64_t inc = xn;
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t y = __shfl_up_sync(full, inc, o);
            if (lane >= o) inc += y;
        }
        const int64_t total = __shfl_sync(full, inc, 31);
        const int64_t before = inc - xn;
        for (int64_t p0 = 0; p0 < total; p0 += 32) {
            const int64_t p = p0 + lane;
            int own = 0;  // the last lane with before <= p and candidates of its own
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const int64_t b = __shfl_sync(full, before, own + o);
                if (b <= p) own += o;
            }
            const int32_t oxb = __shfl_sync(full, xb, own), oyb = __shfl_sync(full, yb, own);
            const int32_t oyn = __shfl_sync(full, yn, own), oof = __shfl_sync(full, of_u, own);
            const int64_t ob = __shfl_sync(full, before, own);
            const int32_t ou = __shfl_sync(full, u, own), ov = __shfl_sync(full, v, own), oe = __shfl_sync(full, e, own);
            const int32_t px = oxb + (int32_t)(p - ob);
            int32_t w = 0;
            int lo = 0;
            bool hit = false;
            if (p < total) {
                const int32_t* ys = g.dg_col + oyb;
                int hi = oyn;
                w = g.dg_col[px];
#pragma unroll 1
                while (lo < hi) {
                    const int mid = (lo + hi) >> 1;
                    if (__ldg(ys + mid) < w)
                        lo = mid + 1;
                    else
                        hi = mid;
                }
                hit = lo < oyn && __ldg(ys + lo) == w;
            }
            sink.tri(hit, own, oe, px, oyb + lo, oof != 0, ou, ov, w);
        }
        __syncwarp();
        if (j < g.m) sink.end(lane, e, u, v);
        __syncwarp();
    }
}
