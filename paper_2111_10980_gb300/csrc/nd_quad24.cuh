// The 4-cliques of the oriented graph with the ids of their edges, for (2,4): counted by nd_count.cu,
// put into incidence lists by nd_inc.cu.
#pragma once

#include "nd_common.cuh"

constexpr int kQuadThreads = 256;

// (2,4), one warp per DG edge u -> v: the 4-cliques whose two lowest vertices (in the orientation)
// are u and v are u, v plus a DG edge w -> x inside I = N_DG(u) ∩ N_DG(v). The warp stages I in
// shared memory (ascending ids, with the edge ids u-w and v-w and the out-list bounds of each w),
// numbers the candidate pairs (w, k-th out-neighbour of w) through a prefix sum of the out-degrees
// and spreads them evenly over its lanes; a lane finds x in the staged I by bisection. A sink that
// tallies (kTally) gets w-x of every 4-clique, and at the end the numbers of u-w, v-w (the same for
// both, kept in shared memory meanwhile) and u-v: one global atomic for each 4-clique instead of five
// (R-MAT of 50,001 vertices, 131 M 4-cliques: the count call 7.0 -> 5.2 ms, with the vertex u read
// from the edge instead of bisected). Another sink gets the six edges, u-v
// first, from the whole warp, with each lane saying whether it has a 4-clique.
// An edge whose I does not fit the stage (more than kC24 vertices) is listed by the lanes walking
// out-lists instead; a tallying sink's clique() then adds to all but u-v.
constexpr int kC24 = 128;

__device__ __forceinline__ int stage_find24(const int32_t* a, int n, int32_t x) {
    int lo = 0, hi = n;
    while (lo < hi) {
        int mid = (lo + hi) >> 1;
        if (a[mid] < x)
            lo = mid + 1;
        else
            hi = mid;
    }
    return (lo < n && a[lo] == x) ? lo : -1;
}

// With `every` > 1 only one DG edge in that many is taken, for an estimate.
template <typename Sink>
__device__ __forceinline__ void quad24_list(const GraphView& g, Sink& sink, int64_t every = 1) {
    constexpr int kWarpsPerBlock = kQuadThreads / 32;
    __shared__ int32_t s_w[kWarpsPerBlock][kC24], s_eu[kWarpsPerBlock][kC24], s_ev[kWarpsPerBlock][kC24],
        s_b[kWarpsPerBlock][kC24], s_p[kWarpsPerBlock][kC24 + 1];
    __shared__ int32_t s_c[Sink::kTally ? kWarpsPerBlock : 1][Sink::kTally ? kC24 : 1];
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int32_t *sw = s_w[wid], *seu = s_eu[wid], *sev = s_ev[wid], *sb = s_b[wid], *sp = s_p[wid];
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t j = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * every; j < g.m; j += nwarps * every) {
        const int32_t v = g.dg_col[j], e_uv = g.dg_eid[j];
        const int32_t u = g.eu[e_uv] == v ? g.ev[e_uv] : g.eu[e_uv];
        const int64_t ub = g.dg_rp[u], ue = g.dg_rp[u + 1], vb = g.dg_rp[v], vn = g.dg_rp[v + 1] - vb;
        // stage I = N_DG(u) ∩ N_DG(v) in order
        int c = 0;
        for (int64_t p0 = ub; p0 < ue; p0 += 32) {
            int64_t p = p0 + lane;
            int64_t q = p < ue ? nd_find(g.dg_col + vb, vn, g.dg_col[p]) : -1;
            unsigned mk = __ballot_sync(full, q >= 0);
            if (q >= 0) {
                int at = c + __popc(mk & nd_lanemask_lt());
                if (at < kC24) {
                    int32_t w = g.dg_col[p];
                    sw[at] = w;
                    seu[at] = g.dg_eid[p];
                    sev[at] = g.dg_eid[vb + q];
                    sb[at] = (int32_t)g.dg_rp[w];
                    sp[at] = (int32_t)(g.dg_rp[w + 1] - g.dg_rp[w]);
                }
            }
            c += __popc(mk);
        }
        if (c < 2) {  // a 4-clique needs two vertices of I
            __syncwarp();
            continue;
        }
        if constexpr (Sink::kTally)
            for (int i = lane; i < c && i < kC24; i += 32) s_c[wid][i] = 0;
        __syncwarp();
        unsigned long long c_uv = 0;
        if (c <= kC24) {
            // exclusive prefix of the out-degrees (c <= kC24: at most four 32-wide chunks)
            int32_t carry = 0;
            for (int c0 = 0; c0 < c; c0 += 32) {
                int i = c0 + lane;
                int32_t d = i < c ? sp[i] : 0, inc = d;
                for (int o = 1; o < 32; o <<= 1) {
                    int32_t y = __shfl_up_sync(full, inc, o);
                    if (lane >= o) inc += y;
                }
                if (i < c) sp[i] = carry + inc - d;
                carry += __shfl_sync(full, inc, 31);
            }
            if (lane == 0) sp[c] = carry;
            __syncwarp();
            for (int32_t p0 = 0; p0 < carry; p0 += 32) {
                const int32_t p = p0 + lane;
                int a = 0, b = c, k = -1;  // owner a: the last i with sp[i] <= p
                int64_t jx = 0;
                if (p < carry) {
                    while (b - a > 1) {
                        int mid = (a + b) >> 1;
                        if (sp[mid] <= p)
                            a = mid;
                        else
                            b = mid;
                    }
                    jx = (int64_t)sb[a] + (p - sp[a]);
                    k = stage_find24(sw, c, g.dg_col[jx]);
                }
                if constexpr (Sink::kTally) {
                    if (k < 0) continue;
                    ++c_uv;
                    sink.pair(g.dg_eid[jx]);
                    atomicAdd(&s_c[wid][k], 1);
                    atomicAdd(&s_c[wid][a], 1);
                } else {
                    const bool hit = k >= 0;
                    const int32_t e[6] = {e_uv, hit ? seu[k] : 0, hit ? sev[k] : 0, seu[a], sev[a], hit ? g.dg_eid[jx] : 0};
                    sink.clique(hit, e);
                }
            }
            if constexpr (Sink::kTally) {
                // w's 4-cliques with u and v count for u-w and for v-w alike
                __syncwarp();
                for (int i = lane; i < c; i += 32)
                    if (const int32_t n = s_c[wid][i]) {
                        sink.add(seu[i], n);
                        sink.add(sev[i], n);
                    }
            }
        } else {
            // I does not fit the stage: the lanes take the w of N_DG(u) ∩ N_DG(v) and walk their
            // out-lists, searching x in both lists
            for (int64_t p0 = ub; p0 < ue; p0 += 32) {
                const int64_t p = p0 + lane;
                const int32_t w = p < ue ? g.dg_col[p] : 0;
                const int64_t q = p < ue ? nd_find(g.dg_col + vb, vn, w) : -1;
                int64_t jx = q < 0 ? 0 : g.dg_rp[w];
                const int64_t je = q < 0 ? 0 : g.dg_rp[w + 1];
                const int32_t e_uw = q < 0 ? 0 : g.dg_eid[p], e_vw = q < 0 ? 0 : g.dg_eid[vb + q];
                for (; __any_sync(full, jx < je); ++jx) {
                    int64_t pux = -1, pvx = -1;
                    if (jx < je) {
                        const int32_t x = g.dg_col[jx];
                        pux = nd_find(g.dg_col + ub, ue - ub, x);
                        if (pux >= 0) pvx = nd_find(g.dg_col + vb, vn, x);
                    }
                    const bool hit = pvx >= 0;
                    int32_t e[6] = {e_uv, 0, 0, e_uw, e_vw, 0};
                    if (hit) {
                        e[1] = g.dg_eid[ub + pux];
                        e[2] = g.dg_eid[vb + pvx];
                        e[5] = g.dg_eid[jx];
                        ++c_uv;
                    }
                    sink.clique(hit, e);
                }
            }
        }
        if constexpr (!Sink::kTally) {
            __syncwarp();
            continue;
        }
        for (int o = 16; o > 0; o >>= 1) c_uv += __shfl_down_sync(full, c_uv, o);
        if constexpr (Sink::kTally)
            if (lane == 0 && c_uv) sink.add(e_uv, (int64_t)c_uv);
        __syncwarp();
    }
}
