// Per-vertex (orbit) counts of the connected induced 4-vertex motifs: an output mode beside the
// global counts of Section III-F (the paper's closure is global; this refines every induced
// occurrence S by the role of each of its vertices, the role being the vertex's automorphism class
// in the motif, which for 4-vertex motifs its degree inside G[S] decides).  Eleven roles, in order:
//   0 star centre  1 star leaf  2 path end  3 path inner  4 paw pendant  5 paw hub (degree 3)
//   6 paw side (degree-2 triangle vertex)  7 cycle  8 diamond spine (degree 3)  9 diamond tip
//   10 clique
// The same closure idea as the global counts, per vertex: eleven non-induced statistics N_i(v) (copies
// of a pattern in which v plays role i) are sums of degrees, per-edge triangle counts t_e, per-vertex
// triangle, 4-cycle and 4-clique counts, and their containment in the induced roles is a unit
// upper-triangular integer matrix, so the roles follow by back-substitution without division:
//   N0 = C(d_v, 3)                                N1 = sum_{c in N(v)} C(d_c - 1, 2)
//   N2 = sum_{a in N(v)} S1(a) - d_v (d_v - 1) - 2 t_v,  S1(a) = sum_{b in N(a)} (d_b - 1)
//   N3 = (d_v - 1) S1(v) - 2 t_v                  N4 = sum_{h in N(v)} t_h - 2 t_v
//   N5 = t_v (d_v - 2)                            N6 = sum_{h in N(v)} t_vh (d_h - 2)
//   N7 = 4-cycles through v                       N8 = sum_{s in N(v)} C(t_vs, 2)
//   N9 = sum over triangles {v, a, b} of (t_ab - 1)
//   N10 = 4-cliques through v = tau(H_v), gathered six-fold in tau6
// with t_v = (1/2) sum_{h in N(v)} t_vh the triangles on v.
//
// Passes after orientation and the triangle pass (which leaves t_e of every out-arc in ws.te):
//   orbit_triangles  (tri.cu) every triangle {u, a, b} once, anchored at its lowest vertex u, routes t_ab - 1,
//                 t_ub - 1, t_ua - 1 to N9 of u, a, b and the 4-cliques on u, a, b found from the anchor's
//                 bitmap to tau6; k_orb_tri_big does the same for anchors of out-degree above 1024, a warp per
//                 out-arc
//   k_orb_vertex  t_v, S1(v), N1, N6, N8 (k_orb_vertex_hub: rows of more than 256 neighbours)
//   k_orb_c4w     warp per root u with wedge work W(u) <= kMidMax (a shared-memory hash, two sizes),
//   k_orb_c4win   a block per heavier root, counters of a window of ranks in shared memory, or, for graphs of
//                 more than kWinMax windows,
//   k_orb_c4b     a block per heavier root, dense counters over all ranks in a per-block global array: every
//                 4-cycle has one top vertex u, opposite corner x and middles w1, w2 below u; with cnt(x) the
//                 wedges u - w - x, u gets sum_x C(cnt(x), 2), x gets C(cnt(x), 2) and each middle w gets
//                 sum_{x in its segment} (cnt(x) - 1)
//   k_orb_close   warp per vertex: N2, N4, N0, N3, N5, N9, N10 and the back-substitution, written to
//                 the input id of the vertex.
//
// Per-edge (edge orbit) counts use the same passes with routing to edges instead of vertices: ten
// roles of an edge inside G[S] (its endpoints' degrees there decide them), ten statistics E_i(e) for
// e = (a, b) and a unit upper-triangular 10 x 10 containment system:
//   E0 = C(d_a - 1, 2) + C(d_b - 1, 2)          E1 = S1(a) + S1(b) - d_a - d_b + 2 - 2 t_ab
//   E2 = (d_a - 1)(d_b - 1) - t_ab              E3 = t_a + t_b - 2 t_ab
//   E4 = t_ab (d_a + d_b - 4)                   E5 = sum_{h in N(a) n N(b)} (d_h - 2)
//   E6 = 4-cycles through e                     E7 = C(t_ab, 2)
//   E8 = sum_{s in N(a) n N(b)} (t_as - 1) + (t_bs - 1)
//   E9 = 4-cliques through e (gathered twice)
// E5, E8 and E9 are routed from each triangle to its three edges (orbit_triangles), E6 from the wedge walk:
// each wedge u - w - x adds cnt(x) - 1 to the arcs (u, w) and (w, x) (k_orb_c4w / k_orb_c4win / k_orb_c4b), and
// k_eorb_close evaluates one edge per thread and writes it at the edge's index in the input graph's
// edge list ((a, b), a < b, lexicographic by input id).
#include "harp_internal.cuh"

namespace harp {
namespace {

constexpr int kOrbThreads = 256;
constexpr int kOrbWarps = kOrbThreads / 32;
constexpr int kOrbStage = 512;      // C_uv members staged per warp
constexpr int kHashSlots = 1024;    // per-warp wedge hash (roots with W(u) <= kHashMax)
constexpr int kHashMax = 512;
constexpr int kMidSlots = 4096;     // and of the middle tier (W(u) <= kMidMax)
constexpr int kMidMax = 2048;
constexpr int kMidWarps = 4;         // a block of this many warps per root
constexpr int32_t kNoKey = -1;
constexpr int kOrbits = 11;

// the containment matrix of the per-vertex system (row: statistic, column: role), unit upper triangular
__constant__ uint8_t c_contain[kOrbits][kOrbits] = {
    {1, 0, 0, 0, 0, 1, 0, 0, 1, 0, 1}, {0, 1, 0, 0, 1, 0, 1, 0, 1, 2, 3}, {0, 0, 1, 0, 2, 0, 1, 2, 2, 4, 6},
    {0, 0, 0, 1, 0, 2, 1, 2, 4, 2, 6}, {0, 0, 0, 0, 1, 0, 0, 0, 0, 2, 3}, {0, 0, 0, 0, 0, 1, 0, 0, 2, 0, 3},
    {0, 0, 0, 0, 0, 0, 1, 0, 2, 2, 6}, {0, 0, 0, 0, 0, 0, 0, 1, 1, 1, 3}, {0, 0, 0, 0, 0, 0, 0, 0, 1, 0, 3},
    {0, 0, 0, 0, 0, 0, 0, 0, 0, 1, 3}, {0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 1}};

struct OrbGraph {
    const int64_t* off;    // rank-order CSR, rows sorted
    const int32_t* cols;
    const int32_t* deg;
    const int64_t* offp;   // out-lists N+(v) and t_e of every out-arc
    const int32_t* colsp;
    const uint32_t* te;
};

__device__ __forceinline__ bool has(const int32_t* __restrict__ cols, int64_t b, int64_t e, int32_t x) {
    const int64_t p = b + lower_bound_i32(cols + b, e - b, x);
    return p < e && __ldg(cols + p) == x;
}

// the out-arc of the edge {a, b} (a != b adjacent): the lower rank's out-list holds the higher one
__device__ __forceinline__ int64_t arc_of(const OrbGraph& G, int32_t a, int32_t b) {
    const int32_t lo = a < b ? a : b, hi = a < b ? b : a;
    const int64_t pb = G.offp[lo], pe = G.offp[lo + 1];
    return pb + lower_bound_i32(G.colsp + pb, pe - pb, hi);
}
// t of the edge {a, b}
__device__ __forceinline__ uint64_t t_of(const OrbGraph& G, int32_t a, int32_t b) {
    return (uint64_t)G.te[arc_of(G, a, b)];
}

__device__ __forceinline__ int32_t arc_row(const int64_t* __restrict__ offp, int64_t n, int64_t a) {
    int64_t lo = 0, hi = n;
    while (hi - lo > 1) {
        const int64_t mid = (lo + hi) >> 1;
        if (offp[mid] <= a) lo = mid;
        else hi = mid;
    }
    return (int32_t)lo;
}

// ---------------------------------------------------------------------------------------------
// Triangles: N9 and tau6 routing, for anchors of out-degree above 1024 (the others: orbit_triangles, tri.cu).
// ---------------------------------------------------------------------------------------------
// Per-edge routing targets of the triangle pass (per out-arc; all nullptr for the per-vertex mode).
struct EdgeRoute {
    unsigned long long* e5;  // sum of (d of the third vertex - 2)
    unsigned long long* e8;  // sum of (t - 1) of the other two edges
    unsigned long long* e9;  // twice the 4-cliques through the edge
};

// The queued anchors q[0, *qcnt): a block per anchor, a warp per out-arc.
__global__ void __launch_bounds__(kOrbThreads) k_orb_tri_big(OrbGraph G, const int32_t* __restrict__ q,
                                                             const uint64_t* __restrict__ qcnt,
                                                             unsigned long long* __restrict__ n9,
                                                             unsigned long long* __restrict__ tau6, EdgeRoute er) {
    grid_begin();
    __shared__ int32_t sbuf[kOrbWarps][kOrbStage];
    const int w = threadIdx.x >> 5, l = lane_id();
    for (int64_t i = blockIdx.x; i < (int64_t)*qcnt; i += gridDim.x)
    for (int64_t a = G.offp[q[i]] + w; a < G.offp[q[i] + 1]; a += kOrbWarps) {
        const int32_t u = q[i];
        const int32_t v = G.colsp[a];
        const uint64_t t_uv = G.te[a];
        if (t_uv == 0) continue;
        // the 4-cliques counted here have u as their lowest vertex: only u's neighbours above it are walked
        const int64_t ub = G.off[u + 1] - (G.offp[u + 1] - G.offp[u]), ue = G.off[u + 1];
        const int64_t vb = G.off[v], ve = G.off[v + 1];
        const bool staged = t_uv <= (uint64_t)kOrbStage;
        uint32_t ns = 0;  // members of N+(u) n N(v), staged in rank order
        if (staged) {
            for (int64_t k0 = ub; k0 < ue; k0 += 32) {
                const int64_t k = k0 + l;
                const int32_t x = k < ue ? __ldg(G.cols + k) : -1;
                const bool in = k < ue && has(G.cols, vb, ve, x);
                const uint32_t bal = __ballot_sync(kFull, in);
                const uint32_t pos = ns + __popc(bal & lanemask_lt());
                if (in && pos < (uint32_t)kOrbStage) sbuf[w][pos] = x;  // pos < t_uv <= kOrbStage
                ns += __popc(bal);
            }
            __syncwarp();
        }
        auto triangle = [&](int32_t wv) {
            const int64_t wb = G.off[wv], we = G.off[wv + 1];
            uint32_t c3 = 0;
            if (staged) {
                for (uint32_t k = l; k < ns; k += 32) c3 += has(G.cols, wb, we, sbuf[w][k]) ? 1u : 0u;
            } else {
                for (int64_t k = ub + l; k < ue; k += 32) {
                    const int32_t x = __ldg(G.cols + k);
                    c3 += (has(G.cols, vb, ve, x) && has(G.cols, wb, we, x)) ? 1u : 0u;
                }
            }
            c3 = warp_sum(c3);
            if (l == 0 && n9) {
                const uint64_t t_uw = t_of(G, u, wv), t_vw = t_of(G, v, wv);
                atomicAdd(&n9[u], (unsigned long long)(t_vw - 1));
                atomicAdd(&n9[v], (unsigned long long)(t_uw - 1));
                atomicAdd(&n9[wv], (unsigned long long)(t_uv - 1));
                if (c3) {
                    atomicAdd(&tau6[u], 2ull * c3);
                    atomicAdd(&tau6[v], 3ull * c3);
                    atomicAdd(&tau6[wv], 3ull * c3);
                }
            }
            if (l == 0 && er.e5) {  // the triangle's three edges: (u, v) = arc a, (u, w), (v, w)
                const int64_t a_uw = arc_of(G, u, wv), a_vw = arc_of(G, v, wv);
                const uint64_t t_uw = G.te[a_uw], t_vw = G.te[a_vw];
                const uint64_t du = (uint64_t)G.deg[u], dv = (uint64_t)G.deg[v], dw = (uint64_t)G.deg[wv];
                atomicAdd(&er.e5[a], (unsigned long long)(dw - 2));
                atomicAdd(&er.e5[a_uw], (unsigned long long)(dv - 2));
                atomicAdd(&er.e5[a_vw], (unsigned long long)(du - 2));
                atomicAdd(&er.e8[a], (unsigned long long)((t_uw - 1) + (t_vw - 1)));
                atomicAdd(&er.e8[a_uw], (unsigned long long)((t_uv - 1) + (t_vw - 1)));
                atomicAdd(&er.e8[a_vw], (unsigned long long)((t_uv - 1) + (t_uw - 1)));
                if (c3) {
                    atomicAdd(&er.e9[a], (unsigned long long)c3);
                    atomicAdd(&er.e9[a_uw], (unsigned long long)c3);
                    atomicAdd(&er.e9[a_vw], 2ull * c3);
                }
            }
        };
        if (staged) {
            uint32_t below = 0;
            for (uint32_t k = l; k < ns; k += 32) below += sbuf[w][k] < v ? 1u : 0u;
            for (uint32_t i = warp_sum(below); i < ns; ++i) triangle(sbuf[w][i]);
        } else {
            for (int64_t k0 = ub + lower_bound_i32(G.cols + ub, ue - ub, v + 1); k0 < ue; k0 += 32) {
                const int64_t k = k0 + l;
                const int32_t x = k < ue ? __ldg(G.cols + k) : -1;
                uint32_t bal = __ballot_sync(kFull, k < ue && has(G.cols, vb, ve, x));
                while (bal) {
                    const int src = __ffs(bal) - 1;
                    bal &= bal - 1;
                    triangle(__shfl_sync(kFull, x, src));
                }
            }
        }
        __syncwarp();
    }
}

// ---------------------------------------------------------------------------------------------
// Per-vertex sums over the neighbourhood.
// ---------------------------------------------------------------------------------------------
// t of the arc at position p of v's row (its k-th, to h): an out-arc of v, or the out-arc of h at which v stands
// (rev[p] is v's position in h's row).
__device__ __forceinline__ uint64_t arc_t(const OrbGraph& G, const int32_t* __restrict__ rev, int64_t v, int64_t p,
                                          int64_t k, int64_t dm, int32_t h) {
    if (k >= dm) return (uint64_t)G.te[G.offp[v] + (k - dm)];
    const int64_t ph = G.offp[h];
    return (uint64_t)G.te[ph + rev[p] - ((int64_t)G.deg[h] - (G.offp[h + 1] - ph))];
}

struct VertexSums {
    uint64_t ts = 0, sa = 0, n1 = 0, n6 = 0, n8 = 0;
    __device__ __forceinline__ void add(const OrbGraph& G, const int32_t* __restrict__ rev, int64_t v, int64_t vb, int64_t k,
                                        int64_t dm) {
        const int32_t h = __ldg(G.cols + vb + k);
        const uint64_t dh = (uint64_t)G.deg[h];
        const uint64_t t = arc_t(G, rev, v, vb + k, k, dm, h);
        ts += t;
        sa += dh - 1;
        n1 += choose2_u64(dh - 1);
        n6 += t * (dh - 2);  // dh >= 2 whenever t > 0
        n8 += choose2_u64(t);
    }
    __device__ __forceinline__ void reduce(int width) {  // over aligned groups of width lanes
        for (int o = width / 2; o > 0; o >>= 1) {
            ts += __shfl_xor_sync(kFull, ts, o);
            sa += __shfl_xor_sync(kFull, sa, o);
            n1 += __shfl_xor_sync(kFull, n1, o);
            n6 += __shfl_xor_sync(kFull, n6, o);
            n8 += __shfl_xor_sync(kFull, n8, o);
        }
    }
};

// Rows of at most kRowLane neighbours by 8 lanes (4 rows to a warp), up to kRowWarp by a warp; longer ones by
// k_orb_vertex_hub (a warp per hub row took 350 us on R-MAT scale 15: the largest row has 5,962 entries).
constexpr int kRowLane = 64, kRowWarp = 256;

__global__ void __launch_bounds__(kOrbThreads) k_orb_vertex(OrbGraph G, const int32_t* __restrict__ rev, int64_t n,
                                                            uint64_t* __restrict__ tsum, uint64_t* __restrict__ s1,
                                                            uint64_t* __restrict__ N) {
    grid_begin();
    const int l = lane_id();
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    auto store = [&](int64_t v, const VertexSums& x) {
        tsum[v] = x.ts;
        s1[v] = x.sa;
        N[v * kOrbits + 1] = x.n1;
        N[v * kOrbits + 6] = x.n6;
        N[v * kOrbits + 8] = x.n8;
    };
    for (int64_t v0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 4; v0 < n; v0 += nw * 4) {
        const int64_t v = v0 + (l >> 3);
        const int64_t d = v < n ? G.deg[v] : 0;
        VertexSums x;
        if (d <= kRowLane && d > 0) {
            const int64_t vb = G.off[v], dm = d - (G.offp[v + 1] - G.offp[v]);
            for (int64_t k = l & 7; k < d; k += 8) x.add(G, rev, v, vb, k, dm);
        }
        x.reduce(8);
        if ((l & 7) == 0 && v < n && d <= kRowLane) store(v, x);
        uint32_t big = __ballot_sync(kFull, (l & 7) == 0 && d > kRowLane && d <= kRowWarp);
        while (big) {
            const int src = __ffs(big) - 1;
            big &= big - 1;
            const int64_t r = v0 + (src >> 3);
            const int64_t rd = __shfl_sync(kFull, d, src);
            const int64_t rb = G.off[r], dm = rd - (G.offp[r + 1] - G.offp[r]);
            VertexSums y;
            for (int64_t k = l; k < rd; k += 32) y.add(G, rev, r, rb, k, dm);
            y.reduce(32);
            if (l == 0) store(r, y);
        }
    }
}

// Rows of more than kRowWarp neighbours: the last ranks, whose arcs are one contiguous range; a warp per 256 arcs
// (at most two rows), added to the zeroed sums.
__global__ void __launch_bounds__(kOrbThreads) k_orb_vertex_hub(OrbGraph G, const int32_t* __restrict__ rev, int64_t n,
                                                                unsigned long long* __restrict__ tsum,
                                                                unsigned long long* __restrict__ s1,
                                                                unsigned long long* __restrict__ N) {
    grid_begin();
    const int l = lane_id();
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    int64_t lo = 0, hi = n;  // first rank of degree above kRowWarp
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (G.deg[mid] <= kRowWarp) lo = mid + 1;
        else hi = mid;
    }
    const int64_t vh = lo;
    if (vh >= n) return;
    const int64_t end = G.off[n];
    for (int64_t a0 = G.off[vh] + (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 256; a0 < end; a0 += nw * 256) {
        const int64_t a1 = a0 + 256 < end ? a0 + 256 : end;
        int64_t v = vh, h = n;  // row of a0
        while (h - v > 1) {
            const int64_t mid = (v + h) >> 1;
            if (G.off[mid] <= a0) v = mid;
            else h = mid;
        }
        for (int64_t b = a0; b < a1; ++v) {
            const int64_t vb = G.off[v], ve = G.off[v + 1];
            const int64_t e = ve < a1 ? ve : a1;
            const int64_t dm = (ve - vb) - (G.offp[v + 1] - G.offp[v]);
            VertexSums x;
            for (int64_t k = b - vb + l; k < e - vb; k += 32) x.add(G, rev, v, vb, k, dm);
            x.reduce(32);
            if (l == 0) {
                atomicAdd(&tsum[v], (unsigned long long)x.ts);
                atomicAdd(&s1[v], (unsigned long long)x.sa);
                atomicAdd(&N[v * kOrbits + 1], (unsigned long long)x.n1);
                atomicAdd(&N[v * kOrbits + 6], (unsigned long long)x.n6);
                atomicAdd(&N[v * kOrbits + 8], (unsigned long long)x.n8);
            }
            b = e;
        }
    }
}

// ---------------------------------------------------------------------------------------------
// 4-cycles through each vertex (N7), by the wedge anchor with per-role routing.
// ---------------------------------------------------------------------------------------------
// Wedge work of root u: sum over w in N-(u) of |{x in N(w) : x < u}| = rev of the arc (u, w).  Light roots are
// queued (with W) for the warp kernel from the front of q_light, middle ones from its back; heavy roots in
// q_heavy, the heaviest (W > kHugeWork) from the front, the others from the back, so that the block kernels
// take the heaviest first.  A lane sums a short list itself.
constexpr uint64_t kHugeWork = 16384;
enum : int { QO_LIGHT = 0, QO_MID, QO_HUGE, QO_HEAVY, QO_TICKET };

__global__ void k_orb_classify(OrbGraph G, const int32_t* __restrict__ rev, int64_t n, int32_t* __restrict__ q_light,
                               int32_t* __restrict__ w_light, int32_t* __restrict__ q_heavy,
                               unsigned long long* __restrict__ qcnt) {
    grid_begin();
    const int l = lane_id();
    const int64_t wid = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t k0 = wid; k0 < n; k0 += nw * 32) {  // ranks spaced by the warps: the hubs fall to different warps
        const int64_t u = n - 1 - (k0 + (int64_t)l * nw);
        int64_t dm = 0, ub = 0;
        if (u >= 0) {
            ub = G.off[u];
            dm = (int64_t)G.deg[u] - (G.offp[u + 1] - G.offp[u]);  // |N-(u)|
        }
        uint64_t W = 0;
        if (dm >= 2 && dm <= 32)
            for (int64_t k = 0; k < dm; ++k) W += (uint64_t)rev[ub + k];
        uint32_t big = __ballot_sync(kFull, dm > 32);
        while (big) {
            const int src = __ffs(big) - 1;
            big &= big - 1;
            const int64_t bd = __shfl_sync(kFull, dm, src), bb = __shfl_sync(kFull, ub, src);
            uint64_t x = 0;
            for (int64_t k = l; k < bd; k += 32) x += (uint64_t)rev[bb + k];
            x = warp_sum(x);
            if (l == src) W = x;
        }
        const int cls = W == 0 ? -1 : (W <= (uint64_t)kHashMax ? QO_LIGHT : (W <= (uint64_t)kMidMax ? QO_MID
                                                                           : (W > kHugeWork ? QO_HUGE : QO_HEAVY)));
#pragma unroll
        for (int c = QO_LIGHT; c <= QO_HEAVY; ++c) {  // one atomic per class and warp
            const uint32_t mask = __ballot_sync(kFull, cls == c);
            if (!mask) continue;
            unsigned long long start = 0;
            const int leader = __ffs(mask) - 1;
            if (l == leader) start = atomicAdd(&qcnt[c], (unsigned long long)__popc(mask));
            start = __shfl_sync(kFull, start, leader);
            if (cls != c) continue;
            const int64_t k = (int64_t)start + __popc(mask & lanemask_lt());
            if (c == QO_LIGHT || c == QO_MID) {
                q_light[c == QO_LIGHT ? k : n - 1 - k] = (int32_t)u;
                w_light[c == QO_LIGHT ? k : n - 1 - k] = (int32_t)W;
            } else {
                q_heavy[c == QO_HUGE ? k : n - 1 - k] = (int32_t)u;
            }
        }
    }
}

// root `item` of the heavy queue, the heaviest first
__device__ __forceinline__ int32_t heavy_root(const int32_t* __restrict__ q, const unsigned long long* __restrict__ qcnt,
                                              int64_t n, int64_t item) {
    const int64_t huge = (int64_t)qcnt[QO_HUGE];
    return item < huge ? q[item] : q[n - 1 - (item - huge)];
}

// Flattens 32 segments (lane l owns positions base_l .. base_l + len_l - 1 of cols): f(position, element, owner).
template <typename F>
__device__ __forceinline__ void flat_segments(const int32_t* __restrict__ cols, int64_t base, int len, F&& f) {
    const int l = lane_id();
    int incl = len;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kFull, incl, o);
        if (l >= o) incl += y;
    }
    const int excl = incl - len;
    const int total = __shfl_sync(kFull, incl, 31);
    for (int t0 = 0; t0 < total; t0 += 128) {  // four loads in flight
        int64_t p[4];
        int32_t x[4];
        int own[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int t = t0 + 32 * r + l;
            int o = 0;
            if (t0 + 32 * r < total) {  // uniform
#pragma unroll
                for (int s = 16; s >= 1; s >>= 1) {
                    const int e = __shfl_sync(kFull, excl, o + s);
                    if (e <= t) o += s;
                }
                p[r] = __shfl_sync(kFull, base, o) + (t - __shfl_sync(kFull, excl, o));
            }
            own[r] = t < total ? o : -1;
            x[r] = t < total ? __ldg(cols + p[r]) : 0;
        }
#pragma unroll
        for (int r = 0; r < 4; ++r)
            if (own[r] >= 0) f(p[r], x[r], own[r]);
    }
}

__device__ __forceinline__ uint32_t* hash_slot(int32_t* keys, uint32_t* cnt, uint32_t mask, int32_t x, bool insert) {
    uint32_t h = hash32((uint32_t)x) & mask;
    for (;;) {
        int32_t k = keys[h];
        if (k == kNoKey) {
            if (!insert) return nullptr;
            const int32_t prev = atomicCAS(&keys[h], kNoKey, x);
            if (prev == kNoKey || prev == x) return &cnt[h];
            k = prev;
        }
        if (k == x) return &cnt[h];
        h = (h + 1) & mask;
    }
}

// Light roots: a warp each; middle roots (MID): a block each (a warp took 265 us for the 1,280 middle roots of a
// Barabasi-Albert graph with 100,001 vertices).  A hash of the power of two >= 2 W slots.  Pass 1 counts cnt(x) over the wedges
// u - w - x, x < u; pass 2 gives each middle w the sum of cnt(x) - 1 over its segment (and, per edge, each arc
// its part); then every x with cnt >= 2 gets cnt (cnt - 1) in its doubled count and the root half the total.
template <int SLOTS, int WARPS, bool MID>
__global__ void __launch_bounds__(WARPS * 32) k_orb_c4w(OrbGraph G, const int32_t* __restrict__ rev, int64_t n,
                                                        const int32_t* __restrict__ q, const int32_t* __restrict__ qw,
                                                        const unsigned long long* __restrict__ qcnt,
                                                        unsigned long long* __restrict__ n7,
                                                        unsigned long long* __restrict__ n7x2,
                                                        unsigned long long* __restrict__ e6a) {
    grid_begin();
    constexpr int TEAMS = MID ? 1 : WARPS, TW = MID ? WARPS : 1;  // roots per block, warps per root
    extern __shared__ __align__(16) uint32_t smem[];
    __shared__ uint32_t s_sw[WARPS][32];
    const int w = threadIdx.x >> 5, l = lane_id();
    const int team = MID ? 0 : w, tw = MID ? w : 0, tl = MID ? (int)threadIdx.x : l;
    int32_t* keys = reinterpret_cast<int32_t*>(smem) + team * SLOTS;
    uint32_t* cnt = smem + (TEAMS + team) * SLOTS;
    auto sync = [] {
        if (MID) __syncthreads();
        else __syncwarp();
    };
    const int64_t nq = (int64_t)qcnt[MID ? QO_MID : QO_LIGHT];
    s_sw[w][l] = 0;
    for (int64_t i = (int64_t)blockIdx.x * TEAMS + team; i < nq; i += (int64_t)gridDim.x * TEAMS) {
        const int64_t slot = MID ? n - 1 - i : i;
        const int32_t u = q[slot];
        const uint32_t W = (uint32_t)qw[slot];
        uint32_t P = 32;
        while (P < 2 * W) P <<= 1;
        for (uint32_t k = tl; k < P; k += 32 * TW) {
            keys[k] = kNoKey;
            cnt[k] = 0;
        }
        sync();
        const int64_t ub = G.off[u];
        const int64_t dm = (int64_t)G.deg[u] - (G.offp[u + 1] - G.offp[u]);
        for (int64_t k0 = tw * 32; k0 < dm; k0 += 32 * TW) {
            const bool in = k0 + l < dm;
            const int64_t base = in ? G.off[__ldg(G.cols + ub + k0 + l)] : 0;
            flat_segments(G.cols, base, in ? rev[ub + k0 + l] : 0, [&](int64_t, int32_t x, int) {
                atomicAdd(hash_slot(keys, cnt, P - 1, x, true), 1u);
            });
        }
        sync();
        for (int64_t k0 = tw * 32; k0 < dm; k0 += 32 * TW) {
            const bool in = k0 + l < dm;
            const int32_t wv = in ? __ldg(G.cols + ub + k0 + l) : 0;
            flat_segments(G.cols, in ? G.off[wv] : 0, in ? rev[ub + k0 + l] : 0, [&](int64_t p, int32_t x, int o) {
                const uint32_t c = *hash_slot(keys, cnt, P - 1, x, false) - 1u;
                if (c) {
                    atomicAdd(&s_sw[w][o], c);
                    if (e6a) atomicAdd(&e6a[p], (unsigned long long)c);  // the arc (w, x)
                }
            });
            __syncwarp();
            const uint32_t sw = s_sw[w][l];
            s_sw[w][l] = 0;
            if (sw && n7) atomicAdd(&n7[wv], (unsigned long long)sw);
            if (sw && e6a) atomicAdd(&e6a[ub + k0 + l], (unsigned long long)sw);  // the arc (u, w)
            __syncwarp();
        }
        if (n7) {
            uint64_t root2 = 0;
            for (uint32_t k = tl; k < P; k += 32 * TW) {
                const uint64_t c = cnt[k];
                if (c < 2) continue;
                root2 += c * (c - 1);
                atomicAdd(&n7x2[keys[k]], (unsigned long long)(c * (c - 1)));
            }
            root2 = warp_sum(root2);  // even: cnt (cnt - 1) is
            if (l == 0 && root2) atomicAdd(&n7[u], (unsigned long long)(root2 >> 1));
        }
        sync();
    }
}

// Heavy roots of graphs up to kWinMax windows of ranks: a block per root, counters of a window of x in shared
// memory (16-bit while every degree is below 65,536: cnt(x) <= d(x); else 32-bit), the window's segments walked
// twice (count, route), then the counters scanned and cleared.  (Counters of every rank in global memory, three
// walks: 5.2 ms on R-MAT scale 15, 1.7 ms on Barabasi-Albert with 100,001 vertices.)
constexpr int kWinThreads = 512;
constexpr int kWinWarps = kWinThreads / 32;
constexpr int kWinWords = 24576;  // 96 KiB: two blocks to an SM
constexpr int kWinMax = 8;

template <int BITS>
__global__ void __launch_bounds__(kWinThreads, 2) k_orb_c4win(OrbGraph G, const int32_t* __restrict__ rev,
                                                              int64_t n, const int32_t* __restrict__ q,
                                                              unsigned long long* __restrict__ qcnt,
                                                              unsigned long long* __restrict__ n7,
                                                              unsigned long long* __restrict__ n7x2,
                                                              unsigned long long* __restrict__ e6a) {
    grid_begin();
    constexpr int PER = 32 / BITS;
    constexpr int64_t X = (int64_t)kWinWords * PER;
    extern __shared__ uint32_t ctr[];
    __shared__ uint64_t red[32];
    __shared__ uint32_t s_sw[kWinWarps][32];
    __shared__ int64_t s_item;
    const int w = threadIdx.x >> 5, l = lane_id();
    for (int i = threadIdx.x; i < kWinWords; i += kWinThreads) ctr[i] = 0;
    s_sw[w][l] = 0;
    const int64_t nq = (int64_t)(qcnt[QO_HUGE] + qcnt[QO_HEAVY]);
    auto shift = [](uint32_t r) { return PER == 2 ? (r & 1u) * 16u : 0u; };
    for (;;) {
        if (threadIdx.x == 0) s_item = (int64_t)atomicAdd(&qcnt[QO_TICKET], 1ull);
        __syncthreads();
        const int64_t item = s_item;
        if (item >= nq) break;
        const int32_t u = heavy_root(q, qcnt, n, item);
        const int64_t ub = G.off[u];
        const int64_t dm = (int64_t)G.deg[u] - (G.offp[u + 1] - G.offp[u]);
        uint64_t root2 = 0;
        for (int64_t xlo = 0; xlo < u; xlo += X) {
            const int64_t xhi = xlo + X < u ? xlo + X : u;
            for (int pass = 0; pass < 2; ++pass) {
                for (int64_t k0 = w * 32; k0 < dm; k0 += kWinThreads) {
                    const bool in = k0 + l < dm;
                    int32_t wv = 0;
                    int64_t base = 0;
                    int len = 0;
                    if (in) {
                        wv = __ldg(G.cols + ub + k0 + l);
                        base = G.off[wv];
                        len = rev[ub + k0 + l];
                        if (xhi < u) len = (int)lower_bound_i32(G.cols + base, len, (int32_t)xhi);
                        if (xlo > 0) {
                            const int p = (int)lower_bound_i32(G.cols + base, len, (int32_t)xlo);
                            base += p;
                            len -= p;
                        }
                    }
                    uint32_t longs = __ballot_sync(kFull, len >= 32);
                    const int slen = len >= 32 ? 0 : len;
                    if (pass == 0) {
                        auto add = [&](int32_t x) {
                            const uint32_t r = (uint32_t)(x - xlo);
                            atomicAdd(&ctr[r / PER], 1u << shift(r));
                        };
                        while (longs) {
                            const int src = __ffs(longs) - 1;
                            longs &= longs - 1;
                            const int64_t b = __shfl_sync(kFull, base, src);
                            const int c = __shfl_sync(kFull, len, src);
                            for (int k = l; k < c; k += 128) {  // four loads in flight
                                int32_t x[4];
#pragma unroll
                                for (int t = 0; t < 4; ++t) x[t] = k + 32 * t < c ? __ldg(G.cols + b + k + 32 * t) : -1;
#pragma unroll
                                for (int t = 0; t < 4; ++t)
                                    if (x[t] >= 0) add(x[t]);
                            }
                        }
                        flat_segments(G.cols, base, slen, [&](int64_t, int32_t x, int) { add(x); });
                    } else {
                        auto others = [&](int32_t x) {  // cnt(x) - 1
                            const uint32_t r = (uint32_t)(x - xlo);
                            return (BITS == 32 ? ctr[r] : (ctr[r / PER] >> shift(r)) & 0xffffu) - 1u;
                        };
                        uint64_t sw = 0;
                        while (longs) {
                            const int src = __ffs(longs) - 1;
                            longs &= longs - 1;
                            const int64_t b = __shfl_sync(kFull, base, src);
                            const int c = __shfl_sync(kFull, len, src);
                            uint64_t sum = 0;
                            for (int k = l; k < c; k += 128) {
                                int32_t x[4];
#pragma unroll
                                for (int t = 0; t < 4; ++t) x[t] = k + 32 * t < c ? __ldg(G.cols + b + k + 32 * t) : -1;
#pragma unroll
                                for (int t = 0; t < 4; ++t) {
                                    if (x[t] < 0) continue;
                                    const uint32_t o = others(x[t]);
                                    sum += o;
                                    if (o && e6a) atomicAdd(&e6a[b + k + 32 * t], (unsigned long long)o);  // the arc (w, x)
                                }
                            }
                            sum = warp_sum(sum);
                            if (l == src) sw = sum;
                        }
                        flat_segments(G.cols, base, slen, [&](int64_t p, int32_t x, int o) {
                            const uint32_t c = others(x);
                            if (!c) return;
                            if (BITS == 16) atomicAdd(&s_sw[w][o], c);  // at most 31 * 65535
                            else if (n7) atomicAdd(&n7[__ldg(G.cols + ub + k0 + o)], (unsigned long long)c);
                            else atomicAdd(&e6a[ub + k0 + o], (unsigned long long)c);
                            if (e6a) atomicAdd(&e6a[p], (unsigned long long)c);
                        });
                        __syncwarp();
                        sw += s_sw[w][l];
                        s_sw[w][l] = 0;
                        if (sw && n7) atomicAdd(&n7[wv], (unsigned long long)sw);
                        if (sw && e6a) atomicAdd(&e6a[ub + k0 + l], (unsigned long long)sw);  // the arc (u, w)
                        __syncwarp();
                    }
                }
                __syncthreads();  // every counter is final before it is read, every read done before the scan
            }
            const int words = (int)((xhi - xlo + PER - 1) / PER);
            for (int i = threadIdx.x; i < words; i += kWinThreads) {
                const uint32_t v = ctr[i];
                if (!v) continue;
                ctr[i] = 0;
                if (!n7) continue;
#pragma unroll
                for (int h = 0; h < PER; ++h) {
                    const uint64_t c = BITS == 32 ? v : (v >> (16 * h)) & 0xffffu;
                    if (c < 2) continue;
                    root2 += c * (c - 1);
                    atomicAdd(&n7x2[xlo + (int64_t)i * PER + h], (unsigned long long)(c * (c - 1)));
                }
            }
            __syncthreads();
        }
        if (n7) {
            root2 = block_sum_u64(root2, red);
            if (threadIdx.x == 0 && root2) atomicAdd(&n7[u], (unsigned long long)(root2 >> 1));
        }
    }
}

// Heavy roots of larger graphs: one block each (persistent blocks over the queue), dense counters over every
// rank in the block's slice of a global array (cleared again by a third walk).
__global__ void __launch_bounds__(kOrbThreads) k_orb_c4b(OrbGraph G, int64_t n, const int32_t* __restrict__ q,
                                                         const unsigned long long* __restrict__ qcnt,
                                                         uint32_t* __restrict__ dense,
                                                         unsigned long long* __restrict__ n7,
                                                         unsigned long long* __restrict__ n7x2,
                                                         unsigned long long* __restrict__ e6a) {
    grid_begin();
    __shared__ uint64_t red[32];
    uint32_t* cntv = dense + (size_t)blockIdx.x * (size_t)n;
    const int64_t nq = (int64_t)(qcnt[QO_HUGE] + qcnt[QO_HEAVY]);
    const int w = threadIdx.x >> 5, l = lane_id();
    for (int64_t i = blockIdx.x; i < nq; i += gridDim.x) {
        const int32_t u = heavy_root(q, qcnt, n, i);
        const int64_t ub = G.off[u];
        const int64_t dm = (int64_t)G.deg[u] - (G.offp[u + 1] - G.offp[u]);
        // warp per lower neighbour, lanes along its segment
        for (int pass = 0; pass < 3; ++pass) {
            uint64_t root2 = 0;
            for (int64_t k = w; k < dm; k += kOrbWarps) {
                const int32_t wv = __ldg(G.cols + ub + k);
                const int64_t wb = G.off[wv];
                const int64_t we = wb + lower_bound_i32(G.cols + wb, G.off[wv + 1] - wb, u);
                uint64_t sw = 0;
                for (int64_t p = wb + l; p < we; p += 32) {
                    const int32_t x = __ldg(G.cols + p);
                    if (pass == 0) {
                        atomicAdd(&cntv[x], 1u);
                    } else if (pass == 1) {
                        const uint32_t c = cntv[x] - 1u;
                        sw += c;
                        if (c && n7x2) atomicAdd(&n7x2[x], (unsigned long long)c);
                        if (c && e6a) atomicAdd(&e6a[p], (unsigned long long)c);  // the arc (w, x)
                    } else {
                        cntv[x] = 0;
                    }
                }
                if (pass == 1) {
                    sw = warp_sum(sw);
                    if (l == 0 && sw && n7) atomicAdd(&n7[wv], (unsigned long long)sw);
                    if (l == 0 && sw && e6a) atomicAdd(&e6a[ub + k], (unsigned long long)sw);  // the arc (u, w)
                    root2 += sw;
                }
            }
            __syncthreads();  // every counter of the pass is final before the next reads it
            if (pass == 1) {
                root2 = block_sum_u64(l == 0 ? root2 : 0, red);
                if (threadIdx.x == 0 && root2 && n7) atomicAdd(&n7[u], (unsigned long long)(root2 >> 1));
            }
        }
    }
}

// ---------------------------------------------------------------------------------------------
// The remaining statistics and the back-substitution.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kOrbThreads) k_orb_close(OrbGraph G, int64_t n, const uint64_t* __restrict__ tsum,
                                                           const uint64_t* __restrict__ s1,
                                                           const unsigned long long* __restrict__ n9,
                                                           const unsigned long long* __restrict__ tau6,
                                                           const unsigned long long* __restrict__ n7,
                                                           const unsigned long long* __restrict__ n7x2,
                                                           const int32_t* __restrict__ order,
                                                           uint64_t* __restrict__ N, uint64_t* __restrict__ out,
                                                           uint64_t* __restrict__ acc) {
    grid_begin();
    const int l = lane_id();
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t v = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < n; v += nw) {
        const int64_t vb = G.off[v], ve = G.off[v + 1];
        uint64_t sa = 0, st = 0;  // sum of S1 and of t_h over the neighbours
        for (int64_t k = vb + l; k < ve; k += 32) {
            const int32_t h = __ldg(G.cols + k);
            sa += s1[h];
            st += tsum[h];
        }
        sa = warp_sum(sa);
        st = warp_sum(st);
        if (l != 0) continue;
        const uint64_t d = (uint64_t)(ve - vb);
        const uint64_t ts = tsum[v];       // 2 t_v
        const uint64_t tv = ts >> 1;
        uint64_t* Nv = N + v * kOrbits;
        uint64_t S[kOrbits];
        S[0] = choose3_u64(d);
        S[1] = Nv[1];
        S[2] = sa - d * (d - 1) - ts;      // sum_a S1(a) - d (d - 1) - 2 t_v
        S[3] = (d - 1) * s1[v] - ts;       // d >= 1 whenever v has a neighbour
        S[4] = (st >> 1) - ts;             // sum_h t_h - 2 t_v (every tsum is even)
        S[5] = tv * (d >= 2 ? d - 2 : 0);
        S[6] = Nv[6];
        S[7] = n7[v] + (n7x2[v] >> 1);
        S[8] = Nv[8];
        S[9] = n9[v];
        S[10] = tau6[v] / 6;
        if ((ts & 1) || (tau6[v] % 6) || (n7x2[v] & 1))
            atomicOr((unsigned long long*)&acc[ACC_ERR], (unsigned long long)kErrLitDiv);
        uint64_t o[kOrbits];
#pragma unroll
        for (int i = kOrbits - 1; i >= 0; --i) {
            uint64_t x = S[i];
#pragma unroll
            for (int j = i + 1; j < kOrbits; ++j) x -= (uint64_t)c_contain[i][j] * o[j];
            o[i] = x;
        }
        uint64_t* dst = out + (int64_t)order[v] * kOrbits;
#pragma unroll
        for (int i = 0; i < kOrbits; ++i) dst[i] = o[i];
    }
}

// ---------------------------------------------------------------------------------------------
// Per-edge statistics and back-substitution.
// ---------------------------------------------------------------------------------------------
constexpr int kEdgeOrbits = 10;
__constant__ uint8_t c_econtain[kEdgeOrbits][kEdgeOrbits] = {
    {1, 0, 0, 1, 1, 0, 0, 2, 1, 2}, {0, 1, 0, 2, 0, 2, 2, 0, 3, 4}, {0, 0, 1, 0, 1, 0, 1, 2, 1, 2},
    {0, 0, 0, 1, 0, 0, 0, 0, 1, 2}, {0, 0, 0, 0, 1, 0, 0, 4, 1, 4}, {0, 0, 0, 0, 0, 1, 0, 0, 1, 2},
    {0, 0, 0, 0, 0, 0, 1, 0, 1, 2}, {0, 0, 0, 0, 0, 0, 0, 1, 0, 1}, {0, 0, 0, 0, 0, 0, 0, 0, 1, 4},
    {0, 0, 0, 0, 0, 0, 0, 0, 0, 1}};

// up[x] = neighbours of input vertex x above x (its row's suffix in the input CSR)
__global__ void k_eorb_up(const int64_t* __restrict__ off_in, const int32_t* __restrict__ cols_in, int64_t n,
                          int32_t* __restrict__ up) {
    grid_begin();
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n; x += (int64_t)gridDim.x * blockDim.x) {
        const int64_t b = off_in[x], e = off_in[x + 1];
        up[x] = (int32_t)(e - b - lower_bound_i32(cols_in + b, e - b, (int32_t)x + 1));
    }
}

// One thread per out-arc (u, v) of the rank-order graph: the ten statistics, the back-substitution,
// and the write at the edge's index in the input edge list.
__global__ void k_eorb_close(OrbGraph G, int64_t n, int64_t m, const int32_t* __restrict__ dplus,
                             const uint64_t* __restrict__ tsum, const uint64_t* __restrict__ s1,
                             const unsigned long long* __restrict__ e5, const unsigned long long* __restrict__ e8,
                             const unsigned long long* __restrict__ e9, const unsigned long long* __restrict__ e6a,
                             const int32_t* __restrict__ order, const int64_t* __restrict__ off_in,
                             const int32_t* __restrict__ cols_in, const int32_t* __restrict__ up,
                             const int64_t* __restrict__ ebase, uint64_t* __restrict__ out,
                             uint64_t* __restrict__ acc) {
    grid_begin();
    for (int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; a < m; a += (int64_t)gridDim.x * blockDim.x) {
        const int32_t u = arc_row(G.offp, n, a);
        const int32_t v = G.colsp[a];
        const uint64_t du = (uint64_t)G.deg[u], dv = (uint64_t)G.deg[v];
        const uint64_t t = (uint64_t)G.te[a];
        const uint64_t tu = tsum[u] >> 1, tv = tsum[v] >> 1;
        // the two arcs of the edge in the rank-order CSR: (u, v) in u's suffix, (v, u) in v's prefix
        const int64_t p_uv = G.off[u] + ((int64_t)G.deg[u] - dplus[u]) + (a - G.offp[u]);
        const int64_t vb = G.off[v];
        const int64_t p_vu = vb + lower_bound_i32(G.cols + vb, (int64_t)G.deg[v] - dplus[v], u);
        uint64_t E[kEdgeOrbits];
        E[0] = choose2_u64(du - 1) + choose2_u64(dv - 1);
        E[1] = s1[u] + s1[v] - du - dv + 2 - 2 * t;
        E[2] = (du - 1) * (dv - 1) - t;
        E[3] = tu + tv - 2 * t;
        E[4] = t * (du + dv - 4);
        E[5] = e5[a];
        E[6] = e6a[p_uv] + e6a[p_vu];
        E[7] = choose2_u64(t);
        E[8] = e8[a];
        E[9] = e9[a] >> 1;
        if (e9[a] & 1) atomicOr((unsigned long long*)&acc[ACC_ERR], (unsigned long long)kErrLitDiv);
        uint64_t o[kEdgeOrbits];
#pragma unroll
        for (int i = kEdgeOrbits - 1; i >= 0; --i) {
            uint64_t x = E[i];
#pragma unroll
            for (int j = i + 1; j < kEdgeOrbits; ++j) x -= (uint64_t)c_econtain[i][j] * o[j];
            o[i] = x;
        }
        // index of the edge in the input edge list: (lo, hi) by input id, rows' upper suffixes in order
        const int32_t ia = order[u], ib = order[v];
        const int32_t lo = ia < ib ? ia : ib, hi = ia < ib ? ib : ia;
        const int64_t rb = off_in[lo], re = off_in[lo + 1];
        const int64_t pos = lower_bound_i32(cols_in + rb, re - rb, hi);  // within lo's row
        const int64_t idx = ebase[lo] + (pos - ((re - rb) - up[lo]));
        uint64_t* dst = out + idx * kEdgeOrbits;
#pragma unroll
        for (int i = 0; i < kEdgeOrbits; ++i) dst[i] = o[i];
    }
}

unsigned orb_grid(int64_t warps) {
    int64_t b = (warps * 32 + kOrbThreads - 1) / kOrbThreads;
    if (b < 1) b = 1;
    const int64_t cap = (int64_t)num_sms() * 8;
    return (unsigned)(b > cap ? cap : b);
}

}  // namespace

namespace {

// The passes both outputs share, on scratch that starts at zero: triangles, vertex sums and the wedge walk.
struct OrbScratch {
    uint64_t *tsum, *s1, *N;
    unsigned long long *n9, *tau6, *n7, *n7x2;  // per vertex (nullptr per edge)
    unsigned long long *e5, *e8, *e9, *e6a;     // per edge (nullptr per vertex)
    int32_t *q_light, *w_light, *q_heavy;
    unsigned long long* qcnt;                   // QO_*: lengths of the queues, the window kernel's ticket
    uint32_t* dense;                            // global counters of heavy roots (nullptr: windows)
    int heavy_blocks;
};

// Whether the heavy roots' counters go through shared-memory windows.
bool orbit_windows(const harp_csr* g) {
    const int64_t per = g->max_deg < 65536 ? 2 : 1;
    return g->n <= (int64_t)kWinWords * per * kWinMax;
}

// Blocks of the heavy roots' global counters (n uint32 each): at most 4 GiB in all; 0 with windows.
int orbit_heavy_blocks(const harp_csr* g) {
    if (orbit_windows(g)) return 0;
    int64_t hb = ((int64_t)4 << 30) / (4 * g->n);
    if (hb > num_sms()) hb = num_sms();
    return hb < 1 ? 1 : (int)hb;
}

harp_status orbit_passes(const harp_csr* g, Workspace& ws, const OrbScratch& o, cudaStream_t s) {
    const int64_t n = g->n, m = g->m;
    const OrbGraph G{ws.off, ws.cols, ws.deg, ws.offp, ws.colsp, ws.te};
    if (m == 0) return HARP_OK;  // every sum is zero
    HARP_TRY(orbit_triangles(g, ws, OrbTri{o.n9, o.tau6, o.e5, o.e8, o.e9}, s));
    if (max_out_degree(g) > 1024) {
        const EdgeRoute er{o.e5, o.e8, o.e9};
        launch(k_orb_tri_big, num_sms() * 4, kOrbThreads, 0, s, G, ws.q_mid + n, ws.acc + Q_TRI_BIG, o.n9, o.tau6, er);
        HARP_LAUNCHED();
        launch(k_orb_tri_big, num_sms() * 4, kOrbThreads, 0, s, G, ws.q_mid, ws.acc + Q_TRI_FB, o.n9, o.tau6, er);
        HARP_LAUNCHED();
    }
    HARP_TRY(wedge_positions(g, ws, s));
    launch(k_orb_vertex, orb_grid((n + 3) / 4), kOrbThreads, 0, s, G, ws.rev, n, o.tsum, o.s1, o.N);
    HARP_LAUNCHED();
    if (g->max_deg > kRowWarp) {
        launch(k_orb_vertex_hub, num_sms() * 4, kOrbThreads, 0, s, G, ws.rev, n, (unsigned long long*)o.tsum,
               (unsigned long long*)o.s1, (unsigned long long*)o.N);
        HARP_LAUNCHED();
    }
    launch(k_orb_classify, orb_grid((n + 31) / 32), kOrbThreads, 0, s, G, ws.rev, n, o.q_light, o.w_light, o.q_heavy,
           o.qcnt);
    HARP_LAUNCHED();
    const size_t light_smem = (size_t)kOrbWarps * kHashSlots * 8, mid_smem = (size_t)kMidSlots * 8;
    auto light = k_orb_c4w<kHashSlots, kOrbWarps, false>;
    auto mid = k_orb_c4w<kMidSlots, kMidWarps, true>;
    HARP_CK(cudaFuncSetAttribute(light, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)light_smem));
    HARP_CK(cudaFuncSetAttribute(mid, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)mid_smem));
    launch(light, orb_grid(n), kOrbThreads, light_smem, s, G, ws.rev, n, o.q_light, o.w_light, o.qcnt, o.n7, o.n7x2,
           o.e6a);
    HARP_LAUNCHED();
    launch(mid, num_sms() * 6, kMidWarps * 32, mid_smem, s, G, ws.rev, n, o.q_light, o.w_light, o.qcnt, o.n7, o.n7x2,
           o.e6a);
    HARP_LAUNCHED();
    if (o.dense) {
        launch(k_orb_c4b, o.heavy_blocks, kOrbThreads, 0, s, G, n, o.q_heavy, o.qcnt, o.dense, o.n7, o.n7x2, o.e6a);
    } else {
        const size_t smem = (size_t)kWinWords * sizeof(uint32_t);
        auto kernel = g->max_deg < 65536 ? k_orb_c4win<16> : k_orb_c4win<32>;
        HARP_CK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        launch(kernel, num_sms() * 2, kWinThreads, smem, s, G, ws.rev, n, o.q_heavy, o.qcnt, o.n7, o.n7x2, o.e6a);
    }
    HARP_LAUNCHED();
    return HARP_OK;
}

}  // namespace

harp_status count_orbits(const harp_csr* g, Workspace& ws, uint64_t* d_out, cudaStream_t s) {
    const int64_t n = g->n;
    if (n == 0) return HARP_OK;
    // per-vertex scratch: tsum, s1, n9, tau6, n7, n7x2 (uint64), N (11 uint64), the queue counters, three int32
    // queue arrays (rounded to 8 bytes) and the heavy roots' global counters, if any
    OrbScratch o{};
    o.heavy_blocks = orbit_heavy_blocks(g);
    const size_t dense_bytes = (size_t)o.heavy_blocks * (size_t)n * 4;
    const size_t words = (size_t)n * (6 + kOrbits) + 8;
    const size_t bytes = 8 * words + 4 * (size_t)(3 * n + (n & 1)) + dense_bytes;
    unsigned char* base = nullptr;
    HARP_CK(cudaMallocAsync((void**)&base, bytes, s));
    o.tsum = reinterpret_cast<uint64_t*>(base);
    o.s1 = o.tsum + n;
    o.n9 = reinterpret_cast<unsigned long long*>(o.s1 + n);
    o.tau6 = o.n9 + n;
    o.n7 = o.tau6 + n;
    o.n7x2 = o.n7 + n;
    o.N = reinterpret_cast<uint64_t*>(o.n7x2 + n);
    o.qcnt = reinterpret_cast<unsigned long long*>(o.N + kOrbits * n);
    o.q_light = reinterpret_cast<int32_t*>(o.qcnt + 8);
    o.w_light = o.q_light + n;
    o.q_heavy = o.w_light + n;
    o.dense = dense_bytes ? reinterpret_cast<uint32_t*>(o.q_heavy + n + (n & 1)) : nullptr;
    harp_status st = HARP_OK;
    cudaError_t e = cudaMemsetAsync(base, 0, bytes, s);  // every accumulator and the dense counters
    if (e == cudaSuccess) st = orbit_passes(g, ws, o, s);
    if (e == cudaSuccess && st == HARP_OK) {
        const OrbGraph G{ws.off, ws.cols, ws.deg, ws.offp, ws.colsp, ws.te};
        launch(k_orb_close, orb_grid(n), kOrbThreads, 0, s, G, n, o.tsum, o.s1, o.n9, o.tau6, o.n7, o.n7x2, ws.order,
               o.N, d_out, ws.acc);
        note_launch();
        e = cudaGetLastError();
    }
    cudaFreeAsync(base, s);
    if (e != cudaSuccess) {
        record_cuda_error(e);
        return e == cudaErrorMemoryAllocation ? HARP_ENOMEM : HARP_ECUDA;
    }
    return st;
}

harp_status count_edge_orbits(const harp_csr* g, Workspace& ws, uint64_t* d_out, cudaStream_t s) {
    const int64_t n = g->n, m = g->m;
    if (m == 0) return HARP_OK;
    // scratch: tsum, s1, N (13 n uint64; of N only the vertex sums are written), e5, e8, e9 (m), e6a (2 m), ebase
    // (int64 n + 1), the queue counters, up and three queue arrays (int32 n), the heavy roots' global counters
    OrbScratch o{};
    o.heavy_blocks = orbit_heavy_blocks(g);
    const size_t dense_bytes = (size_t)o.heavy_blocks * (size_t)n * 4;
    const size_t words = (size_t)n * (2 + kOrbits) + 5 * (size_t)m + (size_t)n + 1 + 8;
    const size_t bytes = 8 * words + 4 * (size_t)(4 * n) + dense_bytes;
    unsigned char* base = nullptr;
    HARP_CK(cudaMallocAsync((void**)&base, bytes, s));
    o.tsum = reinterpret_cast<uint64_t*>(base);
    o.s1 = o.tsum + n;
    o.N = o.s1 + n;
    o.e5 = reinterpret_cast<unsigned long long*>(o.N + kOrbits * n);
    o.e8 = o.e5 + m;
    o.e9 = o.e8 + m;
    o.e6a = o.e9 + m;
    int64_t* ebase = reinterpret_cast<int64_t*>(o.e6a + 2 * m);
    o.qcnt = reinterpret_cast<unsigned long long*>(ebase + n + 1);
    int32_t* up = reinterpret_cast<int32_t*>(o.qcnt + 8);
    o.q_light = up + n;
    o.w_light = o.q_light + n;
    o.q_heavy = o.w_light + n;
    o.dense = dense_bytes ? reinterpret_cast<uint32_t*>(o.q_heavy + n) : nullptr;
    harp_status st = HARP_OK;
    cudaError_t e = cudaMemsetAsync(base, 0, bytes, s);
    if (e == cudaSuccess) st = orbit_passes(g, ws, o, s);
    if (e == cudaSuccess && st == HARP_OK) {
        const int64_t blocks = (n + 255) / 256;
        launch(k_eorb_up, (unsigned)(blocks < 4096 ? blocks : 4096), 256, 0, s, g->off, g->cols, n, up);
        note_launch();
        e = cudaGetLastError();
    }
    if (e == cudaSuccess && st == HARP_OK) st = exclusive_scan_i32_to_i64(up, ebase, n, ws.scan_tmp, ws.scan_tmp_len, s);
    if (e == cudaSuccess && st == HARP_OK) {
        const OrbGraph G{ws.off, ws.cols, ws.deg, ws.offp, ws.colsp, ws.te};
        const int64_t blocks = (m + 255) / 256;
        launch(k_eorb_close, (unsigned)(blocks < (int64_t)num_sms() * 16 ? blocks : (int64_t)num_sms() * 16), 256, 0,
               s, G, n, m, ws.dplus, o.tsum, o.s1, o.e5, o.e8, o.e9, o.e6a, ws.order, g->off, g->cols, up, ebase,
               d_out, ws.acc);
        note_launch();
        e = cudaGetLastError();
    }
    cudaFreeAsync(base, s);
    if (e != cudaSuccess) {
        record_cuda_error(e);
        return e == cudaErrorMemoryAllocation ? HARP_ENOMEM : HARP_ECUDA;
    }
    return st;
}

}  // namespace harp
