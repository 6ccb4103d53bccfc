// Steps a3 + a4: triangle anchors with per-edge triangle statistics, and their 4-clique extension
// (Section III-B: "for 4-node motifs, anchors include ordered wedges and triangles"; Section III-F:
// X_3 / 4-cliques; Section III-D: warp-local vs CTA mode, ordered set intersection, compaction,
// block-local aggregation).
//
// In rank order every triangle {u < v < w} is anchored once at its lowest vertex u.  For an anchor
// vertex u with out-neighbourhood L = N+(u) (sorted, d = |L|) we build the oriented adjacency of
// G[L] as a bitmap: row i has bit j (j > i) iff L[j] is in N+(L[i]).  Row i is the candidate
// frontier of the partial embedding (u, L[i]) (its signature: j = 2, frontier generator (u, L[i]),
// required adjacency to both, no forbidden edge); it is computed once by an ordered intersection of
// N+(L[i]) with L and then reused for
//   * triangles:   T_u = sum_i popc(row_i)
//   * t_e:         arc (u, L[i]) gets popc(row_i) + (# rows with bit i); arc (L[i], L[j]) gets +1
//                  per set bit (global atomic at the position where the intersection found it)
//   * 4-cliques:   K4_u = sum over set bits (i, j) of popc(row_i & row_j)   (the X_3 extension)
//   * paw sums:    sum over triangles of (d_a + d_b + d_c)
// Where L[i] lies in the wedge core (CoreTable), row i is read from the core's bitmap, a bit per pair (gather_rows).
// Otherwise the intersection either probes the exact range of N+(L[i]) in [L[i+1], max L] (16-byte loads, a
// membership filter while hits are rare, then the index j of each element in L), or, where few keys
// of L remain after L[i], searches each of those keys in N+(L[i]) (row_searches).
// Warp-local mode: d <= tri_warp_max (<= 32), rows are single words, one warp per anchor.
// CTA mode: up to tri_cta_max (<= 1024) in three sizes (256 / 512 / 1024), rows in shared memory, one
// block per anchor; the 4-clique sum is dealt to the block as (word, row) units of the bitmap.  Global-staged
// mode (up to tri_big_max <= 4096, hubs of very large skewed graphs): the same rows in a per-block scratch that stays in L2 (d^2 / 8 bytes), each row built in
// a per-warp shared buffer and written out once.  Fallback (larger d): per out-arc ordered
// intersections through global memory with binary-searched membership; 4-cliques by binary search
// in N+(w).  Membership of y in L is a hash lookup (HARP_PROBE_HASH) or a binary search of the
// sorted L in shared memory (HARP_PROBE_BSEARCH); with the hash, a CTA anchor whose L spans few ranks
// uses a direct table indexed by y - L[0] in the hash's bytes instead.
//
// Signature reuse (Section III-C): the extension of (u, v, w) to a 4-clique needs
// |N+(w) n S_uv|, and since S_uv is a subset of L this is popc(row_v & row_w): the staged frontier of
// the signature (u, w) answers it.  Every triangle is one such lookup; it is a hit when the anchor's
// rows are staged (warp and CTA modes) and a miss in the fallback, which recomputes the
// intersection from N+(w).  With reuse switched off (HARP_PLAN_NO_REUSE) the staged modes recompute
// too, by walking N+(w) in global memory; the counts are identical either way.  acc[ACC_SIG_HITS]
// counts hits; the lookups are the triangles.
#include "harp_internal.cuh"

namespace harp {
namespace {

constexpr int kCta1 = 256;
// Block shape of the 256 mode: 128 threads, 9 resident blocks per SM.  An anchor's rows spread over fewer warps wait
// less at its block barriers, and more blocks share each SM: Chung-Lu of 2,000,000 vertices 5.58 ms, against 6.05 ms
// for 192 x 7 and 7.9 ms for 256 x 5; R-MAT scale 20 2.98, 3.10 and 4.0 ms.
constexpr int kCta1Threads = 128;
constexpr int kCta1Blocks = 9;
constexpr int kCta2 = 512;
constexpr int kCtaMax = 1024;
constexpr int kInf = 0x7fffffff;
constexpr int32_t kNoKey = -1;

// Anchor queues: in ws.q_tri (n entries) warp-mode anchors (2 <= d <= tri_warp_max) from the front
// and CTA-mode anchors from the back; fallback anchors in ws.q_mid[0, n) and global-staged anchors in
// ws.q_mid[n, 2n) (q_mid is free until the wedge pass).  Vertices are scanned in descending rank, so
// high-degree anchors tend to be queued (and taken) first.
//
// Tier of an anchor of out-degree d: -1 none, 0 warp, 1/2/3 CTA 256/512/1024, 4 global-staged,
// 5 fallback.  wmax <= 32, cmax <= kCtaMax, bmax <= kBigMax (tri_warp_max / tri_cta_max / tri_big_max).
constexpr int kBigMax = 4096;
__device__ __forceinline__ int tri_class(int d, int wmax, int cmax, int bmax) {
    if (d < 2) return -1;
    if (d <= wmax) return 0;
    if (d > cmax) return d <= bmax ? 4 : 5;
    return d <= kCta1 ? 1 : (d <= kCta2 ? 2 : 3);
}

__global__ void k_tri_classify(const int32_t* __restrict__ dplus, int64_t n, int64_t own_lo, int64_t own_hi,
                               int wmax, int cmax, int bmax, int32_t* __restrict__ q, int32_t* __restrict__ q_fb,
                               unsigned long long* __restrict__ cnt, unsigned long long* __restrict__ cnt_fb,
                               unsigned long long* __restrict__ cnt_big) {
    grid_begin();
    const int l = lane_id();
    for (int64_t base = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) - l; base < n;
         base += (int64_t)gridDim.x * blockDim.x) {
        const int64_t u = n - 1 - (base + l);
        int cls = -1;
        if (u >= own_lo && u < own_hi && u < n) cls = tri_class(dplus[u], wmax, cmax, bmax);
        // 0: warp queue, 1: CTA queue, 2: fallback queue, 3: global-staged queue
        cls = cls == 5 ? 2 : (cls == 4 ? 3 : (cls > 0 ? 1 : cls));
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const uint32_t mask = __ballot_sync(kFull, cls == c);
            if (!mask) continue;
            unsigned long long start = 0;
            const int leader = __ffs(mask) - 1;
            unsigned long long* ctr = c < 2 ? &cnt[c] : (c == 2 ? cnt_fb : cnt_big);
            if (l == leader) start = atomicAdd(ctr, (unsigned long long)__popc(mask));
            start = __shfl_sync(kFull, start, leader);
            if (cls == c) {
                const unsigned long long k = start + __popc(mask & lanemask_lt());
                if (c == 0) q[k] = (int32_t)u;
                else if (c == 1) q[n - 1 - (int64_t)k] = (int32_t)u;
                else if (c == 2) q_fb[k] = (int32_t)u;
                else q_fb[n + (int64_t)k] = (int32_t)u;
            }
        }
    }
}

// Shared-memory hash of the anchor list: key = vertex, value = its index in L.  2^bits slots.
template <typename V>
__device__ __forceinline__ void hash_put(int32_t* hk, V* hv, int bits, int32_t key, int idx) {
    const uint32_t mask = (1u << bits) - 1;
    uint32_t h = hash32((uint32_t)key) >> (32 - bits);
    for (;;) {
        if (atomicCAS(&hk[h], kNoKey, key) == kNoKey) {
            hv[h] = (V)idx;
            return;
        }
        h = (h + 1) & mask;
    }
}

template <typename V>
__device__ __forceinline__ int hash_get(const int32_t* hk, const V* hv, int bits, int32_t key) {
    const uint32_t mask = (1u << bits) - 1;
    uint32_t h = hash32((uint32_t)key) >> (32 - bits);
    for (;;) {
        const int32_t k = hk[h];
        if (k == key) return (int)hv[h];
        if (k == kNoKey) return -1;
        h = (h + 1) & mask;
    }
}

// Index of y in the sorted list L[0, d) (shared memory), or -1.
__device__ __forceinline__ int find_sorted(const int32_t* L, int d, int32_t y) {
    int lo = 0, hi = d;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (L[mid] < y) lo = mid + 1;
        else hi = mid;
    }
    return (lo < d && L[lo] == y) ? lo : -1;
}

// First position p in [lo, hi) with a[p] >= t, found by the whole warp (32-ary search).
__device__ __forceinline__ int64_t warp_lower_bound(const int32_t* __restrict__ a, int64_t lo, int64_t hi, int32_t t) {
    const int l = lane_id();
    while (hi - lo > 32) {
        const int64_t step = (hi - lo + 31) >> 5;
        const int64_t idx = lo + (int64_t)(l + 1) * step - 1;
        const bool pred = idx >= hi || a[idx] >= t;
        const uint32_t m = __ballot_sync(kFull, pred);
        if (!m) return hi;  // every probed element (the last one included) is below t
        const int k = __ffs(m) - 1;
        const int64_t nlo = lo + (int64_t)k * step;
        const int64_t nhi = nlo + step < hi ? nlo + step : hi;
        lo = nlo;
        hi = nhi;
    }
    const bool pred = lo + l < hi && a[lo + l] >= t;
    const uint32_t m = __ballot_sync(kFull, pred);
    return m ? lo + __ffs(m) - 1 : hi;
}

// Walk the sorted list colsp[b, e) in warp-wide chunks with kProbeUnroll chunks' loads in flight,
// calling probe(y, position) for every element, and stop after the chunk that passes `last`.
constexpr int kProbeUnroll = 2;

template <typename F>
__device__ __forceinline__ void probe_list(const int32_t* __restrict__ colsp, int64_t b, int64_t e, int32_t last,
                                           F&& probe) {
    const int l = lane_id();
    for (int64_t p0 = b; p0 < e; p0 += 32 * kProbeUnroll) {
        int32_t ys[kProbeUnroll];
#pragma unroll
        for (int r = 0; r < kProbeUnroll; ++r) {
            const int64_t p = p0 + r * 32 + l;
            ys[r] = p < e ? colsp[p] : kInf;
        }
        bool done = false;
#pragma unroll
        for (int r = 0; r < kProbeUnroll; ++r) {
            if (!done) {
                probe(ys[r], p0 + r * 32 + l);
                done = __shfl_sync(kFull, ys[r], 31) >= last;  // rows are sorted: past the largest candidate
            }
        }
        if (done) break;
    }
}

// Probe every element of colsp[b, e) (an exact range) with 16-byte loads.  The range is widened to
// 4-element boundaries: colsp starts on a 256-byte boundary and its allocation is padded to a multiple
// of 256 bytes, so the wider loads stay inside it; lane l takes elements a + 128 k + 4 l .. + 3 (a = b
// rounded down to a multiple of 4) and masks those outside [b, e).  visit(y, p) gets the element and
// its position in colsp.
// With `filter` (warp-uniform) the membership test may_hold(y) (a filter bit: 0 proves y absent) runs
// first on all four elements and the lane then visits only those that pass, so 128 elements pay for
// the divergent lookup and hit paths once per candidate of the busiest lane, instead of once per 32
// elements whenever any lane holds a candidate.  Without it (rows where hits are common) every
// element is visited.
template <typename Filter, typename Visit>
__device__ __forceinline__ void probe_filtered(const int32_t* __restrict__ colsp, int64_t b, int64_t e, bool filter,
                                               Filter&& may_hold, Visit&& visit) {
    const int64_t a = b & ~(int64_t)3;
    const int4* __restrict__ v = reinterpret_cast<const int4*>(colsp + a);
    const int lo = (int)(b - a), hi = (int)(e - a);  // the range's offsets from a: lo <= 3
    for (int q = 4 * lane_id(); q < hi; q += 128) {
        const int4 y = __ldg(v + (q >> 2));
        uint32_t valid = hi - q >= 4 ? 0xfu : (1u << (hi - q)) - 1u;
        if (q < lo) valid &= 0xfu << (lo - q);
        if (filter) {
            uint32_t cand = may_hold(y.x) | (may_hold(y.y) << 1) | (may_hold(y.z) << 2) | (may_hold(y.w) << 3);
            cand &= valid;
            while (cand) {
                const int r = __ffs(cand) - 1;
                cand &= cand - 1;
                const int32_t x = r == 0 ? y.x : (r == 1 ? y.y : (r == 2 ? y.z : y.w));
                visit(x, a + q + r);
            }
        } else {
            if (valid & 1u) visit(y.x, a + q);
            if (valid & 2u) visit(y.y, a + q + 1);
            if (valid & 4u) visit(y.z, a + q + 2);
            if (valid & 8u) visit(y.w, a + q + 3);
        }
    }
}

// Whether the next row is probed through the membership filter: the filter pays while hits are rare.
// Each warp keeps its own probe and hit totals over the rows it has taken (halved past 2^20 probes, so
// they follow the current anchors) and filters while fewer than one probe in eight has hit.
struct FilterChoice {
    uint32_t probes = 0, hits = 0;
    __device__ __forceinline__ bool use() const { return 8u * hits <= probes; }
    __device__ __forceinline__ void add(int64_t row_probes, uint32_t row_hits) {
        probes += (uint32_t)row_probes;
        hits += row_hits;
        if (probes > (1u << 20)) {
            probes >>= 1;
            hits >>= 1;
        }
    }
};

// Row i's hits can be found from either side: probe every element of its range (one load and a
// filter or hash lookup each), or search each of the keys of L left after L[i] in the range (a binary
// search of about log2(len) + 1 dependent loads each, which the row's few cache lines keep in L1).
// Searching costs less when keys * (log2(len) + 1) < 2 * len: rows near the end of L and rows of long
// ranges.  Both find exactly the members of L in the range.
__device__ __forceinline__ bool row_searches(int keys, int64_t len) {
    if (len <= 0) return false;  // no element: nothing to do either way
    const int lg = 64 - __clzll(len);  // floor(log2(len)) + 1
    return (int64_t)keys * lg < 2 * len;
}

// Position of key in the sorted colsp[b, b + len), or -1.
__device__ __forceinline__ int64_t find_in_range(const int32_t* __restrict__ colsp, int64_t b, int len, int32_t key) {
    int lo = 0, hi = len;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(colsp + b + mid) < key) lo = mid + 1;
        else hi = mid;
    }
    return (lo < len && __ldg(colsp + b + lo) == key) ? b + lo : -1;
}

// Membership filter in front of the hash lookup: bit (top FB bits of hash32(y)) is set for every key,
// so a clear bit proves y is not in L (most probes miss; a miss then costs one shared load).
template <int FB>
__device__ __forceinline__ uint32_t filter_may_hold(const uint32_t* filt, int32_t y) {
    const uint32_t h = hash32((uint32_t)y) >> (32 - FB);
    const uint32_t w = filt[h >> 5];
    return __funnelshift_r(w, w, h) & 1u;  // bit (h mod 32) of the word: the rotate takes h mod 32
}

// single-graph mode: one block reduction and one atomic per statistic at the end of the kernel;
// the signature hits go to acc[ACC_SIG_HITS] in both modes
__device__ __forceinline__ void flush_block(const Sink& sink, uint64_t tri, uint64_t k4, uint64_t paw, uint64_t hits,
                                            uint64_t* red) {
    tri = block_sum_u64(tri, red);
    k4 = block_sum_u64(k4, red);
    paw = block_sum_u64(paw, red);
    hits = block_sum_u64(hits, red);
    if (threadIdx.x == 0) {
        if (hits) atomicAdd((unsigned long long*)&sink.acc[ACC_SIG_HITS], (unsigned long long)hits);
        if (!sink.batch()) {
            if (tri) atomicAdd((unsigned long long*)&sink.acc[ACC_T], (unsigned long long)tri);
            if (k4) atomicAdd((unsigned long long*)&sink.acc[ACC_K4], (unsigned long long)k4);
            if (paw) atomicAdd((unsigned long long*)&sink.acc[ACC_PAWSUM], (unsigned long long)paw);
        }
    }
}

// ---------------------------------------------------------------------------------------------
// Warp-local mode.
// ---------------------------------------------------------------------------------------------
constexpr int kWarpThreads = 256;
constexpr int kWarpsPerBlock = kWarpThreads / 32;
constexpr int kWarpHashBits = 7;  // 128 slots for <= 32 keys: load <= 1/4, ~1.4 slot reads per miss
constexpr int kWarpFilterBits = 10;  // membership filter of 1024 bits: false positives <= 32 / 1024

// Anchors are short chains of dependent loads (the anchor, its list, the lists' bounds, their elements), so a warp
// takes kWarpChunk consecutive anchors of the queue: their headers are loaded side by side, the next anchor's
// list while the current one is worked on, and in a batch their sums (mostly of one graph) meet in registers.
// Fewer where the queue would not give every warp two chunks.  Chunks are taken by ticket: the heavy anchors come
// first in the queue (dealt in turn, the batch below took 11.1 ms).
// Batch of 4,096 graphs: 22.5 -> 8.75 ms; random geometric, 1,000,003 vertices: 1.56 -> 0.71 ms; Chung-Lu,
// 2,000,000 vertices: 4.39 -> 3.31 ms.
constexpr int kWarpChunk = 8;
// A probing row this long is read by the whole warp behind the membership filter; shorter ones by 8 lanes each.
constexpr int kLongRow = 64;

template <bool BS>
__global__ void __launch_bounds__(kWarpThreads, 4) k_tri_warp(const int64_t* __restrict__ offp,
                                                           const int32_t* __restrict__ colsp,
                                                           const int32_t* __restrict__ deg,
                                                           const int32_t* __restrict__ q,
                                                           const unsigned long long* __restrict__ cnt,
                                                           bool reuse, uint32_t* __restrict__ te, Sink sink) {
    grid_begin();
    __shared__ int32_t sL[kWarpsPerBlock][32];
    __shared__ uint32_t sRow[kWarpsPerBlock][32];  // row i: bit j (j > i) iff L[j] in N+(L[i])
    __shared__ uint32_t sCol[kWarpsPerBlock][32];  // its transpose
    __shared__ int32_t sHk[kWarpsPerBlock][1 << kWarpHashBits];
    __shared__ uint8_t sHv[kWarpsPerBlock][1 << kWarpHashBits];
    __shared__ uint32_t sFilt[kWarpsPerBlock][(1 << kWarpFilterBits) / 32];
    __shared__ uint64_t red[32];
    const int w = threadIdx.x >> 5, l = lane_id();
    const int64_t nq = (int64_t)cnt[0];
    uint64_t tri = 0, k4 = 0, paw = 0, hits = 0;  // since the last flush (batch) or in all
    int32_t g = -1;
    FilterChoice fc;
    auto flush_graph = [&] {
        const uint64_t t1 = warp_sum(tri), t2 = warp_sum(k4), t3 = warp_sum(paw);
        if (l == 0 && g >= 0) {
            unsigned long long* a = (unsigned long long*)&sink.accG[(int64_t)g * kGStride];
            if (t1) atomicAdd(&a[G_T], (unsigned long long)t1);
            if (t2) atomicAdd(&a[G_K4], (unsigned long long)t2);
            if (t3) atomicAdd(&a[G_PAWSUM], (unsigned long long)t3);
        }
        tri = k4 = paw = 0;
    };
    const int64_t share = nq / (2 * (int64_t)gridDim.x * kWarpsPerBlock);
    const int chunk = share < 1 ? 1 : (share < kWarpChunk ? (int)share : kWarpChunk);
    const int64_t nchunk = (nq + chunk - 1) / chunk;
    unsigned long long* ticket = (unsigned long long*)&sink.acc[T_TRI_W];
    auto next_ticket = [&] { return l == 0 ? (int64_t)atomicAdd(ticket, 1ull) : 0; };
    int64_t c_next = next_ticket();
    for (;;) {
        const int64_t c = __shfl_sync(kFull, c_next, 0);
        if (c >= nchunk) break;
        c_next = next_ticket();  // in flight while this chunk is worked on
        const int cn = nq - c * chunk < chunk ? (int)(nq - c * chunk) : chunk;
        int32_t hu = 0, hg = -1, hdeg = 0;
        int64_t hb = 0;
        int hd = 0;
        if (l < cn) {
            hu = q[c * chunk + l];
            hb = offp[hu];
            hd = (int)(offp[hu + 1] - hb);
            hdeg = deg[hu];
            if (sink.batch()) hg = sink.gid[hu];
        }
        int64_t ub = __shfl_sync(kFull, hb, 0);
        int d = __shfl_sync(kFull, hd, 0);
        int32_t x_next = l < d ? colsp[ub + l] : kInf;
        for (int ai = 0; ai < cn; ++ai) {
            const int32_t x = x_next;  // lane l holds L[l] (kInf past the list)
            ub = __shfl_sync(kFull, hb, ai);
            d = __shfl_sync(kFull, hd, ai);
            int64_t b = 0;
            int len = 0;
            if (l < d - 1) {
                b = offp[x];
                len = (int)(offp[x + 1] - b);
            }
            const uint64_t dx = l < d ? (uint64_t)deg[x] : 0;
            {
                const int nd = ai + 1 < cn ? __shfl_sync(kFull, hd, ai + 1) : 0;
                const int64_t nb = __shfl_sync(kFull, hb, (ai + 1) & 31);
                x_next = l < nd ? colsp[nb + l] : kInf;
            }
            if (sink.batch()) {
                const int32_t ag = __shfl_sync(kFull, hg, ai);
                if (ag != g) {
                    flush_graph();
                    g = ag;
                }
            }
            sRow[w][l] = 0;
            sCol[w][l] = 0;
            __syncwarp();
            const int32_t last = __shfl_sync(kFull, x, d - 1);
            auto found = [&](int i, int j, int64_t p) {  // L[j] at position p of N+(L[i])
                atomicAdd(&te[p], 1u);  // arc (L[i], L[j]): top edge of triangle (u, L[i], L[j])
                atomicOr(&sRow[w][i], 1u << j);
                atomicOr(&sCol[w][j], 1u << i);
            };
            // A member of L found anywhere in N+(L[i]) is an edge, so short rows and searches need no exact range.
            const bool search = len > 0 && row_searches(d - 1 - l, len);
            // the searching rows' (row, key) pairs are flattened over the lanes, so one round of binary
            // searches covers several short rows; pair t belongs to the last row whose first pair is at or
            // before t
            if (__any_sync(kFull, search)) {
                const int npairs = search ? d - 1 - l : 0;
                int incl = npairs;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(kFull, incl, o);
                    if (l >= o) incl += y;
                }
                const int excl = incl - npairs;
                const int total = __shfl_sync(kFull, incl, 31);
                for (int t0 = 0; t0 < total; t0 += 32) {
                    const int t = t0 + l;
                    int o = 0;
#pragma unroll
                    for (int sft = 16; sft >= 1; sft >>= 1) {
                        const int e = __shfl_sync(kFull, excl, o + sft);
                        if (e <= t) o += sft;
                    }
                    const int64_t rb = __shfl_sync(kFull, b, o);
                    const int rl = __shfl_sync(kFull, len, o);
                    const int j = o + 1 + (t - __shfl_sync(kFull, excl, o));
                    const int32_t key = __shfl_sync(kFull, x, j & 31);
                    if (t < total) {
                        const int64_t p = find_in_range(colsp, rb, rl, key);
                        if (p >= 0) found(o, j, p);
                    }
                }
            }
            // short probing rows: 8 lanes each, two elements a lane at once; the place of y in L by a search over
            // the lanes (a few dozen elements do not pay for building a hash)
            uint32_t shorts = __ballot_sync(kFull, len > 0 && !search && len < kLongRow);
            while (shorts) {
                int r = -1;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if (k == (l >> 3)) r = __ffs(shorts) - 1;
                    shorts &= shorts - 1;
                }
                const int64_t rb = __shfl_sync(kFull, b, r & 31);
                int rl = __shfl_sync(kFull, len, r & 31);
                if (r < 0) rl = 0;
                for (int k = l & 7; __any_sync(kFull, k < rl); k += 16) {
                    int32_t y[2];
#pragma unroll
                    for (int h = 0; h < 2; ++h) y[h] = k + 8 * h < rl ? __ldg(colsp + rb + k + 8 * h) : kInf;
                    if (y[0] > last) rl = 0;  // rows are sorted: this lane's further elements are larger still
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        int pos = 0;
#pragma unroll
                        for (int sft = 16; sft >= 1; sft >>= 1) {
                            const int32_t v = __shfl_sync(kFull, x, pos + sft - 1);
                            if (v < y[h]) pos += sft;
                        }
                        const int32_t v = __shfl_sync(kFull, x, pos);  // kInf elements stop at a lane past the list
                        if (v == y[h] && v != kInf) found(r, pos, rb + k + 8 * h);
                    }
                }
            }
            uint32_t longs = __ballot_sync(kFull, len >= kLongRow && !search);
            if (longs || !reuse) {
                sL[w][l] = x;
#pragma unroll
                for (int hs = 0; hs < (1 << kWarpHashBits); hs += 32) sHk[w][l + hs] = kNoKey;
                sFilt[w][l] = 0;
                __syncwarp();
                if (l < d) {
                    if (!BS) hash_put(sHk[w], sHv[w], kWarpHashBits, x, l);
                    const uint32_t h = hash32((uint32_t)x) >> (32 - kWarpFilterBits);
                    atomicOr(&sFilt[w][h >> 5], 1u << (h & 31));
                }
                __syncwarp();
            }
            auto lookup = [&](int32_t y) {
                return BS ? find_sorted(sL[w], d, y) : hash_get(sHk[w], sHv[w], kWarpHashBits, y);
            };
            // long probing rows: the exact range [rb, re) of N+(L[i]) in [L[i+1], max L], lane i for row i (the lanes'
            // dependent loads overlap)
            if (longs) {
                int64_t rb = 0, re = 0;
                if ((longs >> l) & 1u) {
                    rb = b + lower_bound_i32(colsp + b, len, sL[w][l + 1]);
                    re = rb + lower_bound_i32(colsp + rb, b + len - rb, last + 1);
                }
                while (longs) {
                    const int i = __ffs(longs) - 1;
                    longs &= longs - 1;
                    const int64_t pb = __shfl_sync(kFull, rb, i), pe = __shfl_sync(kFull, re, i);
                    uint32_t row_hits = 0;
                    probe_filtered(colsp, pb, pe, fc.use(),
                                   [&](int32_t y) { return filter_may_hold<kWarpFilterBits>(sFilt[w], y); },
                                   [&](int32_t y, int64_t p) {
                                       const int j = lookup(y);
                                       if (j >= 0) {
                                           found(i, j, p);
                                           ++row_hits;
                                       }
                                   });
                    fc.add(pe - pb, __reduce_add_sync(kFull, row_hits));
                }
            }
            __syncwarp();
            const uint32_t myrow = sRow[w][l];
            const uint32_t own = (uint32_t)(__popc(myrow) + __popc(sCol[w][l]));
            if (own) atomicAdd(&te[ub + l], own);
            const uint64_t a_tri = (uint64_t)__popc(myrow);
            uint64_t a_k4 = 0;
            uint32_t bits = myrow;
            if (reuse) {
                while (bits) {  // the staged frontier of (u, L[j]) answers the extension
                    const int j = __ffs(bits) - 1;
                    bits &= bits - 1;
                    a_k4 += (uint64_t)__popc(myrow & sRow[w][j]);
                }
                hits += a_tri;
            } else {
                while (bits) {  // recompute |N+(L[j]) n S_uv| from N+(L[j]) in global memory
                    const int j = __ffs(bits) - 1;
                    bits &= bits - 1;
                    const int32_t wv = sL[w][j];
                    for (int64_t p = offp[wv], pe = offp[wv + 1]; p < pe; ++p) {
                        const int32_t y = colsp[p];
                        if (y > last) break;
                        const int jj = lookup(y);
                        if (jj >= 0 && ((myrow >> jj) & 1u)) ++a_k4;
                    }
                }
            }
            tri += a_tri;
            k4 += a_k4;
            paw += (uint64_t)own * dx + a_tri * (uint64_t)__shfl_sync(kFull, hdeg, ai);
            __syncwarp();
        }
    }
    if (sink.batch()) flush_graph();
    flush_block(sink, tri, k4, paw, hits, red);
}

// ---------------------------------------------------------------------------------------------
// CTA mode: rows of the anchor's out-neighbourhood bitmap in shared memory.
// ---------------------------------------------------------------------------------------------
template <int DMAX>
struct CtaSmem {
    static constexpr int W = DMAX / 32;             // words per row
    static constexpr int WS = W | 1;                // odd row stride: no bank conflicts
    static constexpr int HB = (DMAX <= 256) ? 10 : ((DMAX <= 512) ? 11 : 12);  // 4 * DMAX hash slots
    // filter: 64 bits per key (2, 4 and 8 KB); false positives at most d / 2^FB <= 1 / 64
    static constexpr int FB = HB + 4;
    // The 256 and 1024 modes resolve every row's exact probe range up front (one binary search per
    // thread per bound); the 512 mode does so only for direct-table anchors (in the filter's bytes,
    // below) and otherwise finds each row's range with the warp-wide search when the row is taken:
    // two more range arrays would cost it a resident block per SM.
    static constexpr bool PRE = DMAX <= 256 || DMAX >= 1024;
    int32_t L[DMAX];
    uint32_t own[DMAX];
    uint32_t R[DMAX * WS];
    // membership of y in L: a direct table indexed by y - L[0] when L's span fits (tab[y - L[0]] = index
    // + 1, 0 = absent; 3 * 2^HB entries), else a hash of 2^HB slots in the same bytes
    static constexpr int TAB = 3 << HB;
    union {
        struct {
            int32_t hk[1 << HB];
            uint16_t hv[1 << HB];
        } h;
        uint16_t tab[TAB];
    } m;
    // the filter (hash and binary-search anchors) or, for direct-table anchors of the 512 mode, every
    // row's probe range as offsets into N+(L[i]): lo in rel[i], hi in rel[DMAX + i] (the same 8 * DMAX
    // bytes)
    union {
        uint32_t filt[(1 << FB) / 32];
        int32_t rel[2 * DMAX];
    };
    static_assert((1 << FB) / 32 == 2 * DMAX, "the filter and the relative ranges share their bytes");
    // row i probes colsp[rb[i], re[i]): the elements of N+(L[i]) in [L[i+1], max L]
    int64_t rb[PRE ? DMAX : 1];
    int64_t re[PRE ? DMAX : 1];
    uint64_t red[32];
    int walk;
};

// The anchor a block works on: its list L = N+(u) of d members, of which the first `walk` have their rows walked (the
// others are in the core and have theirs read from its bitmap); direct: membership by the table indexed by
// y - L0 (where L's span fits: dense anchors, high ranks close together) instead of the hash.
struct CtaAnchor {
    int d, walk;
    int32_t L0;
    uint32_t span;
    bool direct;
};

// Stages L and, where rows are walked, the membership structure and these rows' probe ranges; clears own and the
// bitmap (d rows of WS words).  c0: the core's first rank (s.walk is then INT_MAX on entry), or INT_MAX.  Ends with a
// block barrier.
template <int DMAX, int THREADS, bool BS>
__device__ __forceinline__ CtaAnchor stage_anchor(CtaSmem<DMAX>& s, const int64_t* __restrict__ offp,
                                                  const int32_t* __restrict__ colsp, int64_t ub, int d, int WS,
                                                  int32_t c0) {
    using S = CtaSmem<DMAX>;
    CtaAnchor A;
    A.d = d;
    A.L0 = colsp[ub];
    A.span = (uint32_t)(colsp[ub + d - 1] - A.L0) + 1u;
    A.direct = !BS && A.span <= (uint32_t)S::TAB;
    for (int i = threadIdx.x; i < d; i += THREADS) {
        const int32_t x = colsp[ub + i];
        s.L[i] = x;
        s.own[i] = 0;
        if (x >= c0 && (i == 0 || colsp[ub + i - 1] < c0)) s.walk = i;
    }
    for (int i = threadIdx.x; i < d * WS; i += THREADS) s.R[i] = 0;
    if (A.L0 >= c0) {
        __syncthreads();
        A.walk = 0;
        return A;
    }
    if (A.direct) {
        for (int i = threadIdx.x; i < (int)A.span; i += THREADS) s.m.tab[i] = 0;
    } else {
        for (int i = threadIdx.x; i < (1 << S::HB); i += THREADS) s.m.h.hk[i] = kNoKey;
        for (int i = threadIdx.x; i < (1 << S::FB) / 32; i += THREADS) s.filt[i] = 0;
    }
    __syncthreads();
    A.walk = c0 == kInf || s.walk > d - 1 ? d - 1 : s.walk;  // row d - 1 is empty
    for (int i = threadIdx.x; i < d; i += THREADS) {
        if (A.direct) {
            s.m.tab[s.L[i] - A.L0] = (uint16_t)(i + 1);
        } else {
            if (!BS) hash_put(s.m.h.hk, s.m.h.hv, S::HB, s.L[i], i);
            const uint32_t h = hash32((uint32_t)s.L[i]) >> (32 - S::FB);
            atomicOr(&s.filt[h >> 5], 1u << (h & 31));
        }
        if (!S::PRE && A.direct && i < A.walk) {  // as offsets into N+(L[i]) (rows are short)
            const int32_t v = s.L[i];
            const int64_t b = offp[v], e = offp[v + 1];
            const int32_t lo = (int32_t)lower_bound_i32(colsp + b, e - b, s.L[i + 1]);
            s.rel[i] = lo;
            s.rel[DMAX + i] = lo + (int32_t)lower_bound_i32(colsp + b + lo, e - b - lo, s.L[d - 1] + 1);
        }
        if (S::PRE && i < A.walk) {  // every row's probe range at once: dependent loads overlap across rows
            const int32_t v = s.L[i];
            const int64_t b = offp[v], e = offp[v + 1];
            const int64_t lo = b + lower_bound_i32(colsp + b, e - b, s.L[i + 1]);
            s.rb[i] = lo;
            s.re[i] = lo + lower_bound_i32(colsp + lo, e - lo, s.L[d - 1] + 1);  // elements <= max L
        }
    }
    __syncthreads();
    return A;
}

// index of y in the staged list, or -1
template <int DMAX, bool BS>
__device__ __forceinline__ int anchor_find(const CtaSmem<DMAX>& s, const CtaAnchor& A, int32_t y) {
    if (A.direct) {
        const uint32_t o = (uint32_t)(y - A.L0);
        return o < A.span ? (int)s.m.tab[o] - 1 : -1;
    }
    return BS ? find_sorted(s.L, A.d, y) : hash_get(s.m.h.hk, s.m.h.hv, CtaSmem<DMAX>::HB, y);
}

// Row i by a warp: the ordered intersection of N+(L[i]) with L over the exact range of N+(L[i]) in
// [L[i+1], max L] (no smaller element can be in L after L[i], no larger one at all).  hit(j, p) is called for
// every j > i with L[j] at position p of colsp; returns this lane's hits summed over the warp.
template <int DMAX, bool BS, typename Hit>
__device__ __forceinline__ uint32_t walk_row(const CtaSmem<DMAX>& s, const CtaAnchor& A, const int64_t* __restrict__ offp,
                                             const int32_t* __restrict__ colsp, int i, FilterChoice& fc, Hit&& hit) {
    using S = CtaSmem<DMAX>;
    const int d = A.d, l = lane_id();
    int64_t b = 0, e = 0;
    if (S::PRE) {
        b = s.rb[i];
        e = s.re[i];
    } else if (A.direct) {
        const int64_t o = offp[s.L[i]];
        b = o + s.rel[i];
        e = o + s.rel[DMAX + i];
    } else {
        const int32_t v = s.L[i];
        const int64_t e0 = offp[v + 1];
        b = warp_lower_bound(colsp, offp[v], e0, s.L[i + 1]);
        e = warp_lower_bound(colsp, b, e0, s.L[d - 1] + 1);
    }
    uint32_t hits = 0;
    if (row_searches(d - 1 - i, e - b)) {  // the keys after L[i] searched in the range
        const int len = (int)(e - b);
        for (int j = i + 1 + l; j < d; j += 32) {
            const int64_t p = find_in_range(colsp, b, len, s.L[j]);
            if (p >= 0) {
                hit(j, p);
                ++hits;
            }
        }
        hits = warp_sum(hits);
    } else {
        // the filter is built and used only with the hash or the binary search
        probe_filtered(colsp, b, e, !A.direct && fc.use(),
                       [&](int32_t y) { return filter_may_hold<S::FB>(s.filt, y); },
                       [&](int32_t y, int64_t p) {
                           const int j = anchor_find<DMAX, BS>(s, A, y);
                           if (j >= 0) {
                               hit(j, p);
                               ++hits;
                           }
                       });
        hits = warp_sum(hits);
        fc.add(e - b, hits);
    }
    return hits;
}

// The rows i >= walk, whose L[i] are in the core: the core's bitmap has a bit for each pair (L[i], L[j]), so they are
// gathered, one word a pair.  A warp takes a tile of ROWS rows and the 32 keys of a word of the row: a lane keeps
// its key, the tile's words are loaded side by side, the ballots are the words of R and the keys' counts meet in
// registers.

template <int DMAX, int ROWS>
__device__ __forceinline__ void gather_rows(CtaSmem<DMAX>& s, const CoreTable& t, int d, int walk, int WS, int warp,
                                            int nwarps, const int64_t* __restrict__ offp, uint32_t* __restrict__ te) {
    const int l = lane_id();
    int unit = warp;
    for (int c = walk >> 5; 32 * c < d; ++c) {
        const int end = 32 * c + 31 < d - 1 ? 32 * c + 31 : d - 1;  // rows below have keys in word c
        const int tiles = (end - walk + ROWS - 1) / ROWS;
        for (; unit < tiles; unit += nwarps) {
            const int j = 32 * c + l, below = j < d ? j : 0;  // the lane's rows
            const uint32_t o = j < d ? (uint32_t)(s.L[j] - t.c0) : 0u, bit = 1u << (o & 31);
            const uint32_t base = (o >> 5) - (uint32_t)t.c0 * (uint32_t)t.KW;  // + L[i] * KW, modulo 2^32
            const int r0 = walk + unit * ROWS;
            uint32_t word[ROWS], mine = 0, mrow = 0;
#pragma unroll
            for (int k = 0; k < ROWS; ++k) {
                word[k] = 0;
                if (r0 + k < below) word[k] = __ldg(t.bits + ((uint32_t)s.L[r0 + k] * (uint32_t)t.KW + base));
            }
#pragma unroll
            for (int k = 0; k < ROWS; ++k) {
                const bool is = (word[k] & bit) != 0;
                const uint32_t m = __ballot_sync(kFull, is);
                if (l == k) mrow = m;
                if (is) {  // arc (L[i], L[j]): top edge of triangle (u, L[i], L[j])
                    const int32_t v = s.L[r0 + k];
                    const uint32_t before = __ldg(t.before + ((uint32_t)v * (uint32_t)t.KW + base));
                    atomicAdd(&te[offp[v] + before + __popc(word[k] & (bit - 1))], 1u);
                    ++mine;
                }
            }
            if (mrow) {
                s.R[(r0 + l) * WS + c] = mrow;
                atomicAdd(&s.own[r0 + l], (uint32_t)__popc(mrow));
            }
            if (mine) atomicAdd(&s.own[j], mine);
        }
        unit -= tiles;
    }
}

template <int DMAX, int THREADS, int MINB, bool BS>
__global__ void __launch_bounds__(THREADS, MINB) k_tri_cta(const int64_t* __restrict__ offp,
                                                     const int32_t* __restrict__ colsp,
                                                     const int32_t* __restrict__ deg,
                                                     const int32_t* __restrict__ q, int64_t n, int cls,
                                                     int wmax, int cmax, int bmax, bool reuse,
                                                     const unsigned long long* __restrict__ cnt,
                                                     unsigned long long* __restrict__ ticket,
                                                     const int64_t* __restrict__ ginfo,
                                                     const uint32_t* __restrict__ region,
                                                     uint32_t* __restrict__ te, Sink sink) {
    grid_begin();
    using S = CtaSmem<DMAX>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    S& s = *reinterpret_cast<S*>(smem_raw);
    __shared__ int64_t s_item;
    constexpr int NW = THREADS / 32;
    const int w = threadIdx.x >> 5, l = lane_id();
    const int64_t nq = (int64_t)cnt[1];
    uint64_t tri = 0, k4 = 0, paw = 0, hits = 0;
    FilterChoice fc;
    CoreTable core = sink.batch() ? CoreTable{} : core_table(ginfo, 0, region);
    for (;;) {
        if (threadIdx.x == 0) {
            s_item = (int64_t)atomicAdd(ticket, 1ull);
            s.walk = kInf;
        }
        __syncthreads();
        const int64_t k = s_item;
        __syncthreads();
        if (k >= nq) break;
        const int32_t u = q[n - 1 - k];
        const int64_t ub = offp[u];
        const int d = (int)(offp[u + 1] - ub);
        if (tri_class(d, wmax, cmax, bmax) != cls) continue;
        const int W = (d + 31) >> 5;
        const int WS = W | 1;
        if (region && sink.batch()) core = core_table(ginfo, sink.gid[u], region);
        const CtaAnchor A = stage_anchor<DMAX, THREADS, BS>(s, offp, colsp, ub, d, WS, core.c0);
        const int32_t last = s.L[d - 1];
        auto lookup = [&](int32_t y) {
            if (!A.direct && !filter_may_hold<S::FB>(s.filt, y)) return -1;
            return anchor_find<DMAX, BS>(s, A, y);
        };
        for (int i = w; i < A.walk; i += NW) {  // a warp per row
            uint32_t* Ri = &s.R[i * WS];
            const uint32_t row_hits = walk_row<DMAX, BS>(s, A, offp, colsp, i, fc, [&](int j, int64_t p) {
                atomicAdd(&te[p], 1u);  // arc (L[i], L[j]): top edge of triangle (u, L[i], L[j])
                atomicOr(&Ri[j >> 5], 1u << (j & 31));
                atomicAdd(&s.own[j], 1u);
            });
            if (l == 0 && row_hits) atomicAdd(&s.own[i], row_hits);
        }
        if (A.walk < d - 1) gather_rows<DMAX, (DMAX <= 256 ? 8 : 16)>(s, core, d, A.walk, WS, w, NW, offp, te);
        __syncthreads();
        // triangles and 4-cliques (the X_3 extension): the bitmap's (word, row) units are dealt to all the
        // block's threads.  Unit (x, i) counts the set bits j of word x of row i (the triangles (u, L[i],
        // L[j])) and adds |row_i n row_j| for each, over the words from x on (row j has no bit at or
        // below j), so the work is spread by the bits themselves and no lane searches for its bit.  A
        // warp's lanes take one word of consecutive rows: equal word spans, conflict-free row reads.
        uint64_t a_tri = 0, a_k4 = 0, a_paw = 0;
        const int rows = d - 1;  // row d - 1 is empty
        for (int t = threadIdx.x; t < rows * W; t += THREADS) {
            const int x = t / rows, i = t - x * rows;
            if ((x << 5) + 31 <= i) continue;  // row i has no bit at or below i
            const uint32_t* Ri = &s.R[i * WS];
            uint32_t bits = Ri[x];
            a_tri += (uint64_t)__popc(bits);
            while (bits) {
                const int j = (x << 5) + __ffs(bits) - 1;
                bits &= bits - 1;
                uint32_t cnt = 0;
                if (reuse) {  // the staged frontier of (u, L[j])
                    const uint32_t* Rj = &s.R[j * WS];
                    for (int y = x; y < W; ++y) cnt += __popc(Ri[y] & Rj[y]);
                } else {      // recompute from N+(L[j]) in global memory
                    const int32_t wv = s.L[j];
                    for (int64_t p = offp[wv], pe = offp[wv + 1]; p < pe; ++p) {
                        const int32_t y = colsp[p];
                        if (y > last) break;
                        const int jj = lookup(y);
                        if (jj >= 0 && ((Ri[jj >> 5] >> (jj & 31)) & 1u)) ++cnt;
                    }
                }
                a_k4 += cnt;
            }
        }
        for (int i = threadIdx.x; i < d; i += THREADS) {
            const uint32_t o = s.own[i];
            if (o) {
                atomicAdd(&te[ub + i], o);
                a_paw += (uint64_t)o * (uint64_t)deg[s.L[i]];
            }
        }
        // the anchor's own degree term: T_u * d_u
        a_paw += a_tri * (uint64_t)deg[u];
        if (reuse) hits += a_tri;
        __syncthreads();
        if (sink.batch()) {
            const uint64_t t1 = block_sum_u64(a_tri, s.red);
            const uint64_t t2 = block_sum_u64(a_k4, s.red);
            const uint64_t t3 = block_sum_u64(a_paw, s.red);
            if (threadIdx.x == 0) {
                sink_add(sink, u, G_T, t1);
                sink_add(sink, u, G_K4, t2);
                sink_add(sink, u, G_PAWSUM, t3);
            }
        } else {
            tri += a_tri;
            k4 += a_k4;
            paw += a_paw;
        }
    }
    flush_block(sink, tri, k4, paw, hits, s.red);
}

// ---------------------------------------------------------------------------------------------
// Global-staged mode (kCtaMax < d <= kBigMax): one 512-thread block per anchor, the d rows of d bits
// in the block's slice of a global scratch (row stride W = ceil(d / 32) words; at most 2 MiB, so it
// stays in L2).  A warp builds one row at a time in its shared buffer (membership of y in L by binary
// search of the sorted L in shared memory) and writes it out; after a block barrier the 4-clique
// extension reads the staged rows back, exactly as the CTA mode does from shared memory.
// ---------------------------------------------------------------------------------------------
constexpr int kBigThreads = 512;
constexpr int kBigWarps = kBigThreads / 32;
constexpr int kBigWords = kBigMax / 32;

struct BigSmem {
    int32_t L[kBigMax];
    uint32_t own[kBigMax];
    uint32_t row[kBigWarps][kBigWords];
    uint64_t red[32];
};

__global__ void __launch_bounds__(kBigThreads, 1) k_tri_big(const int64_t* __restrict__ offp,
                                                            const int32_t* __restrict__ colsp,
                                                            const int32_t* __restrict__ deg,
                                                            const int32_t* __restrict__ q_big,
                                                            const unsigned long long* __restrict__ cnt_big,
                                                            unsigned long long* __restrict__ ticket, bool reuse,
                                                            uint32_t* __restrict__ scratch,
                                                            uint32_t* __restrict__ te, Sink sink) {
    grid_begin();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    BigSmem& s = *reinterpret_cast<BigSmem*>(smem_raw);
    __shared__ int64_t s_item;
    const int w = threadIdx.x >> 5, l = lane_id();
    uint32_t* R = scratch + (size_t)blockIdx.x * kBigMax * kBigWords;
    uint32_t* buf = s.row[w];
    const int64_t nq = (int64_t)*cnt_big;
    uint64_t tri = 0, k4 = 0, paw = 0, hits = 0;
    for (;;) {
        if (threadIdx.x == 0) s_item = (int64_t)atomicAdd(ticket, 1ull);
        __syncthreads();
        const int64_t k = s_item;
        __syncthreads();
        if (k >= nq) break;
        const int32_t u = q_big[k];
        const int64_t ub = offp[u];
        const int d = (int)(offp[u + 1] - ub);  // cmax < d <= kBigMax by classification
        const int W = (d + 31) >> 5;
        for (int i = threadIdx.x; i < d; i += kBigThreads) {
            s.L[i] = colsp[ub + i];
            s.own[i] = 0;
        }
        __syncthreads();
        const int32_t last = s.L[d - 1];
        // rows: warp per row, built in the warp's shared buffer, then written to the scratch
        for (int i = w; i < d; i += kBigWarps) {
            for (int x = l; x < W; x += 32) buf[x] = 0;
            __syncwarp();
            uint32_t hits_i = 0;
            if (i < d - 1) {
                const int32_t v = s.L[i];
                const int32_t next = s.L[i + 1];
                const int64_t e = offp[v + 1];
                int64_t b = offp[v];
                if (e - b > 64) b = warp_lower_bound(colsp, b, e, next);
                auto probe = [&](int32_t y, int64_t p) {
                    if (y >= next && y <= last) {
                        const int j = find_sorted(s.L, d, y);
                        if (j >= 0) {
                            atomicAdd(&te[p], 1u);
                            atomicOr(&buf[j >> 5], 1u << (j & 31));
                            atomicAdd(&s.own[j], 1u);
                            ++hits_i;
                        }
                    }
                };
                probe_list(colsp, b, e, last, probe);
            }
            hits_i = warp_sum(hits_i);
            if (l == 0 && hits_i) atomicAdd(&s.own[i], hits_i);
            __syncwarp();
            for (int x = l; x < W; x += 32) R[(size_t)i * W + x] = buf[x];
            __syncwarp();
        }
        __syncthreads();  // every row is in the scratch
        uint64_t a_tri = 0, a_k4 = 0, a_paw = 0;
        for (int i = w; i < d - 1; i += kBigWarps) {
            const uint32_t* Ri = R + (size_t)i * W;
            for (int x = l; x < W; x += 32) buf[x] = Ri[x];
            __syncwarp();
            // the set bits of row i in chunks of 32 words (one word per lane), dealt to the lanes
            for (int c0 = 0; c0 < W; c0 += 32) {
                const uint32_t myw = c0 + l < W ? buf[c0 + l] : 0u;
                const int cnt_w = __popc(myw);
                int pre = cnt_w;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(kFull, pre, o);
                    if (l >= o) pre += y;
                }
                const int B = __shfl_sync(kFull, pre, 31);
                pre -= cnt_w;
                a_tri += (l == 0) ? (uint64_t)B : 0;
                for (int k0 = 0; k0 < B; k0 += 32) {
                    const int kk = k0 + l;
                    int o = 0;
#pragma unroll
                    for (int sft = 16; sft >= 1; sft >>= 1) {
                        const int e = __shfl_sync(kFull, pre, o + sft);
                        if (e <= kk) o += sft;
                    }
                    const uint32_t word = __shfl_sync(kFull, myw, o);
                    const int rank = kk - __shfl_sync(kFull, pre, o);
                    if (kk < B) {
                        const int j = ((c0 + o) << 5) + (int)__fns(word, 0, rank + 1);
                        uint32_t cnt = 0;
                        if (reuse) {  // the staged frontier of (u, L[j])
                            const uint32_t* Rj = R + (size_t)j * W;
                            for (int x = c0 + o; x < W; ++x) cnt += __popc(buf[x] & Rj[x]);
                        } else {      // recompute from N+(L[j]) in global memory
                            const int32_t wv = s.L[j];
                            for (int64_t p = offp[wv], pe = offp[wv + 1]; p < pe; ++p) {
                                const int32_t y = colsp[p];
                                if (y > last) break;
                                const int jj = find_sorted(s.L, d, y);
                                if (jj >= 0 && ((buf[jj >> 5] >> (jj & 31)) & 1u)) ++cnt;
                            }
                        }
                        a_k4 += cnt;
                    }
                }
            }
            __syncwarp();
        }
        for (int i = threadIdx.x; i < d; i += kBigThreads) {
            const uint32_t o = s.own[i];
            if (o) {
                atomicAdd(&te[ub + i], o);
                a_paw += (uint64_t)o * (uint64_t)deg[s.L[i]];
            }
        }
        a_paw += a_tri * (uint64_t)deg[u];
        if (reuse) hits += a_tri;
        __syncthreads();
        if (sink.batch()) {
            const uint64_t t1 = block_sum_u64(a_tri, s.red);
            const uint64_t t2 = block_sum_u64(a_k4, s.red);
            const uint64_t t3 = block_sum_u64(a_paw, s.red);
            if (threadIdx.x == 0) {
                sink_add(sink, u, G_T, t1);
                sink_add(sink, u, G_K4, t2);
                sink_add(sink, u, G_PAWSUM, t3);
            }
        } else {
            tri += a_tri;
            k4 += a_k4;
            paw += a_paw;
        }
    }
    flush_block(sink, tri, k4, paw, hits, s.red);
}

// ---------------------------------------------------------------------------------------------
// Fallback for out-degree > kCtaMax (1024): per out-arc (u, v) the frontier S_uv = N+(u) n N+(v) is
// materialised (compaction) in a per-warp global buffer, then reused for the 4-clique extension.
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ int64_t lb_global(const int32_t* __restrict__ a, int64_t lo, int64_t hi, int32_t y) {
    while (lo < hi) {
        int64_t mid = (lo + hi) >> 1;
        if (a[mid] < y) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

__global__ void __launch_bounds__(256) k_tri_fallback(const int64_t* __restrict__ offp,
                                                      const int32_t* __restrict__ colsp,
                                                      const int32_t* __restrict__ deg,
                                                      const int32_t* __restrict__ q_fb,
                                                      const unsigned long long* __restrict__ cnt_fb,
                                                      int32_t* __restrict__ scratch, int64_t scratch_per_warp,
                                                      uint32_t* __restrict__ te, Sink sink) {
    grid_begin();
    __shared__ uint64_t red[32];
    const int w = threadIdx.x >> 5, l = lane_id();
    const int nw = blockDim.x >> 5;
    int32_t* S = scratch + ((int64_t)blockIdx.x * nw + w) * scratch_per_warp;
    const int64_t nq = (int64_t)*cnt_fb;
    uint64_t tri = 0, k4 = 0, paw = 0;
    for (int64_t k = blockIdx.x; k < nq; k += gridDim.x) {
        const int32_t u = q_fb[k];
        const int64_t ub = offp[u], ue = offp[u + 1];
        const uint64_t du = (uint64_t)deg[u];
        const uint64_t tri0 = tri, k40 = k4, paw0 = paw;
        for (int64_t a = ub + w; a < ue; a += nw) {  // warp per out-arc (u, v)
            const int32_t v = colsp[a];
            const int64_t b = offp[v], e = offp[v + 1];
            const uint64_t dv = (uint64_t)deg[v];
            int64_t ns = 0;
            uint32_t own_uv = 0;
            for (int64_t p0 = b; p0 < e; p0 += 32) {
                const int64_t p = p0 + l;
                bool hit = false;
                int32_t y = kInf;
                int64_t pu = 0;
                if (p < e) {
                    y = colsp[p];
                    pu = lb_global(colsp, ub, ue, y);
                    hit = pu < ue && colsp[pu] == y;
                }
                const uint32_t hm = __ballot_sync(kFull, hit);
                if (hit) {
                    atomicAdd(&te[p], 1u);   // (v, y)
                    atomicAdd(&te[pu], 1u);  // (u, y)
                    S[ns + __popc(hm & lanemask_lt())] = y;
                    paw += du + dv + (uint64_t)deg[y];
                }
                ns += __popc(hm);
                own_uv += __popc(hm);
            }
            if (l == 0 && own_uv) atomicAdd(&te[a], own_uv);
            tri += (l == 0) ? (uint64_t)own_uv : 0;
            __syncwarp();
            // 4-cliques through (u, v): pairs w < x of S_uv with x in N+(w)
            for (int64_t s1 = 0; s1 < ns; ++s1) {
                const int32_t wv = S[s1];
                const int64_t wb = offp[wv], we = offp[wv + 1];
                for (int64_t s2 = s1 + 1 + l; s2 < ns; s2 += 32) {
                    const int32_t xv = S[s2];
                    const int64_t px = lb_global(colsp, wb, we, xv);
                    k4 += (px < we && colsp[px] == xv) ? 1 : 0;
                }
            }
            __syncwarp();
        }
        if (sink.batch()) {  // this anchor's part goes to its graph; the running sums stay unchanged
            const uint64_t t1 = block_sum_u64(tri - tri0, red);
            const uint64_t t2 = block_sum_u64(k4 - k40, red);
            const uint64_t t3 = block_sum_u64(paw - paw0, red);
            if (threadIdx.x == 0) {
                sink_add(sink, u, G_T, t1);
                sink_add(sink, u, G_K4, t2);
                sink_add(sink, u, G_PAWSUM, t3);
            }
            tri = tri0;
            k4 = k40;
            paw = paw0;
        }
    }
    flush_block(sink, tri, k4, paw, 0, red);
}

// ---------------------------------------------------------------------------------------------
// Orbit statistics of the triangles and 4-cliques (orbits.cu), anchored like the counts, after t_e is final.
// With the symmetric bitmap of G[L], c_ij = |row_i n row_j| is the number of 4-cliques {u, L[i], L[j], .}, so
// every triangle (u, a = L[i], b = L[j]) at position p of colsp gives, in one visit,
//   per vertex: N9(u) += t_ab - 1, N9(a) += t_ub - 1, N9(b) += t_ua - 1 (t from t_e); 3 K4(u) += c_ij; and
//               2 K4(a), 2 K4(b) += c_ij over the anchors u (the 4-cliques on a with u lowest are the
//               triangles of G[L] through a: half of sum_j c_ij)
//   per edge:   e5 (sum of d - 2 of the third vertex) and e8 (sum of t - 1 of the other two edges) of its three
//               edges, e9 (twice the 4-cliques) of (a, b) += 2 c_ij and of (u, a), (u, b) += c_ij.
// What goes to L[j] is gathered in shared memory, 16 bits of the value to each of two words (at most 1024
// terms), and added to global memory once per anchor; only the (a, b) edge needs an atomic per triangle.
// (A warp per edge that walked the common neighbours per triangle took 13.2 ms on R-MAT scale 15.)
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ void split_add(uint32_t* lo, uint32_t* hi, int j, uint32_t v) {
    atomicAdd(&lo[j], v & 0xffffu);
    if (v >> 16) atomicAdd(&hi[j], v >> 16);
}
__device__ __forceinline__ uint64_t split_sum(const uint32_t* lo, const uint32_t* hi, int j) {
    return (uint64_t)lo[j] + ((uint64_t)hi[j] << 16);
}
__device__ __forceinline__ void add_u64(unsigned long long* p, uint64_t v) {
    if (v) atomicAdd(p, (unsigned long long)v);
}

// Warp-local anchors (2 <= d <= 32): every (row, key) pair searched once, its position kept in shared memory
// while the bitmap is completed.
constexpr int kOrbWarps = 8;

template <bool EDGE>
__global__ void __launch_bounds__(kOrbWarps * 32) k_orb_tri_warp(const int64_t* __restrict__ offp,
                                                                 const int32_t* __restrict__ colsp,
                                                                 const int32_t* __restrict__ deg,
                                                                 const uint32_t* __restrict__ te,
                                                                 const int32_t* __restrict__ q,
                                                                 const unsigned long long* __restrict__ cnt, OrbTri o) {
    grid_begin();
    __shared__ int32_t s_L[kOrbWarps][32], s_pos[kOrbWarps][32 * 31 / 2];
    __shared__ uint32_t s_row[kOrbWarps][32], s_k[kOrbWarps][32], s_t[kOrbWarps][32], s_d[kOrbWarps][32];
    __shared__ uint32_t s_lo[kOrbWarps][32], s_hi[kOrbWarps][32], s_lo2[kOrbWarps][32], s_hi2[kOrbWarps][32];
    const int w = threadIdx.x >> 5, l = lane_id();
    const int64_t nq = (int64_t)cnt[0];
    for (int64_t k = (int64_t)blockIdx.x * kOrbWarps + w; k < nq; k += (int64_t)gridDim.x * kOrbWarps) {
        const int32_t u = q[k];
        const int64_t ub = offp[u];
        const int d = (int)(offp[u + 1] - ub);
        const int32_t x = l < d ? colsp[ub + l] : 0;
        int64_t b = 0;
        int len = 0;
        if (l < d) {
            b = offp[x];
            len = (int)(offp[x + 1] - b);
        }
        s_L[w][l] = x;
        s_row[w][l] = s_k[w][l] = s_lo[w][l] = s_hi[w][l] = s_lo2[w][l] = s_hi2[w][l] = 0;
        s_t[w][l] = l < d ? te[ub + l] - 1u : 0u;  // used only where the edge has a triangle
        s_d[w][l] = l < d ? (uint32_t)deg[x] - 2u : 0u;
        __syncwarp();
        // pairs (i, j), i < j, flattened: row i's first pair is excl(i)
        const int npairs = l < d ? d - 1 - l : 0;
        int incl = npairs;
#pragma unroll
        for (int s = 1; s < 32; s <<= 1) {
            const int y = __shfl_up_sync(kFull, incl, s);
            if (l >= s) incl += y;
        }
        const int excl = incl - npairs;
        const int total = d * (d - 1) / 2;
        auto each_pair = [&](auto&& f) {
            for (int t0 = 0; t0 < total; t0 += 32) {
                const int t = t0 + l;
                int i = 0;
#pragma unroll
                for (int s = 16; s >= 1; s >>= 1) {
                    const int e = __shfl_sync(kFull, excl, i + s);
                    if (i + s < d && e <= t) i += s;
                }
                const int64_t rb = __shfl_sync(kFull, b, i);
                const int rl = __shfl_sync(kFull, len, i), e = __shfl_sync(kFull, excl, i);
                if (t < total) f(t, i, i + 1 + (t - e), rb, rl);
            }
        };
        each_pair([&](int t, int i, int j, int64_t rb, int rl) {
            const int64_t p = find_in_range(colsp, rb, rl, s_L[w][j]);
            s_pos[w][t] = p < 0 ? -1 : (int32_t)(p - rb);
            if (p >= 0) {
                atomicOr(&s_row[w][i], 1u << j);
                atomicOr(&s_row[w][j], 1u << i);
            }
        });
        __syncwarp();
        uint64_t n9u = 0, k3u = 0;
        const uint32_t du2 = (uint32_t)deg[u] - 2u;
        each_pair([&](int t, int i, int j, int64_t rb, int) {
            const int32_t rel = s_pos[w][t];
            if (rel < 0) return;
            const int64_t p = rb + rel;
            const uint32_t c = (uint32_t)__popc(s_row[w][i] & s_row[w][j]);
            const uint32_t ti = s_t[w][i], tj = s_t[w][j], tp = te[p] - 1u;
            if (c) {
                atomicAdd(&s_k[w][i], c);
                atomicAdd(&s_k[w][j], c);
            }
            if (EDGE) {
                split_add(s_lo[w], s_hi[w], i, s_d[w][j]);
                split_add(s_lo[w], s_hi[w], j, s_d[w][i]);
                split_add(s_lo2[w], s_hi2[w], i, tp);
                split_add(s_lo2[w], s_hi2[w], i, tj);
                split_add(s_lo2[w], s_hi2[w], j, tp);
                split_add(s_lo2[w], s_hi2[w], j, ti);
                add_u64(&o.e5[p], du2);
                add_u64(&o.e8[p], (uint64_t)ti + tj);
                add_u64(&o.e9[p], 2ull * c);
            } else {
                split_add(s_lo[w], s_hi[w], i, tj);
                split_add(s_lo[w], s_hi[w], j, ti);
                n9u += tp;
                k3u += c;
            }
        });
        __syncwarp();
        if (l < d) {
            if (EDGE) {
                add_u64(&o.e5[ub + l], split_sum(s_lo[w], s_hi[w], l));
                add_u64(&o.e8[ub + l], split_sum(s_lo2[w], s_hi2[w], l));
                add_u64(&o.e9[ub + l], s_k[w][l]);
            } else {
                add_u64(&o.n9[x], split_sum(s_lo[w], s_hi[w], l));
                add_u64(&o.tau6[x], 3ull * s_k[w][l]);
            }
        }
        if (!EDGE) {
            n9u = warp_sum(n9u);
            k3u = warp_sum(k3u);
            if (l == 0) {
                add_u64(&o.n9[u], n9u);
                add_u64(&o.tau6[u], 2 * k3u);
            }
        }
        __syncwarp();
    }
}

template <int DMAX>
struct OrbSmem {
    CtaSmem<DMAX> c;
    uint32_t t[DMAX], d[DMAX];                            // t_e - 1 of (u, L[i]) and deg - 2 of L[i]
    uint32_t lo[DMAX], hi[DMAX], lo2[DMAX], hi2[DMAX];
};

template <int DMAX, int THREADS, bool EDGE>
__global__ void __launch_bounds__(THREADS) k_orb_tri_cta(const int64_t* __restrict__ offp,
                                                         const int32_t* __restrict__ colsp,
                                                         const int32_t* __restrict__ deg, const uint32_t* __restrict__ te,
                                                         const int32_t* __restrict__ q, int64_t n, int cls,
                                                         const unsigned long long* __restrict__ cnt,
                                                         unsigned long long* __restrict__ ticket, OrbTri o) {
    grid_begin();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    OrbSmem<DMAX>& s = *reinterpret_cast<OrbSmem<DMAX>*>(smem_raw);
    __shared__ int64_t s_item;
    constexpr int NW = THREADS / 32;
    const int w = threadIdx.x >> 5, l = lane_id();
    const int64_t nq = (int64_t)cnt[1];
    FilterChoice fc;
    for (;;) {
        if (threadIdx.x == 0) s_item = (int64_t)atomicAdd(ticket, 1ull);
        __syncthreads();
        const int64_t k = s_item;
        __syncthreads();
        if (k >= nq) break;
        const int32_t u = q[n - 1 - k];
        const int64_t ub = offp[u];
        const int d = (int)(offp[u + 1] - ub);
        if (tri_class(d, 32, kCtaMax, kBigMax) != cls) continue;
        const int W = (d + 31) >> 5;
        const int WS = W | 1;
        for (int i = threadIdx.x; i < d; i += THREADS) {
            s.t[i] = te[ub + i] - 1u;
            s.d[i] = (uint32_t)deg[colsp[ub + i]] - 2u;
            s.lo[i] = s.hi[i] = s.lo2[i] = s.hi2[i] = 0;
        }
        const CtaAnchor A = stage_anchor<DMAX, THREADS, false>(s.c, offp, colsp, ub, d, WS, kInf);
        for (int i = w; i < d - 1; i += NW)
            walk_row<DMAX, false>(s.c, A, offp, colsp, i, fc, [&](int j, int64_t) {
                atomicOr(&s.c.R[i * WS + (j >> 5)], 1u << (j & 31));
                atomicOr(&s.c.R[j * WS + (i >> 5)], 1u << (i & 31));
            });
        __syncthreads();
        uint64_t n9u = 0, k3u = 0;
        const uint32_t du2 = (uint32_t)deg[u] - 2u;
        for (int i = w; i < d - 1; i += NW) {
            const uint32_t* Ri = &s.c.R[i * WS];
            const uint32_t ti = s.t[i];
            uint64_t a5 = 0, a8 = 0;  // to L[i]: N9, or e5 and e8
            uint32_t ki = 0;
            walk_row<DMAX, false>(s.c, A, offp, colsp, i, fc, [&](int j, int64_t p) {
                const uint32_t* Rj = &s.c.R[j * WS];
                uint32_t c = 0;
                for (int y = 0; y < W; ++y) c += __popc(Ri[y] & Rj[y]);
                const uint32_t tj = s.t[j], tp = te[p] - 1u;
                if (c) atomicAdd(&s.c.own[j], c);
                ki += c;
                if (EDGE) {
                    a5 += s.d[j];
                    a8 += (uint64_t)tp + tj;
                    split_add(s.lo, s.hi, j, s.d[i]);
                    split_add(s.lo2, s.hi2, j, tp);
                    split_add(s.lo2, s.hi2, j, ti);
                    add_u64(&o.e5[p], du2);
                    add_u64(&o.e8[p], (uint64_t)ti + tj);
                    add_u64(&o.e9[p], 2ull * c);
                } else {
                    a5 += tj;
                    split_add(s.lo, s.hi, j, ti);
                    n9u += tp;
                }
            });
            if (!EDGE) k3u += ki;
            ki = warp_sum(ki);
            a5 = warp_sum(a5);
            if (EDGE) a8 = warp_sum(a8);
            if (l == 0) {
                if (ki) atomicAdd(&s.c.own[i], ki);
                if (EDGE) {
                    add_u64(&o.e5[ub + i], a5);
                    add_u64(&o.e8[ub + i], a8);
                } else {
                    add_u64(&o.n9[s.c.L[i]], a5);
                }
            }
        }
        __syncthreads();
        for (int i = threadIdx.x; i < d; i += THREADS) {
            if (EDGE) {
                add_u64(&o.e5[ub + i], split_sum(s.lo, s.hi, i));
                add_u64(&o.e8[ub + i], split_sum(s.lo2, s.hi2, i));
                add_u64(&o.e9[ub + i], s.c.own[i]);
            } else {
                add_u64(&o.n9[s.c.L[i]], split_sum(s.lo, s.hi, i));
                add_u64(&o.tau6[s.c.L[i]], 3ull * s.c.own[i]);
            }
        }
        if (!EDGE) {
            n9u = block_sum_u64(n9u, s.c.red);
            k3u = block_sum_u64(k3u, s.c.red);
            if (threadIdx.x == 0) {
                add_u64(&o.n9[u], n9u);
                add_u64(&o.tau6[u], 2 * k3u);
            }
        }
        __syncthreads();  // the shared arrays are read before the next anchor fills them
    }
}

template <int DMAX, int THREADS, bool EDGE>
harp_status launch_orb_cta(const harp_csr* g, Workspace& ws, int cls, int ticket_slot, int per_sm, const OrbTri& o,
                           cudaStream_t s) {
    const size_t smem = sizeof(OrbSmem<DMAX>);
    HARP_CK(cudaFuncSetAttribute(k_orb_tri_cta<DMAX, THREADS, EDGE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    launch(k_orb_tri_cta<DMAX, THREADS, EDGE>, num_sms() * per_sm, THREADS, smem, s, ws.offp, ws.colsp, ws.deg, ws.te,
           ws.q_tri, g->n, cls, (const unsigned long long*)&ws.acc[Q_TRI_WARP],
           (unsigned long long*)&ws.acc[ticket_slot], o);
    HARP_LAUNCHED();
    return HARP_OK;
}

template <bool EDGE>
harp_status orbit_tiers(const harp_csr* g, Workspace& ws, const OrbTri& o, int64_t dmax, cudaStream_t s) {
    launch(k_orb_tri_warp<EDGE>, num_sms() * 8, kOrbWarps * 32, 0, s, ws.offp, ws.colsp, ws.deg, ws.te, ws.q_tri,
           (const unsigned long long*)&ws.acc[Q_TRI_WARP], o);
    HARP_LAUNCHED();
    if (dmax > 32) HARP_TRY((launch_orb_cta<kCta1, 256, EDGE>(g, ws, 1, T_TRI_S, 5, o, s)));
    if (dmax > kCta1) HARP_TRY((launch_orb_cta<kCta2, 256, EDGE>(g, ws, 2, T_TRI_M, 3, o, s)));
    if (dmax > kCta2) HARP_TRY((launch_orb_cta<kCtaMax, 512, EDGE>(g, ws, 3, T_TRI_L, 1, o, s)));
    return HARP_OK;
}

template <int DMAX, int THREADS, int MINB, bool BS>
harp_status launch_cta(const harp_csr* g, Workspace& ws, int cls, int ticket_slot, int wmax, int cmax, int bmax,
                       bool reuse, cudaStream_t s) {
    const size_t smem = sizeof(CtaSmem<DMAX>);
    HARP_CK(cudaFuncSetAttribute(k_tri_cta<DMAX, THREADS, MINB, BS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem));
    launch(k_tri_cta<DMAX, THREADS, MINB, BS>, num_sms() * MINB, THREADS, smem, s, ws.offp, ws.colsp, ws.deg, ws.q_tri,
           g->n, cls, wmax, cmax, bmax, reuse, (const unsigned long long*)&ws.acc[Q_TRI_WARP],
           (unsigned long long*)&ws.acc[ticket_slot], ws.ginfo,
           ws.core && reuse ? reinterpret_cast<const uint32_t*>(ws.rev) : nullptr, ws.te, Sink{ws.acc, ws.gid,
           ws.accG});
    HARP_LAUNCHED();
    return HARP_OK;
}

// The four staged tiers, each with its bin's membership probe (plan.tri_probe_bin[k]: bsearch or hash).
harp_status launch_tiers(const harp_csr* g, Workspace& ws, int wmax, int cmax, int bmax, bool reuse,
                         const uint8_t* probe_bin, int64_t dmax, cudaStream_t s) {
    const Sink sink{ws.acc, ws.gid, ws.accG};
    const bool bs0 = probe_bin[0] == HARP_PROBE_BSEARCH, bs1 = probe_bin[1] == HARP_PROBE_BSEARCH;
    const bool bs2 = probe_bin[2] == HARP_PROBE_BSEARCH, bs3 = probe_bin[3] == HARP_PROBE_BSEARCH;
    const unsigned wgrid = (unsigned)num_sms() * 4;
    const unsigned long long* qcnt = (const unsigned long long*)&ws.acc[Q_TRI_WARP];
    if (bs0) launch(k_tri_warp<true>, wgrid, kWarpThreads, 0, s, ws.offp, ws.colsp, ws.deg, ws.q_tri, qcnt, reuse,
                    ws.te, sink);
    else launch(k_tri_warp<false>, wgrid, kWarpThreads, 0, s, ws.offp, ws.colsp, ws.deg, ws.q_tri, qcnt, reuse, ws.te,
                sink);
    HARP_LAUNCHED();
    HARP_CK(prof_mark(s, SEG_TRI_WARP));
    // tiers that the largest possible out-degree does not reach have no anchors
    if (dmax > wmax) {
        if (bs1) HARP_TRY((launch_cta<kCta1, kCta1Threads, kCta1Blocks, true>(g, ws, 1, T_TRI_S, wmax, cmax, bmax, reuse, s)));
        else HARP_TRY((launch_cta<kCta1, kCta1Threads, kCta1Blocks, false>(g, ws, 1, T_TRI_S, wmax, cmax, bmax, reuse, s)));
    }
    HARP_CK(prof_mark(s, SEG_TRI_CTA_S));
    if (dmax > kCta1) {
        if (bs2) HARP_TRY((launch_cta<kCta2, 256, 4, true>(g, ws, 2, T_TRI_M, wmax, cmax, bmax, reuse, s)));
        else HARP_TRY((launch_cta<kCta2, 256, 4, false>(g, ws, 2, T_TRI_M, wmax, cmax, bmax, reuse, s)));
    }
    if (dmax > kCta2) {
        if (bs3) HARP_TRY((launch_cta<kCtaMax, 1024, 1, true>(g, ws, 3, T_TRI_L, wmax, cmax, bmax, reuse, s)));
        else HARP_TRY((launch_cta<kCtaMax, 1024, 1, false>(g, ws, 3, T_TRI_L, wmax, cmax, bmax, reuse, s)));
    }
    HARP_CK(prof_mark(s, SEG_TRI_CTA_L));
    return HARP_OK;
}

}  // namespace

int64_t max_out_degree(const harp_csr* g) {
    int64_t dmax = 1;
    while (dmax * dmax < 2 * g->m) ++dmax;
    return dmax > g->max_deg ? g->max_deg : dmax;
}

harp_status orbit_triangles(const harp_csr* g, Workspace& ws, const OrbTri& o, cudaStream_t s) {
    // the tickets of the triangle pass (slots T_TRI_S .. T_TRI_M) start again
    HARP_CK(cudaMemsetAsync(&ws.acc[T_TRI_S], 0, sizeof(uint64_t) * (T_TRI_M - T_TRI_S + 1), s));
    const int64_t dmax = max_out_degree(g);
    return o.n9 ? orbit_tiers<false>(g, ws, o, dmax, s) : orbit_tiers<true>(g, ws, o, dmax, s);
}

// acc[Q_TRI_WARP], acc[Q_TRI_CTA] hold the queue lengths, acc[T_TRI_*] the CTA tickets (all cleared
// with the accumulators before the count).
harp_status count_triangles_k4(const harp_csr* g, Workspace& ws, const harp_plan& plan, cudaStream_t s) {
    const int64_t n = g->n;
    if (n == 0 || g->m == 0) return HARP_OK;  // no marks: the segments read as zero
    const int wmax = (int)plan.tri_warp_max;  // normalised: 1..32
    const int cmax = (int)plan.tri_cta_max;   // normalised: 1..kCtaMax
    const int bmax = (int)plan.tri_big_max;   // normalised: 1..kBigMax
    const bool reuse = !(plan.flags & HARP_PLAN_NO_REUSE);
    unsigned long long* cnt = (unsigned long long*)&ws.acc[Q_TRI_WARP];
    int64_t blocks = (n + 255) / 256;
    if (blocks > (int64_t)num_sms() * 16) blocks = (int64_t)num_sms() * 16;
    unsigned long long* cnt_fb = (unsigned long long*)&ws.acc[Q_TRI_FB];
    unsigned long long* cnt_big = (unsigned long long*)&ws.acc[Q_TRI_BIG];
    launch(k_tri_classify, (unsigned)blocks, 256, 0, s, ws.dplus, n, ws.own_lo, ws.own_hi, wmax, cmax, bmax, ws.q_tri,
           ws.q_mid, cnt, cnt_fb, cnt_big);
    HARP_LAUNCHED();
    const Sink sink{ws.acc, ws.gid, ws.accG};
    const int64_t dmax = max_out_degree(g);
    HARP_TRY(launch_tiers(g, ws, wmax, cmax, bmax, reuse, plan.tri_probe_bin, dmax, s));
    // the largest possible out-degree is bounded by sqrt(2m) and by the maximum degree
    if (dmax > cmax && bmax > cmax) {  // global-staged tier: one block per SM, scratch of kBigMax rows
        const size_t bytes = (size_t)num_sms() * kBigMax * kBigWords * sizeof(uint32_t);
        uint32_t* scratch = nullptr;
        HARP_CK(cudaMallocAsync((void**)&scratch, bytes, s));
        const size_t smem = sizeof(BigSmem);
        cudaError_t e = cudaFuncSetAttribute(k_tri_big, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e == cudaSuccess) {
            launch(k_tri_big, num_sms(), kBigThreads, smem, s, ws.offp, ws.colsp, ws.deg, ws.q_mid + n, cnt_big,
                   (unsigned long long*)&ws.acc[T_TRI_BIG], reuse, scratch, ws.te, sink);
            note_launch();
            e = cudaGetLastError();
        }
        cudaFreeAsync(scratch, s);
        if (e != cudaSuccess) {
            record_cuda_error(e);
            return HARP_ECUDA;
        }
    }
    // fallback: per-warp frontier buffers of the largest possible out-degree
    if (dmax > cmax && dmax > bmax) {
        const int fb_blocks = num_sms();
        const int64_t per_warp = dmax + 32;
        const size_t bytes = (size_t)fb_blocks * 8 * (size_t)per_warp * sizeof(int32_t);
        int32_t* scratch = nullptr;
        HARP_CK(cudaMallocAsync((void**)&scratch, bytes, s));
        launch(k_tri_fallback, fb_blocks, 256, 0, s, ws.offp, ws.colsp, ws.deg, ws.q_mid, cnt_fb, scratch, per_warp,
               ws.te, sink);
        note_launch();
        cudaError_t e = cudaGetLastError();
        cudaFreeAsync(scratch, s);
        if (e != cudaSuccess) {
            record_cuda_error(e);
            return HARP_ECUDA;
        }
    }
    HARP_CK(prof_mark(s, SEG_TRI_FALLBACK));
    return HARP_OK;
}

}  // namespace harp
