// Step a5: the ordered-wedge anchor (Section III-B) and non-induced 4-cycles.
//
// In rank order, every 4-cycle has a unique top vertex u; its opposite corner x and both middle
// vertices w1, w2 rank below u.  For a root u, an ordered wedge is u - w - x with w in N-(u) and
// x in N(w), x < u; because rows are sorted in rank order, the x of one w are a contiguous range of
// w's row ending at pos_w(u), the position of u in that row.  With cnt(x) = number of wedges ending
// in x, the root contributes sum_x C(cnt(x), 2) 4-cycles; each increment adds the counter's previous
// value, which sums to the same total without a second pass.
//
// Two bounds shape the work: cnt(x) <= d(x) (every wedge into x uses a distinct neighbour of x) and
// cnt(x) <= d-(u).  Rank order sorts each graph's vertices by degree, so inside a graph's rank range
//   * x of degree 1 never complete a cycle: x runs over [n1, u) with n1 the graph's first rank of
//     degree >= 2, and every row's segment starts at fpos[w] (its first neighbour of degree >= 2);
//   * a dense counter for x needs only as many bits as d(x) has, so the x-range splits into bands
//     by degree (d <= 7, 15, 31, 63, 255, 65535, larger) with 3-, 4-, 5-, 6-, 8-, 16- and 32-bit
//     counters packed floor(32 / bits) to a word.  The bands cut into windows of 48-100 KiB of
//     counters form a fixed grid per graph, so the row position of every grid boundary is computed
//     once per row (bpos) instead of being searched for every (root, lower neighbour, window).
// pos_w(u) itself is computed once per lower arc (rev, as the segment length) by a fully parallel pass.
//
// The frontier (the set of x) is not an induced class: whether u ~ x or w1 ~ w2 holds decides
// whether the cycle is induced, a diamond or part of a 4-clique; the closure resolves that mix
// (Section III-C explains why a frontier alone must not be reused as an induced state).
//
// Work per root W(u) = sum_{w in N-(u)} (pos_w(u) - fpos[w]) picks the execution mode:
//   W <= warp_max   one warp, hash table of 1024 slots in shared memory (warp-local mode)
//   W <= mid_max    a block of four warps, hash table of 4096 slots (the middle tier: roots with few wedges
//                   spread over many windows would otherwise cost a whole window pass per window)
//   W <= 16384      the wide tier, where two or more windows lie below the root: hash tables of 16384 and 32768
//                   slots
//   larger          one block per (root, grid window): dense packed counters in shared memory
//                   (CTA mode); lower neighbours are handed to warps in groups of 32, heaviest first,
//                   and segments of 2048+ elements are split across all warps of the block.  The
//                   window (100, 64 or 48 KiB) sets how many blocks share an SM (2, 3 or 4).
#include <type_traits>

#include "harp_internal.cuh"

namespace harp {
namespace {

constexpr int32_t kEmpty = -1;
// Window sizes by resident blocks per SM (plan.c4_window_bytes picks one): 200 KiB for one
// 1024-thread block, 100 KiB at 2 blocks of 512 threads (the default), 64 KiB at 3, 48 KiB at 4
// (counters plus ~3 KiB of static and reserved shared memory per block).  On R-MAT scale 20 the
// 200 KiB window measured 15.7 ms against 13.2 ms for 100 KiB: its fewer (root, window) items do not
// pay for the 32-warp end-of-item barrier there; it is kept for graphs whose x-range spans many windows.
constexpr int kWinWords1 = 51200;
constexpr int kWinWords2 = 25600;
constexpr int kWinWords3 = 16384;
constexpr int kWinWords4 = 12288;
__host__ __device__ constexpr int win_words(int minb) {
    return minb == 1 ? kWinWords1 : (minb == 2 ? kWinWords2 : (minb == 3 ? kWinWords3 : kWinWords4));
}
__host__ __device__ constexpr int win_threads(int minb) { return minb == 1 ? 1024 : 512; }
constexpr int kSmallThreads = 256;
constexpr int kSmallWarps = kSmallThreads / 32;
constexpr int kSmallSlots = 1024;            // per-warp hash table of the light roots (W <= 512)
constexpr int kMidSlots = 4096;              // hash table of the middle tier (W <= 2048)
constexpr int kMidWarps = 4;                 // warps of the block that takes a middle root
constexpr int kWideSlots = 16384;            // hash tables of the wide tier: W <= 8192,
constexpr int kWideWarps = 16;
constexpr int kWide2Slots = 32768;           // and W <= 16384
constexpr int kWide2Warps = 32;
constexpr int kWideBits = 10;                // its counts: at most 1,024 lower neighbours
constexpr int kLong = 32;                    // segments this long are read warp-coalesced
constexpr int kSplit = 2048;                 // segments this long are split across the block
constexpr int kSplitQ = 128;                 // split-queue capacity per window item
constexpr int kChunk = 1024;                 // elements per split chunk

// ---------------------------------------------------------------------------------------------
// Per-graph band and grid geometry (ginfo: kGInfo int64 per graph).
// ---------------------------------------------------------------------------------------------
// The window size is a template parameter (WORDS 32-bit words of counters) of every kernel that
// computes window geometry, so each size is its own compiled instance with constant spans.
// The x-range [n1, hi) splits into bands by degree, each with the narrowest counter that is exact
// there (cnt(x) <= d(x) < 2^width): a band of width b packs floor(32 / b) counters into a word.
// ginfo slots: GI_HI, GI_NWIN, then the band starts GI_BAND + b (b = 0 .. kBands - 1; band b
// ends where band b + 1 starts, the last band at GI_HI).  GI_N1 = GI_BAND: the first band starts at n1.
constexpr int kBands = 7;
enum : int { GI_HI = 0, GI_NWIN = 1, GI_BAND = 2, GI_N1 = GI_BAND };
static_assert(GI_BAND + kBands <= GI_CORE && kBands < 32, "ginfo slots; one search per lane");

// counter bits of band b and the largest degree the band holds
__host__ __device__ constexpr int band_width(int b) {
    return b == 0 ? 3 : (b == 1 ? 4 : (b == 2 ? 5 : (b == 3 ? 6 : (b == 4 ? 8 : (b == 5 ? 16 : 32)))));
}
__host__ __device__ constexpr int band_per_word(int b) { return 32 / band_width(b); }
__host__ __device__ constexpr int32_t band_max_degree(int b) {
    return band_width(b) >= 31 ? INT32_MAX : (int32_t)((1u << band_width(b)) - 1u);
}

// first position in [lo, hi) of the ascending deg above t, by a whole warp (32 probes a round)
__device__ __forceinline__ int64_t warp_first_above(const int32_t* __restrict__ deg, int64_t lo, int64_t hi, int32_t t) {
    const int l = lane_id();
    while (hi - lo > 32) {
        const int64_t step = (hi - lo + 31) >> 5;
        const int64_t i = lo + (int64_t)(l + 1) * step - 1;
        const uint32_t m = __ballot_sync(kFull, i >= hi || deg[i] > t);
        if (!m) return hi;
        lo += (int64_t)(__ffs(m) - 1) * step;
        hi = lo + step < hi ? lo + step : hi;
    }
    const uint32_t m = __ballot_sync(kFull, lo + l < hi && deg[lo + l] > t);
    return m ? lo + __ffs(m) - 1 : hi;
}

// x-values one window of band b covers: the window's words times counters per word
template <int WORDS>
__device__ __forceinline__ int64_t span_of(int b) { return (int64_t)WORDS * band_per_word(b); }

__device__ __forceinline__ int64_t band_end(const int64_t* gi, int b) {
    return b + 1 < kBands ? gi[GI_BAND + b + 1] : gi[GI_HI];
}

// window j of the graph's grid: [xlo, xhi) and its band; false if j is past the grid.  The band loops
// are unrolled, so every span is a compile-time constant.
template <int WORDS>
__device__ __forceinline__ bool grid_window(const int64_t* gi, int64_t j, int64_t& xlo, int64_t& xhi, int& band) {
#pragma unroll
    for (int b = 0; b < kBands; ++b) {
        const int64_t bs = gi[GI_BAND + b], be = band_end(gi, b);
        if (be <= bs) continue;
        const int64_t S = span_of<WORDS>(b);
        const int64_t nb = (be - bs + S - 1) / S;
        if (j < nb) {
            xlo = bs + j * S;
            xhi = xlo + S < be ? xlo + S : be;
            band = b;
            return true;
        }
        j -= nb;
    }
    return false;
}

// number of grid windows that intersect [n1, u)
template <int WORDS>
__device__ __forceinline__ int64_t windows_below(const int64_t* gi, int64_t u) {
    int64_t total = 0;
#pragma unroll
    for (int b = 0; b < kBands; ++b) {
        const int64_t bs = gi[GI_BAND + b], be = band_end(gi, b);
        const int64_t e = be < u ? be : u;
        if (e <= bs) continue;
        const int64_t S = span_of<WORDS>(b);
        total += (e - bs + S - 1) / S;
    }
    return total;
}

// Windows intersecting [n1, u) when bands are merged upwards by mask (bit b set: band b joins band
// b + 1 and takes its wider counters).  st[0 .. kBands] are the unmerged band starts and hi.
template <int WORDS>
__device__ __forceinline__ int64_t merged_windows(const int64_t* st, unsigned mask, int64_t u) {
    int64_t total = 0, gs = st[0];
#pragma unroll
    for (int b = 0; b < kBands; ++b) {
        if (b + 1 < kBands && ((mask >> b) & 1u)) continue;  // the group goes on into band b + 1
        const int64_t e = st[b + 1] < u ? st[b + 1] : u;
        const uint32_t S = (uint32_t)WORDS * (uint32_t)band_per_word(b);  // constant once unrolled
        if (e > gs) total += ((uint32_t)(e - gs) + (S - 1u)) / S;  // ranks and spans fit 31 bits
        gs = st[b + 1];
    }
    return total;
}

constexpr int kMergeMasks = 1 << (kBands - 1);
constexpr int kMergeSamples = 64;
constexpr int kGinfoThreads = 128;
constexpr int kGinfoWarps = kGinfoThreads / 32;

// The graph's wedge core (c4core.cu), by one warp: ranks [lo, gend), arcs [alo, ahi) of the rank-order CSR.
// The core is the largest K = 2^10 .. 2^14 (at most half the graph) with
//   * deg >= K / 64 at the core's first rank: a core row's words then hold enough bits to beat walking
//     its list (R-MAT scale 15: 728 us a count at K / 64, 746 at K / 128; Chung-Lu with 500,000 vertices:
//     5.08 ms against 5.23 at K / 256; R-MAT 16 to 20 choose the same K with each),
//   * an eighth of the graph's arcs at core vertices, else the wedges are elsewhere (Barabasi-Albert,
//     100,000 vertices: 637 us with its core of 17 % of the arcs, 710 without; random geometric graphs
//     have about 0.1 %),
//   * K * K bits and K * K / 32 prefix counts in the graph's share of the region (4 bytes an arc and 64 a vertex).
__device__ __forceinline__ void choose_core(const int32_t* __restrict__ deg, const int64_t* __restrict__ off,
                                            int64_t lo, int64_t gend, int64_t* gi, uint64_t* acc) {
    const int l = lane_id();
    int64_t c0 = INT64_MAX, K = 0, base = 0;
    if (off) {  // uniform: a kernel argument
        const int64_t alo = off[lo], ahi = off[gend], ng = gend - lo;
        const int64_t b0 = (4 * alo + 64 * lo + 15) & ~(int64_t)15;
        const int64_t cap = 4 * ahi + 64 * gend - b0;
        bool ok = false;
        const int64_t k = (int64_t)1024 << l;
        if (l < 5 && ahi - alo >= 2 * kCoreMinM && 2 * k <= ng && 3 * k * k / 16 <= cap &&
            deg[gend - 1] >= kCoreMinMaxDeg)
            ok = (int64_t)deg[gend - k] >= k / 64 && 8 * (ahi - off[gend - k]) >= ahi - alo;
        const uint32_t m = __ballot_sync(kFull, ok);
        if (m) {
            K = (int64_t)1024 << (31 - __clz(m));
            c0 = gend - K;
            base = b0 / 4;
        }
    }
    if (l == 0) {
        gi[GI_CORE] = c0;
        gi[GI_CORE_K] = K;
        gi[GI_CORE_BASE] = base;
        if (K > 0) atomicAdd((unsigned long long*)&acc[A_CORE_ANY], 1ull);
    }
}

// One block per graph.  The x-range of a graph's grid is [n1, hi) intersected with [x_lo, x_hi) (a
// partitioned wedge block owns only the opposite vertices in that slice; a whole graph passes
// [0, INT64_MAX)).  A narrow band holding few vertices costs a partly filled window for every root
// that reaches past it, so bands may merge into the next wider one: each lane scores two merge masks by
// the windows of kMergeSamples roots spread evenly over the graph's ranks of degree >= 64 (the roots
// that take the windowed mode), each weighted by its degree; the cheapest mask (lowest on a tie) wins.
// The samples are dealt to the block's warps and the scores are integers: by one warp in FP64 the scoring
// took 55 us, a fifth of a whole count of a graph of 8,000 edges.
// merge = false keeps every band separate (mask 0).  off (nullptr: no core): see choose_core.
template <int WORDS>
__global__ void __launch_bounds__(kGinfoThreads) k_c4_ginfo(const int32_t* __restrict__ deg, int64_t n,
                                                            const int64_t* __restrict__ gbase, int64_t G, int64_t x_lo,
                                                            int64_t x_hi, bool merge, const int64_t* __restrict__ off,
                                                            int64_t* __restrict__ ginfo, uint64_t* __restrict__ acc) {
    grid_begin();
    __shared__ uint64_t s_score[kGinfoWarps][kMergeMasks];
    __shared__ int64_t s_rank[kBands + 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int64_t g = blockIdx.x; g < G; g += gridDim.x) {
        const int64_t lo = gbase ? gbase[g] : 0, gend = gbase ? gbase[g + 1] : n;
        int64_t* gi = ginfo + g * kGInfo;
        if (warp == kGinfoWarps - 1 && gend > lo) choose_core(deg, off, lo, gend, gi, acc);
        if (warp == kGinfoWarps - 1 && gend <= lo && lane == 0) {
            gi[GI_CORE] = INT64_MAX;
            gi[GI_CORE_K] = gi[GI_CORE_BASE] = 0;
        }
        auto clamp = [&](int64_t v) { return v < x_lo ? x_lo : (v > x_hi ? x_hi : v); };
        const int64_t hi = gend < x_hi ? gend : x_hi;
        // threshold 0: n1 (first rank of degree >= 2); b < kBands: the first rank above band b - 1's degrees
        // (band b's start); kBands: the first rank of degree >= 64.  A warp-wide search each.
        for (int b = warp; b <= kBands; b += kGinfoWarps) {
            const int64_t r = warp_first_above(deg, lo, gend, b == 0 ? 1 : (b < kBands ? band_max_degree(b - 1) : 63));
            if (lane == 0) s_rank[b] = r;
        }
        __syncthreads();
        int64_t n1 = clamp(s_rank[0]);
        n1 = n1 < hi ? n1 : hi;
        int64_t st[kBands + 1];
        st[0] = n1;
        st[kBands] = hi;
#pragma unroll
        for (int b = 1; b < kBands; ++b) {
            const int64_t r = clamp(s_rank[b]);
            st[b] = r > n1 ? (r < hi ? r : hi) : n1;
        }
        unsigned best_mask = 0;  // mask 0: every band separate
        if (merge && hi - n1 <= WORDS) {
            best_mask = kMergeMasks - 1;  // all in one window of 32-bit counters
        } else if (merge) {               // uniform over the block
            int64_t s0 = s_rank[kBands];
            if (s0 >= gend) s0 = lo;
            const int64_t span = gend - s0;  // samples u lie in [s0, gend); none for an empty graph
            constexpr int kPer = kMergeSamples / kGinfoWarps;  // this warp's samples, one per lane
            static_assert(kPer <= 32 && kMergeMasks == 64, "a sample and two masks per lane");
            const int64_t u_l = s0 + (span * (2 * (warp * kPer + lane) + 1)) / (2 * kMergeSamples);
            const uint32_t w_l = span > 0 && lane < kPer ? (uint32_t)deg[u_l] : 0u;
            uint64_t c[2] = {0, 0};
            for (int k = 0; k < kPer; ++k) {  // uniform over the warp: every lane shuffles
                const int64_t u = __shfl_sync(0xffffffffu, u_l, k);
                const uint32_t w = __shfl_sync(0xffffffffu, w_l, k);
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    c[h] += (uint64_t)w * (uint64_t)merged_windows<WORDS>(st, (unsigned)(lane + 32 * h), u);
            }
            s_score[warp][lane] = c[0];
            s_score[warp][lane + 32] = c[1];
            __syncthreads();
            if (warp == 0) {
                uint64_t best = 0;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    uint64_t v = 0;
#pragma unroll
                    for (int k = 0; k < kGinfoWarps; ++k) v += s_score[k][lane + 32 * h];
                    if (h == 0 || v < best) {
                        best = v;
                        best_mask = (unsigned)(lane + 32 * h);
                    }
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const uint64_t oc = __shfl_xor_sync(0xffffffffu, best, o);
                    const unsigned om = __shfl_xor_sync(0xffffffffu, best_mask, o);
                    if (oc < best || (oc == best && om < best_mask)) {
                        best = oc;
                        best_mask = om;
                    }
                }
            }
        }
        __syncthreads();  // the scores and ranks are read before the next graph's are written
        if (threadIdx.x == 0) {
#pragma unroll
            for (int b = 0; b + 1 < kBands; ++b)
                if ((best_mask >> b) & 1u) st[b + 1] = st[b];  // band b becomes empty, b + 1 starts at its start
            gi[GI_HI] = hi;
#pragma unroll
            for (int b = 0; b < kBands; ++b) gi[GI_BAND + b] = st[b];
            gi[GI_NWIN] = windows_below<WORDS>(gi, hi);
        }
    }
}

// fpos[w] = row position of w's first neighbour of degree >= 2 (the graph's n1 boundary); vinfo[w] (whole graphs) =
// what a lower arc to w needs, side by side: the start and length of N+(w), d-(w) - fpos[w], and the start of
// w's segments in cols.  Positions fit 32 bits.  Without ginfo every segment starts at its row (fpos = 0).
__global__ void __launch_bounds__(256) k_c4_fpos(const int64_t* __restrict__ off, const int32_t* __restrict__ cols,
                                                 const int64_t* __restrict__ offp, const int32_t* __restrict__ gid,
                                                 const int64_t* __restrict__ ginfo, int64_t n,
                                                 int32_t* __restrict__ fpos, uint4* __restrict__ vinfo) {
    grid_begin();
    for (int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; w < n; w += (int64_t)gridDim.x * blockDim.x) {
        const int64_t wb = off[w], we = off[w + 1];
        int32_t f = 0;
        if (ginfo) {
            const int64_t n1 = ginfo[(gid ? (int64_t)gid[w] : 0) * kGInfo + GI_N1];
            f = (int32_t)lower_bound_i32(cols + wb, we - wb, (int32_t)n1);
            fpos[w] = f;
        }
        if (vinfo) {
            const int64_t pb = offp[w];
            const int32_t dp = (int32_t)(offp[w + 1] - pb);
            vinfo[w] = make_uint4((uint32_t)pb, (uint32_t)dp, (uint32_t)((int32_t)(we - wb) - dp - f), (uint32_t)(wb + f));
        }
    }
}

// rev[a] = the wedge segment's length for every lower arc (u -> w) at position a of u's list: the position of u in
// w's row less fpos[w] (0 where u stands before it).
// Whole graph: the lower arcs of all rows are numbered through, row u's from off[u] - offp[u] on.  A warp takes a run
// of steps, a step being a lower arc or a row's end (runs of rows without lower arcs are as long as the graph's
// isolated vertices), a lane per arc: the rows are held by the lanes, 32 at a time, and an arc finds its row by a
// search over the lanes.  The position comes from N+(w): d-(w) + rank of u in N+(w).  (A thread per 16 arcs that
// walked its rows and gathered four arrays per arc: 2.59 ms on the batch of 4,096 graphs, 0.25 ms on the random
// geometric graph with 1,000,003 vertices.)  Core roots and roots of one lower neighbour need no length.
__device__ __forceinline__ int64_t lower_start(const int64_t* __restrict__ off, const int64_t* __restrict__ offp, int64_t u) {
    return off[u] - offp[u];
}

__global__ void __launch_bounds__(256) k_c4_seglen(const int64_t* __restrict__ off, const int32_t* __restrict__ cols,
                                                   const int64_t* __restrict__ offp, const int32_t* __restrict__ colsp,
                                                   const uint4* __restrict__ vinfo, const int32_t* __restrict__ gid,
                                                   const int64_t* __restrict__ ginfo, int64_t n, int run,
                                                   int32_t* __restrict__ rev) {
    grid_begin();
    const int l = lane_id();
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    // one graph: the arcs of its core rows come last and are left out
    int64_t rows = n;
    if (ginfo && !gid && ginfo[GI_CORE] < n) rows = ginfo[GI_CORE];
    // first row u in [lo, hi) whose place lower_start(u) + u lies past t, less one: the row of step t; 32 probes a round
    auto row_of = [&](int64_t lo, int64_t hi, int64_t t) {
        while (hi - lo > 1) {
            const int64_t step = (hi - lo + 31) >> 5;
            const int64_t p = lo + (int64_t)(l + 1) * step;
            const uint32_t m = __ballot_sync(kFull, p >= hi || lower_start(off, offp, p) + p > t);
            const int k = __ffs(m) - 1;  // lane 31 probes at or past hi
            lo += (int64_t)k * step;
            hi = lo + step < hi ? lo + step : hi;
        }
        return lo;
    };
    const int64_t steps = lower_start(off, offp, rows) + rows;  // row u: its lower arcs, then one step
    for (int64_t t0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * run; t0 < steps; t0 += nw * run) {
        const int64_t t1 = t0 + run < steps ? t0 + run : steps;
        int64_t r0 = row_of(0, rows, t0);
        const int64_t a1 = t1 - (t1 < steps ? row_of(r0, r0 + run + 1 < rows ? r0 + run + 1 : rows, t1) : rows);
        int64_t s = 0, e = 0, ob = 0;  // the lanes hold rows r0 .. r0 + 31
        uint32_t valid = 0;
        for (int64_t cur = t0 - r0; cur < a1; r0 += 32) {
            {
                const int64_t r = r0 + l;
                s = lower_start(off, offp, r < rows ? r : rows);
                e = lower_start(off, offp, r + 1 < rows ? r + 1 : rows);
                if (__shfl_sync(kFull, e, 31) <= cur) continue;  // no arc left in these rows
            }
            {
                const int64_t r = r0 + l;
                ob = r < rows ? off[r] : 0;
                bool want = r < rows && e - s >= (ginfo ? 2 : 1);
                if (want && gid) want = r < ginfo[(int64_t)gid[r] * kGInfo + GI_CORE];
                valid = __ballot_sync(kFull, want);
            }
            const int64_t end0 = __shfl_sync(kFull, e, 31);
            const int64_t end = end0 < a1 ? end0 : a1;
            for (int64_t b = cur; b < end; b += 32) {
                const int64_t a = b + l;
                int k = 0;  // last row with s <= a
#pragma unroll
                for (int sft = 16; sft >= 1; sft >>= 1) {
                    const int64_t v = __shfl_sync(kFull, s, k + sft);
                    if (v <= a) k += sft;
                }
                const int64_t pos = __shfl_sync(kFull, ob, k) + (a - __shfl_sync(kFull, s, k));
                if (a < end && ((valid >> k) & 1u)) {
                    const uint4 vi = __ldg(vinfo + cols[pos]);
                    const int32_t len = (int32_t)vi.z + (int32_t)lower_bound_i32(colsp + vi.x, vi.y, (int32_t)(r0 + k));
                    rev[pos] = len > 0 ? len : 0;
                }
            }
            cur = end;
        }
    }
}

// Partitioned blocks: the lists are the roots' lower lists (loff, lcols), the position is searched in w's row of
// the halo.  Each thread takes a run of kRevRun consecutive arcs.  arcs must equal loff[n].
constexpr int kRevRun = 16;

__global__ void __launch_bounds__(256) k_c4_seglen_rows(const int64_t* __restrict__ loff, const int32_t* __restrict__ lcols,
                                                        const int64_t* __restrict__ off, const int32_t* __restrict__ cols,
                                                        const int32_t* __restrict__ fpos, int64_t n, int64_t arcs,
                                                        int32_t* __restrict__ rev) {
    grid_begin();
    const int64_t runs = (arcs + kRevRun - 1) / kRevRun;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < runs; r += (int64_t)gridDim.x * blockDim.x) {
        const int64_t a0 = r * kRevRun;
        const int64_t a1 = a0 + kRevRun < arcs ? a0 + kRevRun : arcs;
        int64_t u = 0, hi = n;  // row of arc a0: last u with loff[u] <= a0
        while (hi - u > 1) {
            const int64_t mid = (u + hi) >> 1;
            if (loff[mid] <= a0) u = mid;
            else hi = mid;
        }
        int64_t ub = loff[u], ue = loff[u + 1];
        for (int64_t a = a0; a < a1; ++a) {
            if (a >= ue) {  // the row of arc a: last u with loff[u] <= a, searched outward from u + 1 (rows that the
                            // block does not own are empty and come in long runs)
                if (u + 1 >= n) return;  // only if arcs > loff[n]
                int64_t p = u + 1, step = 1;
                while (p + step < n && loff[p + step] <= a) {
                    p += step;
                    step <<= 1;
                }
                int64_t q = p + step < n ? p + step : n;  // loff[p] <= a < loff[q], or q = n
                while (q - p > 1) {
                    const int64_t mid = (p + q) >> 1;
                    if (loff[mid] <= a) p = mid;
                    else q = mid;
                }
                u = p;
                ub = loff[u];
                ue = loff[u + 1];
                if (a >= ue) return;  // only if arcs > loff[n]
            }
            if (ue - ub < 2) continue;  // only roots with d- >= 2
            const int32_t w = lcols[a];
            const int64_t pb = off[w];
            const int32_t len = (int32_t)lower_bound_i32(cols + pb, off[w + 1] - pb, (int32_t)u) - fpos[w];
            rev[a] = len > 0 ? len : 0;
        }
    }
}

// The boundary table keeps kGridCap entries per row: entry k is the row position of grid boundary
// k << s, where s is the smallest shift with ceil((nwin + 1) / 2^s) <= kGridCap (boundary i < nwin is
// the start of window i, boundary nwin the end of the grid).  s = 0 (every boundary) for grids of at
// most kGridCap - 1 windows; larger grids keep every 2^s-th boundary and the rest is found from the
// nearest kept one by a galloping search.
__device__ __forceinline__ int table_shift(int64_t nwin) {
    int sl = 0;
    while (((nwin + 1 + ((int64_t)1 << sl) - 1) >> sl) > kGridCap) ++sl;
    return sl;
}

// First index in [lo, hi) whose element is >= key (a sorted), searching outward from lo: cost grows
// with the log of the distance, not of the row length.
__device__ __forceinline__ int64_t gallop_i32(const int32_t* __restrict__ a, int64_t lo, int64_t hi, int32_t key) {
    if (lo >= hi || __ldg(a + lo) >= key) return lo;
    int64_t prev = lo, step = 1;  // a[prev] < key
    while (prev + step < hi && __ldg(a + prev + step) < key) {
        prev += step;
        step <<= 1;
    }
    int64_t l = prev + 1, r = prev + step < hi ? prev + step : hi;  // the answer lies in [l, r]
    while (l < r) {
        const int64_t mid = (l + r) >> 1;
        if (__ldg(a + mid) < key) l = mid + 1;
        else r = mid;
    }
    return l;
}

// The table pays for its 16 searches a row only where the windowed roots make many visits: it is built and used
// from kTableVisits visits per row on.  (R-MAT scale 20, whose core leaves few windowed roots: 0.20 ms to build,
// 0.15 ms saved; a random geometric graph has none; Chung-Lu with 2,000,000 vertices needs it.)
constexpr uint64_t kTableVisits = 8;
__device__ __forceinline__ bool table_pays(const uint64_t* acc, int64_t n) {
    return acc[C4_VISITS] >= kTableVisits * (uint64_t)n;
}

// bpos[w * kGridCap + k] = row position of grid boundary k << s (see table_shift)
template <int WORDS>
__global__ void k_c4_bpos(const int64_t* __restrict__ off, const int32_t* __restrict__ cols,
                          const int32_t* __restrict__ gid, const int64_t* __restrict__ ginfo, int64_t n,
                          const int32_t* __restrict__ fpos, const uint64_t* __restrict__ acc, int32_t* __restrict__ bpos) {
    grid_begin();
    if (!table_pays(acc, n)) return;
    const int64_t total = n * kGridCap;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t w = t / kGridCap;
        const int k = (int)(t % kGridCap);
        if (k == 0) {
            bpos[t] = fpos[w];
            continue;
        }
        const int64_t* gi = ginfo + (gid ? (int64_t)gid[w] : 0) * kGInfo;
        const int64_t nwin = gi[GI_NWIN];
        const int64_t i = (int64_t)k << table_shift(nwin);
        if (i > nwin) continue;
        int64_t bound = gi[GI_HI];
        if (i < nwin) {
            int64_t xhi;
            int band;
            grid_window<WORDS>(gi, i, bound, xhi, band);
        }
        const int64_t wb = off[w];
        bpos[t] = (int32_t)lower_bound_i32(cols + wb, off[w + 1] - wb, (int32_t)bound);
    }
}

// ---------------------------------------------------------------------------------------------
// Segment traversal helpers.  Every loop issues kUnroll independent loads per lane before it uses
// any of them: the per-element work is a load followed by a dependent shared-memory atomic, and
// without the unrolling one load per warp in flight bounds the throughput by latency.
// ---------------------------------------------------------------------------------------------
constexpr int kUnroll = 4;

// Every visitor f(x) returns the previous value of x's counter; the helpers add those values into
// sum.  NARROW: a value fits 16 bits (8- and 16-bit counters, hash counters), so kUnroll of them are
// summed in 32 bits before one 64-bit add.

// Warp-cooperative traversal of 32 segments (lane l owns cols[base_l .. base_l + len_l)):
// flattened so that every lane takes one element per round.
template <bool NARROW, typename F>
__device__ __forceinline__ void warp_flat(const int32_t* __restrict__ cols, int64_t base, int len, F&& f,
                                          uint64_t& sum) {
    const int l = lane_id();
    int incl = len;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(kFull, incl, o);
        if (l >= o) incl += y;
    }
    const int excl = incl - len;
    const int total = __shfl_sync(kFull, incl, 31);
    for (int t0 = 0; t0 < total; t0 += 32 * kUnroll) {
        int32_t xs[kUnroll];
#pragma unroll
        for (int r = 0; r < kUnroll; ++r) {
            const int t = t0 + r * 32 + l;
            int o = 0;
#pragma unroll
            for (int s = 16; s >= 1; s >>= 1) {
                const int e = __shfl_sync(kFull, excl, o + s);
                if (e <= t) o += s;
            }
            const int64_t ob = __shfl_sync(kFull, base, o);
            const int oe = __shfl_sync(kFull, excl, o);
            xs[r] = t < total ? __ldg(cols + ob + (t - oe)) : 0;
        }
        uint32_t part = 0;
#pragma unroll
        for (int r = 0; r < kUnroll; ++r)
            if (t0 + r * 32 + l < total) {
                if (NARROW) part += f(xs[r]);
                else sum += f(xs[r]);
            }
        if (NARROW) sum += part;
    }
}

// n consecutive elements from b, read by the whole warp (coalesced), kUnroll loads in flight per
// lane: whole chunks of 32 * kUnroll without bounds tests, then one guarded tail chunk.
template <bool NARROW, typename F>
__device__ __forceinline__ void warp_run(const int32_t* __restrict__ cols, int64_t b, int n, F&& f, uint64_t& sum) {
    const int l = lane_id();
    const int32_t* __restrict__ p = cols + b + l;
    constexpr int kCh = 32 * kUnroll;
    int k0 = 0;
    for (; k0 + kCh <= n; k0 += kCh) {
        int32_t xs[kUnroll];
#pragma unroll
        for (int r = 0; r < kUnroll; ++r) xs[r] = __ldg(p + k0 + r * 32);
        uint32_t part = 0;
#pragma unroll
        for (int r = 0; r < kUnroll; ++r) {
            if (NARROW) part += f(xs[r]);
            else sum += f(xs[r]);
        }
        if (NARROW) sum += part;
    }
    if (k0 < n) {
        int32_t xs[kUnroll];
#pragma unroll
        for (int r = 0; r < kUnroll; ++r) xs[r] = k0 + r * 32 + l < n ? __ldg(p + k0 + r * 32) : 0;
#pragma unroll
        for (int r = 0; r < kUnroll; ++r)
            if (k0 + r * 32 + l < n) sum += f(xs[r]);
    }
}

// Long segments one after the other, each read by the whole warp (coalesced); short ones flattened.
template <bool NARROW, typename F>
__device__ __forceinline__ void warp_segments(const int32_t* __restrict__ cols, int64_t base, int len, F&& f,
                                              uint64_t& sum) {
    uint32_t longs = __ballot_sync(kFull, len >= kLong);
    while (longs) {
        const int src = __ffs(longs) - 1;
        longs &= longs - 1;
        const int64_t b = __shfl_sync(kFull, base, src);
        const int n = __shfl_sync(kFull, len, src);
        warp_run<NARROW>(cols, b, n, f, sum);
    }
    warp_flat<NARROW>(cols, base, len >= kLong ? 0 : len, f, sum);
}

// shared-memory hash table: keys[] (kEmpty = free), cnt[]; returns the counter's previous value
__device__ __forceinline__ uint32_t hash_add(int32_t* keys, uint32_t* cnt, uint32_t mask, int32_t x) {
    uint32_t h = hash32((uint32_t)x) & mask;
    for (;;) {
        int32_t k = keys[h];
        if (k == kEmpty) {
            const int32_t prev = atomicCAS(&keys[h], kEmpty, x);
            if (prev == kEmpty || prev == x) return atomicAdd(&cnt[h], 1u);
            k = prev;
        }
        if (k == x) return atomicAdd(&cnt[h], 1u);
        h = (h + 1) & mask;
    }
}

// ---------------------------------------------------------------------------------------------
// Classification: every root (a lane per root, descending rank so heavy roots are queued first).
// ---------------------------------------------------------------------------------------------
template <int WORDS>
__global__ void __launch_bounds__(256) k_c4_classify(const int64_t* __restrict__ loff, const int32_t* __restrict__ deg,
                                                     const int32_t* __restrict__ dplus,
                                                     const int32_t* __restrict__ rev,
                                                     const int32_t* __restrict__ gid,
                                                     const int64_t* __restrict__ ginfo, int64_t n, int64_t own_lo,
                                                     int64_t own_hi, uint32_t warp_max, uint32_t mid_max,
                                                     uint32_t wide_max,
                                                     int32_t* __restrict__ q_small, int32_t* __restrict__ q_win,
                                                     int32_t* __restrict__ wcount, uint64_t* __restrict__ acc) {
    grid_begin();
    const int l = lane_id();
    const int64_t wid = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    unsigned long long* qcnt_small = (unsigned long long*)&acc[Q_C4_MID];
    unsigned long long* qcnt_mid = (unsigned long long*)&acc[Q_C4_MIDW];
    unsigned long long* qcnt_win = (unsigned long long*)&acc[Q_C4_WIN];
    unsigned long long* qcnt_wide = (unsigned long long*)&acc[Q_C4_WIDE];
    // a warp takes 32 ranks, one root per lane, spaced by the number of warps (so the hubs at the top
    // ranks fall to different warps): a lane sums W(u) itself when u has at most 32 lower neighbours,
    // the warp sums the larger roots together; queue slots are taken in lane order (descending rank).
    // A warp per root left most lanes idle on the many small roots of a batch of small graphs.
    uint64_t visits = 0;
    for (int64_t k0 = wid; k0 < n; k0 += nw * 32) {
        const int64_t k = k0 + (int64_t)l * nw;
        const int32_t u = (int32_t)(n - 1 - k);
        int64_t dm = 0;
        if (k < n && u >= own_lo && u < own_hi &&                       // the owner rule
            u < ginfo[(gid ? (int64_t)gid[u] : 0) * kGInfo + GI_CORE])  // core roots are counted by the core pass
            dm = (int64_t)deg[u] - dplus[u];
        const int64_t ub = dm >= 2 ? loff[u] : 0;
        uint64_t W = 0;
        if (dm >= 2 && dm <= 32) {
            for (int64_t a = 0; a < dm; ++a) W += (uint64_t)rev[ub + a];
        }
        uint32_t big = __ballot_sync(kFull, dm > 32);
        while (big) {
            const int src = __ffs(big) - 1;
            big &= big - 1;
            const int64_t bdm = __shfl_sync(kFull, dm, src), bub = __shfl_sync(kFull, ub, src);
            uint64_t bw = 0;
            for (int64_t a = l; a < bdm; a += 32) bw += (uint64_t)rev[bub + a];
            bw = warp_sum(bw);
            if (l == src) W = bw;
        }
        int cls = W == 0 ? -1 : (W <= warp_max ? 0 : (W <= mid_max ? 1 : 2));
        int64_t windows = 0;
        if (cls == 2) {
            windows = windows_below<WORDS>(ginfo + (gid ? (int64_t)gid[u] : 0) * kGInfo, u);
            if (W <= wide_max && windows >= 2 && dm <= (1 << kWideBits)) cls = 3;
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const uint32_t mask = __ballot_sync(kFull, cls == c);
            if (!mask) continue;
            unsigned long long base = 0;
            const int leader = __ffs(mask) - 1;
            unsigned long long* ctr = c == 0 ? qcnt_small : (c == 1 ? qcnt_mid : (c == 2 ? qcnt_win : qcnt_wide));
            if (l == leader) base = atomicAdd(ctr, (unsigned long long)__popc(mask));
            base = __shfl_sync(kFull, base, leader);
            if (cls == c) {
                const int64_t slot = (int64_t)(base + __popc(mask & lanemask_lt()));
                if (c == 0) {
                    q_small[slot] = u;
                    q_small[n + slot] = (int32_t)W;
                } else if (c == 1) {  // the middle tier fills the same queue from the back
                    q_small[n - 1 - slot] = u;
                    q_small[2 * n - 1 - slot] = (int32_t)W;
                } else if (c == 2) {
                    q_win[slot] = u;
                    wcount[slot] = (int32_t)windows;
                    visits += (uint64_t)(windows * dm);
                } else {
                    q_win[n - 1 - slot] = u;
                    wcount[n - 1 - slot] = (int32_t)W;
                }
            }
        }
    }
    visits = warp_sum(visits);
    if (l == 0 && visits) atomicAdd((unsigned long long*)&acc[C4_VISITS], (unsigned long long)visits);
}

// ---------------------------------------------------------------------------------------------
// Hash modes: roots of few wedges, a hash table in shared memory.
// ---------------------------------------------------------------------------------------------
// Counters of x by open addressing.  PACKED: one word per slot, (x - x0) << CB | (count - 1): one load finds the
// key and one atomic counts it, and the table takes half the bytes; needs x - x0 < 2^(32 - CB) - 1 and counts
// of at most 2^CB.  Else a key and a count word.  add() returns the counter's previous value.
template <int SLOTS, int CB, bool PACKED>
struct HashTable {
    static constexpr int kWords = PACKED ? SLOTS : 2 * SLOTS;
    static constexpr uint32_t kFree = 0xffffffffu;
    uint32_t* t;
    uint32_t mask;
    int32_t x0;
    __device__ __forceinline__ void clear(int tid, int threads) {  // mask + 1 slots, a multiple of 32
        const uint32_t P = mask + 1;
        for (uint32_t i = 4 * tid; i < P; i += 4 * threads)
            *reinterpret_cast<uint4*>(t + i) = make_uint4(kFree, kFree, kFree, kFree);
        if (!PACKED)
            for (uint32_t i = 4 * tid; i < P; i += 4 * threads)
                *reinterpret_cast<uint4*>(t + SLOTS + i) = make_uint4(0, 0, 0, 0);
    }
    __device__ __forceinline__ uint32_t add(int32_t x) {
        uint32_t h = (hash32((uint32_t)x) >> 8) & mask;
        if (!PACKED) return hash_add(reinterpret_cast<int32_t*>(t), t + SLOTS, mask, x);
        const uint32_t key = (uint32_t)(x - x0);
        for (;;) {
            uint32_t v = t[h];
            if (v == kFree) {
                v = atomicCAS(&t[h], kFree, key << CB);
                if (v == kFree) return 0;
            }
            if ((v >> CB) == key) return (atomicAdd(&t[h], 1u) & ((1u << CB) - 1u)) + 1u;
            h = (h + 1) & mask;
        }
    }
};
static_assert(kEmpty == -1, "a free key is all ones in both layouts");

// 32 segments (lane l owns cols[base_l .. base_l + len_l)) flattened so that every lane takes one element per
// round, kUnroll rounds in flight.  The owner of an element is found from the segment starts that fall into
// its round (one or-reduction) and a compacted list of the nonempty segments in shared memory (rel[32]),
// about 9 instructions a round where a search over the lanes takes 25.  Positions fit 32 bits.
template <typename F>
__device__ __forceinline__ void warp_flat_rel(const int32_t* __restrict__ cols, uint32_t base, int len, uint32_t* rel,
                                              F&& f) {
    const int l = lane_id();
    int incl = len;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kFull, incl, o);
        if (l >= o) incl += y;
    }
    const int excl = incl - len;
    const int total = __shfl_sync(kFull, incl, 31);
    const uint32_t some = __ballot_sync(kFull, len > 0);
    if (len > 0) rel[__popc(some & lanemask_lt())] = base - (uint32_t)excl;
    __syncwarp();
    int before = 0;  // nonempty segments that start before the round
    const uint32_t le = lanemask_lt() | (1u << l);
    for (int t0 = 0; t0 < total; t0 += 32 * kUnroll) {
        int32_t xs[kUnroll];
#pragma unroll
        for (int r = 0; r < kUnroll; ++r) {
            const int t = t0 + r * 32 + l;
            const int s = excl - (t0 + r * 32);
            const uint32_t starts = __reduce_or_sync(kFull, len > 0 && s >= 0 && s < 32 ? 1u << s : 0u);
            const int k = before + __popc(starts & le) - 1;
            before += __popc(starts);
            xs[r] = t < total ? __ldg(cols + (rel[k] + (uint32_t)t)) : -1;
        }
#pragma unroll
        for (int r = 0; r < kUnroll; ++r) f(xs[r], t0 + r * 32 + l < total);
    }
    __syncwarp();  // rel is read before the next call writes it
}

// Sums of one graph at a time (batch): a running sum that goes to its graph when the next root's differs.
struct GraphSum {
    uint64_t v = 0;
    int32_t g = -1;
    __device__ __forceinline__ void flush(const Sink& sink) {  // by a whole warp
        const uint64_t t = warp_sum(v);
        if (lane_id() == 0 && g >= 0 && t) atomicAdd((unsigned long long*)&sink.accG[(int64_t)g * kGStride + G_C4], (unsigned long long)t);
        v = 0;
    }
    __device__ __forceinline__ void enter(const Sink& sink, int32_t graph) {
        if (graph != g) {
            flush(sink);
            g = graph;
        }
    }
};

// Light roots (W <= 512): a warp each.  A root is a short chain of dependent loads, so a warp takes kLightChunk
// consecutive roots of the queue, loads their headers side by side and the next root's lower list while it
// works on the current one.  W <= 32 (and one group of lower neighbours) needs no table: equal x are found
// among the lanes.  Light and middle roots of the batch of 4,096 graphs: 12.4 + 8.9 -> 5.8 + 2.2 ms; light roots
// of the random geometric graph with 1,000,003 vertices: 0.90 -> 0.52 ms.
constexpr int kLightChunk = 8;
constexpr int kLightBits = 9;  // counts of at most 512

template <bool PACKED>
__global__ void __launch_bounds__(kSmallThreads, PACKED ? 5 : 3) k_c4_light(const int64_t* __restrict__ off,
                                                                            const int32_t* __restrict__ cols,
                                                                            const int64_t* __restrict__ loff,
                                                                            const int32_t* __restrict__ lcols,
                                                                            const int32_t* __restrict__ deg,
                                                                            const int32_t* __restrict__ dplus,
                                                                            const int32_t* __restrict__ fpos,
                                                                            const int32_t* __restrict__ rev,
                                                                            const uint4* __restrict__ vinfo,
                                                                            const int64_t* __restrict__ ginfo,
                                                                            const int32_t* __restrict__ q_small,
                                                                            int64_t n, uint64_t* __restrict__ acc,
                                                                            Sink sink) {
    grid_begin();
    using Table = HashTable<kSmallSlots, kLightBits, PACKED>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ uint32_t s_rel[kSmallWarps][32];
    __shared__ uint64_t red[32];
    const int w = threadIdx.x >> 5, l = lane_id();
    Table table;
    table.t = reinterpret_cast<uint32_t*>(smem_raw) + w * Table::kWords;
    const int64_t nq = (int64_t)acc[Q_C4_MID];
    const int64_t share = nq / (2 * (int64_t)gridDim.x * kSmallWarps);
    const int chunk = share < 1 ? 1 : (share < kLightChunk ? (int)share : kLightChunk);
    const int64_t nchunk = (nq + chunk - 1) / chunk;
    unsigned long long* ticket = (unsigned long long*)&acc[T_C4_LIGHT];
    auto next_ticket = [&] { return l == 0 ? (int64_t)atomicAdd(ticket, 1ull) : 0; };
    GraphSum sum;
    int64_t c_next = next_ticket();
    for (;;) {
        const int64_t c = __shfl_sync(kFull, c_next, 0);
        if (c >= nchunk) break;
        c_next = next_ticket();  // in flight while this chunk is worked on
        const int cn = nq - c * chunk < chunk ? (int)(nq - c * chunk) : chunk;
        int32_t hW = 0, hg = 0, hx0 = 0;
        int hdm = 0;
        int64_t hub = 0;
        if (l < cn) {
            const int32_t u = q_small[c * chunk + l];
            hW = q_small[n + c * chunk + l];
            hdm = deg[u] - dplus[u];
            hub = loff[u];
            if (sink.batch()) hg = sink.gid[u];
            hx0 = (int32_t)ginfo[(int64_t)hg * kGInfo + GI_N1];
        }
        int dm = __shfl_sync(kFull, hdm, 0);
        int64_t ub = __shfl_sync(kFull, hub, 0);
        int32_t w_next = l < dm ? lcols[ub + l] : 0, r_next = l < dm ? rev[ub + l] : 0;
        for (int i = 0; i < cn; ++i) {
            dm = __shfl_sync(kFull, hdm, i);
            ub = __shfl_sync(kFull, hub, i);
            const uint32_t W = (uint32_t)__shfl_sync(kFull, hW, i);
            int32_t wv = w_next, rv = r_next;
            {
                const int nd = i + 1 < cn ? __shfl_sync(kFull, hdm, i + 1) : 0;
                const int64_t nb = __shfl_sync(kFull, hub, (i + 1) & 31);
                w_next = l < nd ? lcols[nb + l] : 0;
                r_next = l < nd ? rev[nb + l] : 0;
            }
            if (sink.batch()) sum.enter(sink, __shfl_sync(kFull, hg, i));
            table.x0 = __shfl_sync(kFull, hx0, i);
            const bool tabled = W > 32 || dm > 32;
            if (tabled) {
                uint32_t P = 64;
                while (P < 2 * W) P <<= 1;
                table.mask = P - 1;
                table.clear(l, 32);
                __syncwarp();
            }
            for (int a0 = 0; a0 < dm; a0 += 32) {
                if (a0 > 0) {
                    wv = a0 + l < dm ? lcols[ub + a0 + l] : 0;
                    rv = a0 + l < dm ? rev[ub + a0 + l] : 0;
                }
                uint32_t base = 0;
                int len = 0;
                if (a0 + l < dm) {
                    base = vinfo ? __ldg(&vinfo[wv].w) : (uint32_t)(off[wv] + fpos[wv]);
                    len = rv;
                }
                if (tabled) {
                    uint32_t part = 0;
                    warp_flat_rel(cols, base, len, s_rel[w], [&](int32_t x, bool in) {
                        if (in) part += table.add(x);
                    });
                    sum.v += part;
                } else {  // the root's only group, and at most one round of it
                    uint32_t part = 0;
                    warp_flat_rel(cols, base, len, s_rel[w], [&](int32_t x, bool in) {
                        if (!__any_sync(kFull, in)) return;
                        const uint32_t same = __match_any_sync(kFull, in ? x : -1 - l);
                        if (in) part += (uint32_t)__popc(same & lanemask_lt());
                    });
                    sum.v += part;
                }
            }
            __syncwarp();
        }
    }
    if (sink.batch()) {
        sum.flush(sink);
        return;
    }
    const uint64_t c4 = block_sum_u64(sum.v, red);
    if (threadIdx.x == 0 && c4) atomicAdd((unsigned long long*)&acc[ACC_C4], (unsigned long long)c4);
}

// Middle roots (512 < W <= 2048, the back of q_mid) and wide ones (2048 < W <= 16384, the back of q_win): a block each,
// the lower neighbours dealt to its warps.  A wide root would else cost a pass over its lower neighbours and a scan of
// the counters for every window of ranks below it: Chung-Lu of 2,000,000 vertices, 40,000 such roots over up to 40
// windows, 10.4 ms of window passes against 2.3 ms (its whole count 50.6 -> 42.4 ms); R-MAT scale 20 0.72 and 0.28 ms.
// One table size of 32,768 slots for both halves took 3.1 ms, blocks of 8 warps for the lower half 1.33 instead of 0.99.
constexpr int kMidThreads = kMidWarps * 32;
constexpr int kMidBits = 11;  // counts of at most 2048

template <int SLOTS, int WARPS, int BITS, bool PACKED>
__global__ void __launch_bounds__(WARPS * 32) k_c4_mid(const int64_t* __restrict__ off, const int32_t* __restrict__ cols,
                                                        const int64_t* __restrict__ loff,
                                                        const int32_t* __restrict__ lcols,
                                                        const int32_t* __restrict__ deg, const int32_t* __restrict__ dplus,
                                                        const int32_t* __restrict__ fpos, const int32_t* __restrict__ rev,
                                                        const uint4* __restrict__ vinfo, const int64_t* __restrict__ ginfo,
                                                        const int32_t* __restrict__ q, int64_t n, uint32_t wlo,
                                                        uint32_t whi, int qslot, int tslot,
                                                        uint64_t* __restrict__ acc, Sink sink) {
    grid_begin();
    using Table = HashTable<SLOTS, BITS, PACKED>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ uint32_t s_rel[WARPS][32];
    __shared__ uint64_t red[32];
    __shared__ int64_t s_item;
    const int w = threadIdx.x >> 5, l = lane_id();
    Table table;
    table.t = reinterpret_cast<uint32_t*>(smem_raw);
    const int64_t nq = (int64_t)acc[qslot];
    unsigned long long* ticket = (unsigned long long*)&acc[tslot];
    GraphSum sum;
    auto take = [&] {  // the next root with wlo < W <= whi
        int64_t k;
        uint32_t W = 0;
        do {
            k = (int64_t)atomicAdd(ticket, 1ull);
            if (k < nq) W = (uint32_t)q[2 * n - 1 - k];
        } while (k < nq && (W <= wlo || W > whi));
        s_item = k;
    };
    if (threadIdx.x == 0) take();
    __syncthreads();
    for (;;) {
        const int64_t k = s_item;
        if (k >= nq) break;
        const int32_t u = q[n - 1 - k];
        const uint32_t W = (uint32_t)q[2 * n - 1 - k];
        const int64_t dm = (int64_t)deg[u] - dplus[u];
        const int64_t ub = loff[u];
        const int32_t g = sink.batch() ? sink.gid[u] : 0;
        if (sink.batch()) sum.enter(sink, g);
        table.x0 = (int32_t)ginfo[(int64_t)g * kGInfo + GI_N1];
        uint32_t P = 64;
        while (P < 2 * W) P <<= 1;
        table.mask = P - 1;
        table.clear(threadIdx.x, WARPS * 32);
        __syncthreads();  // the table is clear, every thread has read s_item
        if (threadIdx.x == 0) take();
        uint64_t part = 0;
        for (int64_t a0 = 0; a0 < dm; a0 += WARPS * 32) {
            const int64_t a = a0 + l * WARPS + w;
            uint32_t base = 0;
            int len = 0;
            if (a < dm) {
                const int32_t wv = lcols[ub + a];
                base = vinfo ? __ldg(&vinfo[wv].w) : (uint32_t)(off[wv] + fpos[wv]);
                len = rev[ub + a];
            }
            warp_flat_rel(cols, base, len, s_rel[w], [&](int32_t x, bool in) {
                if (in) part += table.add(x);
            });
        }
        sum.v += part;
        __syncthreads();  // the root is counted before the table is cleared; s_item is set
    }
    if (sink.batch()) {
        sum.flush(sink);
        return;
    }
    const uint64_t c4 = block_sum_u64(sum.v, red);
    if (threadIdx.x == 0 && c4) atomicAdd((unsigned long long*)&acc[ACC_C4], (unsigned long long)c4);
}

// ---------------------------------------------------------------------------------------------
// Windowed CTA mode: one block per (root, grid window); dense packed counters in shared memory.
// ---------------------------------------------------------------------------------------------
// Packed counters: a band of width b packs floor(32 / b) counters into a word (3-bit ten, 4-bit
// eight, 5-bit six, 6-bit five, 8-bit four, 16-bit two).  (A byte-plane layout that
// puts consecutive x in consecutive banks was measured no faster: the kernel is bound by load
// latency and the end-of-item barrier, not by shared-memory bank conflicts.)
template <int WIDTH, int WORDS>
__device__ __forceinline__ uint32_t counter_add(uint32_t* cw, uint32_t r) {
    constexpr uint32_t K = 32 / WIDTH;  // counters per word
    if constexpr (K == 1) {
        return atomicAdd(&cw[r], 1u);
    } else {
        const uint32_t q = r / K;  // a constant divisor: a multiply and a shift
        const uint32_t sh = (r - q * K) * WIDTH;
        return (atomicAdd(&cw[q], 1u << sh) >> sh) & ((1u << WIDTH) - 1u);
    }
}

// Calls f(std::integral_constant<int, width>) for band b's counter width, so each width is its own
// compiled instance of the window and split passes.
template <typename F>
__device__ __forceinline__ void with_band(int b, F&& f) {
    switch (b) {
        case 0: f(std::integral_constant<int, band_width(0)>{}); break;
        case 1: f(std::integral_constant<int, band_width(1)>{}); break;
        case 2: f(std::integral_constant<int, band_width(2)>{}); break;
        case 3: f(std::integral_constant<int, band_width(3)>{}); break;
        case 4: f(std::integral_constant<int, band_width(4)>{}); break;
        case 5: f(std::integral_constant<int, band_width(5)>{}); break;
        default: f(std::integral_constant<int, band_width(6)>{}); break;
    }
}
static_assert(kBands == 7, "with_band covers every band");

struct WinShared {
    int group;                 // next group of 32 lower neighbours
    int nsplit;                // entries pushed to the split queue
    int chunk;                 // next split chunk
    int64_t split_base[kSplitQ];
    int32_t split_len[kSplitQ];
    int32_t split_pre[kSplitQ + 1];
};

// Self-check: a segment outside its row, or one whose first or last element lies outside the window
// (rows are sorted, so these two bound every element of the segment), is skipped and recorded in
// acc[ACC_ERR]; the host then reports HARP_EDEVICE.
__device__ __forceinline__ void flag_error(uint64_t* acc, unsigned long long bit) {
    atomicOr((unsigned long long*)&acc[ACC_ERR], bit);
}

template <int WIDTH, int WORDS>
__device__ __forceinline__ void window_pass(const int64_t* __restrict__ off, const int32_t* __restrict__ cols,
                                            const int32_t* __restrict__ lcols,
                                            const int32_t* __restrict__ fpos, const int32_t* __restrict__ rev,
                                            const int32_t* __restrict__ bpos, bool table, int sl, int64_t nwin,
                                            int64_t j, int64_t ub,
                                            int64_t dm, int32_t xlo, int32_t xhi, bool first, bool last, uint32_t* cw,
                                            WinShared& sh, uint64_t& c4, uint64_t* acc) {
    const int l = lane_id();
    auto add = [&](int32_t x) { return counter_add<WIDTH, WORDS>(cw, (uint32_t)(x - xlo)); };
    const int ngroups = (int)((dm + 31) >> 5);
    for (;;) {
        int g = 0;
        if (l == 0) g = atomicAdd(&sh.group, 1);
        g = __shfl_sync(kFull, g, 0);
        if (g >= ngroups) break;
        const int64_t a = (int64_t)(ngroups - 1 - g) * 32 + l;  // heaviest groups first
        int64_t base = 0;
        int len = 0;
        if (a < dm) {
            const int32_t wv = lcols[ub + a];
            const int64_t wb = off[wv];
            int64_t p0, p1;
            const int64_t rowlen = off[wv + 1] - wb;
            const int64_t mask = ((int64_t)1 << sl) - 1;
            if (first) p0 = fpos[wv];
            else if (table && (j & mask) == 0) p0 = bpos[(int64_t)wv * kGridCap + (j >> sl)];
            else if (table) p0 = gallop_i32(cols + wb, bpos[(int64_t)wv * kGridCap + (j >> sl)], rowlen, xlo);
            else p0 = lower_bound_i32(cols + wb, rowlen, xlo);
            if (last) p1 = (int64_t)(first ? p0 : fpos[wv]) + rev[ub + a];
            else if (table && ((j + 1) & mask) == 0 && j + 1 <= nwin) p1 = bpos[(int64_t)wv * kGridCap + ((j + 1) >> sl)];
            else if (table) p1 = gallop_i32(cols + wb, p0 < 0 ? 0 : p0, rowlen, xhi);
            else p1 = lower_bound_i32(cols + wb, rowlen, xhi);
            if (p0 < 0 || p1 > rowlen) {
                flag_error(acc, kErrRow);
                p0 = p1 = 0;
            }
            if (p1 > p0 && (cols[wb + p0] < xlo || cols[wb + p1 - 1] >= xhi)) {
                flag_error(acc, kErrSegment);
                p1 = p0;
            }
            base = wb + p0;
            len = p1 > p0 ? (int)(p1 - p0) : 0;
        }
        if (len >= kSplit) {  // hand very long segments to the whole block
            const int slot = atomicAdd(&sh.nsplit, 1);
            if (slot < kSplitQ) {
                sh.split_base[slot] = base;
                sh.split_len[slot] = len;
                len = 0;
            }
        }
        warp_segments<WIDTH != 32>(cols, base, len, add, c4);
    }
}

template <int WIDTH, int WORDS>
__device__ __forceinline__ void split_pass(const int32_t* __restrict__ cols, int32_t xlo, uint32_t* cw, WinShared& sh,
                                           uint64_t& c4) {
    const int l = lane_id();
    const int ns = sh.nsplit < kSplitQ ? sh.nsplit : kSplitQ;
    const int total = sh.split_pre[ns];
    for (;;) {
        int t = 0;
        if (l == 0) t = atomicAdd(&sh.chunk, 1);
        t = __shfl_sync(kFull, t, 0);
        if (t >= total) break;
        int e = 0;  // entry owning chunk t: last e with split_pre[e] <= t
        int hi = ns;
        while (hi - e > 1) {
            const int mid = (e + hi) >> 1;
            if (sh.split_pre[mid] <= t) e = mid;
            else hi = mid;
        }
        const int64_t b = sh.split_base[e] + (int64_t)(t - sh.split_pre[e]) * kChunk;
        const int64_t end = sh.split_base[e] + sh.split_len[e];
        const int64_t stop = b + kChunk < end ? b + kChunk : end;
        warp_run<WIDTH != 32>(cols, b, (int)(stop - b),
                              [&](int32_t x) { return counter_add<WIDTH, WORDS>(cw, (uint32_t)(x - xlo)); }, c4);
    }
}

// Everything an item (root, grid window) needs before its lower neighbours are walked.  Resolving it
// is a chain of dependent loads (ticket, search of the item's root, the root, its grid window, its
// list), so one thread resolves the next item while the block works on the current one.
struct WinItem {
    int64_t t;  // ticket; >= the item total: no more items
    int64_t j, xlo, xhi, nwin, dm, ub;
    int32_t u;
    int band, sl, first, last;
};

template <int WORDS>
__device__ __forceinline__ void resolve_item(WinItem& it, int64_t t, int64_t total, int64_t nroots,
                                             const int64_t* __restrict__ win_prefix,
                                             const int32_t* __restrict__ q_win, const int32_t* __restrict__ gid,
                                             const int64_t* __restrict__ ginfo, const int32_t* __restrict__ deg,
                                             const int32_t* __restrict__ dplus, const int64_t* __restrict__ loff) {
    it.t = t;
    if (t >= total) return;
    int64_t lo = 0, hi = nroots;  // root index: last k with win_prefix[k] <= t
    while (hi - lo > 1) {
        const int64_t mid = (lo + hi) >> 1;
        if (win_prefix[mid] <= t) lo = mid;
        else hi = mid;
    }
    const int32_t u = q_win[lo];
    const int64_t j = t - win_prefix[lo];
    const int64_t* gi = ginfo + (gid ? (int64_t)gid[u] : 0) * kGInfo;
    int64_t xlo = 0, xhi = 0;
    int band = kBands - 1;
    grid_window<WORDS>(gi, j, xlo, xhi, band);
    it.last = xhi >= (int64_t)u;
    it.xhi = it.last ? u : xhi;
    it.xlo = xlo;
    it.first = j == 0;
    it.j = j;
    it.u = u;
    it.band = band;
    it.nwin = gi[GI_NWIN];
    it.sl = table_shift(it.nwin);
    it.dm = (int64_t)deg[u] - dplus[u];
    it.ub = loff[u];
}

template <int MINB>
__global__ void __launch_bounds__(win_threads(MINB), MINB) k_c4_window(const int64_t* __restrict__ off,
                                                              const int32_t* __restrict__ cols,
                                                              const int64_t* __restrict__ loff,
                                                              const int32_t* __restrict__ lcols,
                                                              const int32_t* __restrict__ deg,
                                                              const int32_t* __restrict__ dplus,
                                                              const int32_t* __restrict__ fpos,
                                                              const int32_t* __restrict__ rev,
                                                              const int32_t* __restrict__ bpos,
                                                              const int32_t* __restrict__ gid,
                                                              const int64_t* __restrict__ ginfo,
                                                              const int32_t* __restrict__ q_win,
                                                              const int64_t* __restrict__ win_prefix, int64_t n,
                                                              uint64_t* __restrict__ acc, Sink sink) {
    grid_begin();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    uint32_t* cw = reinterpret_cast<uint32_t*>(smem_raw);
    constexpr int WORDS = win_words(MINB);
    __shared__ WinItem s_next;
    __shared__ WinShared sh;
    __shared__ uint64_t red[32];
    const int64_t nroots = (int64_t)acc[Q_C4_WIN];
    const int64_t total = win_prefix[nroots];
    unsigned long long* ticket = (unsigned long long*)&acc[T_C4_WIN];
    const bool table = bpos != nullptr && table_pays(acc, n);
    uint64_t c4 = 0;
    if (threadIdx.x == 0)
        resolve_item<WORDS>(s_next, (int64_t)atomicAdd(ticket, 1ull), total, nroots, win_prefix, q_win, gid, ginfo,
                            deg, dplus, loff);
    __syncthreads();
    for (;;) {
        const WinItem it = s_next;
        if (it.t >= total) break;
        const int32_t u = it.u;
        const int64_t j = it.j, xlo = it.xlo, xhi = it.xhi, nwin = it.nwin, dm = it.dm, ub = it.ub;
        const int band = it.band, sl = it.sl;
        const bool first = it.first, last = it.last;
        if (threadIdx.x == 0) {
            sh.group = 0;
            sh.nsplit = 0;
            sh.chunk = 0;
        }
        int words = 0;
        with_band(band, [&](auto wc) {
            constexpr int per = 32 / decltype(wc)::value;
            words = (int)((xhi - xlo + per - 1) / per);
        });
        for (int i = threadIdx.x; i < words; i += win_threads(MINB)) cw[i] = 0;
        __syncthreads();  // every thread holds this item; counters and work counters are reset
        if (threadIdx.x == 0)  // the next item, resolved while the block walks this one
            resolve_item<WORDS>(s_next, (int64_t)atomicAdd(ticket, 1ull), total, nroots, win_prefix, q_win, gid,
                                ginfo, deg, dplus, loff);
        uint64_t a_c4 = 0;
        with_band(band, [&](auto wc) {
            window_pass<decltype(wc)::value, WORDS>(off, cols, lcols, fpos, rev, bpos, table, sl, nwin, j, ub, dm,
                                                    (int32_t)xlo, (int32_t)xhi, first, last, cw, sh, a_c4, acc);
        });
        __syncthreads();
        if (sh.nsplit > 0) {
            if (threadIdx.x == 0) {
                const int ns = sh.nsplit < kSplitQ ? sh.nsplit : kSplitQ;
                int run = 0;
                for (int e = 0; e < ns; ++e) {
                    sh.split_pre[e] = run;
                    run += (sh.split_len[e] + kChunk - 1) / kChunk;
                }
                sh.split_pre[ns] = run;
            }
            __syncthreads();
            with_band(band, [&](auto wc) { split_pass<decltype(wc)::value, WORDS>(cols, (int32_t)xlo, cw, sh, a_c4); });
            __syncthreads();
        }
        if (sink.batch()) {
            const uint64_t s = block_sum_u64(a_c4, red);
            if (threadIdx.x == 0) sink_add(sink, u, G_C4, s);
        } else {
            c4 += a_c4;
        }
        __syncthreads();  // every thread is done with this item's shared state; s_next is resolved
    }
    c4 = block_sum_u64(c4, red);
    if (threadIdx.x == 0 && c4) atomicAdd((unsigned long long*)&acc[ACC_C4], (unsigned long long)c4);
}

unsigned grid_cap(int64_t work, int threads, int64_t cap) {
    int64_t b = (work + threads - 1) / threads;
    if (b < 1) b = 1;
    if (b > cap) b = cap;
    return (unsigned)b;
}

// k_c4_seglen over a whole graph's lower arcs; runs long enough to pay for finding their rows, short enough to give
// every warp one.
harp_status segment_lengths(const harp_csr* g, Workspace& ws, const uint4* vinfo, const int64_t* ginfo, cudaStream_t s) {
    const int64_t warps = (int64_t)num_sms() * 64;
    int64_t run = ((g->m + g->n) / warps + 31) / 32 * 32;
    run = run < 32 ? 32 : (run > 256 ? 256 : run);
    launch(k_c4_seglen, grid_cap((g->m + g->n + run - 1) / run * 32, 256, (int64_t)num_sms() * 64), 256, 0, s, ws.off,
           ws.cols, ws.offp, ws.colsp, vinfo, ginfo ? ws.gid : nullptr, ginfo, g->n, (int)run, ws.rev);
    HARP_LAUNCHED();
    return HARP_OK;
}

// The whole wedge pass for one window size (MINB resident window blocks per SM).
template <int MINB>
harp_status wedge_pass(const harp_csr* g, Workspace& ws, uint32_t warp_max, uint32_t mid_max, cudaStream_t s) {
    constexpr int WORDS = win_words(MINB);
    const int64_t n = g->n;
    const Sink sink{ws.acc, ws.gid, ws.accG};
    const int sms = num_sms();
    const int64_t most_n = ws.G > 1 ? ws.max_member_n : n;  // vertices of the largest graph
    int32_t* wcount = ws.q_win + n;
    // the wide tier: where a graph can have several windows (fewer vertices than a window has words fit one at any
    // width but the last) and its ranks fit beside the counts; a middle tier set lower turns it off
    const bool wide_on = mid_max == kMidSlots / 2 && most_n >= WORDS && most_n < ((int64_t)1 << (32 - kWideBits)) - 1;
    const uint32_t wide_max = wide_on ? kWide2Slots / 2 : 0;
    if (ws.core) HARP_TRY(count_wedge_core(g, ws, s));  // uses rev, bpos and the queues before they are filled below
    // the roots' lower lists: row prefixes of a whole graph, or their own CSR in a partitioned block
    const bool lists = ws.loff != nullptr;
    const int64_t* loff = lists ? ws.loff : ws.off;
    const int32_t* lcols = lists ? ws.lcols : ws.cols;
    uint4* vinfo = lists ? nullptr : reinterpret_cast<uint4*>(ws.vkeys);  // the sort keys' two arrays are done with
    launch(k_c4_fpos, grid_cap(n, 256, (int64_t)sms * 64), 256, 0, s, ws.off, ws.cols, ws.offp, ws.gid, ws.ginfo, n,
           ws.fpos, vinfo);
    HARP_LAUNCHED();
    if (lists) {
        const int64_t la = ws.lower_arcs;  // == loff[n]
        launch(k_c4_seglen_rows, grid_cap((la + kRevRun - 1) / kRevRun, 256, (int64_t)sms * 64), 256, 0, s, ws.loff,
               ws.lcols, ws.off, ws.cols, ws.fpos, n, la, ws.rev);
        HARP_LAUNCHED();
    } else {
        HARP_TRY(segment_lengths(g, ws, vinfo, ws.ginfo, s));
    }
    launch(k_c4_classify<WORDS>, grid_cap(n, 256, (int64_t)sms * 32), 256, 0, s, loff, ws.deg, ws.dplus, ws.rev, ws.gid,
           ws.ginfo, n, ws.own_lo, ws.own_hi, warp_max, mid_max, wide_max, ws.q_mid, ws.q_win, wcount,
           ws.acc);  // a lane per root
    HARP_LAUNCHED();
    // the three tiers read the same arrays and meet only in the accumulators (count_passes joins the sides)
    cudaStream_t s_light = s, s_mid = s;
    if (ws.fork) {
        HARP_TRY(ws.fork->go(1, s));
        HARP_TRY(ws.fork->go(2, s));
        s_light = ws.fork->side[1];
        s_mid = ws.fork->side[2];
    }
    // one word per hash slot where every graph's ranks fit beside the count
    const bool packed_light = most_n < ((int64_t)1 << (32 - kLightBits)) - 1;
    const bool packed_mid = most_n < ((int64_t)1 << (32 - kMidBits)) - 1;
    const size_t light_smem = (size_t)kSmallWarps * kSmallSlots * (packed_light ? 4 : 8);
    auto light = packed_light ? k_c4_light<true> : k_c4_light<false>;
    HARP_CK(cudaFuncSetAttribute(light, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)light_smem));
    launch(light, sms * (packed_light ? 5 : 3), kSmallThreads, light_smem, s_light, ws.off, ws.cols, loff, lcols, ws.deg,
           ws.dplus, ws.fpos, ws.rev, vinfo, ws.ginfo, ws.q_mid, n, ws.acc, sink);
    HARP_LAUNCHED();
    HARP_CK(prof_mark(s, SEG_C4_SMALL));
    if (mid_max > warp_max) {
        const size_t mid_smem = (size_t)kMidSlots * (packed_mid ? 4 : 8);
        auto mid = packed_mid ? k_c4_mid<kMidSlots, kMidWarps, kMidBits, true>
                              : k_c4_mid<kMidSlots, kMidWarps, kMidBits, false>;
        HARP_CK(cudaFuncSetAttribute(mid, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)mid_smem));
        launch(mid, sms * (packed_mid ? 12 : 6), kMidThreads, mid_smem, s_mid, ws.off, ws.cols, loff, lcols, ws.deg,
               ws.dplus, ws.fpos, ws.rev, vinfo, ws.ginfo, ws.q_mid, n, 0u, (uint32_t)kMidSlots / 2, (int)Q_C4_MIDW,
               (int)T_C4_MID, ws.acc, sink);
        HARP_LAUNCHED();
    }
    if (wide_on) {
        auto wide2 = k_c4_mid<kWide2Slots, kWide2Warps, kWideBits, true>;
        HARP_CK(cudaFuncSetAttribute(wide2, cudaFuncAttributeMaxDynamicSharedMemorySize, kWide2Slots * 4));
        launch(wide2, sms, kWide2Warps * 32, (size_t)kWide2Slots * 4, s_mid, ws.off, ws.cols, loff, lcols, ws.deg,
               ws.dplus, ws.fpos, ws.rev, vinfo, ws.ginfo, ws.q_win, n, (uint32_t)kWideSlots / 2,
               (uint32_t)kWide2Slots / 2, (int)Q_C4_WIDE, (int)T_C4_WIDE2, ws.acc, sink);
        HARP_LAUNCHED();
        auto wide = k_c4_mid<kWideSlots, kWideWarps, kWideBits, true>;
        HARP_CK(cudaFuncSetAttribute(wide, cudaFuncAttributeMaxDynamicSharedMemorySize, kWideSlots * 4));
        launch(wide, sms * 3, kWideWarps * 32, (size_t)kWideSlots * 4, s_mid, ws.off, ws.cols, loff, lcols, ws.deg,
               ws.dplus, ws.fpos, ws.rev, vinfo, ws.ginfo, ws.q_win, n, 0u, (uint32_t)kWideSlots / 2, (int)Q_C4_WIDE,
               (int)T_C4_WIDE, ws.acc, sink);
        HARP_LAUNCHED();
    }
    HARP_CK(prof_mark(s, SEG_C4_MID));
    // only the queued roots' counts matter (and are set); what follows them in the scan is never read
    HARP_TRY(exclusive_scan_i32_to_i64(wcount, ws.win_prefix, n, ws.scan_tmp, ws.scan_tmp_len, s));
    if (ws.bpos) {
        launch(k_c4_bpos<WORDS>, grid_cap(n * kGridCap, 256, (int64_t)sms * 64), 256, 0, s, ws.off, ws.cols, ws.gid,
               ws.ginfo, n, ws.fpos, ws.acc, ws.bpos);
        HARP_LAUNCHED();
    }
    const size_t win_smem = (size_t)WORDS * sizeof(uint32_t);
    HARP_CK(cudaFuncSetAttribute(k_c4_window<MINB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)win_smem));
    launch(k_c4_window<MINB>, sms * MINB, win_threads(MINB), win_smem, s, ws.off, ws.cols, loff, lcols, ws.deg,
           ws.dplus, ws.fpos, ws.rev, ws.bpos, ws.gid, ws.ginfo, ws.q_win, ws.win_prefix, n, ws.acc, sink);
    HARP_LAUNCHED();
    HARP_CK(prof_mark(s, SEG_C4_WINDOW));
    return HARP_OK;
}

}  // namespace

harp_status wedge_positions(const harp_csr* g, Workspace& ws, cudaStream_t s) {
    uint4* vinfo = reinterpret_cast<uint4*>(ws.vkeys);
    launch(k_c4_fpos, grid_cap(g->n, 256, (int64_t)num_sms() * 64), 256, 0, s, ws.off, ws.cols, ws.offp, nullptr,
           nullptr, g->n, nullptr, vinfo);
    HARP_LAUNCHED();
    return segment_lengths(g, ws, vinfo, nullptr, s);
}

namespace {

// Resident window blocks per SM (MINB) for this plan and workspace, which fixes the window size: the largest of the
// four that fits plan.c4_window_bytes (at least the smallest).
// 0 = by graph: a single graph of more than 2^22 vertices takes 200 KiB (its x-range spans tens to
// hundreds of 100 KiB windows, and halving the (root, window) visits measured 37.7 -> 26.1 s on
// the 5e7-vertex Chung-Lu graph), anything smaller and every batch 100 KiB (R-MAT scale 20: 13.2
// ms at 100 KiB against 15.7 ms at 200 KiB)
int window_blocks(const harp_csr* g, const Workspace& ws, const harp_plan& plan) {
    uint32_t wbytes = plan.c4_window_bytes;
    if (wbytes == 0) wbytes = (ws.G <= 1 && g->n > ((int64_t)1 << 22)) ? (uint32_t)kWinWords1 * 4 : (uint32_t)kWinWords2 * 4;
    if (wbytes >= (uint32_t)kWinWords1 * 4) return 1;
    if (wbytes >= (uint32_t)kWinWords2 * 4) return 2;
    return wbytes >= (uint32_t)kWinWords3 * 4 ? 3 : 4;
}

template <int MINB>
harp_status launch_ginfo(const harp_csr* g, Workspace& ws, bool merge, bool core, cudaStream_t s) {
    const int64_t G = ws.G > 0 ? ws.G : 1;
    launch(k_c4_ginfo<win_words(MINB)>, (unsigned)(G < 8192 ? G : 8192), kGinfoThreads, 0, s, ws.deg, g->n, ws.gbase,
           G, ws.x_lo, ws.x_hi, merge, core ? ws.off : nullptr, ws.ginfo, ws.acc);
    HARP_LAUNCHED();
    return HARP_OK;
}

}  // namespace

harp_status wedge_geometry(const harp_csr* g, Workspace& ws, const harp_plan& plan, cudaStream_t s) {
    ws.core = false;
    if (g->n == 0 || g->m == 0) return HARP_OK;
    const bool merge = !(plan.flags & HARP_PLAN_NO_BAND_MERGE), core = wedge_core_applies(g, ws);
    switch (window_blocks(g, ws, plan)) {
        case 1: HARP_TRY(launch_ginfo<1>(g, ws, merge, core, s)); break;
        case 2: HARP_TRY(launch_ginfo<2>(g, ws, merge, core, s)); break;
        case 3: HARP_TRY(launch_ginfo<3>(g, ws, merge, core, s)); break;
        default: HARP_TRY(launch_ginfo<4>(g, ws, merge, core, s));
    }
    if (core) HARP_TRY(build_core_bits(ws, s));
    ws.core = core;
    return HARP_OK;
}

harp_status count_wedge_c4(const harp_csr* g, Workspace& ws, const harp_plan& plan, cudaStream_t s) {
    if (g->n == 0 || g->m == 0) return HARP_OK;
    uint32_t warp_max = plan.c4_warp_max_work ? plan.c4_warp_max_work : 512;
    if (warp_max > kSmallSlots / 2) warp_max = kSmallSlots / 2;
    // the middle tier takes kMidSlots / 2 wedges at most; c4_cta_max_work <= warp_max turns it off
    uint32_t mid_max = plan.c4_cta_max_work;
    if (mid_max > kMidSlots / 2) mid_max = kMidSlots / 2;
    if (mid_max < warp_max) mid_max = warp_max;
    switch (window_blocks(g, ws, plan)) {
        case 1: return wedge_pass<1>(g, ws, warp_max, mid_max, s);
        case 2: return wedge_pass<2>(g, ws, warp_max, mid_max, s);
        case 3: return wedge_pass<3>(g, ws, warp_max, mid_max, s);
        default: return wedge_pass<4>(g, ws, warp_max, mid_max, s);
    }
}

}  // namespace harp
