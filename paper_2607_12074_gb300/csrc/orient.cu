// Step a1: degree ordering and orientation (Section III-D, "sorted CSR adjacency and canonical
// ordering constraints").
//
// Vertices are renumbered by rank(v) = (d(v), v) ascending, so that in the new numbering
//   * N+(v) = neighbours ranked above v = the suffix of v's sorted row after v itself,
//   * N-(v) = neighbours ranked below v = the prefix of the row,
//   * the neighbours of w ranked below u form a prefix of w's row (the ordered wedges of the
//     4-cycle anchor, Section III-B, read contiguous memory).
// Output (workspace): deg, order (new -> old), perm (old -> new), off/cols (relabelled CSR with
// every row sorted), dplus, offp/colsp (out-CSR: only N+), te zeroed, S = sum_v C(d_v, 3).
//
// Rows are sorted by four kernels chosen by degree: for d <= 32 a lane's bitonic network in registers
// (d <= 16) or the warp's over its lanes (every row is visited), a warp's bitonic network over up to 32
// registers a lane for d <= 1024, a block's for d <= 4096 (16 warps' networks joined through shared memory),
// and for hubs a bitmap of the ranks, or a per-row LSD radix sort through global memory where the graph
// has too many ranks for one (the last three from queues filled by the relabel pass).
#include "harp_internal.cuh"
#include "rowsort.cuh"

namespace harp {
namespace {


int bits_for(int64_t x) {
    int b = 0;
    while (b < 63 && ((int64_t)1 << b) <= x) ++b;
    return b < 1 ? 1 : b;
}

unsigned grid_for(int64_t work, int threads, int64_t cap = -1) {
    if (cap < 0) cap = (int64_t)num_sms() * 64;
    int64_t b = (work + threads - 1) / threads;
    if (b < 1) b = 1;
    if (b > cap) b = cap;
    return (unsigned)b;
}

__global__ void k_vertex_keys(const int64_t* __restrict__ off, int64_t n, int b, int bd,
                              uint64_t* __restrict__ keys, uint64_t* __restrict__ acc,
                              const int32_t* __restrict__ gid_in, uint64_t* __restrict__ accG) {
    grid_begin();
    uint64_t s3 = 0;
    // a caller-built CSR that failed its check (harp_count4_noalloc) is counted as edgeless: every
    // later kernel then stays inside the arrays sized for its (n, m)
    const bool bad_csr = (acc[ACC_ERR] & kErrBadCsr) != 0;
    const int l = lane_id();
    for (int64_t base = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) - l; base < n;
         base += (int64_t)gridDim.x * blockDim.x) {
        const int64_t v = base + l;
        uint64_t c3 = 0;
        int32_t g = 0;
        if (v < n) {
            const uint64_t d = bad_csr ? 0 : (uint64_t)(off[v + 1] - off[v]);
            if (gid_in) g = gid_in[v];
            keys[v] = ((uint64_t)g << (bd + b)) | (d << b) | (uint64_t)v;
            c3 = choose3_u64(d);
        }
        if (gid_in) warp_add_by_graph(accG, G_S, g, c3);
        else s3 += c3;
    }
    __shared__ uint64_t red[32];
    uint64_t t = block_sum_u64(s3, red);
    if (threadIdx.x == 0 && t) atomicAdd((unsigned long long*)&acc[ACC_S], (unsigned long long)t);
}

// New ids = sorted key order.  Rows of more than kTierA neighbours are queued: q holds the warp sort's rows from
// the front and hub rows from the back, q_block the block sort's.
__global__ void k_relabel(const uint64_t* __restrict__ keys, int64_t n, int b, int bd, int32_t* __restrict__ order,
                          int32_t* __restrict__ perm, int32_t* __restrict__ deg,
                          const int32_t* __restrict__ gid_in, int32_t* __restrict__ gid,
                          int32_t* __restrict__ q, int32_t* __restrict__ q_block, uint64_t* __restrict__ acc) {
    grid_begin();
    const uint64_t mask = ((uint64_t)1 << b) - 1;
    const uint64_t dmask = ((uint64_t)1 << bd) - 1;
    const int l = lane_id();
    for (int64_t base = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) - l; base < n;
         base += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = base + l;
        int cls = -1;
        if (i < n) {
            const uint64_t k = keys[i];
            const int32_t old = (int32_t)(k & mask);
            const int32_t d = (int32_t)((k >> b) & dmask);
            order[i] = old;
            perm[old] = (int32_t)i;
            deg[i] = d;
            if (gid_in) gid[i] = gid_in[old];
            cls = d > kTierB ? 1 : (d > kTierB1 ? 2 : (d > kTierA ? 0 : -1));
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const uint32_t m = __ballot_sync(kFull, cls == c);
            if (!m) continue;
            unsigned long long start = 0;
            const int leader = __ffs(m) - 1;
            unsigned long long* ctr = (unsigned long long*)&acc[c == 2 ? Q_SORT_BLOCK : Q_SORT_WARP + c];
            if (l == leader) start = atomicAdd(ctr, (unsigned long long)__popc(m));
            start = __shfl_sync(kFull, start, leader);
            if (cls == c) {
                const unsigned long long k = start + __popc(m & lanemask_lt());
                if (c == 0) q[k] = (int32_t)i;
                else if (c == 1) q[n - 1 - (int64_t)k] = (int32_t)i;
                else q_block[k] = (int32_t)i;
            }
        }
    }
}

// Tier A: rows with 1 <= d <= 32, 32 consecutive rows per warp (consecutive ranks have similar
// degrees).  A row of at most 16 neighbours is sorted by its own lane, a bitonic network over 8 or 16
// registers padded with +inf; the warp then sorts its rows of 17..32 together, a bitonic network over
// the lanes.  A warp per row left most lanes idle on the many short rows of sparse graphs.
template <int P>
__device__ __forceinline__ void lane_sort_row(int64_t i, int d, const int64_t* __restrict__ goff,
                                              const int32_t* __restrict__ gcols, const int32_t* __restrict__ order,
                                              const int32_t* __restrict__ perm, const int64_t* __restrict__ off,
                                              int32_t* __restrict__ cols, int32_t* __restrict__ dplus) {
    const int64_t src = goff[order[i]];
    int32_t a[P];
#pragma unroll
    for (int r = 0; r < P; ++r) a[r] = r < d ? perm[gcols[src + r]] : 0x7fffffff;
    sort_regs<P>(a);
    const int64_t ob = off[i];
    int above = 0;
#pragma unroll
    for (int r = 0; r < P; ++r) {
        if (r < d) {
            cols[ob + r] = a[r];
            above += a[r] > (int32_t)i;
        }
    }
    dplus[i] = above;
}

__global__ void __launch_bounds__(256) k_sort_rows_warp(const int64_t* __restrict__ goff,
                                                        const int32_t* __restrict__ gcols,
                                                        const int32_t* __restrict__ order,
                                                        const int32_t* __restrict__ perm,
                                                        const int32_t* __restrict__ deg,
                                                        const int64_t* __restrict__ off, int64_t n,
                                                        int32_t* __restrict__ cols,
                                                        int32_t* __restrict__ dplus) {
    grid_begin();
    const int l = lane_id();
    const int64_t wid = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i0 = wid * 32; i0 < n; i0 += nw * 32) {
        const int64_t i = i0 + l;
        const int d = i < n ? deg[i] : -1;  // CTA and hub rows (d > 32) are sorted by the queued kernels
        if (d == 0) dplus[i] = 0;
        else if (d >= 1 && d <= 8) lane_sort_row<8>(i, d, goff, gcols, order, perm, off, cols, dplus);
        else if (d > 8 && d <= 16) lane_sort_row<16>(i, d, goff, gcols, order, perm, off, cols, dplus);
        const bool wide = d > 16 && d <= kTierA;
        uint32_t rest = __ballot_sync(kFull, wide);
        if (!rest) continue;
        const int64_t mysrc = wide ? goff[order[i]] : 0, myoff = wide ? off[i] : 0;
        while (rest) {  // four rows at a time: their loads overlap
            int row[4], dr[4];
            int32_t v[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                row[t] = rest ? __ffs(rest) - 1 : -1;
                rest &= rest - 1;
                dr[t] = row[t] >= 0 ? __shfl_sync(kFull, d, row[t] & 31) : 0;
                const int64_t rsrc = __shfl_sync(kFull, mysrc, row[t] & 31);
                v[t] = l < dr[t] ? gcols[rsrc + l] : -1;
            }
#pragma unroll
            for (int t = 0; t < 4; ++t) v[t] = v[t] >= 0 ? perm[v[t]] : 0x7fffffff;
#pragma unroll
            for (int k = 2; k <= 32; k <<= 1) {
#pragma unroll
                for (int j = k >> 1; j > 0; j >>= 1) {
                    const bool keep_min = ((l & j) == 0) == ((l & k) == 0);
#pragma unroll
                    for (int t = 0; t < 4; ++t) {
                        const int32_t o = __shfl_xor_sync(kFull, v[t], j);
                        v[t] = keep_min ? min(v[t], o) : max(v[t], o);
                    }
                }
            }
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                if (row[t] < 0) continue;  // uniform
                const int64_t r = i0 + row[t];
                const int64_t ob = __shfl_sync(kFull, myoff, row[t]);
                if (l < dr[t]) cols[ob + l] = v[t];
                const uint32_t above = __ballot_sync(kFull, l < dr[t] && v[t] > (int32_t)r);
                if (l == 0) dplus[r] = __popc(above);
            }
        }
    }
}

// Tier B1: 32 < d <= 1024, a warp per row, E registers a lane.  (Through shared memory, a warp barrier per
// stage up to 256 and a block barrier per stage above: 0.23 + 0.87 ms on R-MAT scale 20.)
constexpr int kMidWarps = 4;

template <int E>
__device__ __forceinline__ void warp_sort_row(int64_t i, int d, int64_t src, int64_t dst,
                                              const int32_t* __restrict__ gcols, const int32_t* __restrict__ perm,
                                              int32_t* __restrict__ cols, int32_t* __restrict__ dplus) {
    const int l = lane_id();
    int32_t v[E];
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = e * 32 + l < d ? gcols[src + e * 32 + l] : -1;  // any order will do
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = v[e] >= 0 ? perm[v[e]] : 0x7fffffff;
    warp_bitonic_sort<E>(v, true);
    int above = 0;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        if (l * E + e < d) {
            cols[dst + l * E + e] = v[e];
            above += v[e] > (int32_t)i;
        }
    }
    above = warp_sum(above);
    if (l == 0) dplus[i] = above;
}

__global__ void __launch_bounds__(kMidWarps * 32) k_sort_rows_mid(const int64_t* __restrict__ goff,
                                                                   const int32_t* __restrict__ gcols,
                                                                   const int32_t* __restrict__ order,
                                                                   const int32_t* __restrict__ perm,
                                                                   const int32_t* __restrict__ deg,
                                                                   const int64_t* __restrict__ off,
                                                                   int32_t* __restrict__ cols,
                                                                   int32_t* __restrict__ dplus,
                                                                   const int32_t* __restrict__ q,
                                                                   const uint64_t* __restrict__ acc) {
    grid_begin();
    const int64_t nq = (int64_t)acc[Q_SORT_WARP];
    for (int64_t qi = (int64_t)blockIdx.x * kMidWarps + (threadIdx.x >> 5); qi < nq; qi += (int64_t)gridDim.x * kMidWarps) {
        const int64_t i = q[qi];
        const int d = deg[i];
        const int64_t src = goff[order[i]], dst = off[i];
        if (d <= 64) warp_sort_row<2>(i, d, src, dst, gcols, perm, cols, dplus);
        else if (d <= 128) warp_sort_row<4>(i, d, src, dst, gcols, perm, cols, dplus);
        else if (d <= 256) warp_sort_row<8>(i, d, src, dst, gcols, perm, cols, dplus);
        else if (d <= 512) warp_sort_row<16>(i, d, src, dst, gcols, perm, cols, dplus);
        else warp_sort_row<32>(i, d, src, dst, gcols, perm, cols, dplus);
    }
}

// Tier B: 1024 < d <= 4096, one block per row (block_bitonic_sort).

__global__ void __launch_bounds__(kBlockWarps * 32) k_sort_rows_block(const int64_t* __restrict__ goff,
                                                                      const int32_t* __restrict__ gcols,
                                                                      const int32_t* __restrict__ order,
                                                                      const int32_t* __restrict__ perm,
                                                                      const int32_t* __restrict__ deg,
                                                                      const int64_t* __restrict__ off,
                                                                      int32_t* __restrict__ cols,
                                                                      int32_t* __restrict__ dplus,
                                                                      const int32_t* __restrict__ q,
                                                                      const uint64_t* __restrict__ acc) {
    grid_begin();
    constexpr int E = kBlockE, RUN = 32 * E;
    __shared__ int32_t buf[kTierB];
    __shared__ int s_above[kBlockWarps];
    const int w = threadIdx.x >> 5, l = lane_id();
    const int64_t nq = (int64_t)acc[Q_SORT_BLOCK];
    for (int64_t qi = blockIdx.x; qi < nq; qi += gridDim.x) {
        const int64_t i = q[qi];
        const int d = deg[i];
        const int64_t src = goff[order[i]], dst = off[i];
        int32_t v[E];
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int k = w * RUN + e * 32 + l;
            v[e] = k < d ? gcols[src + k] : -1;
        }
#pragma unroll
        for (int e = 0; e < E; ++e) v[e] = v[e] >= 0 ? perm[v[e]] : 0x7fffffff;
        block_bitonic_sort(v, buf);
        int above = 0;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int k = w * RUN + l * E + e;
            if (k < d) {
                cols[dst + k] = v[e];
                above += v[e] > (int32_t)i;
            }
        }
        above = warp_sum(above);
        if (l == 0) s_above[w] = above;
        __syncthreads();
        if (threadIdx.x == 0) {
            int t = 0;
            for (int x = 0; x < kBlockWarps; ++x) t += s_above[x];
            dplus[i] = t;
        }
        __syncthreads();
    }
}

// Tier C: hubs (d > 4096) of graphs of at most kBitmapRanks ranks: a block per row sets the row's ranks in a bitmap
// in shared memory and writes them out in order, a window of ranks at a time (one for up to 1.6 M ranks).
// again (rows of a caller's CSR, which may hold a rank more than once; nullptr: such rows cannot occur): a row that
// comes out short is queued from the back for the radix sort below, which keeps repeats, so that all of
// its deg entries are written.
__global__ void __launch_bounds__(kBitmapThreads) k_sort_rows_bitmap(const int64_t* __restrict__ goff,
                                                                     const int32_t* __restrict__ gcols,
                                                                     const int32_t* __restrict__ order,
                                                                     const int32_t* __restrict__ perm,
                                                                     const int32_t* __restrict__ deg,
                                                                     const int64_t* __restrict__ off, int64_t n,
                                                                     const int32_t* __restrict__ gid,
                                                                     const int64_t* __restrict__ gbase,
                                                                     int32_t* __restrict__ cols,
                                                                     int32_t* __restrict__ dplus,
                                                                     const int32_t* __restrict__ q,
                                                                     int32_t* __restrict__ again,
                                                                     uint64_t* __restrict__ acc) {
    grid_begin();
    extern __shared__ uint32_t bm[];
    __shared__ int s_count[kBitmapWarps];
    __shared__ int s_above;
    const int w = threadIdx.x >> 5, l = lane_id();
    const int64_t nq = (int64_t)acc[Q_SORT_WARP + 1];
    for (int64_t qi = blockIdx.x; qi < nq; qi += gridDim.x) {
        const int64_t i = q[n - 1 - qi];
        const int64_t d = deg[i], src = goff[order[i]];
        const int64_t r0 = gid ? gbase[gid[i]] : 0, r1 = gid ? gbase[gid[i] + 1] : n;  // the graph's ranks
        int64_t dst = off[i];
        if (threadIdx.x == 0) s_above = 0;
        int above = 0;
        for (int64_t lo = r0; lo < r1; lo += 32 * (int64_t)kBitmapWords) {
            const int64_t hi = lo + 32 * (int64_t)kBitmapWords < r1 ? lo + 32 * (int64_t)kBitmapWords : r1;
            // each warp's share of the words: whole groups of 32
            const int groups = (int)((hi - lo + 1023) / 1024), per = (groups + kBitmapWarps - 1) / kBitmapWarps;
            for (int k = threadIdx.x; k < per * kBitmapThreads; k += kBitmapThreads) bm[k] = 0;
            __syncthreads();
            for (int64_t k0 = threadIdx.x; k0 < d; k0 += 4 * kBitmapThreads) {
                int32_t x[4];
#pragma unroll
                for (int t = 0; t < 4; ++t) x[t] = k0 + t * kBitmapThreads < d ? gcols[src + k0 + t * kBitmapThreads] : -1;
#pragma unroll
                for (int t = 0; t < 4; ++t) x[t] = x[t] >= 0 ? perm[x[t]] : -1;
#pragma unroll
                for (int t = 0; t < 4; ++t)
                    if (x[t] >= lo && x[t] < hi) {
                        const uint32_t b = (uint32_t)(x[t] - lo);
                        atomicOr(&bm[b >> 5], 1u << (b & 31));
                    }
            }
            __syncthreads();
            dst += bitmap_write(bm, per, lo, cols + dst, s_count, [&](int32_t x) { above += x > (int32_t)i; });
            __syncthreads();  // the bitmap is read before the next window clears it
        }
        above = warp_sum(above);
        if (l == 0 && above) atomicAdd(&s_above, above);
        __syncthreads();
        if (threadIdx.x == 0) {
            dplus[i] = s_above;
            if (again && dst - off[i] != d)
                again[n - 1 - (int64_t)atomicAdd((unsigned long long*)&acc[Q_SORT_AGAIN], 1ull)] = (int32_t)i;
        }
        __syncthreads();
    }
}

// Tier C, graphs of more ranks (and rows with repeats): one block per hub row, LSD radix sort (8-bit digits) through global memory.
// Pass p reads the previous pass's output; pass 0 reads the old row through perm.  The pass count
// decides which buffer each pass writes so that the last one lands in `cols`.
constexpr int kHubThreads = 512;
constexpr int kHubWarps = kHubThreads / 32;

__global__ void __launch_bounds__(kHubThreads) k_sort_rows_hub(const int64_t* __restrict__ goff,
                                                               const int32_t* __restrict__ gcols,
                                                               const int32_t* __restrict__ order,
                                                               const int32_t* __restrict__ perm,
                                                               const int32_t* __restrict__ deg,
                                                               const int64_t* __restrict__ off, int64_t n,
                                                               int nbits, int32_t* __restrict__ cols,
                                                               int32_t* __restrict__ tmp,
                                                               int32_t* __restrict__ dplus,
                                                               const int32_t* __restrict__ q,
                                                               const uint64_t* __restrict__ qcnt) {
    grid_begin();
    __shared__ uint32_t base[256];
    __shared__ uint32_t wcnt[kHubWarps][256];
    __shared__ int cnt_below;
    const int npass = (nbits + 7) / 8;
    const int w = threadIdx.x >> 5, l = lane_id();
    const uint32_t lt = lanemask_lt();
    const int64_t nq = (int64_t)*qcnt;
    for (int64_t qi = blockIdx.x; qi < nq; qi += gridDim.x) {
        const int64_t i = q[n - 1 - qi];
        const int64_t d = deg[i];
        const int64_t src = goff[order[i]];
        const int64_t dst0 = off[i];
        for (int p = 0; p < npass; ++p) {
            const int shift = 8 * p;
            const bool to_cols = ((npass - 1 - p) & 1) == 0;
            int32_t* out = (to_cols ? cols : tmp) + dst0;
            const int32_t* in = (p == 0) ? nullptr : ((to_cols ? tmp : cols) + dst0);
            // histogram of the row
            for (int k = threadIdx.x; k < 256; k += blockDim.x) base[k] = 0;
            __syncthreads();
            for (int64_t k = threadIdx.x; k < d; k += blockDim.x) {
                int32_t x = in ? in[k] : perm[gcols[src + k]];
                atomicAdd(&base[((uint32_t)x >> shift) & 255u], 1u);
            }
            __syncthreads();
            if (threadIdx.x < 32) {  // exclusive scan of 256 counters by one warp
                uint32_t c[8], s = 0;
#pragma unroll
                for (int q = 0; q < 8; ++q) { c[q] = base[threadIdx.x * 8 + q]; s += c[q]; }
                uint32_t inc = s;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    uint32_t u = __shfl_up_sync(kFull, inc, o);
                    if (threadIdx.x >= o) inc += u;
                }
                uint32_t run = inc - s;
#pragma unroll
                for (int q = 0; q < 8; ++q) { base[threadIdx.x * 8 + q] = run; run += c[q]; }
            }
            __syncthreads();
            // stable scatter, tile by tile (tile = kHubThreads keys, warp-contiguous)
            for (int64_t t0 = 0; t0 < d; t0 += kHubThreads) {
                for (int k = threadIdx.x; k < kHubWarps * 256; k += blockDim.x) (&wcnt[0][0])[k] = 0;
                __syncthreads();
                const int64_t k = t0 + w * 32 + l;
                const bool valid = k < d;
                int32_t x = 0;
                if (valid) x = in ? in[k] : perm[gcols[src + k]];
                const uint32_t dg = valid ? (((uint32_t)x >> shift) & 255u) : 256u;
                const uint32_t peers = __match_any_sync(kFull, dg);
                const uint32_t r = __popc(peers & lt);
                if (valid && r == 0) wcnt[w][dg] = __popc(peers);
                __syncthreads();
                if (threadIdx.x < 256) {  // exclusive over warps, add the running digit base
                    uint32_t run = base[threadIdx.x];
                    for (int ww = 0; ww < kHubWarps; ++ww) {
                        uint32_t c = wcnt[ww][threadIdx.x];
                        wcnt[ww][threadIdx.x] = run;
                        run += c;
                    }
                    base[threadIdx.x] = run;
                }
                __syncthreads();
                if (valid) out[wcnt[w][dg] + r] = x;
                __syncthreads();
            }
            __syncthreads();
        }
        // out-degree: elements above i in the sorted row
        if (threadIdx.x == 0) cnt_below = 0;
        __syncthreads();
        int below = 0;
        for (int64_t k = threadIdx.x; k < d; k += blockDim.x) below += cols[dst0 + k] < (int32_t)i;
        below = warp_sum(below);
        if (l == 0 && below) atomicAdd(&cnt_below, below);
        __syncthreads();
        if (threadIdx.x == 0) dplus[i] = (int32_t)(d - cnt_below);
        __syncthreads();
    }
}

// N+ of every vertex (the end of its sorted row) into colsp, t_e cleared, and the sum over the arcs of
// (d_u - 1)(d_v - 1).  A warp per `run` consecutive out-arcs: the row of the first is searched (32 probes a round), then
// the lanes hold 32 rows and each arc looks its row up among them.  Bound by the loads' latency (four in flight) and
// the scattered reads of degrees.  Before (32 rows per warp, short ones a lane each, long ones in
// turn) and now: R-MAT scale 20 212 and 88 us, Chung-Lu of 2,000,000 vertices 468 and 225 us, the union of 4,096 graphs 830 and
// 650 us.
__global__ void __launch_bounds__(256) k_out_csr(const int64_t* __restrict__ off, const int32_t* __restrict__ cols,
                                                 const int32_t* __restrict__ deg, const int64_t* __restrict__ offp,
                                                 int64_t n, int run, int32_t* __restrict__ colsp,
                                                 uint32_t* __restrict__ te, Sink sink) {
    grid_begin();
    __shared__ uint64_t red[32];
    const int l = lane_id();
    const int64_t M = offp[n], nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    uint64_t pw = 0;  // of graph g in a batch
    int32_t g = -1;
    auto flush = [&] {
        const uint64_t t = warp_sum(pw);
        if (l == 0 && g >= 0 && t) atomicAdd((unsigned long long*)&sink.accG[(int64_t)g * kGStride + G_PW], (unsigned long long)t);
        pw = 0;
    };
    for (int64_t t0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * run; t0 < M; t0 += nw * run) {
        const int64_t t1 = t0 + run < M ? t0 + run : M;
        int64_t r0 = 0, hi = n;  // the last row that begins at or before t0: offp[r0] <= t0 < offp[hi]
        while (hi - r0 > 1) {
            const int64_t step = (hi - r0 + 31) >> 5, p = r0 + (int64_t)(l + 1) * step;
            const uint32_t m = __ballot_sync(kFull, p >= hi || offp[p] > t0);
            r0 += (int64_t)(__ffs(m) - 1) * step;
            hi = r0 + step < hi ? r0 + step : hi;
        }
        for (int64_t cur = t0; cur < t1; r0 += 32) {
            const int64_t r = r0 + l < n ? r0 + l : n;
            const int64_t o = offp[r];
            const int64_t next = offp[r0 + 32 < n ? r0 + 32 : n];
            if (next <= cur) continue;  // these rows are empty
            const int64_t shift = r < n ? off[r + 1] - offp[r + 1] : 0;  // the row's end in cols less its end in colsp
            const uint32_t du = r < n ? (uint32_t)deg[r] - 1u : 0u;
            const int32_t gr = sink.batch() && r < n ? sink.gid[r] : 0;
            const int64_t end = next < t1 ? next : t1;
            for (int64_t b = cur; b < end; b += 128) {
                int32_t v[4];
                int k[4];
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    const int64_t t = b + 32 * h + l;
                    k[h] = 0;  // last row with o <= t
#pragma unroll
                    for (int sft = 16; sft >= 1; sft >>= 1) {
                        const int64_t x = __shfl_sync(kFull, o, k[h] + sft);
                        if (x <= t) k[h] += sft;
                    }
                    const int64_t at = t + __shfl_sync(kFull, shift, k[h]);
                    v[h] = t < end ? cols[at] : -1;
                }
                uint32_t dv[4];
#pragma unroll
                for (int h = 0; h < 4; ++h) dv[h] = v[h] >= 0 ? (uint32_t)deg[v[h]] - 1u : 0u;
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    if (b + 32 * h >= end) break;
                    const int64_t t = b + 32 * h + l;
                    if (v[h] >= 0) {
                        colsp[t] = v[h];
                        te[t] = 0;
                    }
                    const uint64_t x = (uint64_t)__shfl_sync(kFull, du, k[h]) * dv[h];
                    if (sink.batch()) {
                        const int32_t ge = __shfl_sync(kFull, gr, k[h]);
                        const int32_t first = __shfl_sync(kFull, ge, 0);
                        if (first != g) {
                            flush();
                            g = first;
                        }
                        if (!__all_sync(kFull, v[h] < 0 || ge == g)) {  // rows of several graphs
                            warp_add_by_graph(sink.accG, G_PW, v[h] >= 0 ? ge : -1, x);
                            continue;
                        }
                    }
                    pw += x;
                }
            }
            cur = end;
        }
    }
    if (sink.batch()) {
        flush();
        return;
    }
    pw = block_sum_u64(pw, red);
    if (threadIdx.x == 0 && pw) atomicAdd((unsigned long long*)&sink.acc[ACC_PW], (unsigned long long)pw);
}

// A caller's CSR need not list every edge in both rows: then more than m arcs may point upwards in rank, and what is laid
// out for m of them (t_e above all) would be written past its end.  Such a graph is counted as edgeless
// and flagged.  One block: the rest of the device has nothing to do here.
__global__ void __launch_bounds__(1024) k_check_out_arcs(int64_t n, int64_t m, int32_t* __restrict__ deg,
                                                         int32_t* __restrict__ dplus, int64_t* __restrict__ off,
                                                         int64_t* __restrict__ offp, uint64_t* __restrict__ acc) {
    grid_begin();
    const bool bad = offp[n] > m;
    __syncthreads();  // every thread has read offp[n]
    if (!bad) return;
    for (int64_t v = threadIdx.x; v <= n; v += 1024) {
        off[v] = offp[v] = 0;
        if (v < n) deg[v] = dplus[v] = 0;
    }
    if (threadIdx.x == 0) {
        acc[ACC_S] = 0;
        acc[ACC_ERR] |= kErrBadCsr;
    }
}

}  // namespace

harp_status orient(const harp_csr* g, Workspace& ws, cudaStream_t s) {
    const int64_t n = g->n, m = g->m;
    if (n == 0) return HARP_OK;
    const int b = bits_for(n);
    const int bd = bits_for(g->max_deg);
    const int bg = ws.gid_in && ws.G > 1 ? bits_for(ws.G - 1) : 0;
    if (b + bd + bg > 64) return HARP_EOVERFLOW;

    // rank = (graph, degree, id): each graph's vertices form one contiguous rank range, sorted by
    // degree (a single graph is graph 0)
    launch(k_vertex_keys, grid_for(n, 256), 256, 0, s, g->off, n, b, bd, ws.vkeys, ws.acc, ws.gid_in, ws.accG);
    HARP_LAUNCHED();
    uint64_t* k0 = ws.vkeys;
    uint64_t* k1 = ws.vkeys_alt;
    // the keys are written in id order and every pass is stable, so only the graph and degree bits
    // need sorting: equal (graph, degree) keep ascending ids
    HARP_TRY(radix_sort_u64(&k0, &k1, n, b, b + bd + bg, ws.hist, ws.scan_tmp, ws.scan_tmp_len, s));
    launch(k_relabel, grid_for(n, 256), 256, 0, s, k0, n, b, bd, ws.order, ws.perm, ws.deg, ws.gid_in, ws.gid,
           ws.q_tri, ws.q_mid, ws.acc);
    HARP_LAUNCHED();
    HARP_TRY(exclusive_scan_i32_to_i64(ws.deg, ws.off, n, ws.scan_tmp, ws.scan_tmp_len, s));
    if (m > 0) {
        // 32 rows per warp
        launch(k_sort_rows_warp, grid_for(n, 256), 256, 0, s, g->off, g->cols, ws.order, ws.perm, ws.deg, ws.off, n,
               ws.cols, ws.dplus);
        HARP_LAUNCHED();
        if (g->max_deg > kTierA) {
            launch(k_sort_rows_mid, num_sms() * 8, kMidWarps * 32, 0, s, g->off, g->cols, ws.order, ws.perm, ws.deg,
                   ws.off, ws.cols, ws.dplus, ws.q_tri, ws.acc);
            HARP_LAUNCHED();
        }
        if (g->max_deg > kTierB1) {
            launch(k_sort_rows_block, num_sms() * 4, kBlockWarps * 32, 0, s, g->off, g->cols, ws.order, ws.perm,
                   ws.deg, ws.off, ws.cols, ws.dplus, ws.q_mid, ws.acc);
            HARP_LAUNCHED();
        }
        const int64_t most_n = ws.G > 1 ? ws.max_member_n : n;  // ranks of the largest graph
        const bool bitmap = most_n <= kBitmapRanks;
        int32_t* again = g->simple ? nullptr : ws.q_mid + n;
        if (g->max_deg > kTierB && bitmap) {
            const size_t smem = sizeof(uint32_t) * (size_t)kBitmapWords;
            HARP_CK(cudaFuncSetAttribute(k_sort_rows_bitmap, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
            launch(k_sort_rows_bitmap, num_sms(), kBitmapThreads, smem, s, g->off, g->cols, ws.order, ws.perm, ws.deg,
                   ws.off, n, ws.G > 1 ? ws.gid : nullptr, ws.gbase, ws.cols, ws.dplus, ws.q_tri, again, ws.acc);
            HARP_LAUNCHED();
        }
        if (g->max_deg > kTierB && (!bitmap || again)) {
            // the out-CSR columns + t_e region (2m int32) is free until k_out_csr: hub sort ping-pong
            launch(k_sort_rows_hub, num_sms(), kHubThreads, 0, s, g->off, g->cols, ws.order, ws.perm, ws.deg, ws.off,
                   n, b, ws.cols, ws.colsp, ws.dplus, bitmap ? again : ws.q_tri,
                   &ws.acc[bitmap ? Q_SORT_AGAIN : Q_SORT_WARP + 1]);
            HARP_LAUNCHED();
        }
    } else {
        HARP_CK(cudaMemsetAsync(ws.dplus, 0, (size_t)n * sizeof(int32_t), s));
    }
    HARP_TRY(exclusive_scan_i32_to_i64(ws.dplus, ws.offp, n, ws.scan_tmp, ws.scan_tmp_len, s));
    if (!g->simple) {
        launch(k_check_out_arcs, 1, 1024, 0, s, n, m, ws.deg, ws.dplus, ws.off, ws.offp, ws.acc);
        HARP_LAUNCHED();
    }
    if (m > 0) {
        const Sink sink{ws.acc, ws.gid, ws.accG};
        const int run = m >= (1 << 20) ? 1024 : (m >= (1 << 17) ? 256 : 32);  // small graphs: enough warps
        launch(k_out_csr, grid_for((m + run - 1) / run * 32, 256), 256, 0, s, ws.off, ws.cols, ws.deg, ws.offp, n, run,
               ws.colsp, ws.te, sink);
        HARP_LAUNCHED();
    }
    return HARP_OK;
}

}  // namespace harp
