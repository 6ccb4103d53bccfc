// harp_build_csr on the device: degrees -> offsets -> scatter -> rows sorted and deduplicated -> CSR.
//
// Every input pair (u, v), u != v, counts towards both degrees and is scattered into both rows at slots taken by
// atomics (equal endpoints within a warp take theirs together: edge lists often run along one vertex).  Self-loops
// are skipped; out-of-range ids are skipped and raise a flag that turns into HARP_EINVAL.  Rows are then sorted by
// the tiers of rowsort.cuh (very long ones, and hubs among very many ids, by one radix sort of them all), equal
// neighbours dropped while they are written, and, where any were, the rows closed up.  The rows' order makes the result independent of the order in which slots were taken.
// (A radix sort of all arcs as 64-bit keys moved every arc 2 * bits(n) / 8 times.)  Kernels of a build, with the sort and
// now: R-MAT scale 20 2.8 and 1.6 ms, Chung-Lu of 1,347,423 vertices (hubs of close ids) 2.2 and 1.4 ms, random
// geometric of 1,000,003 vertices 1.24 and 0.30 ms.
#include "harp_internal.cuh"
#include "rowsort.cuh"

namespace harp {
namespace {

// Words of the build's summary, read back by the host.
enum : int { B_BAD = 0, B_MAXDEG, B_ARCS, B_Q_WARP, B_Q_BLOCK, B_Q_HUB, B_Q_LONG, B_LONG_LEN, B_WORDS = 8 };

// Fewer vertices keep their counters by id: the copy back costs a launch and there is little to contend for.
constexpr int64_t kSpreadMinN = 1 << 14;

// An input pair's endpoints; valid: in range and not a self-loop.
struct Pair {
    int32_t u, v;
    bool valid;
};

__device__ __forceinline__ Pair load_pair(const int32_t* __restrict__ src, const int32_t* __restrict__ dst, int64_t e,
                                          int64_t m_in, int64_t n, bool& bad) {
    Pair p{-1, -1, false};
    if (e < m_in) {
        p.u = src[e];
        p.v = dst[e];
        const bool ok = p.u >= 0 && p.v >= 0 && (int64_t)p.u < n && (int64_t)p.v < n;
        bad |= !ok;
        p.valid = ok && p.u != p.v;
    }
    return p;
}

// Where a vertex's counter lies: ids 32 apart are neighbours, so that hubs of close ids (weights or arrival times that
// fall with the id) are counted in different L2 slices; stride 0: by id.  Chung-Lu of 1,347,423 vertices: degrees 1.07
// -> 0.36 ms, scatter 1.14 -> 0.48 ms.
struct Spread {
    int64_t stride;
    __device__ __forceinline__ int64_t at(int64_t v) const { return stride ? (v & 31) * stride + (v >> 5) : v; }
};

// the counters by id
__global__ void __launch_bounds__(256) k_build_gather(const int32_t* __restrict__ deg, Spread at, int64_t n,
                                                      int32_t* __restrict__ by_id) {
    grid_begin();
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
        by_id[v] = deg[at.at(v)];
}

__global__ void __launch_bounds__(256) k_build_degrees(const int32_t* __restrict__ src, const int32_t* __restrict__ dst,
                                                       int64_t m_in, int64_t n, Spread at, int32_t* __restrict__ deg,
                                                       unsigned long long* __restrict__ summary) {
    grid_begin();
    const int l = lane_id();
    bool bad = false;
    for (int64_t base = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) - l; base < m_in;
         base += (int64_t)gridDim.x * blockDim.x) {
        const Pair p = load_pair(src, dst, base + l, m_in, n, bad);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int32_t x = p.valid ? (h ? p.v : p.u) : -1 - l;
            const uint32_t same = __match_any_sync(kFull, x);
            if (p.valid && l == __ffs(same) - 1) atomicAdd(&deg[at.at(x)], __popc(same));
        }
    }
    if (__any_sync(kFull, bad) && l == 0) atomicOr(&summary[B_BAD], 1ull);
}

// deg counts down to zero: each pair's slot is the value before.
__global__ void __launch_bounds__(256) k_build_scatter(const int32_t* __restrict__ src, const int32_t* __restrict__ dst,
                                                       int64_t m_in, int64_t n, const int64_t* __restrict__ roff,
                                                       Spread at, int32_t* __restrict__ deg, int32_t* __restrict__ out) {
    grid_begin();
    const int l = lane_id();
    bool bad = false;
    for (int64_t base = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) - l; base < m_in;
         base += (int64_t)gridDim.x * blockDim.x) {
        const Pair p = load_pair(src, dst, base + l, m_in, n, bad);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int32_t x = p.valid ? (h ? p.v : p.u) : -1 - l, y = h ? p.u : p.v;
            const uint32_t same = __match_any_sync(kFull, x);
            const int leader = __ffs(same) - 1;
            int left = 0;
            if (p.valid && l == leader) left = atomicSub(&deg[at.at(x)], __popc(same));
            left = __shfl_sync(kFull, left, leader);
            if (p.valid) out[roff[x] + left - 1 - __popc(same & lanemask_lt())] = y;
        }
    }
}

// Hub rows whose bitmap sort may not pay: a block reads its row once for each window of ids, about 1 ns an entry, while
// the rest of the device may have nothing to do, and every window is cleared and searched (5 us) whatever the row
// holds.  Rows of more than 2^18 entry reads, and all hub rows where the ids take more than four windows (the
// bound of the orientation's rows too), wait for the host, which knows their number and length then and takes a
// radix sort of all of them over the device (0.15 ns an entry) where that is estimated to be faster.  Whole builds by
// bitmaps alone and now, the radix sort of all arcs that the build once was in brackets: a star of 5,900,000 leaves
// 10.0 and 1.3 ms [1.5], of 99,000,000 1,134 and 25 [23]; 20,000 rows of 5,000 among 100,000,000 ids 130 and 28 [23], among
// 500,000,000 585 and 45 [26: the other passes here go over the ids]; Chung-Lu of 20,000,000 vertices 28 and 25 [48].  300
// rows of 300,000 among 20,000,000 ids keep to bitmaps: 11 ms, by the radix sort 17 [19].
constexpr int64_t kLongReads = 1 << 18;
int64_t bitmap_windows(int64_t n) { return (n + 32 * (int64_t)kBitmapWords - 1) / (32 * (int64_t)kBitmapWords); }
// hub rows of more entries than this are long
int64_t long_above(int64_t n) { return n > kBitmapRanks ? 0 : kLongReads / bitmap_windows(n); }
// nr long rows of H entries
bool long_by_bitmap(int64_t n, int64_t nr, int64_t H) {
    const double turns = (double)((nr + num_sms() - 1) / num_sms());
    const double bitmap_us = turns * (double)bitmap_windows(n) * (5.0 + 1.0e-3 * (double)H / (double)nr);
    return bitmap_us < 100.0 + 0.15e-3 * (double)H;
}

// Rows of at most kTierA entries, 32 consecutive rows per warp (a lane's network up to 16, the warp's above); longer
// ones are queued: the warp sort's from the front of q, hubs from its back, the block sort's from the front of
// q_block, long rows from its back, with their entries added up.
template <int P>
__device__ __forceinline__ int lane_unique_row(const int32_t* __restrict__ in, int32_t* __restrict__ out, int d) {
    int32_t a[P];
#pragma unroll
    for (int r = 0; r < P; ++r) a[r] = r < d ? in[r] : kPadKey;
    sort_regs<P>(a);
    int k = 0;
#pragma unroll
    for (int r = 0; r < P; ++r)
        if (r < d && (r == 0 || a[r] != a[r - 1])) out[k++] = a[r];
    return k;
}

__global__ void __launch_bounds__(256) k_build_rows_small(const int64_t* __restrict__ roff, int64_t n,
                                                          const int32_t* __restrict__ in, int32_t* __restrict__ out,
                                                          int32_t* __restrict__ ndeg, int32_t* __restrict__ q,
                                                          int32_t* __restrict__ q_block, int64_t long_limit,
                                                          unsigned long long* __restrict__ summary) {
    grid_begin();
    const int l = lane_id();
    const int64_t wid = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i0 = wid * 32; i0 < n; i0 += nw * 32) {
        const int64_t i = i0 + l;
        const int64_t b = i < n ? roff[i] : 0;
        const int d = i < n ? (int)(roff[i + 1] - b) : -1;
        const int cls = d > kTierB ? (d > long_limit ? 3 : 2) : (d > kTierB1 ? 1 : (d > kTierA ? 0 : -1));
        if (d == 0 || cls == 3) ndeg[i] = 0;
        else if (d >= 1 && d <= 8) ndeg[i] = lane_unique_row<8>(in + b, out + b, d);
        else if (d > 8 && d <= 16) ndeg[i] = lane_unique_row<16>(in + b, out + b, d);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const uint32_t m = __ballot_sync(kFull, cls == c);
            if (!m) continue;
            unsigned long long start = 0;
            const int leader = __ffs(m) - 1;
            if (l == leader) start = atomicAdd(&summary[B_Q_WARP + c], (unsigned long long)__popc(m));
            start = __shfl_sync(kFull, start, leader);
            if (cls != c) continue;
            const int64_t k = (int64_t)start + __popc(m & lanemask_lt());
            if (c == 0) q[k] = (int32_t)i;
            else if (c == 1) q_block[k] = (int32_t)i;
            else if (c == 2) q[n - 1 - k] = (int32_t)i;
            else q_block[n - 1 - k] = (int32_t)i;
            if (c == 3) atomicAdd(&summary[B_LONG_LEN], (unsigned long long)d);
        }
        uint32_t rest = __ballot_sync(kFull, d > 16 && d <= kTierA);
        while (rest) {  // four rows at a time: their loads overlap
            int row[4], dr[4];
            int64_t rb[4];
            int32_t v[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                row[t] = rest ? __ffs(rest) - 1 : -1;
                rest &= rest - 1;
                dr[t] = __shfl_sync(kFull, d, row[t] & 31);
                if (row[t] < 0) dr[t] = 0;
                rb[t] = __shfl_sync(kFull, b, row[t] & 31);
                v[t] = l < dr[t] ? in[rb[t] + l] : kPadKey;
            }
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
                const int32_t before = __shfl_up_sync(kFull, v[t], 1);
                const bool first = l < dr[t] && (l == 0 || v[t] != before);
                const uint32_t kept = __ballot_sync(kFull, first);
                if (first) out[rb[t] + __popc(kept & lanemask_lt())] = v[t];
                if (l == 0 && row[t] >= 0) ndeg[i0 + row[t]] = __popc(kept);
            }
        }
    }
}

// Unique members of a sorted run held lane * E + e in v (d of them count); before: the key ahead of the run's
// first (kPadKey: none).  Writes them from out on and returns their number (in every lane).
template <int E>
__device__ __forceinline__ int warp_write_unique(const int32_t (&v)[E], int d, int32_t before, int32_t* __restrict__ out) {
    const int l = lane_id();
    const int32_t up = __shfl_up_sync(kFull, v[E - 1], 1);
    uint32_t keep = 0;  // bit e: register e is the first of its value
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int32_t prev = e > 0 ? v[e > 0 ? e - 1 : 0] : (l > 0 ? up : before);
        if (l * E + e < d && v[e] != prev) keep |= 1u << e;
    }
    const int c = __popc(keep);
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kFull, incl, o);
        if (l >= o) incl += y;
    }
    int at = incl - c;
#pragma unroll
    for (int e = 0; e < E; ++e)
        if ((keep >> e) & 1u) out[at++] = v[e];
    return __shfl_sync(kFull, incl, 31);
}

constexpr int kMidWarps = 4;

template <int E>
__device__ __forceinline__ int warp_unique_row(const int32_t* __restrict__ in, int32_t* __restrict__ out, int d) {
    const int l = lane_id();
    int32_t v[E];
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = e * 32 + l < d ? in[e * 32 + l] : kPadKey;  // any order will do
    warp_bitonic_sort<E>(v, true);
    return warp_write_unique<E>(v, d, kPadKey, out);
}

__global__ void __launch_bounds__(kMidWarps * 32) k_build_rows_mid(const int64_t* __restrict__ roff,
                                                                    const int32_t* __restrict__ in,
                                                                    int32_t* __restrict__ out, int32_t* __restrict__ ndeg,
                                                                    const int32_t* __restrict__ q,
                                                                    const unsigned long long* __restrict__ summary) {
    grid_begin();
    const int64_t nq = (int64_t)summary[B_Q_WARP];
    for (int64_t k = (int64_t)blockIdx.x * kMidWarps + (threadIdx.x >> 5); k < nq; k += (int64_t)gridDim.x * kMidWarps) {
        const int64_t i = q[k], b = roff[i];
        const int d = (int)(roff[i + 1] - b);
        int u;
        if (d <= 64) u = warp_unique_row<2>(in + b, out + b, d);
        else if (d <= 128) u = warp_unique_row<4>(in + b, out + b, d);
        else if (d <= 256) u = warp_unique_row<8>(in + b, out + b, d);
        else if (d <= 512) u = warp_unique_row<16>(in + b, out + b, d);
        else u = warp_unique_row<32>(in + b, out + b, d);
        if (lane_id() == 0) ndeg[i] = u;
    }
}

__global__ void __launch_bounds__(kBlockWarps * 32) k_build_rows_block(const int64_t* __restrict__ roff,
                                                                       const int32_t* __restrict__ in,
                                                                       int32_t* __restrict__ out,
                                                                       int32_t* __restrict__ ndeg,
                                                                       const int32_t* __restrict__ q_block,
                                                                       const unsigned long long* __restrict__ summary) {
    grid_begin();
    constexpr int E = kBlockE, RUN = 32 * E;
    __shared__ int32_t buf[kTierB];
    __shared__ int32_t s_last[kBlockWarps];
    __shared__ int s_kept[kBlockWarps];
    const int w = threadIdx.x >> 5, l = lane_id();
    const int64_t nq = (int64_t)summary[B_Q_BLOCK];
    for (int64_t k = blockIdx.x; k < nq; k += gridDim.x) {
        const int64_t i = q_block[k], b = roff[i];
        const int d = (int)(roff[i + 1] - b);
        int32_t v[E];
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int x = w * RUN + e * 32 + l;
            v[e] = x < d ? in[b + x] : kPadKey;
        }
        block_bitonic_sort(v, buf);
        if (l == 31) s_last[w] = v[E - 1];
        __syncthreads();
        const int32_t before = w > 0 ? s_last[w - 1] : kPadKey;
        const int mine = d - w * RUN < 0 ? 0 : (d - w * RUN < RUN ? d - w * RUN : RUN);
        // the warp's unique keys go to its own part of buf, then behind those of the warps before it
        const int kept = warp_write_unique<E>(v, mine, before, buf + w * RUN);
        if (l == 0) s_kept[w] = kept;
        __syncthreads();
        int at = 0, all = 0;
        for (int x = 0; x < kBlockWarps; ++x) {
            if (x < w) at += s_kept[x];
            all += s_kept[x];
        }
        for (int x = l; x < kept; x += 32) out[b + at + x] = buf[w * RUN + x];
        if (threadIdx.x == 0) ndeg[i] = all;
        __syncthreads();  // buf and the shared words are read before the next row
    }
}

__global__ void __launch_bounds__(kBitmapThreads) k_build_rows_bitmap(const int64_t* __restrict__ roff, int64_t n,
                                                                      const int32_t* __restrict__ in,
                                                                      int32_t* __restrict__ out,
                                                                      int32_t* __restrict__ ndeg,
                                                                      const int32_t* __restrict__ q,
                                                                      const unsigned long long* __restrict__ count) {
    grid_begin();
    extern __shared__ uint32_t bm[];
    __shared__ int s_count[kBitmapWarps];
    const int64_t nq = (int64_t)*count;
    for (int64_t k = blockIdx.x; k < nq; k += gridDim.x) {
        const int64_t i = q[n - 1 - k], b = roff[i], e = roff[i + 1];
        int64_t dst = b;
        for (int64_t lo = 0; lo < n; lo += 32 * (int64_t)kBitmapWords) {
            const int64_t hi = lo + 32 * (int64_t)kBitmapWords < n ? lo + 32 * (int64_t)kBitmapWords : n;
            const int groups = (int)((hi - lo + 1023) / 1024), per = (groups + kBitmapWarps - 1) / kBitmapWarps;
            for (int x = threadIdx.x; x < per * kBitmapThreads; x += kBitmapThreads) bm[x] = 0;
            __syncthreads();
            for (int64_t p = b + threadIdx.x; p < e; p += 4 * kBitmapThreads) {
                int32_t x[4];
#pragma unroll
                for (int t = 0; t < 4; ++t) x[t] = p + t * kBitmapThreads < e ? in[p + t * kBitmapThreads] : -1;
#pragma unroll
                for (int t = 0; t < 4; ++t)
                    if (x[t] >= lo && x[t] < hi) {
                        const uint32_t y = (uint32_t)(x[t] - lo);
                        atomicOr(&bm[y >> 5], 1u << (y & 31));
                    }
            }
            __syncthreads();
            dst += bitmap_write(bm, per, lo, out + dst, s_count, [](int32_t) {});
            __syncthreads();  // the bitmap is read before the next window clears it
        }
        if (threadIdx.x == 0) ndeg[i] = (int32_t)(dst - b);
    }
}

// Long rows by radix sort, nr of them in q_block from the back: their entries as keys (row's place in the queue, id), radix-sorted,
// the first of each value written to its row.
__global__ void __launch_bounds__(256) k_long_lengths(const int64_t* __restrict__ roff, int64_t n,
                                                      const int32_t* __restrict__ q_block, int64_t nr,
                                                      int32_t* __restrict__ len) {
    grid_begin();
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < nr; k += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = q_block[n - 1 - k];
        len[k] = (int32_t)(roff[i + 1] - roff[i]);
    }
}

constexpr int kLongRun = 1024;  // entries per warp and search of the first one's row

__global__ void __launch_bounds__(256) k_long_gather(const int64_t* __restrict__ roff, int64_t n,
                                                     const int32_t* __restrict__ q_block, int64_t nr,
                                                     const int64_t* __restrict__ loff, int b,
                                                     const int32_t* __restrict__ in, uint64_t* __restrict__ keys) {
    grid_begin();
    const int64_t H = loff[nr], nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t e0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * kLongRun; e0 < H; e0 += nw * kLongRun) {
        int64_t k = 0, hi = nr;  // the last row that begins at or before e0
        while (hi - k > 1) {
            const int64_t mid = (k + hi) >> 1;
            if (loff[mid] <= e0) k = mid;
            else hi = mid;
        }
        const int64_t e1 = e0 + kLongRun < H ? e0 + kLongRun : H;
        for (int64_t e = e0 + lane_id(); e < e1; e += 32) {
            while (loff[k + 1] <= e) ++k;  // e < H = loff[nr]
            keys[e] = ((uint64_t)k << b) | (uint64_t)(uint32_t)in[roff[q_block[n - 1 - k]] + (e - loff[k])];
        }
    }
}

__global__ void __launch_bounds__(256) k_long_first(const uint64_t* __restrict__ keys, int64_t H, int32_t* __restrict__ first) {
    grid_begin();
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < H; e += (int64_t)gridDim.x * blockDim.x)
        first[e] = e == 0 || keys[e] != keys[e - 1];
}

__global__ void __launch_bounds__(256) k_long_write(const uint64_t* __restrict__ keys, const int64_t* __restrict__ pos,
                                                    int64_t H, const int64_t* __restrict__ loff, int b,
                                                    const int64_t* __restrict__ roff, int64_t n,
                                                    const int32_t* __restrict__ q_block, int32_t* __restrict__ out,
                                                    int32_t* __restrict__ ndeg) {
    grid_begin();
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < H; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t k = (int64_t)(keys[e] >> b), i = q_block[n - 1 - k], before = pos[loff[k]];
        if (pos[e + 1] != pos[e]) out[roff[i] + (pos[e] - before)] = (int32_t)(keys[e] & (((uint64_t)1 << b) - 1));
        if (e == loff[k]) ndeg[i] = (int32_t)(pos[loff[k + 1]] - before);
    }
}

// Largest degree, and the arcs after dropping repeats.
__global__ void __launch_bounds__(256) k_build_summary(const int32_t* __restrict__ ndeg, const int64_t* __restrict__ off,
                                                       int64_t n, unsigned long long* __restrict__ summary) {
    grid_begin();
    int32_t best = 0;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
        best = max(best, ndeg[v]);
    best = __reduce_max_sync(kFull, best);
    if (lane_id() == 0 && best > 0) atomicMax(&summary[B_MAXDEG], (unsigned long long)best);
    if (blockIdx.x == 0 && threadIdx.x == 0) summary[B_ARCS] = (unsigned long long)off[n];
}

// Rows closed up: a warp per `run` consecutive columns of the result.  The row of the first is searched (32 probes a
// round), then the lanes hold the bounds of 32 rows and each column looks its row up among them.  (A warp per 32 rows
// copied a graph's hubs by itself where their ids are close: Chung-Lu of 1,347,423 vertices, 2.0 ms of the build.)
__global__ void __launch_bounds__(256) k_build_compact(const int64_t* __restrict__ roff, const int64_t* __restrict__ off,
                                                       int64_t n, const int32_t* __restrict__ in, int run,
                                                       int32_t* __restrict__ cols) {
    grid_begin();
    const int l = lane_id();
    const int64_t M = off[n], nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t t0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * run; t0 < M; t0 += nw * run) {
        const int64_t t1 = t0 + run < M ? t0 + run : M;
        int64_t r0 = 0, hi = n;  // the last row that begins at or before t0: off[r0] <= t0 < off[hi]
        while (hi - r0 > 1) {
            const int64_t step = (hi - r0 + 31) >> 5, p = r0 + (int64_t)(l + 1) * step;
            const uint32_t m = __ballot_sync(kFull, p >= hi || off[p] > t0);
            r0 += (int64_t)(__ffs(m) - 1) * step;
            hi = r0 + step < hi ? r0 + step : hi;
        }
        for (int64_t cur = t0; cur < t1; r0 += 32) {
            const int64_t r = r0 + l < n ? r0 + l : n;
            const int64_t o = off[r];
            const int64_t next = off[r0 + 32 < n ? r0 + 32 : n];
            if (next <= cur) continue;  // these rows are empty
            const int64_t shift = roff[r] - o;
            const int64_t end = next < t1 ? next : t1;
            for (int64_t b = cur; b < end; b += 128) {  // four loads in flight
                int32_t x[4];
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    const int64_t t = b + 32 * h + l;
                    int k = 0;  // last row with o <= t
#pragma unroll
                    for (int sft = 16; sft >= 1; sft >>= 1) {
                        const int64_t v = __shfl_sync(kFull, o, k + sft);
                        if (v <= t) k += sft;
                    }
                    const int64_t at = t + __shfl_sync(kFull, shift, k);
                    x[h] = t < end ? in[at] : 0;
                }
#pragma unroll
                for (int h = 0; h < 4; ++h)
                    if (b + 32 * h + l < end) cols[b + 32 * h + l] = x[h];
            }
            cur = end;
        }
    }
}

unsigned grid_for(int64_t work, int threads) {
    int64_t b = (work + threads - 1) / threads;
    if (b < 1) b = 1;
    if (b > (int64_t)num_sms() * 32) b = (int64_t)num_sms() * 32;
    return (unsigned)b;
}

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// The long rows of a build: raw holds the scattered rows (and, gathered, is scratch), sorted receives them.
harp_status sort_long_rows(int64_t n, int64_t nr, int64_t H, const int64_t* roff, const int32_t* q_block, int32_t* raw,
                           int32_t* sorted, int32_t* ndeg, cudaStream_t s) {
    auto bits_for = [](int64_t x) {  // to hold values up to x
        int b = 1;
        while (b < 62 && ((int64_t)1 << b) <= x) ++b;
        return b;
    };
    const int b = bits_for(n - 1), br = bits_for(nr - 1);
    const size_t hist_len = radix_hist_len(H), tmp_len = scan_tmp_needed(H) + scan_tmp_needed((int64_t)hist_len) + 64;
    const size_t keys_b = align256(sizeof(uint64_t) * (size_t)(H + 1)), hist_b = align256(sizeof(uint32_t) * hist_len);
    const size_t tmp_b = align256(sizeof(int64_t) * tmp_len), loff_b = align256(sizeof(int64_t) * (size_t)(nr + 1));
    unsigned char* slab = nullptr;
    cudaError_t e = cudaMallocAsync((void**)&slab, 2 * keys_b + hist_b + tmp_b + loff_b + sizeof(int32_t) * (size_t)nr, s);
    if (e != cudaSuccess) {
        record_cuda_error(e);
        return e == cudaErrorMemoryAllocation ? HARP_ENOMEM : HARP_ECUDA;
    }
    uint64_t *keys = reinterpret_cast<uint64_t*>(slab), *alt = reinterpret_cast<uint64_t*>(slab + keys_b);
    uint32_t* hist = reinterpret_cast<uint32_t*>(slab + 2 * keys_b);
    int64_t* tmp = reinterpret_cast<int64_t*>(slab + 2 * keys_b + hist_b);
    int64_t* loff = reinterpret_cast<int64_t*>(slab + 2 * keys_b + hist_b + tmp_b);
    int32_t* len = reinterpret_cast<int32_t*>(slab + 2 * keys_b + hist_b + tmp_b + loff_b);
    auto run = [&]() -> harp_status {
        launch(k_long_lengths, grid_for(nr, 256), 256, 0, s, roff, n, q_block, nr, len);
        HARP_LAUNCHED();
        HARP_TRY(exclusive_scan_i32_to_i64(len, loff, nr, tmp, tmp_len, s));
        launch(k_long_gather, grid_for((H + kLongRun - 1) / kLongRun * 32, 256), 256, 0, s, roff, n, q_block, nr, loff, b,
               raw, keys);
        HARP_LAUNCHED();
        HARP_TRY(radix_sort_u64(&keys, &alt, H, 0, b + br, hist, tmp, tmp_len, s));
        launch(k_long_first, grid_for(H, 256), 256, 0, s, keys, H, raw);
        HARP_LAUNCHED();
        int64_t* pos = reinterpret_cast<int64_t*>(alt);
        HARP_TRY(exclusive_scan_i32_to_i64(raw, pos, H, tmp, tmp_len, s));
        launch(k_long_write, grid_for(H, 256), 256, 0, s, keys, pos, H, loff, b, roff, n, q_block, sorted, ndeg);
        HARP_LAUNCHED();
        return HARP_OK;
    };
    const harp_status st = run();
    cudaFreeAsync(slab, s);
    return st;
}

}  // namespace

harp_status build_csr_device(harp_csr* g, int64_t n, int64_t m_in, const int32_t* d_src,
                             const int32_t* d_dst, cudaStream_t s) {
    harp_status st = HARP_OK;
    const int64_t nn = n > 0 ? n : 1;
    int32_t *raw = nullptr, *sorted = nullptr;  // [2 m_in] scattered and sorted rows, at roff
    unsigned char* slab = nullptr;              // everything else
    auto cleanup = [&]() {
        if (raw) cudaFreeAsync(raw, s);
        if (sorted) cudaFreeAsync(sorted, s);
        if (slab) cudaFreeAsync(slab, s);
    };
#define BCK(call)                                              \
    do {                                                       \
        cudaError_t e_ = (call);                               \
        if (e_ != cudaSuccess) {                               \
            record_cuda_error(e_);                             \
            cleanup();                                         \
            return e_ == cudaErrorMemoryAllocation ? HARP_ENOMEM : HARP_ECUDA; \
        }                                                      \
    } while (0)
#define BTRY(call)                                             \
    do {                                                       \
        st = (call);                                           \
        if (st != HARP_OK) { cleanup(); return st; }           \
    } while (0)
#define BLAUNCHED()                                            \
    do {                                                       \
        note_launch();                                         \
        BCK(cudaGetLastError());                               \
    } while (0)

    BCK(cudaMallocAsync((void**)&g->off, (size_t)(n + 1) * sizeof(int64_t), s));
    if (m_in == 0) {
        BCK(cudaMemsetAsync(g->off, 0, (size_t)(n + 1) * sizeof(int64_t), s));
        BCK(cudaMallocAsync((void**)&g->cols, sizeof(int32_t), s));
        g->n = n;
        g->csr_bytes = (size_t)(n + 1) * sizeof(int64_t) + sizeof(int32_t);
        BCK(cudaStreamSynchronize(s));
        return HARP_OK;
    }
    const size_t tmp_len = scan_tmp_needed(nn) + 64;
    const size_t head = align256(B_WORDS * sizeof(unsigned long long)), per_n = align256((size_t)(nn + 32) * sizeof(int32_t));
    const size_t offs = align256((size_t)(nn + 1) * sizeof(int64_t));
    BCK(cudaMallocAsync((void**)&slab, head + 4 * per_n + offs + tmp_len * sizeof(int64_t), s));
    unsigned long long* summary = reinterpret_cast<unsigned long long*>(slab);
    int32_t* deg = reinterpret_cast<int32_t*>(slab + head);
    int32_t* ndeg = reinterpret_cast<int32_t*>(slab + head + per_n);
    int32_t* q = reinterpret_cast<int32_t*>(slab + head + 2 * per_n);
    int32_t* q_block = reinterpret_cast<int32_t*>(slab + head + 3 * per_n);
    int64_t* roff = reinterpret_cast<int64_t*>(slab + head + 4 * per_n);
    int64_t* tmp = reinterpret_cast<int64_t*>(slab + head + 4 * per_n + offs);
    BCK(cudaMallocAsync((void**)&raw, 2 * (size_t)m_in * sizeof(int32_t), s));
    BCK(cudaMallocAsync((void**)&sorted, 2 * (size_t)m_in * sizeof(int32_t), s));
    BCK(cudaMemsetAsync(slab, 0, head + per_n, s));  // summary and degrees
    const Spread at{n >= kSpreadMinN ? (n + 31) >> 5 : 0};
    launch(k_build_degrees, grid_for(m_in, 256), 256, 0, s, d_src, d_dst, m_in, n, at, deg, summary);
    BLAUNCHED();
    if (at.stride) {
        launch(k_build_gather, grid_for(n, 256), 256, 0, s, deg, at, n, ndeg);
        BLAUNCHED();
    }
    BTRY(exclusive_scan_i32_to_i64(at.stride ? ndeg : deg, roff, n, tmp, tmp_len, s));
    launch(k_build_scatter, grid_for(m_in, 256), 256, 0, s, d_src, d_dst, m_in, n, roff, at, deg, raw);
    BLAUNCHED();
    launch(k_build_rows_small, grid_for(n, 256), 256, 0, s, roff, n, raw, sorted, ndeg, q, q_block,
           long_above(n), summary);
    BLAUNCHED();
    // a row has at most m_in entries: tiers above that are empty
    if (m_in > kTierA) {
        launch(k_build_rows_mid, num_sms() * 8, kMidWarps * 32, 0, s, roff, raw, sorted, ndeg, q, summary);
        BLAUNCHED();
    }
    if (m_in > kTierB1) {
        launch(k_build_rows_block, num_sms() * 4, kBlockWarps * 32, 0, s, roff, raw, sorted, ndeg, q_block, summary);
        BLAUNCHED();
    }
    auto bitmap_rows = [&](const int32_t* queue, int count) -> harp_status {  // from the back of the queue
        const size_t smem = sizeof(uint32_t) * (size_t)kBitmapWords;
        HARP_CK(cudaFuncSetAttribute(k_build_rows_bitmap, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        launch(k_build_rows_bitmap, num_sms(), kBitmapThreads, smem, s, roff, n, raw, sorted, ndeg, queue, summary + count);
        HARP_LAUNCHED();
        return HARP_OK;
    };
    if (m_in > kTierB && n <= kBitmapRanks) BTRY(bitmap_rows(q, B_Q_HUB));
    unsigned long long host[B_WORDS] = {0};
    for (;;) {
        BTRY(exclusive_scan_i32_to_i64(ndeg, g->off, n, tmp, tmp_len, s));
        launch(k_build_summary, grid_for(n, 256), 256, 0, s, ndeg, g->off, n, summary);
        BLAUNCHED();
        const bool again = host[B_LONG_LEN] > 0;
        BCK(cudaMemcpyAsync(host, summary, sizeof(host), cudaMemcpyDeviceToHost, s));
        BCK(cudaStreamSynchronize(s));
        if (again || host[B_BAD] || host[B_LONG_LEN] == 0) break;
        const int64_t nr = (int64_t)host[B_Q_LONG], H = (int64_t)host[B_LONG_LEN];
        if (long_by_bitmap(n, nr, H)) BTRY(bitmap_rows(q_block, B_Q_LONG));
        else BTRY(sort_long_rows(n, nr, H, roff, q_block, raw, sorted, ndeg, s));
    }
    if (host[B_BAD]) {
        cleanup();
        return HARP_EINVAL;
    }
    const int64_t M = (int64_t)host[B_ARCS];
    g->n = n;
    g->m = M / 2;
    g->max_deg = (int64_t)host[B_MAXDEG];
    g->csr_bytes = (size_t)(n + 1) * sizeof(int64_t) + (size_t)(M > 0 ? M : 1) * sizeof(int32_t);
    if (M == 2 * m_in) {  // nothing was dropped: the sorted rows are the columns
        g->cols = sorted;
        sorted = nullptr;
    } else {
        BCK(cudaMallocAsync((void**)&g->cols, (size_t)(M > 0 ? M : 1) * sizeof(int32_t), s));
        if (M > 0) {
            const int run = M >= (1 << 20) ? 1024 : (M >= (1 << 17) ? 256 : 32);  // small: enough warps
            launch(k_build_compact, grid_for((M + run - 1) / run * 32, 256), 256, 0, s, roff, g->off, n, sorted, run, g->cols);
            BLAUNCHED();
        }
        BCK(cudaStreamSynchronize(s));
    }
    cleanup();
    return HARP_OK;
#undef BCK
#undef BTRY
#undef BLAUNCHED
}

}  // namespace harp
