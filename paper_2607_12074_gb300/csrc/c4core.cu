// Step a5 on the dense end of a skewed graph: 4-cycles whose top vertex u lies in the core, the K
// highest ranks of the graph (ginfo[GI_CORE] on).
//
// c4.cu walks the wedges u - w - x from their top vertex u and counts, per u, how many end in each x < u.
// The same total, sum over pairs x < u of C(cnt(x, u), 2) with cnt(x, u) the common neighbours w < u of
// x and u, can be taken per lower end x: the wedges of x are the lists N+(w) above x, over w in N(x), and
// the counters run over u.  On a skewed graph almost every wedge ends in a hub (R-MAT scale 20: 99 % in
// the top 16384 of 1,048,576 ranks; Chung-Lu 2.1 with 2,000,000 vertices: 97 %), so per x the counters of
// u need only K entries, and for w in the core too, N+(w) is a dense row of K bits.  A core row is then added
// to 32 counters at once: the counters are held as bit planes (plane p holds bit p of 32 counters to a
// word, in registers) and rows are added through carry-save adders, about 4 instructions for each word
// of 32 counters, where a counter per element costs about 28 thread instructions.
//
//   * core rows: K x K bits (CoreTable), in the bytes of ws.rev and ws.bpos (which the walk from the top vertex fills
//     afterwards).  32 MiB for K = 16384: the table stays in L2.  The triangle pass reads it too (tri.cu).
//   * w outside the core: the part of N+(w) inside the core, element by element, in packed counters in
//     shared memory.  A bit transpose turns the counters into planes, the starting value of the register
//     planes, so both kinds of w meet in one exact count.  (Counting these elements in planes as well, by
//     an atomic xor and its carries, measured 54 ms on the 2,000,000-vertex Chung-Lu graph: hubs are
//     dense, and 32 of them share a plane's word.)
//   * at the end sum_u C(cnt, 2) is a sum of popcounts: with planes B_p, C(cnt, 2) summed over a word is
//     sum_p C(2^p, 2) popc(B_p) + sum_{p<q} 2^(p+q) popc(B_p & B_q).
//
// What bounds it: reading core rows from L2 (6.6 GB of row words on R-MAT scale 20 at K = 16384) and the
// element-wise part (13 % of the wedges there).  A larger K moves wedges from the second to the first.
//
// The core is chosen per graph on the device (choose_core, called by k_c4_ginfo).
#include "harp_internal.cuh"

namespace harp {
namespace {

constexpr int kKMaxLog2 = 14;
constexpr int kKWordsMax = (1 << kKMaxLog2) / 32;
// Degree classes of x by the counter bits that hold cnt(x, u) <= d(x).  S: a warp per x; M, L and XL: a block
// per x.
constexpr int kBitsS = 4, kBitsM = 8, kBitsL = 16, kBitsXL = 32;
constexpr int kWarpsS = 4;  // x per block in class S

// One thread per vertex, highest rank first.  Outside the core: cseg[v] = (start, length) of the part of
// N+(v) inside the core.  Every vertex x of a graph with a core joins its degree class (fewer than two neighbours
// close no cycle); below[x] = its neighbours below the core.
__global__ void __launch_bounds__(256) k_core_queue(const int64_t* __restrict__ off, const int32_t* __restrict__ cols,
                                                    const int64_t* __restrict__ offp, const int32_t* __restrict__ colsp,
                                                    const int32_t* __restrict__ deg, const int32_t* __restrict__ gid,
                                                    const int64_t* __restrict__ ginfo, int64_t n,
                                                    uint2* __restrict__ cseg, int32_t* __restrict__ below,
                                                    int32_t* __restrict__ q_s, int32_t* __restrict__ q_m,
                                                    int32_t* __restrict__ q_l, uint64_t* __restrict__ acc) {
    grid_begin();
    if (acc[A_CORE_ANY] == 0) return;
    const int l = lane_id();
    for (int64_t base = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) - l; base < n;
         base += (int64_t)gridDim.x * blockDim.x) {
        const int64_t v = n - 1 - (base + l);
        int cls = -1;
        if (v >= 0) {
            const int64_t* gi = ginfo + (gid ? (int64_t)gid[v] : 0) * kGInfo;
            const int64_t c0 = gi[GI_CORE];
            if (gi[GI_CORE_K] > 0) {
                const int32_t d = deg[v];
                if (d >= 2) {
                    cls = d < (1 << kBitsS) ? 0 : (d < (1 << kBitsM) ? 1 : (d < (1 << kBitsL) ? 2 : 3));
                    const int64_t rb = off[v];
                    below[v] = (int32_t)lower_bound_i32(cols + rb, d, (int32_t)c0);
                }
                if (v < c0) {
                    const int64_t b = offp[v], len = offp[v + 1] - b;
                    const int64_t p = lower_bound_i32(colsp + b, len, (int32_t)c0);
                    cseg[v] = make_uint2((uint32_t)(b + p), (uint32_t)(len - p));
                }
            }
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const uint32_t mask = __ballot_sync(kFull, cls == c);
            if (!mask) continue;
            unsigned long long start = 0;
            const int leader = __ffs(mask) - 1;
            if (l == leader) start = atomicAdd((unsigned long long*)&acc[Q_CORE_S + c], (unsigned long long)__popc(mask));
            start = __shfl_sync(kFull, start, leader);
            const int64_t slot = (int64_t)(start + __popc(mask & lanemask_lt()));
            if (cls != c) continue;
            if (c < 3) (c == 0 ? q_s : (c == 1 ? q_m : q_l))[slot] = (int32_t)v;
            else q_l[n - 1 - slot] = (int32_t)v;
        }
    }
}

// A warp per core row: the row's bits built in shared memory and written with 16-byte stores, with the number of bits
// before each word beside them.  Words before the row's own 4-word group hold no bit and are never read.
// The graphs with a core are found 32 at a time.
constexpr int kRowWarps = 8;

__global__ void __launch_bounds__(kRowWarps * 32) k_core_bits(const int64_t* __restrict__ offp,
                                                              const int32_t* __restrict__ colsp, int64_t G,
                                                              const int64_t* __restrict__ ginfo,
                                                              const uint64_t* __restrict__ acc,
                                                              uint32_t* __restrict__ region) {
    grid_begin();
    __shared__ __align__(16) uint32_t sbuf[kRowWarps][kKWordsMax];
    if (acc[A_CORE_ANY] == 0) return;
    uint32_t* buf = sbuf[threadIdx.x >> 5];
    const int l = lane_id();
    const int64_t wid = (int64_t)blockIdx.x * kRowWarps + (threadIdx.x >> 5), nw = (int64_t)gridDim.x * kRowWarps;
    for (int64_t g0 = 0; g0 < G; g0 += 32) {
        uint32_t with_core = __ballot_sync(kFull, g0 + l < G && ginfo[(g0 + l) * kGInfo + GI_CORE_K] > 0);
        while (with_core) {
            const CoreTable t = core_table(ginfo, g0 + __ffs(with_core) - 1, region);
            with_core &= with_core - 1;
            const int KW = t.KW;
            for (int64_t r = wid; r < 32 * (int64_t)KW; r += nw) {
                const int64_t w = t.c0 + r;
                const int first = (int)(r >> 5) & ~3;
                for (int i = first + l; i < KW; i += 32) buf[i] = 0;
                __syncwarp();
                for (int64_t p = offp[w] + l, e = offp[w + 1]; p < e; p += 32) {
                    const int j = (int)(colsp[p] - t.c0);
                    atomicOr(&buf[j >> 5], 1u << (j & 31));
                }
                __syncwarp();
                uint32_t* out = const_cast<uint32_t*>(t.bits) + r * KW;
                for (int i = first + 4 * l; i < KW; i += 128)
                    *reinterpret_cast<uint4*>(out + i) = *reinterpret_cast<const uint4*>(buf + i);
                uint16_t* before = const_cast<uint16_t*>(t.before) + r * KW;
                int run = 0;
                for (int i = first; i < KW; i += 32) {
                    const int c = i + l < KW ? __popc(buf[i + l]) : 0;
                    int incl = c;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int y = __shfl_up_sync(kFull, incl, o);
                        if (l >= o) incl += y;
                    }
                    if (i + l < KW) before[i + l] = (uint16_t)(run + incl - c);
                    run += __shfl_sync(kFull, incl, 31);
                }
                __syncwarp();
            }
        }
    }
}

// sum + carry of three bits in every position
__device__ __forceinline__ void csa(uint32_t& carry, uint32_t& sum, uint32_t a, uint32_t b, uint32_t c) {
    const uint32_t t = a ^ b;
    carry = (a & b) | (t & c);
    sum = t ^ c;
}

template <int VEC>
struct Words {
    uint32_t v[VEC];
};

template <int VEC>
__device__ __forceinline__ Words<VEC> load_words(const uint32_t* p) {
    Words<VEC> r;
    if constexpr (VEC == 4) {
        const uint4 x = __ldg(reinterpret_cast<const uint4*>(p));
        r.v[0] = x.x;
        r.v[1] = x.y;
        r.v[2] = x.z;
        r.v[3] = x.w;
    } else if constexpr (VEC == 2) {
        const uint2 x = __ldg(reinterpret_cast<const uint2*>(p));
        r.v[0] = x.x;
        r.v[1] = x.y;
    } else {
        r.v[0] = __ldg(p);
    }
    return r;
}

// Counters of CB bits in shared memory: the CB words of plane word W hold its 32 counters, counter b (of
// core vertex 32 W + b) in word b mod CB at bit b - b mod CB.  Transposing every CB x CB block of bits
// then turns word p into plane p.  Consecutive core vertices lie in consecutive words (hubs are dense:
// one word for all 32 would serialise a warp's adds).
// ctr: the counters' shared-memory address.
template <int CB>
__device__ __forceinline__ void counter_add(uint32_t ctr, uint32_t j) {
    asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(ctr + 4u * ((j >> 5) * CB + (j & (CB - 1)))),
                 "r"(1u << (j & 31 & ~(CB - 1)))
                 : "memory");
}

// The planes of VEC plane words from wi, taken out of the counters (left clear).
template <int CB, int VEC>
__device__ __forceinline__ void take_counters(uint32_t* ctr, int wi, uint32_t (&B)[CB][VEC]) {
#pragma unroll
    for (int v = 0; v < VEC; ++v) {
        uint32_t w[CB];
        uint4* c = reinterpret_cast<uint4*>(ctr + (wi + v) * CB);
#pragma unroll
        for (int k = 0; k < CB; k += 4) {
            const uint4 x = c[k / 4];
            w[k] = x.x;
            w[k + 1] = x.y;
            w[k + 2] = x.z;
            w[k + 3] = x.w;
            c[k / 4] = make_uint4(0, 0, 0, 0);
        }
#pragma unroll
        for (int s = CB / 2; s >= 1; s >>= 1) {  // swap the off-diagonal s x s blocks
            const uint32_t m = s == 16 ? 0x0000ffffu : (s == 8 ? 0x00ff00ffu : (s == 4 ? 0x0f0f0f0fu : (s == 2 ? 0x33333333u : 0x55555555u)));
#pragma unroll
            for (int k = 0; k < CB; ++k) {
                if (k & s) continue;
                const uint32_t t = ((w[k] >> s) ^ w[k + s]) & m;
                w[k + s] ^= t;
                w[k] ^= t << s;
            }
        }
#pragma unroll
        for (int p = 0; p < CB; ++p) B[p][v] = w[p];
    }
}

// Adds the core rows cols[rb, re) (rank order, all >= c0) to the planes of VEC words from wi.  Called by a
// whole warp whose words end before warp_end.  Four rows are in flight per lane (with eight, the registers cost
// more resident x than the loads gained).
template <int P, int VEC>
__device__ __forceinline__ void add_rows(const uint32_t* __restrict__ bits, const int32_t* __restrict__ cols, int64_t rb,
                                         int64_t re, int32_t c0, int KW, int wi, int warp_end, int np,
                                         uint32_t (&B)[P][VEC]) {
    constexpr int R = 4;
    const int l = lane_id();
    const uint32_t* mybits = bits + wi;
    for (int64_t i0 = rb; i0 < re; i0 += 32) {
        // rows at or past the warp's last word hold no bit there; rows ascend
        const int32_t r = i0 + l < re ? __ldg(cols + i0 + l) - c0 : INT32_MAX;
        const int cnt = __popc(__ballot_sync(kFull, r < warp_end * 32));
        for (int j = 0; j < cnt; j += R) {
            Words<VEC> a[R];
#pragma unroll
            for (int t = 0; t < R; ++t) {
                const int32_t rr = __shfl_sync(kFull, r, (j + t) & 31);
                if (j + t < cnt && wi + VEC > (rr >> 5)) {
                    a[t] = load_words<VEC>(mybits + (int64_t)rr * KW);
                } else {
#pragma unroll
                    for (int v = 0; v < VEC; ++v) a[t].v[v] = 0;
                }
            }
#pragma unroll
            for (int v = 0; v < VEC; ++v) {
                uint32_t t0, t1, f;
                csa(t0, B[0][v], B[0][v], a[0].v[v], a[1].v[v]);
                csa(t1, B[0][v], B[0][v], a[2].v[v], a[3].v[v]);
                csa(f, B[1][v], B[1][v], t0, t1);
#pragma unroll
                for (int p = 2; p < P; ++p) {
                    if (p >= np) break;  // np is uniform
                    const uint32_t t = B[p][v] & f;
                    B[p][v] ^= f;
                    f = t;
                }
            }
        }
        if (cnt < 32) break;
    }
}

// sum of C(cnt, 2) over the planes' counters of core vertices above xo (an offset from c0; negative: all), by
// a whole warp.  Planes that are empty in all of the warp's words are left out: away from the top hubs the
// counts are far below d(x), and the popcounts grow with the square of the planes.
template <int P, int VEC>
__device__ __forceinline__ uint64_t pairs_sum(uint32_t (&B)[P][VEC], int wi, int32_t xo, int np) {
    uint64_t total = 0;
    if (xo >= wi * 32) {
#pragma unroll
        for (int v = 0; v < VEC; ++v) {
            const int32_t lo = xo + 1 - (wi + v) * 32;  // first bit of this word that counts
            const uint32_t keep = lo <= 0 ? 0xffffffffu : (lo >= 32 ? 0u : 0xffffffffu << lo);
#pragma unroll
            for (int p = 0; p < P; ++p) B[p][v] &= keep;
        }
    }
    int top = 0;
#pragma unroll
    for (int q = 1; q < P; ++q) {
        uint32_t any = 0;
#pragma unroll
        for (int v = 0; v < VEC; ++v) any |= B[q][v];
        if (any) top = q;
    }
    top = __reduce_max_sync(kFull, top) + 1;
    np = top < np ? top : np;
#pragma unroll
    for (int v = 0; v < VEC; ++v) {
        // the pair sums fit 32 bits up to 8 planes: 32 * C(255, 2)
        uint64_t wide = 0;
        uint32_t narrow = 0;
#pragma unroll
        for (int q = 1; q < P; ++q) {
            if (q >= np) break;
            if (P <= 8) {
                uint32_t s = __popc(B[q][v]) * ((1u << q) - 1u);
#pragma unroll
                for (int p = 0; p < q; ++p) s += (uint32_t)__popc(B[p][v] & B[q][v]) << (p + 1);
                narrow += s << (q - 1);  // C(2^q, 2) = 2^(q-1) (2^q - 1)
            } else {
                uint64_t s = (uint64_t)__popc(B[q][v]) * ((1ull << q) - 1ull);
#pragma unroll
                for (int p = 0; p < q; ++p) s += (uint64_t)__popc(B[p][v] & B[q][v]) << (p + 1);
                wide += s << (q - 1);
            }
        }
        total += wide + narrow;
    }
    return total;
}

// The element-wise part of one x: every w in cols[rb, re) (outside the core) adds its list's elements above x
// to the counters.  NT threads (whole warps) share the w; returns whether this warp added anything.
template <int CB, int NT>
__device__ __forceinline__ bool core_elements(const int32_t* __restrict__ cols, int64_t rb, int64_t re,
                                              const int32_t* __restrict__ colsp, const uint2* __restrict__ cseg,
                                              int32_t x, int32_t c0, uint32_t* ctr_ptr) {
    const int l = lane_id();
    const uint32_t ctr = (uint32_t)__cvta_generic_to_shared(ctr_ptr);
    const int warp = NT == 32 ? 0 : (int)(threadIdx.x >> 5);
    bool any = false;
    auto add = [&](int32_t u) { counter_add<CB>(ctr, (uint32_t)(u - c0)); };
    for (int64_t i0 = rb; i0 < re; i0 += NT) {
        uint32_t base = 0;
        int len = 0;
        const int64_t i = i0 + l * (NT / 32) + warp;  // dealt so that few w still spread over all warps
        if (i < re) {
            const uint2 sg = __ldg(cseg + __ldg(cols + i));
            base = sg.x;
            len = (int)sg.y;
            if (len > 0 && x >= c0) {  // x in the core: only the list's elements above x
                if (__ldg(colsp + base + len - 1) <= x) {
                    len = 0;
                } else {
                    const int p = (int)lower_bound_i32(colsp + base, len, x + 1);
                    base += (uint32_t)p;
                    len -= p;
                }
            }
        }
        any |= __any_sync(kFull, len > 0);
        // long lists by the whole warp, coalesced: the first 64 elements of four lists are loaded together
        // (the lists average about 50 elements: one list at a time leaves one load in flight)
        uint32_t longs = __ballot_sync(kFull, len >= 24);
        while (longs) {
            uint32_t b[4];
            int c[4];
            int32_t u[8];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const int src = longs ? __ffs(longs) - 1 : 0;
                b[t] = __shfl_sync(kFull, base, src);
                c[t] = longs ? __shfl_sync(kFull, len, src) : 0;
                longs &= longs - 1;
                u[2 * t] = l < c[t] ? __ldg(colsp + b[t] + l) : -1;
                u[2 * t + 1] = l + 32 < c[t] ? __ldg(colsp + b[t] + l + 32) : -1;
            }
#pragma unroll
            for (int t = 0; t < 8; ++t)
                if (u[t] >= 0) add(u[t]);
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                for (int k = 64 + l; k < c[t]; k += 128) {
#pragma unroll
                    for (int h = 0; h < 4; ++h) u[h] = k + 32 * h < c[t] ? __ldg(colsp + b[t] + k + 32 * h) : -1;
#pragma unroll
                    for (int h = 0; h < 4; ++h)
                        if (u[h] >= 0) add(u[h]);
                }
            }
        }
        // short lists flattened over the lanes
        const int slen = len >= 24 ? 0 : len;
        int incl = slen;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(kFull, incl, o);
            if (l >= o) incl += y;
        }
        const int excl = incl - slen;
        const int total = __shfl_sync(kFull, incl, 31);
        for (int t0 = 0; t0 < total; t0 += 32) {
            const int t = t0 + l;
            int o = 0;
#pragma unroll
            for (int s = 16; s >= 1; s >>= 1) {
                const int e = __shfl_sync(kFull, excl, o + s);
                if (e <= t) o += s;
            }
            const uint32_t ob = __shfl_sync(kFull, base, o);
            const int oe = __shfl_sync(kFull, excl, o);
            if (t < total) add(__ldg(colsp + ob + (t - oe)));
        }
    }
    return any;
}

struct CoreX {
    int32_t x, c0, KW, np;
    int64_t rb, split, re;  // x's row: neighbours below the core in [rb, split), core neighbours in [split, re)
    const uint32_t* bits;
};

__device__ __forceinline__ CoreX core_x(int32_t x, const int64_t* __restrict__ off, const int32_t* __restrict__ gid,
                                        const int64_t* __restrict__ ginfo, const int32_t* __restrict__ below,
                                        const uint32_t* __restrict__ bits) {
    const int64_t* gi = ginfo + (gid ? (int64_t)gid[x] : 0) * kGInfo;
    CoreX c;
    c.x = x;
    c.c0 = (int32_t)gi[GI_CORE];
    c.KW = (int)(gi[GI_CORE_K] >> 5);
    c.bits = bits + gi[GI_CORE_BASE];
    c.rb = off[x];
    c.re = off[x + 1];
    c.split = c.rb + below[x];
    c.np = 32 - __clz((int)(c.re - c.rb));  // cnt(x, u) <= d(x) < 2^np
    return c;
}

// Class S: a warp per x, the row words in groups of 32 * VEC.
template <int VEC>
__device__ __forceinline__ uint64_t warp_words(const CoreX& c, const int32_t* __restrict__ cols, bool dirty,
                                               uint32_t* ctr) {
    uint64_t a = 0;
    const int32_t xo = c.x - c.c0;
    for (int w0 = 0; w0 < c.KW; w0 += 32 * VEC) {
        if (xo >= (w0 + 32 * VEC) * 32 - 1) continue;  // nothing of this group lies above x
        const int wi = w0 + VEC * lane_id();
        uint32_t B[kBitsS][VEC] = {};
        if (dirty) take_counters<kBitsS, VEC>(ctr, wi, B);
        add_rows<kBitsS, VEC>(c.bits, cols, c.split, c.re, c.c0, c.KW, wi, w0 + 32 * VEC, c.np, B);
        a += pairs_sum<kBitsS, VEC>(B, wi, xo, c.np);
    }
    return a;
}

__global__ void __launch_bounds__(kWarpsS * 32, 6) k_core_warp(const int64_t* __restrict__ off,
                                                               const int32_t* __restrict__ cols,
                                                               const int32_t* __restrict__ colsp,
                                                               const uint2* __restrict__ cseg,
                                                               const int32_t* __restrict__ gid,
                                                               const int64_t* __restrict__ ginfo,
                                                               const int32_t* __restrict__ below,
                                                               const uint32_t* __restrict__ bits,
                                                               const int32_t* __restrict__ q, Sink sink) {
    grid_begin();
    extern __shared__ __align__(16) uint32_t smem_ctr[];
    __shared__ uint64_t red[32];
    uint32_t* ctr = smem_ctr + (threadIdx.x >> 5) * (kBitsS * kKWordsMax);
    const int l = lane_id();
    for (int i = l; i < kBitsS * kKWordsMax; i += 32) ctr[i] = 0;
    __syncwarp();
    const int64_t nq = (int64_t)sink.acc[Q_CORE_S];
    uint64_t c4 = 0;
    for (int64_t k = (int64_t)blockIdx.x * kWarpsS + (threadIdx.x >> 5); k < nq; k += (int64_t)gridDim.x * kWarpsS) {
        const CoreX c = core_x(q[k], off, gid, ginfo, below, bits);
        const bool dirty = core_elements<kBitsS, 32>(cols, c.rb, c.split, colsp, cseg, c.x, c.c0, ctr);
        __syncwarp();
        uint64_t a = 0;
        if (dirty || c.re - c.split >= 2)
            a = c.KW >= 128 ? warp_words<4>(c, cols, dirty, ctr) : warp_words<1>(c, cols, dirty, ctr);
        if (sink.batch()) {
            a = warp_sum(a);
            if (l == 0) sink_add(sink, c.x, G_C4, a);
        } else {
            c4 += a;
        }
        __syncwarp();
    }
    c4 = block_sum_u64(c4, red);
    if (threadIdx.x == 0 && c4) atomicAdd((unsigned long long*)&sink.acc[ACC_C4], (unsigned long long)c4);
}

// The words of one x by a block (classes M, L, XL): groups of 32 * VEC words above x, one warp each.  Where x
// is so high that fewer groups than warps are left, the rows (many, for such an x) are split as well and
// the parts' planes added up through the counters' shared memory.
template <int CB, int NT, int VEC>
__device__ __forceinline__ uint64_t block_words(const CoreX& c, const int32_t* __restrict__ cols, bool dirty,
                                                uint32_t* ctr) {
    constexpr int NW = NT / 32, GW = 32 * VEC;
    const int warp = threadIdx.x >> 5, l = lane_id();
    const int32_t xo = c.x - c.c0;
    const int groups = c.KW / GW;
    int g0 = xo < 0 ? 0 : (xo + 1) / (GW * 32);  // first group with a counter above x
    const int live = groups - g0;
    if (live <= 0) return 0;  // x is the last rank
    const int64_t R = c.re - c.split;
    int parts = live < NW ? NW / live : 1;
    if (parts > 1 + (int)(R >> 6)) parts = 1 + (int)(R >> 6);
    uint64_t a = 0;
    if (parts == 1) {
        for (int g = g0 + warp; g < groups; g += NW) {
            const int wi = g * GW + VEC * l;
            uint32_t B[CB][VEC] = {};
            if (dirty) take_counters<CB, VEC>(ctr, wi, B);
            add_rows<CB, VEC>(c.bits, cols, c.split, c.re, c.c0, c.KW, wi, (g + 1) * GW, c.np, B);
            a += pairs_sum<CB, VEC>(B, wi, xo, c.np);
        }
        return a;
    }
    const int g = g0 + warp % live, part = warp / live;
    const int wi = g * GW + VEC * l;
    uint32_t B[CB][VEC] = {};
    if (part == 0 && dirty) take_counters<CB, VEC>(ctr, wi, B);
    if (part < parts)
        add_rows<CB, VEC>(c.bits, cols, c.split + R * part / parts, c.split + R * (part + 1) / parts, c.c0, c.KW, wi,
                          (g + 1) * GW, c.np, B);
    __syncthreads();  // the counters are all taken: their bytes hold the parts' planes now
    if (part > 0 && part < parts) {
#pragma unroll
        for (int p = 0; p < CB; ++p) {
            if (p >= c.np) break;
#pragma unroll
            for (int v = 0; v < VEC; ++v) ctr[(warp * CB + p) * GW + v * 32 + l] = B[p][v];
        }
    }
    __syncthreads();
    if (part == 0) {
        for (int o = warp + live; o < live * parts; o += live) {
            uint32_t carry[VEC] = {};
#pragma unroll
            for (int p = 0; p < CB; ++p) {
                if (p >= c.np) break;
#pragma unroll
                for (int v = 0; v < VEC; ++v) {
                    uint32_t* s = &ctr[(o * CB + p) * GW + v * 32 + l];
                    csa(carry[v], B[p][v], B[p][v], *s, carry[v]);
                    *s = 0;
                }
            }
        }
        a = pairs_sum<CB, VEC>(B, wi, xo, c.np);
    }
    return a;
}

// Classes M, L and XL: a block of NT threads per x, highest ranks first.
template <int CB, int NT, int VEC, int MINB>
__global__ void __launch_bounds__(NT, MINB) k_core_block(const int64_t* __restrict__ off, const int32_t* __restrict__ cols,
                                                   const int32_t* __restrict__ colsp, const uint2* __restrict__ cseg,
                                                   const int32_t* __restrict__ gid, const int64_t* __restrict__ ginfo,
                                                   const int32_t* __restrict__ below, const uint32_t* __restrict__ bits,
                                                   const int32_t* __restrict__ q,
                                                   int qslot, int tslot, Sink sink) {
    grid_begin();
    // the parts' planes of block_words fit the counters' bytes
    static_assert((NT / 32) * 32 * VEC <= kKWordsMax, "scratch of the row parts");
    extern __shared__ __align__(16) uint32_t ctr[];
    __shared__ uint64_t red[32];
    __shared__ int64_t s_item;
    for (int i = threadIdx.x; i < CB * kKWordsMax; i += NT) ctr[i] = 0;
    const int64_t nq = (int64_t)sink.acc[qslot];
    uint64_t c4 = 0;
    if (threadIdx.x == 0) s_item = (int64_t)atomicAdd((unsigned long long*)&sink.acc[tslot], 1ull);
    __syncthreads();
    for (;;) {
        const int64_t k = s_item;
        if (k >= nq) break;
        const CoreX c = core_x(CB == kBitsXL ? q[-k] : q[k], off, gid, ginfo, below, bits);  // XL: filled from the back
        const bool mine = core_elements<CB, NT>(cols, c.rb, c.split, colsp, cseg, c.x, c.c0, ctr);
        const bool dirty = __syncthreads_or(mine);  // also: every add is done, every thread has read s_item
        if (threadIdx.x == 0) s_item = (int64_t)atomicAdd((unsigned long long*)&sink.acc[tslot], 1ull);  // the next x
        uint64_t a = 0;
        if (dirty || c.re - c.split >= 2)
            a = c.KW >= 32 * VEC ? block_words<CB, NT, VEC>(c, cols, dirty, ctr)
                                 : block_words<CB, NT, 1>(c, cols, dirty, ctr);
        if (sink.batch()) {
            const uint64_t s = block_sum_u64(a, red);
            if (threadIdx.x == 0) sink_add(sink, c.x, G_C4, s);
        } else {
            c4 += a;
        }
        __syncthreads();  // the counters are clear again before the next x adds to them; s_item is set
    }
    c4 = block_sum_u64(c4, red);
    if (threadIdx.x == 0 && c4) atomicAdd((unsigned long long*)&sink.acc[ACC_C4], (unsigned long long)c4);
}

template <int CB, int NT, int VEC, int MINB>
harp_status launch_block(const Workspace& ws, const uint32_t* bits, const uint2* cseg, const int32_t* q, int qslot,
                         int tslot, const Sink& sink, cudaStream_t s) {
    const size_t smem = (size_t)CB * kKWordsMax * sizeof(uint32_t);
    HARP_CK(cudaFuncSetAttribute(k_core_block<CB, NT, VEC, MINB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    launch(k_core_block<CB, NT, VEC, MINB>, num_sms() * MINB, NT, smem, s, ws.off, ws.cols, ws.colsp, cseg, ws.gid,
           ws.ginfo, ws.fpos, bits, q, qslot, tslot, sink);
    HARP_LAUNCHED();
    return HARP_OK;
}

}  // namespace

bool wedge_core_applies(const harp_csr* g, const Workspace& ws) {
    const bool whole = !ws.loff && ws.arcs < 0 && ws.own_lo <= 0 && ws.own_hi >= g->n && ws.x_lo <= 0 && ws.x_hi >= g->n;
    const int64_t m = ws.G > 1 ? ws.max_member_m : g->m;
    return whole && m >= kCoreMinM && g->max_deg >= kCoreMinMaxDeg;
}

harp_status build_core_bits(Workspace& ws, cudaStream_t s) {
    launch(k_core_bits, num_sms() * 4, kRowWarps * 32, 0, s, ws.offp, ws.colsp, ws.G > 0 ? ws.G : 1, ws.ginfo, ws.acc,
           reinterpret_cast<uint32_t*>(ws.rev));
    HARP_LAUNCHED();
    return HARP_OK;
}

harp_status count_wedge_core(const harp_csr* g, Workspace& ws, cudaStream_t s) {
    const int64_t n = g->n;
    const int sms = num_sms();
    const Sink sink{ws.acc, ws.gid, ws.accG};
    // the bitmaps that build_core_bits wrote; rev and bpos are adjacent (ws_layout) and filled after this pass
    uint32_t* bits = reinterpret_cast<uint32_t*>(ws.rev);
    uint2* cseg = reinterpret_cast<uint2*>(ws.vkeys);      // the sort keys are done with
    int32_t *q_s = ws.q_mid, *q_m = ws.q_mid + n, *q_l = ws.q_win;
    int64_t blocks = (n + 255) / 256;
    if (blocks > (int64_t)sms * 16) blocks = (int64_t)sms * 16;
    launch(k_core_queue, (unsigned)blocks, 256, 0, s, ws.off, ws.cols, ws.offp, ws.colsp, ws.deg, ws.gid, ws.ginfo, n,
           cseg, ws.fpos, q_s, q_m, q_l, ws.acc);
    HARP_LAUNCHED();
    if (g->max_deg >= (1 << kBitsL))
        HARP_TRY((launch_block<kBitsXL, 512, 1, 1>(ws, bits, cseg, q_l + n - 1, Q_CORE_XL, T_CORE_XL, sink, s)));
    HARP_TRY((launch_block<kBitsL, 256, 2, 4>(ws, bits, cseg, q_l, Q_CORE_L, T_CORE_L, sink, s)));
    HARP_TRY((launch_block<kBitsM, 64, 4, 12>(ws, bits, cseg, q_m, Q_CORE_M, T_CORE_M, sink, s)));
    const size_t smem = (size_t)kWarpsS * kBitsS * kKWordsMax * sizeof(uint32_t);
    HARP_CK(cudaFuncSetAttribute(k_core_warp, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    launch(k_core_warp, sms * 6, kWarpsS * 32, smem, s, ws.off, ws.cols, ws.colsp, cseg, ws.gid, ws.ginfo, ws.fpos,
           bits, q_s, sink);
    HARP_LAUNCHED();
    return HARP_OK;
}

}  // namespace harp
