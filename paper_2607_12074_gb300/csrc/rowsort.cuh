// Row sorts shared by the CSR build and the orientation: bitonic networks in the registers of a lane, of a warp and
// of a block, and the shape of the bitmap sort of hub rows.  Rows are sorted by the tier of their length:
// at most kTierA entries by a lane or across a warp's lanes, kTierB1 by a warp, kTierB by a block, longer ones by
// a bitmap of the ids they may hold.
#pragma once

#include "harp_internal.cuh"

namespace harp {

constexpr int kTierA = 32;
constexpr int kTierB1 = 1024;
constexpr int kTierB = 4096;
constexpr int32_t kPadKey = 0x7fffffff;  // sorts after every id

// Bitonic network over the P registers of a lane.
template <int P>
__device__ __forceinline__ void sort_regs(int32_t (&a)[P]) {
#pragma unroll
    for (int k = 2; k <= P; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
#pragma unroll
            for (int i = 0; i < P; ++i) {
                const int p = i ^ j;
                if (p > i) {
                    const int32_t lo = min(a[i], a[p]), hi = max(a[i], a[p]);
                    const bool up = (i & k) == 0;
                    a[i] = up ? lo : hi;
                    a[p] = up ? hi : lo;
                }
            }
        }
    }
}

// Bitonic network over 32 * E keys held by a warp, key lane * E + e in register e: steps of stride below E stay in
// a lane's registers, the others exchange over the lanes.  Sorts blocks of 2, 4, .. up to 32 * E; up: the final
// order of the whole (descending where false, for a larger network's alternate halves).
template <int E>
__device__ __forceinline__ void bitonic_step(int32_t (&v)[E], int j, bool up_all, int k) {
    const int l = lane_id();
    if (j >= E) {
        const int jl = j / E;
        const bool lower = (l & jl) == 0;
        const bool up = k >= 32 * E ? up_all : ((l * E) & k) == 0;  // k > j >= E: a bit of the lane
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int32_t o = __shfl_xor_sync(kFull, v[e], jl);
            v[e] = lower == up ? min(v[e], o) : max(v[e], o);
        }
    } else {
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int p = e ^ j;
            if (p > e && p < E) {
                const bool up = k >= 32 * E ? up_all : ((l * E + e) & k) == 0;
                const int32_t lo = min(v[e], v[p]), hi = max(v[e], v[p]);
                v[e] = up ? lo : hi;
                v[p] = up ? hi : lo;
            }
        }
    }
}

template <int E>
__device__ __forceinline__ void warp_bitonic_sort(int32_t (&v)[E], bool up) {
#pragma unroll
    for (int k = 2; k <= 32 * E; k <<= 1)
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) bitonic_step<E>(v, j, up, k);
}

// The last merge steps of a larger network: strides 16 * E .. 1, all in one direction.
template <int E>
__device__ __forceinline__ void warp_bitonic_merge(int32_t (&v)[E], bool up) {
#pragma unroll
    for (int j = 16 * E; j > 0; j >>= 1) bitonic_step<E>(v, j, up, 32 * E);
}

// A block's sort of kTierB keys: 16 warps sort 256 keys each (in alternate directions), then the merges of 512, 1024,
// 2048 and 4096 keys exchange through shared memory for strides of 256 and more (10 exchanges instead of a
// barrier per stage of the whole network) and finish in registers.  Key x of the block is in warp x / 256, lane
// (x mod 256) / 8, register x mod 8.
constexpr int kBlockE = 8;
constexpr int kBlockWarps = kTierB / (32 * kBlockE);

__device__ __forceinline__ void block_bitonic_sort(int32_t (&v)[kBlockE], int32_t (&buf)[kTierB]) {
    constexpr int E = kBlockE, RUN = 32 * E;
    const int w = threadIdx.x >> 5, l = lane_id();
    warp_bitonic_sort<E>(v, (w & 1) == 0);
    // buf holds register e of lane l of warp w at w * RUN + e * 32 + l, conflict-free; exchanges of stride >= RUN keep
    // the place in the run, so they only change the warp
    for (int k = 2; k <= kBlockWarps; k <<= 1) {  // merge runs of k warps
        const bool up = (w & k) == 0;             // k = kBlockWarps: every warp
        for (int j = k >> 1; j > 0; j >>= 1) {
            __syncthreads();  // the previous exchange is read
#pragma unroll
            for (int e = 0; e < E; ++e) buf[w * RUN + e * 32 + l] = v[e];
            __syncthreads();
            const bool lower = (w & j) == 0;
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const int32_t o = buf[(w ^ j) * RUN + e * 32 + l];
                v[e] = lower == up ? min(v[e], o) : max(v[e], o);
            }
        }
        warp_bitonic_merge<E>(v, up);
    }
}

// Hub rows: a block sets the row's ids in a bitmap in shared memory and writes them out in order, a window of ids at
// a time (one for up to 1.6 M ids).
constexpr int kBitmapThreads = 1024;
constexpr int kBitmapWarps = kBitmapThreads / 32;
constexpr int kBitmapWords = 50176;  // 196 KiB; a multiple of 32 * kBitmapWarps
// Most ids for which the orientation sorts hub rows this way: each window reads the row again.
constexpr int64_t kBitmapRanks = 4 * 32 * (int64_t)kBitmapWords;
static_assert(kBitmapWords % (32 * kBitmapWarps) == 0, "every warp takes whole groups of 32 words");

static_assert(kBitmapWarps == 32, "a lane per warp in the block's prefix");

// Writes the set bits of the window's bitmap (its words dealt to the warps in whole groups of 32, per groups each) as
// ids from lo on, ascending, from out[0]; each(id) sees every id written.  Returns their number.  Called by the
// whole block after the bitmap is complete.
template <typename Each>
__device__ __forceinline__ int bitmap_write(const uint32_t* bm, int per, int64_t lo, int32_t* __restrict__ out,
                                            int (&s_count)[kBitmapWarps], Each&& each) {
    const int w = threadIdx.x >> 5, l = lane_id();
    int count = 0;
    for (int g = 0; g < per; ++g) count += __popc(bm[(w * per + g) * 32 + l]);
    count = warp_sum(count);
    if (l == 0) s_count[w] = count;
    __syncthreads();
    const int before_me = l < w ? s_count[l] : 0;
    int at = warp_sum(before_me);
    const int all = warp_sum(s_count[l]);
    for (int g = 0; g < per; ++g) {
        const int word = (w * per + g) * 32 + l;
        uint32_t bits = bm[word];
        const int c = __popc(bits);
        int incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(kFull, incl, o);
            if (l >= o) incl += y;
        }
        int p = at + incl - c;
        while (bits) {
            const int32_t x = (int32_t)(lo + (int64_t)word * 32 + __ffs(bits) - 1);
            bits &= bits - 1;
            out[p++] = x;
            each(x);
        }
        at += __shfl_sync(kFull, incl, 31);
    }
    return all;
}

}  // namespace harp
