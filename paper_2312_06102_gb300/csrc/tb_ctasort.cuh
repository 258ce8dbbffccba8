// tb_ctasort.cuh -- a stable LSD radix sort of one contiguous range of
// (64-bit key, 32-bit value) pairs by a single block of T threads (T = 256, 512
// or 1024): every pass takes the range's tiles in order with running per-digit
// offsets, so it needs no coordination with other blocks.  Used for the sets of
// a batched build and for the rare long runs left by the single-tree sort.
#pragma once

#include "tb_device.cuh"

namespace tb {
namespace {

constexpr int kCtaThreads = 1024;                // block of the long-run sort
constexpr int kCtaRadixBits = 8;
constexpr int kCtaRadix = 1 << kCtaRadixBits;
constexpr int kCtaMaxPasses = 8;
constexpr int kCtaItems = 4;                     // keys per thread of a tile

template <int T>
struct CtaSortSharedT {
    static constexpr int WARPS = T / 32;
    static constexpr int TILE = T * kCtaItems;
    uint64_t keys[TILE];
    int32_t vals[TILE];
    uint32_t warp_hist[WARPS][kCtaRadix + 1];
    uint32_t hist[kCtaMaxPasses][kCtaRadix];
    uint32_t run[kCtaRadix];                     // next place of each digit in the range
    uint32_t loc[kCtaRadix];                     // where the digit starts in the tile
    uint32_t base[kCtaRadix];                    // place in the range, less place in the tile
    uint32_t carry[WARPS];
};
using CtaSortShared = CtaSortSharedT<kCtaThreads>;

// Digit counts of every pass over [o, o + ns) into sm.hist.
template <int T>
__device__ void cta_histograms(const uint64_t *keys, int64_t o, int64_t ns, int shift0, int passes,
                               CtaSortSharedT<T> &sm) {
    for (int i = threadIdx.x; i < kCtaMaxPasses * kCtaRadix; i += T) (&sm.hist[0][0])[i] = 0;
    __syncthreads();
    for (int64_t i = o + threadIdx.x; i < o + ns; i += T) {
        const uint64_t k = keys[i];
        for (int p = 0; p < passes; ++p)
            atomicAdd(&sm.hist[p][(k >> (shift0 + p * kCtaRadixBits)) & (kCtaRadix - 1)], 1u);
    }
    __syncthreads();
}

// Inclusive prefix over the digits of v, the count of digit threadIdx.x / L,
// the same in the L = T / 256 lanes of a digit; one block barrier.
template <int T>
__device__ __forceinline__ uint32_t cta_digit_scan(uint32_t v, uint32_t *carry) {
    constexpr int L = T / kCtaRadix;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t y = v;
#pragma unroll
    for (int off = L; off < 32; off <<= 1) {
        const uint32_t z = __shfl_up_sync(0xffffffffu, y, off);
        if (lane >= off) y += z;
    }
    if (lane == 31) carry[warp] = y;
    __syncthreads();
    return y + __reduce_add_sync(0xffffffffu, lane < warp ? carry[lane] : 0u);
}

// Stable LSD sort of [o, o + ns) by the digits at shift0 + 8 p, p < passes,
// with sm.hist holding each pass's digit counts.  Buffers alternate
// (keys, vals) -> (alt_k, alt_v) -> ...; with index_vals the first pass takes
// each element's own position as its value.  Returns the number of passes
// (the result is in alt_k / alt_v when it is odd).  A range of at most one tile
// stays in shared memory from pass to pass, and with `staged` its keys are
// there (sm.keys) to begin with.  Five barriers a tile: what bounds it is
// issue and barriers, as in the single-tree passes.
template <int T>
__device__ int cta_lsd_sort(uint64_t *keys, int32_t *vals, uint64_t *alt_k, int32_t *alt_v,
                            int64_t o, int64_t ns, int shift0, int passes, bool index_vals, bool staged,
                            CtaSortSharedT<T> &sm) {
    constexpr int W = CtaSortSharedT<T>::WARPS;
    constexpr int TILE = CtaSortSharedT<T>::TILE;
    constexpr int L = T / kCtaRadix;             // lanes per digit, W / L warps each
    static_assert(L >= 1 && L <= 32 && W % L == 0, "whole lanes per digit");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int dg = threadIdx.x / L, part = threadIdx.x % L;
    const unsigned lt = lanemask_lt();
    const int n = (int)ns, first = (int)o;       // positions are 31-bit
    const bool one = n <= TILE;
    uint64_t *src = keys + o, *dst = alt_k + o;
    int32_t *vsrc = vals + o, *vdst = alt_v + o;
    for (int i = threadIdx.x; i < W * (kCtaRadix + 1); i += T) (&sm.warp_hist[0][0])[i] = 0;
    for (int p = 0; p < passes; ++p) {
        const int shift = shift0 + p * kCtaRadixBits;
        const bool in_smem = one && (p > 0 || staged), last = p == passes - 1;
        {
            const uint32_t v = sm.hist[p][dg];
            const uint32_t y = cta_digit_scan<T>(v, sm.carry);
            if (part == 0) sm.run[dg] = y - v;
            __syncthreads();
        }
        for (int tb = 0; tb < n; tb += min(TILE, n - tb)) {
            const int valid = min(TILE, n - tb);
            uint64_t key[kCtaItems];
            int32_t val[kCtaItems];
            uint32_t rank[kCtaItems];
            const int wbase = warp * 32 * kCtaItems;
#pragma unroll
            for (int i = 0; i < kCtaItems; ++i) {
                const int e = wbase + i * 32 + lane;
                key[i] = 0;
                val[i] = 0;
                if (e < valid) {
                    const bool index = p == 0 && index_vals;
                    key[i] = in_smem ? sm.keys[e] : src[tb + e];
                    val[i] = index ? first + tb + e : (in_smem ? sm.vals[e] : vsrc[tb + e]);
                }
            }
            // stable warp ranking: ballot peer masks, leader-updated counters
#pragma unroll
            for (int i = 0; i < kCtaItems; ++i) {
                const bool in = wbase + i * 32 + lane < valid;
                const uint32_t d = (uint32_t)(key[i] >> shift) & (kCtaRadix - 1);
                unsigned peers = __ballot_sync(0xffffffffu, in);
                if (!in) peers = 0;
#pragma unroll
                for (int b = 0; b < kCtaRadixBits; ++b) {
                    const bool bit = (d >> b) & 1u;
                    const unsigned v = __ballot_sync(0xffffffffu, bit);
                    peers &= bit ? v : ~v;
                }
                const int leader = __ffs(peers) - 1;
                uint32_t old = 0;
                if (in && lane == leader) old = atomicAdd(&sm.warp_hist[warp][d], (uint32_t)__popc(peers));
                rank[i] = __shfl_sync(0xffffffffu, old, leader & 31) + (uint32_t)__popc(peers & lt);
            }
            __syncthreads();
            // each warp's offset within its digit and the tile's count of the
            // digit, L lanes a digit
            uint32_t c[W / L], sum = 0;
#pragma unroll
            for (int j = 0; j < W / L; ++j) {
                c[j] = sm.warp_hist[part * (W / L) + j][dg];
                sum += c[j];
            }
            uint32_t y = sum;
#pragma unroll
            for (int off = 1; off < L; off <<= 1) {
                const uint32_t z = __shfl_up_sync(0xffffffffu, y, off, L);
                if (part >= off) y += z;
            }
            uint32_t at = y - sum;
#pragma unroll
            for (int j = 0; j < W / L; ++j) {
                sm.warp_hist[part * (W / L) + j][dg] = at;
                at += c[j];
            }
            const uint32_t cnt = __shfl_sync(0xffffffffu, y, L - 1, L);
            y = cta_digit_scan<T>(cnt, sm.carry);
            if (part == 0) {
                const uint32_t r = sm.run[dg];
                sm.loc[dg] = y - cnt;
                sm.base[dg] = r - (y - cnt);
                sm.run[dg] = r + cnt;
            }
            __syncthreads();
#pragma unroll
            for (int i = 0; i < kCtaItems; ++i) {
                if (wbase + i * 32 + lane < valid) {
                    const uint32_t d = (uint32_t)(key[i] >> shift) & (kCtaRadix - 1);
                    const uint32_t ps = sm.loc[d] + sm.warp_hist[warp][d] + rank[i];
                    sm.keys[ps] = key[i];
                    sm.vals[ps] = val[i];
                }
            }
            __syncthreads();
            for (int i = threadIdx.x; i < W * (kCtaRadix + 1); i += T) (&sm.warp_hist[0][0])[i] = 0;
            if (!one || last) {
#pragma unroll
                for (int i = 0; i < kCtaItems; ++i) {
                    const int j = i * T + (int)threadIdx.x;
                    if (j < valid) {
                        const uint64_t k = sm.keys[j];
                        const uint32_t d = (uint32_t)(k >> shift) & (kCtaRadix - 1);
                        const uint32_t to = sm.base[d] + (uint32_t)j;
                        dst[to] = k;
                        vdst[to] = sm.vals[j];
                    }
                }
            }
            __syncthreads();
        }
        uint64_t *t = src; src = dst; dst = t;
        int32_t *u = vsrc; vsrc = vdst; vdst = u;
    }
    return passes;
}

}  // namespace
}  // namespace tb
