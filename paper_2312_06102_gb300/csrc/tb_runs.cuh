// tb_runs.cuh -- the in-place ordering of the runs of equal upper key bits
// left by radix passes over the upper bits only (see tb_runs.cu), one tile of
// 2048 positions at a time by one block; shared by the single-tree sort and
// the per-set sorts of the batched build.
#pragma once

#include "tb_ctasort.cuh"

namespace tb {
namespace {

constexpr int kRunTile = 2048;
constexpr int kRunMax = 128;                                 // longest run ordered in place
constexpr int kRunSpan = kRunTile + kRunMax;                 // positions a tile loads
constexpr int kRunChunks = kRunSpan / 32 + 2;                // 32-position start masks (+ one past), even

// Bits 0..15 of v to the even bits.
__device__ __forceinline__ uint32_t spread16(uint32_t v) {
    v &= 0xffffu;
    v = (v | (v << 8)) & 0x00ff00ffu;
    v = (v | (v << 4)) & 0x0f0f0f0fu;
    v = (v | (v << 2)) & 0x33333333u;
    return (v | (v << 1)) & 0x55555555u;
}

struct RunSmem {
    // sk[x + 2] = keys[s + x] for x in [-1, nw); before the range's first key,
    // that key's complement, whose upper bits differ from it
    __align__(16) uint64_t sk[kRunSpan + 2];
    uint32_t smask[kRunChunks];   // bit l of chunk c: position 32 c + l starts a run
    uint32_t count;               // positions in list
    uint16_t list[kRunSpan];      // the positions in runs of two keys and more
};

// Orders in place, by (low shift0 bits, position), every run of equal
// key >> shift0 that starts in the tile [s, s + 2048) of the range [lo, hi)
// and holds at most kRunMax keys; calls queue_long(a) once for each longer run
// starting at a in the tile.  All THREADS threads of the block take part.
// Returns, the same in every thread, whether a key of the tile is smaller
// than its predecessor in the same run (a descent).
//
// Bound by instruction issue and by the latency of one tile's loads.  In the
// tree workloads 2% to 8% of the keys lie in runs of two and more, yet a
// quarter to a half of all warps hold one, so the members are listed first and
// ranked by full warps (2^24 particles 66 to 61 us); and the start masks come
// from the keys as they are loaded, 64 a warp step, all loads first (56 us;
// each step loading its own keys 70).
template <int THREADS, class QueueLong>
__device__ bool run_tile(uint64_t *__restrict__ keys, int32_t *__restrict__ vals, int64_t lo, int64_t s,
                         int64_t hi, int shift0, RunSmem &S, QueueLong queue_long) {
    constexpr int PER = kRunTile / THREADS;
    uint64_t *sk = S.sk;
    uint32_t *smask = S.smask;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int te = (int)min64(kRunTile, hi - s);
    const int nw = (int)min64(kRunSpan, hi - s);
    const uint64_t lim = uint64_t(1) << shift0;   // equal upper bits <=> xor below lim
    const uint64_t lowm = lim - 1;
    // a run crossing the tile's end: its members past the end move too
    const bool crossing = te == kRunTile && nw > te && (keys[s + te] ^ keys[s + te - 1]) < lim;
    const int tm = crossing ? nw : te;
    const bool vec = (reinterpret_cast<uintptr_t>(keys + s) & 15u) == 0;
    if (threadIdx.x == 0) S.count = 0;
    __syncthreads();
    // keys, start masks (positions past the loaded ones count as starts) and
    // the list of the members of longer runs, in any order: two neighbouring
    // positions a thread, 64 a warp
    bool multi = false;
    constexpr int ROUNDS = (kRunChunks * 32 + 2 * THREADS - 1) / (2 * THREADS);
    uint64_t r0[ROUNDS], r1[ROUNDS], re[ROUNDS];
#pragma unroll
    for (int i = 0; i < ROUNDS; ++i) {
        const int x = warp * 64 + i * 2 * THREADS + 2 * lane;
        r0[i] = r1[i] = re[i] = 0;
        if (vec && x + 1 < nw) {
            const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(keys + s + x);
            r0[i] = v.x;
            r1[i] = v.y;
        } else if (x < nw) {
            r0[i] = keys[s + x];
            if (x + 1 < nw) r1[i] = keys[s + x + 1];
        }
        // lane 0: the key before the warp's first; lane 31: the key after its last
        const int y = lane == 0 ? x - 1 : x + 2;
        if ((lane == 0 || lane == 31) && y < nw && x < nw && s + y >= lo) re[i] = keys[s + y];
    }
#pragma unroll
    for (int i = 0; i < ROUNDS; ++i) {
        const int w0 = warp * 64 + i * 2 * THREADS;
        if (w0 >= kRunChunks * 32) break;
        const int x = w0 + 2 * lane;
        const uint64_t k0 = r0[i], k1 = r1[i];
        const uint64_t edge = x == 0 && s == lo ? ~k0 : re[i];
        if (x + 1 < nw) *reinterpret_cast<ulonglong2 *>(sk + x + 2) = make_ulonglong2(k0, k1);
        else if (x < nw) sk[x + 2] = k0;
        if (x == 0) sk[1] = edge;
        uint64_t before = __shfl_up_sync(0xffffffffu, k1, 1);
        if (lane == 0) before = edge;
        const bool st0 = x >= nw || (k0 ^ before) >= lim;
        const bool st1 = x + 1 >= nw || (k1 ^ k0) >= lim;
        const uint32_t b0 = __ballot_sync(0xffffffffu, st0), b1 = __ballot_sync(0xffffffffu, st1);
        bool st2 = (b0 >> ((lane + 1) & 31)) & 1u;
        if (lane == 31) st2 = x + 2 >= nw || (edge ^ k1) >= lim;
        const bool in0 = x < tm && !(st0 && st1), in1 = x + 1 < tm && !(st1 && st2);
        if (lane < 2) smask[(w0 >> 5) + lane] = spread16(b0 >> (16 * lane)) | (spread16(b1 >> (16 * lane)) << 1);
        const uint32_t m0 = __ballot_sync(0xffffffffu, in0), m1 = __ballot_sync(0xffffffffu, in1);
        if ((m0 | m1) == 0u) continue;
        multi = true;
        uint32_t at = 0;
        if (lane == 0) at = atomicAdd(&S.count, (uint32_t)(__popc(m0) + __popc(m1)));
        at = __shfl_sync(0xffffffffu, at, 0);
        const uint32_t below = (1u << lane) - 1u;
        if (in0) S.list[at + __popc(m0 & below)] = (uint16_t)x;
        if (in1) S.list[at + __popc(m0) + __popc(m1 & below)] = (uint16_t)(x + 1);
    }
    // a tile of single-key runs is done (the barrier also publishes the masks)
    if (!__syncthreads_or(multi)) return false;
    const uint32_t members = S.count;
    int32_t dst[PER + 1];   // new position - s of the key at the list's i-th place, or -1
    int32_t val[PER + 1];
    bool desc = false;
#pragma unroll
    for (int i = 0; i <= PER; ++i) {
        dst[i] = -1;
        const uint32_t e = threadIdx.x + (uint32_t)(i * THREADS);
        if (e >= members) continue;
        const int x = S.list[e];
        const int c = x >> 5, l = x & 31;
        const uint32_t m = smask[c];
        const bool st_here = (m >> l) & 1u;
        const uint64_t kx = sk[x + 2];
        if (!st_here) desc |= (kx & lowm) < (sk[x + 1] & lowm);
        // the run [a, b) from the start masks, looking at most kScan chunks
        // away: a run that reaches further is longer than kRunMax, and the
        // member at its start queues it
        constexpr int kScan = kRunMax / 32 + 2;
        int a = -1;
        const uint32_t le = m & (0xffffffffu >> (31 - l));
        if (le) {
            a = c * 32 + 31 - __clz(le);
        } else {
            for (int cc = c - 1; cc >= 0 && cc >= c - kScan; --cc) {
                const uint32_t mc = smask[cc];
                if (mc) {
                    a = cc * 32 + 31 - __clz(mc);
                    break;
                }
            }
            if (a < 0) continue;                        // began before this tile, or long
        }
        if (a >= te) continue;                          // the run begins after this tile
        const uint32_t gt = l < 31 ? (m & (0xffffffffu << (l + 1))) : 0u;
        int b = -1;                                     // stays -1 for a long run
        if (gt) {
            b = c * 32 + __ffs(gt) - 1;
        } else {
            // the chunk holding position nw starts runs from there on
            for (int cc = c + 1; cc < kRunChunks && cc <= c + kScan; ++cc) {
                const uint32_t mc = smask[cc];
                if (mc) {
                    b = cc * 32 + __ffs(mc) - 1;
                    break;
                }
            }
        }
        if (b > nw) b = nw;
        // longer runs (including any that reach the end of the loaded span
        // before the end of the keys) go to the block sort
        if (b < 0 || b - a > kRunMax) {
            if (x == a) queue_long(s + a);
            continue;
        }
        // rank by (low bits, position); the low bits fit 32 bits (shift0 <= 32)
        const uint32_t lp = (uint32_t)(kx & lowm);
        int r = 0;
#pragma unroll 4
        for (int j = a; j < b; ++j) {
            const uint32_t lj = (uint32_t)(sk[j + 2] & lowm);
            r += (lj < lp) || (lj == lp && j < x);
        }
        if (a + r == x) continue;
        dst[i] = a + r;
        val[i] = vals[s + x];
    }
    desc = __syncthreads_or(desc);   // also: every moved value is read before any is overwritten
#pragma unroll
    for (int i = 0; i <= PER; ++i) {
        if (dst[i] < 0) continue;
        const int x = S.list[threadIdx.x + i * THREADS];
        keys[s + dst[i]] = sk[x + 2];
        vals[s + dst[i]] = val[i];
    }
    __syncthreads();   // the shared tile may be reloaded next
    return desc;
}

// Queue of long runs and the per-tile descent flags, laid out in one buffer.
struct RunBuffers {
    int32_t *queue;      // [n / kRunMax + 2] start positions of long runs
    uint8_t *desc;       // [n / kRunTile + 1] tile holds a descent inside a run
};
__host__ __device__ inline int64_t run_queue_cap(int64_t n) { return n / kRunMax + 2; }
__host__ __device__ inline RunBuffers run_buffers(int32_t *base, int64_t n) {
    return {base, reinterpret_cast<uint8_t *>(base + run_queue_cap(n))};
}

// Sorts by its low shift0 bits the run of equal key >> shift0 that starts at
// a, when one of its tiles holds a descent (`desc`, one flag per tile of the
// n keys); a block of T threads.
template <int T>
__device__ void sort_long_run(uint64_t *keys, int32_t *vals, uint64_t *alt_k, int32_t *alt_v, int64_t n,
                              int shift0, int64_t a, const uint8_t *desc, CtaSortSharedT<T> &sm) {
    __shared__ unsigned long long s_end;
    __shared__ int s_desc;
    const int passes = (shift0 + kCtaRadixBits - 1) / kCtaRadixBits;
    const uint64_t tp = keys[a] >> shift0;
    // the run's end: the first later position with other upper bits;
    // the first 4096 positions are scanned by the block, then binary search
    if (threadIdx.x == 0) { s_end = (unsigned long long)n; s_desc = 0; }
    __syncthreads();
    int64_t base = a + 1;
    for (int it = 0; it < 4 && base < n; ++it, base += T) {
        const int64_t p = base + threadIdx.x;
        if (p < n && (keys[p] >> shift0) != tp) atomicMin(&s_end, (unsigned long long)p);
        __syncthreads();
        const bool done = s_end < (unsigned long long)n;
        __syncthreads();
        if (done) break;
    }
    if (threadIdx.x == 0 && s_end == (unsigned long long)n && base < n) {
        int64_t lo = base, hi = n;                  // first position with top > tp
        while (lo < hi) {
            const int64_t m = (lo + hi) >> 1;
            if ((keys[m] >> shift0) <= tp) lo = m + 1; else hi = m;
        }
        s_end = (unsigned long long)lo;
    }
    __syncthreads();
    const int64_t len = (int64_t)s_end - a;
    // only a run with a descent needs sorting: look at the tile flags
    const int64_t t0 = (a + 1) / kRunTile, t1 = (a + len - 1) / kRunTile;
    for (int64_t t = t0 + threadIdx.x; t <= t1; t += T)
        if (desc[t]) s_desc = 1;
    __syncthreads();
    if (s_desc) {
        cta_histograms(keys, a, len, 0, passes, sm);
        const int np = cta_lsd_sort(keys, vals, alt_k, alt_v, a, len, 0, passes, false, false, sm);
        if (np & 1)
            for (int64_t p = a + threadIdx.x; p < a + len; p += T) {
                keys[p] = alt_k[p];
                vals[p] = alt_v[p];
            }
    }
    __syncthreads();
}

}  // namespace
}  // namespace tb
