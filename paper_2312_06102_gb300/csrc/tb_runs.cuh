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
constexpr int kRunChunks = kRunSpan / 32 + 1;                // 32-position start masks (+ one past)

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
// Bound by instruction issue.  In the tree workloads 2% to 8% of the keys lie
// in runs of two and more, yet a quarter to a half of all warps hold one, so
// the members are listed first and ranked by full warps.
template <int THREADS, class QueueLong>
__device__ bool run_tile(uint64_t *__restrict__ keys, int32_t *__restrict__ vals, int64_t lo, int64_t s,
                         int64_t hi, int shift0, RunSmem &S, QueueLong queue_long) {
    constexpr int PER = kRunTile / THREADS;
    uint64_t *sk = S.sk;
    uint32_t *smask = S.smask;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int te = (int)min64(kRunTile, hi - s);
    const int nw = (int)min64(kRunSpan, hi - s);
    if ((reinterpret_cast<uintptr_t>(keys + s) & 15u) == 0) {
        const ulonglong2 *src2 = reinterpret_cast<const ulonglong2 *>(keys + s);
        ulonglong2 *dst2 = reinterpret_cast<ulonglong2 *>(sk + 2);
        for (int x = threadIdx.x; x < nw / 2; x += THREADS) dst2[x] = src2[x];
        if (threadIdx.x == 0 && (nw & 1)) sk[nw + 1] = keys[s + nw - 1];
    } else {
        for (int x = threadIdx.x; x < nw; x += THREADS) sk[x + 2] = keys[s + x];
    }
    if (threadIdx.x == 0) {
        S.count = 0;
        sk[1] = s > lo ? keys[s - 1] : ~keys[s];
    }
    __syncthreads();
    const uint64_t lim = uint64_t(1) << shift0;   // equal upper bits <=> xor below lim
    const uint64_t lowm = lim - 1;
    // a run crossing the tile's end: its members past the end move too
    const bool crossing = te == kRunTile && nw > te && (sk[te + 2] ^ sk[te + 1]) < lim;
    const int tm = crossing ? nw : te;
    // start masks (positions past the loaded ones count as starts), and the
    // list of the members of longer runs, in any order
    bool multi = false;
    for (int c = warp; c < kRunChunks; c += THREADS / 32) {
        const int x = c * 32 + lane;
        const bool st = x >= nw || ((sk[x + 2] ^ sk[x + 1]) >= lim);
        const uint32_t m = __ballot_sync(0xffffffffu, st);
        if (lane == 0) smask[c] = m;
        bool next = (m >> ((lane + 1) & 31)) & 1u;
        if (lane == 31) next = x + 1 >= nw || ((sk[x + 3] ^ sk[x + 2]) >= lim);
        const bool mem = x < tm && !(st && next);
        const uint32_t mm = __ballot_sync(0xffffffffu, mem);
        if (mm == 0u) continue;
        multi = true;
        uint32_t at = 0;
        if (lane == 0) at = atomicAdd(&S.count, (uint32_t)__popc(mm));
        at = __shfl_sync(0xffffffffu, at, 0);
        if (mem) S.list[at + __popc(mm & ((1u << lane) - 1u))] = (uint16_t)x;
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
