// tb_cells.cuh -- device code shared by the single-tree and the batched cell
// emission: the per-tile derivation of m_k and L_k and of the per-level start
// masks, and the cells one particle opens and closes.  See tb_cells.cu for
// the method.
#pragma once

#include "tb_device.cuh"

namespace tb {
namespace {

constexpr int kLvThreads = 1024;
constexpr int kLvWarps = kLvThreads / 32;
constexpr int kLvTile = kLvThreads;   // one particle per thread

__host__ __device__ inline int lv_pow2(int ncrit) {
    int p = 1;
    while (2 * p <= ncrit + 1) p *= 2;
    return p;
}

// Shared memory of tile_front for tiles of T particles.
template <int T = kLvTile>
__host__ __device__ inline size_t lv_smem_bytes(int ncrit) {
    size_t ext = (size_t)T + 2 * (size_t)ncrit + 1;   // keys of [s-n-1, e+n)
    size_t nc = (size_t)T + ncrit + 1;                // c over [s-n-1, e)
    return ((ext * 8 + 15) & ~size_t(15)) + 2 * ((nc + 15) & ~size_t(15)) + 64;
}

struct Front {
    int m, L;             // this thread's particle k (m = 255 beyond the tile)
    int64_t k;
};

// Shared state of one tile of T particles (one per thread): masks and counts
// per warp and field (fields 0..21 = cell starts per level, 22 = leaf starts).
template <int T>
struct TileSharedT {
    static constexpr int WARPS = T / 32;
    uint32_t mask[WARPS][kLevelFields];
};
using TileShared = TileSharedT<kLvThreads>;

// Per-warp masks of the lanes starting a cell at each level (fields 0..21)
// and of the lanes starting a leaf (field 22).  Each lane holds the interval
// [m, L] as a row of bits; a 32 x 32 bit-matrix transpose across the warp
// (five exchange rounds) leaves in lane d the mask of field d.
template <int T>
__device__ __forceinline__ void store_level_masks(int m, int L, TileSharedT<T> &ts) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t x = (m <= L) ? (((2u << L) - (1u << m)) | (1u << kLevels)) : 0u;
    uint32_t msk = 0x0000ffffu;
#pragma unroll
    for (int j = 16; j > 0; j >>= 1, msk ^= msk << j) {
        const uint32_t y = __shfl_xor_sync(0xffffffffu, x, j);
        if (lane & j) x ^= ((y >> j) ^ x) & msk;
        else x ^= (((x >> j) ^ y) & msk) << j;
    }
    if (lane < kLevelFields) ts.mask[warp][lane] = x;
}

// m and L of particle s + threadIdx.x of the tile [s, e), and the ballot masks of the level starts of every warp.  The
// tile lies in the segment [seg_lo, seg_hi) of sorted keys that forms one
// tree (the whole array, or one set of a batch); keys outside it do not
// exist for this tree.
template <int T>
__device__ Front tile_front(const uint64_t *__restrict__ skeys, int64_t seg_lo, int64_t seg_hi,
                            int ncrit, int64_t s, int64_t e, unsigned char *raw, TileSharedT<T> &ts) {
    const int64_t lo = s - ncrit - 1;
    const int next = (int)(e + ncrit - lo);
    const int nc = (int)(e - lo);
    const size_t ext = (size_t)T + 2 * (size_t)ncrit + 1;
    const size_t ncp = ((size_t)T + ncrit + 1 + 15) & ~size_t(15);
    uint64_t *key = reinterpret_cast<uint64_t *>(raw);
    uint8_t *A = raw + ((ext * 8 + 15) & ~size_t(15));
    uint8_t *B = A + ncp;
    for (int x = threadIdx.x; x < next; x += T) {
        const int64_t i = lo + x;
        key[x] = (i >= seg_lo && i < seg_hi) ? skeys[i] : 0ull;
    }
    __syncthreads();
    for (int x = threadIdx.x; x < nc; x += T) {
        const int64_t i = lo + x;
        int v = 0;
        if (i >= seg_lo && i + ncrit < seg_hi) v = min(kDepthMax, min_depth(key[x], key[x + ncrit]));
        A[x] = (uint8_t)v;
    }
    __syncthreads();
    const int p = lv_pow2(ncrit);
    for (int q = 1; q < p; q *= 2) {
        for (int x = threadIdx.x; x < nc; x += T)
            B[x] = (x + q < nc) ? max(A[x], A[x + q]) : A[x];
        __syncthreads();
        uint8_t *t = A; A = B; B = t;
    }
    // A[x] = max of c over [x, x + p) (truncated at the end)
    Front f;
    f.k = s + threadIdx.x;
    auto window = [&](int64_t k) {   // max c over [k - n, k], k in [s, e)
        const int x0 = (int)(k - ncrit - lo), x1 = (int)(k - p + 1 - lo);
        return (int)max(A[x0], A[x1]);
    };
    if (f.k < e) {
        const int x = (int)(f.k - lo);
        f.m = (f.k == seg_lo) ? 0 : min_depth(key[x - 1], key[x]);
        f.L = window(f.k);
    } else {
        f.m = 255;
        f.L = 0;
    }
    store_level_masks(f.m, f.L, ts);
    __syncthreads();
    return f;
}

// Starts of each field (0..22) in a tile, one warp per field, one lane per
// warp of the tile: tot[f].  Needs a barrier before (masks written) and after
// (results read).
template <int T>
__device__ __forceinline__ void field_totals(const TileSharedT<T> &ts, uint32_t *tot) {
    constexpr int W = TileSharedT<T>::WARPS;
    const int lane = threadIdx.x & 31;
    for (int f = threadIdx.x >> 5; f < kLevelFields; f += W) {
        const uint32_t v = __reduce_add_sync(0xffffffffu, lane < W ? (uint32_t)__popc(ts.mask[lane][f]) : 0u);
        if (lane == 0) tot[f] = v;
    }
}

// m_k and L_k of the particles [s, e) of a tile, and the leaf starts' counts,
// four consecutive particles per thread of a block of T, for n_crit in
// [kLcMinN, kLcMaxN]; s is a multiple of four, e - s at most 4 T, and particles
// before seg_lo take no part (a segment may start inside the tile's first
// four).  c is kept one byte per
// position; the window maxima of four neighbours share all but their ends:
// L_{k0+j} = max(suffix max from byte j of c[k0-n .. k0-n+3],
//                max of c[k0-n+4 .. k0-1],
//                prefix max to byte j of c[k0 .. k0+3]),
// taken four bytes at a time (byte-wise SIMD maxima).
constexpr int kLcMinN = 3, kLcMaxN = 60;

// Histograms of m and of L + 1 over the leaf starts (m <= L):
// #cells started at level d = #{m <= d} - #{L + 1 <= d}.
struct StartCounts {
    uint32_t m[kLevels + 1], l[kLevels + 1];
    // cells started at level f, or (f = kLevels) leaves
    __device__ uint32_t cells(int f) const {
        uint32_t v = 0;
        if (f == kLevels) {
            for (int d = 0; d < kLevels; ++d) v += m[d];
        } else {
            for (int d = 0; d <= f; ++d) v += m[d] - l[d];
        }
        return v;
    }
};

__host__ __device__ inline int lc_halo_words(int ncrit) { return (ncrit + 3) / 4 + 1; }
template <int T>
__host__ __device__ inline size_t lc_keys(int ncrit) {
    return (size_t)4 * T + 4 * lc_halo_words(ncrit) + ncrit + 4;
}
template <int T>
__host__ __device__ inline size_t lc_smem_bytes(int ncrit) {
    return lc_keys<T>(ncrit) * 8 + ((size_t)T + lc_halo_words(ncrit) + 2) * 4;
}

template <int T>
__device__ void count_tile4(const uint64_t *__restrict__ skeys, int64_t seg_lo, int64_t seg_hi, int ncrit,
                            int64_t s, int64_t e, unsigned char *raw, StartCounts &sc,
                            uint16_t *__restrict__ ml) {
    const int H = lc_halo_words(ncrit);
    const int64_t base = s - 4 * H;                     // position of key[0] and of c byte 0
    const int nk = (int)(e + ncrit - base);
    const int nw = (int)((e - base + 3) / 4);
    uint64_t *key = reinterpret_cast<uint64_t *>(raw);
    uint32_t *cw = reinterpret_cast<uint32_t *>(raw + lc_keys<T>(ncrit) * 8);
    // a tile away from both ends of the segment needs no bounds checks: every
    // window [i, i + n] of its span exists and the keys load as 16-byte pairs
    // (base is even, so key + base is 16-byte aligned when skeys is)
    const bool interior = base >= seg_lo && e == s + 4 * T && e + ncrit + 1 <= seg_hi &&
                          (reinterpret_cast<uintptr_t>(skeys) & 15u) == 0;
    if (interior) {
        const ulonglong2 *src = reinterpret_cast<const ulonglong2 *>(skeys + base);
        ulonglong2 *dst = reinterpret_cast<ulonglong2 *>(key);
        for (int x = threadIdx.x; 2 * x < nk; x += T) dst[x] = src[x];
    } else {
        for (int x = threadIdx.x; x < nk; x += T) {
            const int64_t i = base + x;
            key[x] = (i >= seg_lo && i < seg_hi) ? skeys[i] : 0ull;
        }
    }
    __syncthreads();
    // c of four positions per word: min(21, minDepth(i, i+n)) where the
    // window exists, else 0
    for (int w = threadIdx.x; w < nw; w += T) {
        uint32_t v = 0;
        if (interior) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int x = 4 * w + j;
                v |= (uint32_t)min(kDepthMax, min_depth(key[x], key[x + ncrit])) << (8 * j);
            }
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int x = 4 * w + j;
                const int64_t i = base + x;
                if (i >= seg_lo && i + ncrit < seg_hi && i < e)
                    v |= (uint32_t)min(kDepthMax, min_depth(key[x], key[x + ncrit])) << (8 * j);
            }
        }
        cw[w] = v;
    }
    __syncthreads();
    const int64_t k0 = s + 4 * (int64_t)threadIdx.x;
    uint32_t Lw = 0, mw = 0xffffffffu;                  // bytes: L and m of k0 .. k0 + 3
    if (k0 < e) {
        const int x0 = (int)(k0 - base);                // multiple of 4
        const uint32_t Tw = cw[x0 >> 2];
        auto bytes4 = [&](int b) {                      // c bytes b .. b + 3 (b >= 0)
            const int w = b >> 2, sh = (b & 3) * 8;
            return sh ? __funnelshift_r(cw[w], cw[w + 1], sh) : cw[w];
        };
        const uint32_t Hw = bytes4(x0 - ncrit);
        uint32_t I = 0;
        const int mlen = ncrit - 4;                     // middle bytes x0 - n + 4 .. x0 - 1
        if (mlen >= 4) {
            for (int b = x0 - ncrit + 4; b + 4 <= x0; b += 4) I = __vmaxu4(I, bytes4(b));
            I = __vmaxu4(I, bytes4(x0 - 4));
        } else if (mlen > 0) {
            I = bytes4(x0 - ncrit + 4) & ((1u << (8 * mlen)) - 1u);
        }
        I = __vmaxu4(I, I >> 16);
        I = __vmaxu4(I, I >> 8);
        I = (I & 0xffu) * 0x01010101u;
        uint32_t S = __vmaxu4(Hw, Hw >> 8);
        S = __vmaxu4(S, S >> 16);
        uint32_t P = __vmaxu4(Tw, Tw << 8);
        P = __vmaxu4(P, P << 16);
        Lw = __vmaxu4(__vmaxu4(S, P), I);
        mw = 0;
        if (interior) {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                mw |= (uint32_t)min_depth(key[x0 + j - 1], key[x0 + j]) << (8 * j);
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int64_t k = k0 + j;
                uint32_t m = 255u;
                if (k >= seg_lo && k < e)
                    m = (k == seg_lo) ? 0u : (uint32_t)min_depth(key[x0 + j - 1], key[x0 + j]);
                mw |= m << (8 * j);
            }
        }
        // m and L of the four particles, for the emission
        if (k0 >= seg_lo && k0 + 4 <= e) {
            uint2 v;
            v.x = (mw & 0xffu) | ((Lw & 0xffu) << 8) | (((mw >> 8) & 0xffu) << 16) | (((Lw >> 8) & 0xffu) << 24);
            v.y = ((mw >> 16) & 0xffu) | (((Lw >> 16) & 0xffu) << 8) | ((mw >> 24) << 16) | ((Lw >> 24) << 24);
            *reinterpret_cast<uint2 *>(ml + k0) = v;
        } else {
            for (int j = 0; j < 4; ++j)
                if (k0 + j >= seg_lo && k0 + j < e)
                    ml[k0 + j] = (uint16_t)(((mw >> (8 * j)) & 0xffu) | (((Lw >> (8 * j)) & 0xffu) << 8));
        }
    }
    // histograms over the leaf starts: about one
    // particle in seven is a start, so plain shared atomics rarely collide
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int m = (mw >> (8 * j)) & 0xff, L = (Lw >> (8 * j)) & 0xff;
        if (m <= L) {
            atomicAdd(&sc.m[m], 1u);
            atomicAdd(&sc.l[L + 1], 1u);
        }
    }
}

struct EmitOut {
    uint64_t *ckey;
    uint8_t *level;
    int32_t *parent, *child_first, *child_end, *pfirst, *pend;
    int32_t *leaf_cell;
    int32_t *start_cell;     // batched: the leaf cell that starts at each position
};

// Emission over the leaf starts only, 4 T particles by a block of T threads.
// Only a leaf start (m_k <= L_k) opens or closes cells, one particle in four to
// seven on the tree workloads, so each warp first lists the starts of its 128
// particles in order and then works on that list, 32 starts at a time: every
// lane holds a start, and the level masks (a 32 x 32 bit transpose) are built
// for the list, not for every particle.  The warps meet once, to exchange how
// many cells of each level they start; what bound the kernel before, with the
// starts of the whole block in one list, were its seven barriers (2^27
// clustered 0.97 ms, now 0.71; 2^24 120 and 88 us).
constexpr int kEmitSpan = 128;                          // particles of a warp

struct EmitWarp {
    uint32_t entry[kEmitSpan];                          // k - the warp's first | m << 8 | L << 16 | Lprev << 24
    uint32_t mask[kEmitSpan / 32][kLevels];             // level masks of each chunk of 32 starts
    uint32_t base[kLevels + 2];                         // next cell of each level before the chunk
};
template <int T>
struct EmitShared {
    EmitWarp warp[T / 32];
    uint32_t cnt[2][T / 32][kLevelFields];              // cells (leaves) each warp starts per level
};

// The tile of particles [s, s + 4 T) (s a multiple of four) of the tree whose
// sorted particles are [lo, hi).  Lane f's `base` is the next cell of level f
// (f = kLevels: the next leaf), level_end(d) where level d ends.  Returns how
// many of them the tile starts.  Tiles of one block alternate in `parity`; all
// threads of the block call it.  Writes the leaf of each start to
// out.start_cell when START.
template <int T, bool START, class LevelEnd>
__device__ __forceinline__ uint32_t emit_tile(const uint64_t *skeys, const uint16_t *ml, int64_t lo,
                                              int64_t hi, int64_t tile, uint32_t base,
                                              const LevelEnd &level_end, const EmitOut &out,
                                              EmitShared<T> &sm, int parity) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    EmitWarp &W = sm.warp[warp];
    const int64_t s = tile + warp * kEmitSpan;
    // m and L of four particles per lane
    const int64_t k0 = s + 4 * lane;
    uint32_t m[4], L[4];
    if (k0 >= lo && k0 + 4 <= hi) {
        const uint2 v = *reinterpret_cast<const uint2 *>(ml + k0);
        m[0] = v.x & 0xffu; L[0] = (v.x >> 8) & 0xffu; m[1] = (v.x >> 16) & 0xffu; L[1] = v.x >> 24;
        m[2] = v.y & 0xffu; L[2] = (v.y >> 8) & 0xffu; m[3] = (v.y >> 16) & 0xffu; L[3] = v.y >> 24;
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t v = (k0 + j >= lo && k0 + j < hi) ? (uint32_t)ml[k0 + j] : 255u;
            m[j] = v & 0xffu;
            L[j] = v >> 8;
        }
    }
    uint32_t Lp = __shfl_up_sync(0xffffffffu, L[3], 1);
    if (lane == 0) Lp = s > lo && s < hi ? (uint32_t)(ml[s - 1] >> 8) : 0u;
    // the tree's last particle closes the cells holding it: the last cell of
    // each level 0 .. L, whose children end where the next level ends
    if (k0 <= hi - 1 && hi - 1 < k0 + 4) {
        const uint32_t Ll = L[(int)(hi - 1 - k0)];
        for (int d = 0; d <= (int)Ll; ++d) {
            const int64_t idx = level_end(d) - 1;
            out.pend[idx] = (int32_t)hi;
            out.child_end[idx] = (d < (int)Ll) ? (int32_t)level_end(d + 1) : -1;
        }
    }
    // the warp's starts in order
    uint32_t cnt = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) cnt += (m[j] <= L[j]) ? 1u : 0u;
    uint32_t x = cnt;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, off);
        if (lane >= off) x += y;
    }
    const int total = (int)__shfl_sync(0xffffffffu, x, 31);
    uint32_t pos = x - cnt;
#pragma unroll
    for (int j = 0; j < 4; ++j)
        if (m[j] <= L[j])
            W.entry[pos++] = (uint32_t)(4 * lane + j) | (m[j] << 8) | (L[j] << 16) | ((j ? L[j - 1] : Lp) << 24);
    __syncwarp();
    // the keys of the first chunk of starts, loaded now so that the masks and
    // the barrier cover their latency
    uint64_t Kfirst = 0;
    if (lane < total) Kfirst = skeys[s + (W.entry[lane] & 255u)];
    // level masks of every chunk of 32 starts; lane d counts level d
    uint32_t mine = 0;
    for (int c = 0; 32 * c < total; ++c) {
        const int i = c * 32 + lane;
        uint32_t v = 0;
        if (i < total) {
            const uint32_t en = W.entry[i];
            v = (2u << ((en >> 16) & 31u)) - (1u << ((en >> 8) & 31u));
        }
        uint32_t msk = 0x0000ffffu;
#pragma unroll
        for (int j = 16; j > 0; j >>= 1, msk ^= msk << j) {
            const uint32_t y = __shfl_xor_sync(0xffffffffu, v, j);
            if (lane & j) v ^= ((y >> j) ^ v) & msk;
            else v ^= (((v >> j) ^ y) & msk) << j;
        }
        if (lane < kLevels) W.mask[c][lane] = v;
        mine += __popc(v);
    }
    if (lane == kLevels) mine = (uint32_t)total;
    if (lane < kLevelFields) sm.cnt[parity][warp][lane] = mine;
    __syncthreads();
    uint32_t all = 0;
    if (lane < kLevelFields) {
#pragma unroll
        for (int w = 0; w < T / 32; ++w) {
            if (w == warp) W.base[lane] = base + all;
            all += sm.cnt[parity][w][lane];
        }
    }
    __syncwarp();
    const unsigned lt = lanemask_lt();
    for (int c = 0; 32 * c < total; ++c) {
        const int i = c * 32 + lane;
        if (i < total) {
            const uint32_t en = W.entry[i];
            const int64_t k = s + (en & 255u);
            const int mm = (int)((en >> 8) & 31u), LL = (int)((en >> 16) & 31u), Lq = (int)(en >> 24);
            auto P = [&](int d) { return W.base[d] + (uint32_t)__popc(W.mask[c][d] & lt); };
            const uint64_t K = c == 0 ? Kfirst : skeys[k];
            // P(d) of consecutive levels: each loop computes one new level per step
            const uint32_t pm = P(mm);
            if (k > lo) {
                // close the cells holding k-1 but not k
                uint32_t pd = pm;
                for (int d = mm; d <= Lq; ++d) {
                    const uint32_t pn = d < Lq ? P(d + 1) : 0u;
                    out.pend[pd - 1] = (int32_t)k;
                    out.child_end[pd - 1] = (d < Lq) ? (int32_t)pn : -1;
                    pd = pn;
                }
            }
            uint32_t pprev = mm > 0 ? P(mm - 1) : 0u, pd = pm;
            for (int d = mm;; ++d) {
                const uint32_t pn = d < LL ? P(d + 1) : 0u;
                out.ckey[pd] = cell_key(K, d);
                out.level[pd] = (uint8_t)d;
                out.pfirst[pd] = (int32_t)k;
                out.parent[pd] = (d == 0) ? -1 : (int32_t)pprev - (d == mm ? 1 : 0);
                out.child_first[pd] = (d < LL) ? (int32_t)pn : -1;
                if (d == LL) break;
                pprev = pd;
                pd = pn;
            }
            out.leaf_cell[W.base[kLevels] + (uint32_t)i] = (int32_t)pd;
            if constexpr (START) out.start_cell[k] = (int32_t)pd;
        }
        if (32 * (c + 1) < total) {
            __syncwarp();
            if (lane < kLevels) W.base[lane] += (uint32_t)__popc(W.mask[c][lane]);
            __syncwarp();
        }
    }
    __syncwarp();   // the warp's list may be rewritten next
    return all;
}

}  // namespace
}  // namespace tb
