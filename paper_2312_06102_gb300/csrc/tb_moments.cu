// tb_moments.cu -- cell moments without traversing the tree (Sec. 2.3: cell
// properties are computed as cells are created; the centre of mass of a
// parent comes from those of its children, higher multipoles likewise).
//
//   leaf_tile_kernel     : every leaf, one block per tile of 2048 positions in
//                          key order: the tile's permutation bulk-copied (TMA)
//                          into shared memory, its (x, y, z, m) records
//                          gathered beside it (Sec. 2.3 step 3, the reorder),
//                          one thread per leaf summing from there;
//   upward_kernel        : leaves the tiles could not hold, members read
//                          through the permutation (a warp, or a block, per
//                          leaf); then level by level, deepest first, the
//                          children of the level, in tiles bulk-copied (TMA)
//                          into shared memory, and every non-leaf cell of
//                          the level combined from its tile.
//
// Moments of a cell: M = sum m; centre of mass c = sum m x / M; central
// second moment Q = sum m (x - c)(x - c)^T (6 components xx xy xz yy yz zz);
// member bounding box.  Sums run relative to a reference point inside the
// cell (the first member particle for a leaf, the first child's centre for a
// parent), which keeps the FP32 differences small and exact or nearly so.
// Parent from children (parallel-axis theorem):
//   M = sum M_j, c = sum M_j c_j / M, Q = sum [Q_j + M_j (c_j - c)(c_j - c)^T].
//
// Modes:
//   FP32_COMP  -- two-sum / two-product compensated FP32; the centre of mass
//                 is kept as an unevaluated pair com + com_lo (an FP32 value
//                 cannot hold a deep cell's centre to 2e-6 of its side);
//   FP32_PLAIN -- uncompensated FP32, com_lo = 0;
//   FP64       -- FP64 accumulation; FP64 outputs beside the FP32 ones.
// A leaf of more than 2^20 particles is summed in FP64 in every mode, and so
// is a parent of that many in the FP32-plain mode; compensated parents stay
// in FP32 at every size (their error is relative to their own mass and side).
#include "tb_moments.cuh"

namespace tb {

namespace {

// A wait for bulk copies gave up: one thread waits for them again before the
// block leaves, so that none of them lands in shared memory that has gone to
// another block.  The caller's limit, which may be a poll or two
// (tb_set_wait_limit), does not count here: copies depend on no other block.
__device__ __forceinline__ void drain(uint64_t *bar, uint32_t parity) {
    mbar_wait_bounded(bar, parity, kDefaultWaitLimit);
}

// ------------------------------------------------------------ kernels

// Leaves, one block per tile of kLtTile consecutive key-order positions.
//   1. The permutation of the tile and of a halo of kLtHalo positions past
//      it is bulk-copied (TMA) into shared memory, and m_k | L_k << 8 of the
//      same positions is read beside it.
//   2. The records (x, y, z, m) of those particles are gathered into shared
//      memory: xm[perm[k]] (Sec. 2.3 step 3).  When the permutation of the
//      span is one ascending run -- input already in key order, as after a
//      reorder -- the records are one contiguous stretch and come in with one
//      bulk copy instead.  With `xs` set (pos_sorted asked for), the tile's
//      records are bulk-stored to it.
//   3. k starts a leaf iff m_k <= L_k (Alg. 1 as a closed form); leaves tile
//      the key order, so a leaf ends where the next one starts.  The leaves
//      starting in the tile are listed in order; their index among all
//      leaves comes from the scanned per-tile leaf counts of the cell pass (a
//      batched build, which counts per set, noted each leaf's cell by its
//      first position instead).
//   4. One thread per leaf sums its members from shared memory.  A leaf that
//      runs past the staged span (only a depth-21 leaf of identical keys, or
//      n_crit above the halo, can) and, in the compensated mode, a leaf of
//      more than kSplitLeaf members go to the queues of upward_kernel.
constexpr int kLtThreads = 256;
constexpr int kLtPer = kLtTile / kLtThreads;   // positions per thread when listing starts
static_assert(kLtTile == 2 * 1024, "leaf tiles span two tiles of the cell pass");

struct LeafTileSmem {
    float4 rec[kLtSpan];
    int32_t perm[kLtSpan];
    uint16_t ml[kLtSpan];
    uint16_t start[kLtTile];                   // offsets of the leaf starts in the tile
    uint32_t wcount[kLtThreads / 32];
    int32_t next_start;                        // first start at or past the tile end, or -1
    // compensated mode: staged leaves of more than kSplitLeaf members, summed
    // by whole warps after the short ones (at most kLtTile / 17 of them)
    int32_t long_c[kLtTile / (kSplitLeaf + 1) + 1];
    uint32_t long_x[kLtTile / (kSplitLeaf + 1) + 1];   // start | end << 16 (tile offsets)
    uint32_t n_long;
    uint32_t bins[kLtHalo];                    // FP64 mode: leaves by member count
    uint64_t bar;
};
static_assert(kLtHalo == 64, "two member-count bins per lane of a warp");

size_t leaf_tile_smem() { return sizeof(LeafTileSmem); }

// (the FP64 mode holds ten 64-bit sums and their products a thread, which
// spill at the 64 registers of four blocks a SM)
template <int MODE>
__global__ void __launch_bounds__(kLtThreads, MODE == TB_MOM_FP64 ? 3 : 4)
    leaf_tile_kernel(MomOut o, const int32_t *__restrict__ leaf_cell,
                     const int32_t *__restrict__ start_cell,
                     const int32_t *__restrict__ perm, const float4 *__restrict__ xm,
                     const uint16_t *__restrict__ ml, const uint32_t *__restrict__ leaf_off,
                     const int32_t *__restrict__ pend, int64_t n, float4 *__restrict__ xs,
                     int32_t *long_queue, int32_t *big_queue, DevInfo *info, int64_t wait_limit) {
    after_previous();
    if (info->status & (kErrOverflow | kErrNonFinite | kErrTimeout | kErrInvalid)) return;
    // the barrier count of the upward pass that follows starts from zero
    if (blockIdx.x == 0 && threadIdx.x == 0) info->misc_ctr[7] = 0;
    extern __shared__ __align__(128) unsigned char lt_raw[];
    LeafTileSmem &S = *reinterpret_cast<LeafTileSmem *>(lt_raw);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t k0 = (int64_t)blockIdx.x * kLtTile;
    const int span = (int)min64(kLtSpan, n - k0);
    const int te = (int)min64(kLtTile, n - k0);
    // 1. permutation of the span: its whole 16-byte groups by bulk copy
    //    (k0 is a multiple of 4), the rest by plain loads
    const int nbulk = span & ~3;
    if (threadIdx.x == 0) {
        mbar_init(&S.bar, 1);
        mbar_init_fence();
        if (nbulk > 0) {
            mbar_arrive_expect_tx(&S.bar, (uint32_t)nbulk * 4u);
            bulk_load(S.perm, perm + k0, (uint32_t)nbulk * 4u, &S.bar);
        }
    }
    for (int x = nbulk + (int)threadIdx.x; x < span; x += kLtThreads) S.perm[x] = perm[k0 + x];
    for (int x = threadIdx.x; x < span; x += kLtThreads) S.ml[x] = ml[k0 + x];
    __syncthreads();
    uint32_t phase = 0;
    bool ok = true;
    if (nbulk > 0) {
        ok = mbar_wait_bounded(&S.bar, phase, wait_limit);
        phase ^= 1u;
    }
    // a copy that did not complete in time: record it and leave once it has
    if (!__syncthreads_and(ok)) {
        if (threadIdx.x == 0) {
            flag_error(&info->status, kErrTimeout);
            drain(&S.bar, 0);
        }
        return;
    }
    // 2. records of the span
    bool run = true, in_range = true;
    for (int x = threadIdx.x; x < span; x += kLtThreads) {
        const int32_t p = S.perm[x];
        in_range &= (uint32_t)p < (uint32_t)n;
        if (x + 1 < span) run &= S.perm[x + 1] == p + 1;
    }
    if (!__syncthreads_and(in_range)) {
        if (threadIdx.x == 0) flag_error(&info->status, kErrTimeout);
        return;
    }
    if (__syncthreads_and(run)) {
        if (threadIdx.x == 0) {
            mbar_arrive_expect_tx(&S.bar, (uint32_t)span * 16u);
            bulk_load(S.rec, xm + S.perm[0], (uint32_t)span * 16u, &S.bar);
        }
        ok = mbar_wait_bounded(&S.bar, phase, wait_limit);
        if (!__syncthreads_and(ok)) {
            if (threadIdx.x == 0) {
                flag_error(&info->status, kErrTimeout);
                drain(&S.bar, phase);
            }
            return;
        }
    } else {
        // random gather: every record of the span in flight at once, by
        // asynchronous copies that hold no registers
        for (int x = threadIdx.x; x < span; x += kLtThreads) cp_async16(&S.rec[x], xm + S.perm[x]);
        cp_async_wait_all();
        __syncthreads();
    }
    // the reordered records, when asked for, go out by one bulk store (every
    // thread orders its shared-memory writes before the store reads them)
    if (xs) {
        fence_proxy_async_smem();
        __syncthreads();
        if (threadIdx.x == 0) bulk_store(xs + k0, S.rec, (uint32_t)te * 16u);
    }
    // 3. leaf starts of the tile, in order
    uint32_t flags = 0;
#pragma unroll
    for (int j = 0; j < kLtPer; ++j) {
        const int x = threadIdx.x * kLtPer + j;
        if (x < te) {
            const uint32_t v = S.ml[x];
            if ((v & 0xffu) <= (v >> 8)) flags |= 1u << j;
        }
    }
    const uint32_t cnt = __popc(flags);
    uint32_t incl = cnt;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += y;
    }
    if (lane == 31) S.wcount[warp] = incl;
    if (MODE == TB_MOM_FP64 && threadIdx.x < kLtHalo) S.bins[threadIdx.x] = 0;
    // the first start at or past the tile's end, from the halo: warp 0
    if (warp == 0) {
        int32_t nx = -1;
        for (int x0 = te; x0 < span && nx < 0; x0 += 32) {
            const int x = x0 + lane;
            bool st = false;
            if (x < span) {
                const uint32_t v = S.ml[x];
                st = (v & 0xffu) <= (v >> 8);
            }
            const unsigned b = __ballot_sync(0xffffffffu, st);
            if (b) nx = x0 + __ffs(b) - 1;
        }
        // the end of the array ends the last leaf
        if (nx < 0 && k0 + span == n) nx = span;
        if (lane == 0) {
            S.next_start = nx;
            S.n_long = 0;
        }
    }
    __syncthreads();
    uint32_t before = 0, total = 0;
    for (int w = 0; w < kLtThreads / 32; ++w) {
        const uint32_t c = S.wcount[w];
        if (w < warp) before += c;
        total += c;
    }
    uint32_t pos = before + incl - cnt;
#pragma unroll
    for (int j = 0; j < kLtPer; ++j)
        if (flags & (1u << j)) S.start[pos++] = (uint16_t)(threadIdx.x * kLtPer + j);
    __syncthreads();
    // 4. one thread per leaf
    const uint32_t jbase = start_cell ? 0u : leaf_off[2 * blockIdx.x];
    const int32_t nxt = S.next_start;
    // FP64: the leaves in order of their member counts (a counting sort, in
    // the permutation's place), so that the lanes of a warp run equally long.
    // In this mode the kernel is bound by the FP64 pipe (85% busy), which a
    // warp holds as long with few lanes active as with all: 0.49 ms against
    // 0.92 in key order at 6,000,000 particles, n_crit 16.
    uint16_t *order = reinterpret_cast<uint16_t *>(S.perm);
    if constexpr (MODE == TB_MOM_FP64) {
        auto members = [&](uint32_t r) {
            const int xe = (r + 1 < total) ? (int)S.start[r + 1] : nxt;
            return min((int)kLtHalo - 1, xe < 0 ? 0 : xe - (int)S.start[r]);
        };
        for (uint32_t r = threadIdx.x; r < total; r += kLtThreads) atomicAdd(&S.bins[members(r)], 1u);
        __syncthreads();
        if (warp == 0) {
            const uint32_t a = S.bins[2 * lane], b = S.bins[2 * lane + 1];
            uint32_t y = a + b;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const uint32_t z = __shfl_up_sync(0xffffffffu, y, off);
                if (lane >= off) y += z;
            }
            S.bins[2 * lane] = y - a - b;
            S.bins[2 * lane + 1] = y - b;
        }
        __syncthreads();
        for (uint32_t r = threadIdx.x; r < total; r += kLtThreads)
            order[atomicAdd(&S.bins[members(r)], 1u)] = (uint16_t)r;
        __syncthreads();
    }
    for (uint32_t i = threadIdx.x; i < total; i += kLtThreads) {
        const uint32_t r = MODE == TB_MOM_FP64 ? (uint32_t)order[i] : i;
        const int x = S.start[r];
        const int xe = (r + 1 < total) ? (int)S.start[r + 1] : nxt;
        const int64_t c = start_cell ? start_cell[k0 + x] : leaf_cell[jbase + r];
        const bool staged = xe >= 0;
        if (!staged) {
            // the end is past the span: leaves too long for one warp apart
            if (pend[c] - (int32_t)(k0 + x) > kBigLeafThread)
                big_queue[atomicAdd(&info->misc_ctr[2], 1u)] = (int32_t)c;
            else
                long_queue[atomicAdd(&info->misc_ctr[5], 1u)] = (int32_t)c;
            continue;
        }
        if (MODE == TB_MOM_FP32_COMP && xe - x > kSplitLeaf) {
            const uint32_t q = atomicAdd(&S.n_long, 1u);
            S.long_c[q] = (int32_t)c;
            S.long_x[q] = (uint32_t)x | ((uint32_t)xe << 16);
            continue;
        }
        if constexpr (MODE == TB_MOM_FP32_COMP) leaf_sum_split(o, (const float4 *)S.rec, c, x, xe);
        else leaf_sum<MODE>(o, (const float4 *)S.rec, c, x, xe);
    }
    if constexpr (MODE == TB_MOM_FP32_COMP) {
        __syncthreads();
        const uint32_t nl = S.n_long;
        for (uint32_t q = warp; q < nl; q += kLtThreads / 32) {
            const uint32_t xx = S.long_x[q];
            warp_leaf_sum<TB_MOM_FP32_COMP>(o, (const float4 *)S.rec, S.long_c[q], xx & 0xffffu,
                                            xx >> 16);
        }
    }
    if (xs && threadIdx.x == 0) bulk_store_wait_read();
}

// Non-leaf cells level by level, deepest first, each level d from its
// children at level d + 1.  The children of
// consecutive cells are consecutive cells, so level d + 1 is cut into tiles
// of kLmTile children: a block bulk-copies (TMA) the FP32 moments and the
// parent links of its tile -- plus the few children past it that belong to
// its last parents -- into shared memory, lists the parents whose first
// child lies in the tile (a child is the first of its parent iff its parent
// differs from the previous cell's), and combines them there.  Each copy
// covers whole groups of four cells, so that every array's piece starts on a
// 16-byte boundary; the moment and parent arrays are allocated kMomentPad
// cells past the capacity, which the rounding never passes.  The up to three
// cells the rounding adds before a level's first tile belong to level d,
// which is being written: they are copied but never read.  Blocks loop
// over the tiles of the level.
constexpr int kLmThreads = 128;
constexpr int kLmTile = 512, kLmMinTile = kLmTile / 4;
constexpr int kLmSpan = kLmTile + 16;   // 3 before the tile, 7 past it, rounding to 4

struct alignas(128) LevelSmem {
    float mass[kLmSpan];
    float com[3 * kLmSpan];
    float com_lo[3 * kLmSpan];
    float quad[6 * kLmSpan];
    float aabb[6 * kLmSpan];
    int32_t par[kLmSpan + 4];                 // parents of the staged cells and of 4 before
    int32_t own[kLmTile];                     // parents whose first child is in the tile
    uint16_t slot[kLmTile];                   // and that child's place in the tile
    uint32_t wcount[kLmThreads / 32];
    uint64_t bar;
};
static_assert(kLmSpan % 4 == 0, "each staged array spans whole 16-byte groups");
static_assert(kLmTile == 4 * kLmThreads, "the listing takes four children per thread");

// Children's FP32 moments staged in shared memory: cell c at slot c - base.
struct CellsStaged {
    static constexpr bool kAhead = false;
    const LevelSmem *S;
    int64_t base;
    __device__ __forceinline__ float m(int64_t c) const { return S->mass[c - base]; }
    __device__ __forceinline__ float x(int64_t c, int a) const { return S->com[3 * (c - base) + a]; }
    __device__ __forceinline__ float xl(int64_t c, int a) const { return S->com_lo[3 * (c - base) + a]; }
    __device__ __forceinline__ float2 q2(int64_t c, int i) const {
        return reinterpret_cast<const float2 *>(S->quad + 6 * (c - base))[i];
    }
    __device__ __forceinline__ float2 b2(int64_t c, int i) const {
        return reinterpret_cast<const float2 *>(S->aabb + 6 * (c - base))[i];
    }
};

// A tile [c_lo, c_hi) of the children level [off1, off2), as staged: cells
// [s_lo, s_hi) with the moments, parent links from p_lo on (one group of four
// before s_lo, for the cell before c_lo, or the level's start).
struct Staged {
    int64_t off1, off2, c_lo, c_hi, s_lo, s_hi, p_lo;
    __device__ Staged(int64_t off1_, int64_t off2_, int64_t lo, int64_t hi)
        : off1(off1_), off2(off2_), c_lo(lo), c_hi(hi), s_lo(lo & ~int64_t(3)),
          s_hi((min64(hi + 7, off2_) + 3) & ~int64_t(3)),
          p_lo(s_lo >= off1_ + 4 ? s_lo - 4 : (off1_ & ~int64_t(3))) {}
};

// One thread: the bulk copies of a staged tile into S.  The FP64 mode reads its
// sums from the tree, only the boxes from here.
template <int MODE>
__device__ __forceinline__ void stage(const TreeIn &T, const MomOut &o, LevelSmem &S, const Staged &g) {
    constexpr bool f32 = MODE != TB_MOM_FP64;
    const uint32_t len = (uint32_t)(g.s_hi - g.s_lo), plen = (uint32_t)(g.s_hi - g.p_lo);
    mbar_arrive_expect_tx(&S.bar, len * (f32 ? 76u : 24u) + plen * 4u);
    if constexpr (f32) {
        bulk_load(S.mass, o.mass + g.s_lo, len * 4u, &S.bar);
        bulk_load(S.com, o.com + 3 * g.s_lo, len * 12u, &S.bar);
        bulk_load(S.com_lo, o.com_lo + 3 * g.s_lo, len * 12u, &S.bar);
        bulk_load(S.quad, o.quad + 6 * g.s_lo, len * 24u, &S.bar);
    }
    bulk_load(S.aabb, o.aabb + 6 * g.s_lo, len * 24u, &S.bar);
    bulk_load(S.par, T.parent + g.p_lo, plen * 4u, &S.bar);
}

// The block waits for its staged tile; false when a copy did not complete.
__device__ __forceinline__ bool staged_wait(LevelSmem &S, uint32_t &phase, DevInfo *info,
                                            int64_t wait_limit) {
    const bool ok = mbar_wait_bounded(&S.bar, phase, wait_limit);
    phase ^= 1u;
    if (__syncthreads_and(ok)) return true;
    if (threadIdx.x == 0) {
        flag_error(&info->status, kErrTimeout);
        drain(&S.bar, phase ^ 1u);
    }
    return false;
}

// Lists in order the parents whose first child is in the staged tile; returns
// their number.  Four children per thread, a warp prefix and one across the
// warps; ends with a barrier.
__device__ __forceinline__ uint32_t list_parents(LevelSmem &S, const Staged &g) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nt = (int)(g.c_hi - g.c_lo);
    const int32_t *par = S.par + (g.c_lo - g.p_lo);
    uint32_t fl = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int x = 4 * (int)threadIdx.x + j;
        if (x < nt && ((x == 0 && g.c_lo == g.off1) || par[x] != par[x - 1])) fl |= 1u << j;
    }
    const uint32_t cnt = __popc(fl);
    uint32_t incl = cnt;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += y;
    }
    if (lane == 31) S.wcount[warp] = incl;
    __syncthreads();
    uint32_t pos = incl - cnt, total = 0;
#pragma unroll
    for (int w = 0; w < kLmThreads / 32; ++w) {
        const uint32_t v = S.wcount[w];
        if (w < warp) pos += v;
        total += v;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
        if (fl & (1u << j)) {
            const int x = 4 * (int)threadIdx.x + j;
            S.own[pos] = par[x];
            S.slot[pos++] = (uint16_t)x;
        }
    __syncthreads();
    return total;
}

// Children [c0, c1) of the i-th of `total` listed parents: up to the next one's
// first child, or where the links stop naming this parent.
__device__ __forceinline__ void listed_children(const LevelSmem &S, const Staged &g, uint32_t i,
                                                uint32_t total, int32_t &c0, int32_t &c1) {
    c0 = (int32_t)g.c_lo + S.slot[i];
    if (i + 1 < total) {
        c1 = (int32_t)g.c_lo + S.slot[i + 1];
    } else {
        const int32_t p = S.own[i], end = (int32_t)min64(g.c_hi + 7, g.off2);
        c1 = c0 + 1;
        while (c1 < end && S.par[c1 - g.p_lo] == p) ++c1;
    }
}

// The parents of tile t of the children level [off1, off2), staged and
// combined by one block; false when a copy did not complete.
template <int MODE>
__device__ __forceinline__ bool level_tile(const TreeIn &T, const MomOut &o, DevInfo *info, LevelSmem &S,
                                           int64_t off1, int64_t off2, int tile, int64_t t, int64_t step,
                                           uint32_t &phase, int64_t wait_limit) {
    const int64_t lo = off1 + t * tile;
    const Staged g(off1, off2, lo, min64(lo + tile, off2));
    if (threadIdx.x == 0) stage<MODE>(T, o, S, g);
    if (!staged_wait(S, phase, info, wait_limit)) return false;
    // the block's next tile of the level on its way to L2 meanwhile
    const int64_t n_lo = (off1 + (t + step) * tile) & ~int64_t(3);
    if (threadIdx.x == 0 && n_lo < off2) {
        const uint32_t len = (uint32_t)(((min64(n_lo + tile, off2) + 3) & ~int64_t(3)) - n_lo);
        if constexpr (MODE != TB_MOM_FP64) {
            bulk_prefetch(o.mass + n_lo, len * 4u);
            bulk_prefetch(o.com + 3 * n_lo, len * 12u);
            bulk_prefetch(o.com_lo + 3 * n_lo, len * 12u);
            bulk_prefetch(o.quad + 6 * n_lo, len * 24u);
        }
        bulk_prefetch(o.aabb + 6 * n_lo, len * 24u);
        bulk_prefetch(T.parent + n_lo, len * 4u);
    }
    const uint32_t total = list_parents(S, g);
    const CellsStaged src{&S, g.s_lo};
    int32_t c0 = 0, c1 = 0;
    if constexpr (MODE == TB_MOM_FP64) {
        for (uint32_t b = 0; b < total; b += kLmThreads / 4) {
            const uint32_t i = b + threadIdx.x / 4;
            const bool in = i < total;
            if (in) listed_children(S, g, i, total, c0, c1);
            else c0 = c1 = 0;
            combine_f64_quad(o, in ? S.own[i] : -1, c0, c1, src);
        }
    } else {
        for (uint32_t i = threadIdx.x; i < total; i += kLmThreads) {
            listed_children(S, g, i, total, c0, c1);
            combine_range<MODE>(T, o, S.own[i], c0, c1, src);
        }
    }
    return true;
}

// Levels d0 .. 0 by one block, each children level one tile at most, between
// two buffers: while level d is combined from one, the cells of level d (their
// leaves are done) come into the other, and the combined parents are written
// there as well as to the tree.  So a level costs its arithmetic, not a round
// trip through memory.
__device__ __noinline__ void solo_levels(TreeIn T, MomOut o, DevInfo *info, LevelSmem *S,
                                         const int64_t *off, int d0, uint32_t phase0, int64_t wait_limit) {
    uint32_t phase[2] = {phase0, 0u};
    if (threadIdx.x == 0) {
        mbar_init(&S[1].bar, 1);
        mbar_init_fence();
        stage<TB_MOM_FP32_COMP>(T, o, S[0], Staged(off[d0 + 1], off[d0 + 2], off[d0 + 1], off[d0 + 2]));
    }
    __syncthreads();
    int cur = 0;
    for (int d = d0; d >= 0; --d, cur ^= 1) {
        LevelSmem &A = S[cur], &B = S[cur ^ 1];
        const Staged g(off[d + 1], off[d + 2], off[d + 1], off[d + 2]);
        const Staged h(off[d], off[d + 1], off[d], off[d + 1]);
        if (threadIdx.x == 0 && d > 0) stage<TB_MOM_FP32_COMP>(T, o, B, h);
        if (!staged_wait(A, phase[cur], info, wait_limit)) {
            if (threadIdx.x == 0 && d > 0) drain(&B.bar, phase[cur ^ 1]);   // its copies too
            return;
        }
        const uint32_t total = list_parents(A, g);
        if (d > 0 && !staged_wait(B, phase[cur ^ 1], info, wait_limit)) return;
        if (d > 0) phase[cur ^ 1] ^= 1u;   // waited for here, not in the next step
        const CellsStaged src{&A, g.s_lo};
        const MomBoth both{o, MomOut{B.mass, B.com, B.com_lo, B.quad, B.aabb, nullptr, nullptr, nullptr}, h.s_lo};
        int32_t c0, c1;
        for (uint32_t i = threadIdx.x; i < total; i += kLmThreads) {
            listed_children(A, g, i, total, c0, c1);
            combine_range<TB_MOM_FP32_COMP>(T, both, A.own[i], c0, c1, src);
        }
        // A is filled again by the next step's copies
        fence_proxy_async_smem();
        __syncthreads();
    }
}

// Arrival of this block at a barrier of the grid (cooperative launch: every
// block is resident) after which `target` arrivals have been counted in all,
// and with `wait` the wait for them.  What
// the blocks wrote before is then visible, to bulk copies too (the proxy
// fences).  The wait is bounded; false when it ran out.
__device__ __forceinline__ bool grid_meet(uint32_t *ctr, uint32_t target, bool wait, int64_t limit,
                                          DevInfo *info) {
    bool ok = true;
    fence_proxy_async();
    __syncthreads();
    if (threadIdx.x == 0) {
        red_release_u32(ctr, 1u);
        if (wait) {
            int64_t it = 0;
            while (ld_acquire_u32(ctr) < target)
                if (!poll_backoff(it, limit)) {
                    flag_error(&info->status, kErrTimeout);
                    ok = false;
                    break;
                }
            fence_proxy_async();
        }
    }
    return wait ? __syncthreads_and(ok) != 0 : true;
}

constexpr int kBigThreads = kLmThreads;
struct BigLeafSmem {
    double d[kBigThreads][10];
    float f[kBigThreads][20];
    float bb[kBigThreads][6];
};
static_assert(sizeof(BigLeafSmem) <= sizeof(LevelSmem), "shares the level tiles' memory");

// The leaves the leaf launch queued: the long ones one warp per leaf, members
// read through the permutation (32 independent loads per round); those of
// more than kBigLeafThread members -- only depth-21 leaves of identical keys --
// summed by a whole block, one after another.
template <int MODE>
__device__ __noinline__ void queued_leaves(TreeIn T, MomOut o, PermSrc xs,
                                           const int32_t *long_queue, DevInfo *info,
                                           unsigned char *raw) {
    {
        const int64_t nl = info->misc_ctr[5];
        const int64_t nwarps = (int64_t)gridDim.x * (kLmThreads / 32);
        for (int64_t q = (blockIdx.x * (int64_t)kLmThreads + threadIdx.x) / 32; q < nl; q += nwarps) {
            const int64_t c = long_queue[q];
            warp_leaf_sum<MODE>(o, xs, c, T.pfirst[c], T.pend[c]);
        }
    }
    BigLeafSmem &S = *reinterpret_cast<BigLeafSmem *>(raw);
    auto &s_d = S.d;
    auto &s_f = S.f;
    auto &s_bb = S.bb;
    const uint32_t nq = info->misc_ctr[2];
    for (uint32_t q = blockIdx.x; q < nq; q += gridDim.x) {
        const int64_t c = T.big_leaf[q];
        const int64_t pf = T.pfirst[c], pe = T.pend[c];
        const int64_t cnt = pe - pf;
        const int64_t chunk = (cnt + kBigThreads - 1) / kBigThreads;
        const int64_t a0 = pf + threadIdx.x * chunk, a1 = min64(pe, a0 + chunk);
        const float4 r0 = xs[pf];
        const float ref[3] = {r0.x, r0.y, r0.z};
        float bb[6] = {r0.x, r0.y, r0.z, r0.x, r0.y, r0.z};
        const bool f64 = (MODE == TB_MOM_FP64) || cnt > kBigCell;
        AccD D;
        AccC Cc;
        AccP Pp;
        D.init(); Cc.init(); Pp.init();
        for (int64_t k = a0; k < a1; ++k) {
            const float4 v = xs[k];
            const float x[3] = {v.x, v.y, v.z};
            for (int a = 0; a < 3; ++a) { bb[a] = fminf(bb[a], x[a]); bb[3 + a] = fmaxf(bb[3 + a], x[a]); }
            if (f64) {
                double dx[3];
                for (int a = 0; a < 3; ++a) dx[a] = (double)x[a] - (double)ref[a];
                D.add((double)v.w, dx);
            } else {
                float dx[3];
                for (int a = 0; a < 3; ++a) dx[a] = __fsub_rn(x[a], ref[a]);
                if (MODE == TB_MOM_FP32_COMP) Cc.add(v.w, dx);
                else Pp.add(v.w, dx);
            }
        }
        // tree reduction in shared memory, fixed order
        for (int a = 0; a < 6; ++a) s_bb[threadIdx.x][a] = bb[a];
        if (f64) {
            s_d[threadIdx.x][0] = D.M;
            for (int a = 0; a < 3; ++a) s_d[threadIdx.x][1 + a] = D.S[a];
            for (int q2 = 0; q2 < 6; ++q2) s_d[threadIdx.x][4 + q2] = D.Q[q2];
        } else if (MODE == TB_MOM_FP32_COMP) {
            s_f[threadIdx.x][0] = Cc.M; s_f[threadIdx.x][1] = Cc.Mc;
            for (int a = 0; a < 3; ++a) { s_f[threadIdx.x][2 + a] = Cc.S[a]; s_f[threadIdx.x][5 + a] = Cc.Sc[a]; }
            for (int q2 = 0; q2 < 6; ++q2) { s_f[threadIdx.x][8 + q2] = Cc.Q[q2]; s_f[threadIdx.x][14 + q2] = Cc.Qc[q2]; }
        } else {
            s_f[threadIdx.x][0] = Pp.M;
            for (int a = 0; a < 3; ++a) s_f[threadIdx.x][2 + a] = Pp.S[a];
            for (int q2 = 0; q2 < 6; ++q2) s_f[threadIdx.x][8 + q2] = Pp.Q[q2];
        }
        __syncthreads();
        for (int half = kBigThreads / 2; half > 0; half >>= 1) {
            if (threadIdx.x < half) {
                const int u = threadIdx.x, v = threadIdx.x + half;
                for (int a = 0; a < 3; ++a) {
                    s_bb[u][a] = fminf(s_bb[u][a], s_bb[v][a]);
                    s_bb[u][3 + a] = fmaxf(s_bb[u][3 + a], s_bb[v][3 + a]);
                }
                if (f64) {
                    for (int z = 0; z < 10; ++z) s_d[u][z] += s_d[v][z];
                } else if (MODE == TB_MOM_FP32_COMP) {
                    AccC A, B;
                    A.M = s_f[u][0]; A.Mc = s_f[u][1]; B.M = s_f[v][0]; B.Mc = s_f[v][1];
                    for (int a = 0; a < 3; ++a) {
                        A.S[a] = s_f[u][2 + a]; A.Sc[a] = s_f[u][5 + a];
                        B.S[a] = s_f[v][2 + a]; B.Sc[a] = s_f[v][5 + a];
                    }
                    for (int q2 = 0; q2 < 6; ++q2) {
                        A.Q[q2] = s_f[u][8 + q2]; A.Qc[q2] = s_f[u][14 + q2];
                        B.Q[q2] = s_f[v][8 + q2]; B.Qc[q2] = s_f[v][14 + q2];
                    }
                    A.merge(B);
                    s_f[u][0] = A.M; s_f[u][1] = A.Mc;
                    for (int a = 0; a < 3; ++a) { s_f[u][2 + a] = A.S[a]; s_f[u][5 + a] = A.Sc[a]; }
                    for (int q2 = 0; q2 < 6; ++q2) { s_f[u][8 + q2] = A.Q[q2]; s_f[u][14 + q2] = A.Qc[q2]; }
                } else {
                    s_f[u][0] += s_f[v][0];
                    for (int a = 0; a < 3; ++a) s_f[u][2 + a] += s_f[v][2 + a];
                    for (int q2 = 0; q2 < 6; ++q2) s_f[u][8 + q2] += s_f[v][8 + q2];
                }
            }
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            float bbf[6];
            for (int a = 0; a < 6; ++a) bbf[a] = s_bb[0][a];
            if (f64) {
                AccD A;
                A.M = s_d[0][0];
                for (int a = 0; a < 3; ++a) A.S[a] = s_d[0][1 + a];
                for (int q2 = 0; q2 < 6; ++q2) A.Q[q2] = s_d[0][4 + q2];
                finish_d(o, c, A, ref, bbf, MODE == TB_MOM_FP64);
            } else if (MODE == TB_MOM_FP32_COMP) {
                AccC A;
                A.M = s_f[0][0]; A.Mc = s_f[0][1];
                for (int a = 0; a < 3; ++a) { A.S[a] = s_f[0][2 + a]; A.Sc[a] = s_f[0][5 + a]; }
                for (int q2 = 0; q2 < 6; ++q2) { A.Q[q2] = s_f[0][8 + q2]; A.Qc[q2] = s_f[0][14 + q2]; }
                finish_c(o, c, A, ref, bbf);
            } else {
                AccP A;
                A.M = s_f[0][0];
                for (int a = 0; a < 3; ++a) A.S[a] = s_f[0][2 + a];
                for (int q2 = 0; q2 < 6; ++q2) A.Q[q2] = s_f[0][8 + q2];
                finish_p(o, c, A, ref, bbf);
            }
        }
        __syncthreads();
    }
}

// Queued leaves, then the non-leaf cells of levels d_hi .. d_lo, deepest first.
// One cooperative launch takes every level (d_hi = 20, d_lo = 0), with a grid
// barrier between levels; levels that do not exist cost nothing, and blocks
// that no level above needs leave.  From the
// first level on whose children, and those of every level above, fill one
// tile at most, block 0 goes on alone (in the compensated mode, with `two`
// buffers, by solo_levels).  At 65,536 uniform particles this takes 26 us; 21
// launches of one level each took 78 us (16 of them for levels without
// parents, 2.8 us each) and two more for queued leaves 6 us.  At 2^27
// clustered, where the big levels' bytes bound it, 0.75 ms against 0.79.  In
// FP64, bound by latency and
// the FP64 pipe, 0.45 ms against 0.52 at 6,000,000.  A device that
// takes no cooperative launch gets one launch per level (d_hi = d_lo, no
// barrier), queued leaves first (d_hi < 0).
template <int MODE>
__global__ void __launch_bounds__(kLmThreads, 5)
    upward_kernel(TreeIn T, MomOut o, PermSrc src, const int32_t *long_queue, DevInfo *info, int d_hi,
                  int d_lo, bool leaves, bool two, int64_t wait_limit) {
    after_previous();
    if (info->status & (kErrOverflow | kErrNonFinite | kErrTimeout | kErrInvalid)) return;
    extern __shared__ __align__(128) unsigned char lm_raw[];
    LevelSmem &S = *reinterpret_cast<LevelSmem *>(lm_raw);
    __shared__ int64_t s_off[kLevels + 1];
    __shared__ uint32_t s_act[kLevels];
    __shared__ uint32_t s_queued;
    __shared__ int s_solo;
    uint32_t *meet = &info->misc_ctr[7];
    if (threadIdx.x <= kLevels) s_off[threadIdx.x] = info->level_offset[threadIdx.x];
    if (threadIdx.x == 0) s_queued = leaves ? (info->misc_ctr[2] | info->misc_ctr[5]) : 0u;
    __syncthreads();
    uint32_t met = 0, phase = 0;
    if (s_queued) {
        queued_leaves<MODE>(T, o, src, long_queue, info, lm_raw);
        met += gridDim.x;
        if (d_hi >= 0 && !grid_meet(meet, met, true, wait_limit, info)) return;
    }
    if (d_hi < 0) return;
    if (threadIdx.x == 0) {
        mbar_init(&S.bar, 1);
        mbar_init_fence();
        // levels 0 .. solo: at most one tile of children each, block 0 alone;
        // above them as many blocks as the level or one above it has smallest
        // tiles: a barrier costs by the blocks that meet
        int solo = -1;
        while (solo < d_hi && s_off[solo + 3] - s_off[solo + 2] <= kLmTile) ++solo;
        s_solo = solo;
        int64_t most = 1;
        for (int d = 0; d <= d_hi; ++d) {
            const int64_t kids = s_off[d + 2] - s_off[d + 1];
            if (d > solo && (kids + kLmMinTile - 1) / kLmMinTile > most) most = (kids + kLmMinTile - 1) / kLmMinTile;
            s_act[d] = (uint32_t)min64(most, gridDim.x);
        }
    }
    __syncthreads();
    const int solo = s_solo;
    int deepest = d_hi;
    while (deepest > d_lo && s_off[deepest + 1] == s_off[deepest + 2]) --deepest;
    bool tail = d_hi > d_lo;   // the deepest levels, while one tile each: block 0 alone as well
    for (int d = d_hi; d >= d_lo; --d) {
        const int64_t off1 = s_off[d + 1], off2 = s_off[d + 2];
        if (off1 == off2) continue;
        const uint32_t act = s_act[d];
        if (blockIdx.x >= act) return;
        const bool was = tail && d < deepest;
        tail = tail && d > solo && off2 - off1 <= kLmTile;
        if (was && !tail && d > solo) {
            // the first level for all: what block 0 combined is its children
            met += act;
            if (!grid_meet(meet, met, true, wait_limit, info)) return;
        }
        if (tail && blockIdx.x != 0) continue;
        if (MODE == TB_MOM_FP32_COMP && two && d <= solo && d_lo == 0) {
            solo_levels(T, o, info, &S, s_off, d, phase, wait_limit);
            break;
        }
        // smaller tiles where the level would leave blocks idle or give a few
        // of them one tile more
        int tile = kLmTile;
        if (d > solo && !tail)
            while (tile > kLmMinTile && off2 - off1 <= (int64_t)act * tile * 2) tile /= 2;
        const int64_t tiles = (off2 - off1 + tile - 1) / tile;
        for (int64_t t = blockIdx.x; t < tiles; t += act) {
            if (!level_tile<MODE>(T, o, info, S, off1, off2, tile, t, act, phase, wait_limit)) return;
            // the next tile's copies overwrite what this one read
            fence_proxy_async_smem();
            __syncthreads();
        }
        if (d == d_lo) break;
        if (d > solo && !tail) {
            met += act;
            if (!grid_meet(meet, met, blockIdx.x < s_act[d - 1], wait_limit, info)) return;
        } else {
            // this block's own cells are the next level's children
            __threadfence();
            fence_proxy_async();
            __syncthreads();
        }
    }
    // block 0 leaves the queues clear for the next call on this build: every
    // block read their lengths before the first meeting, if they were not zero.
    // (The barrier count is not cleared here, where a block may still be on its
    // way out of that meeting: the next leaf launch does it.)
    if (blockIdx.x == 0 && threadIdx.x == 0 && d_lo == 0) info->misc_ctr[2] = info->misc_ctr[5] = 0;
}

__global__ void wait_selftest_kernel(int64_t limit, uint32_t *status, const uint32_t *flag) {
    int64_t iter = 0;
    while (*(volatile const uint32_t *)flag == 0u) {
        if (!poll_backoff(iter, limit)) {
            flag_error(status, kErrTimeout);
            return;
        }
    }
}

constexpr int64_t kTwoBufferMax = int64_t(1) << 19;   // particles whose upward pass takes two buffers

// The long-leaf queue (at most n / 2 leaves of two or more members past the
// first) sits in the upper half of the big-leaf buffer (at most n / 2049
// entries in the lower).
int32_t *long_queue(Workspace &ws, int64_t n) { return ws.big_leaf + (n + 1) / 2; }

// The leaves' moments (leaf_tile_kernel), long ones queued for upward_kernel.
template <int MODE>
cudaError_t leaves_impl(tb_tree &t, Workspace &ws, const int32_t *start_cell, cudaStream_t s) {
    MomOut o{t.mass, t.com, t.com_lo, t.quad, t.aabb, t.mass64, t.com64, t.quad64};
    const int64_t n = t.n_particles;
    static std::atomic<uint64_t> attr_done{0};
    const cudaError_t set = once_on_device(attr_done, [] {
        const cudaError_t e = allow_smem(leaf_tile_kernel<MODE>, leaf_tile_smem(), true);
        return e == cudaSuccess ? allow_smem(upward_kernel<MODE>, 2 * sizeof(LevelSmem), true) : e;
    });
    if (set != cudaSuccess) return set;
    const int64_t tiles = (n + kLtTile - 1) / kLtTile;
    const int64_t level_tiles = (n + level_tile_size() - 1) / level_tile_size();
    const uint32_t *leaf_off = ws.level_cnt + (int64_t)kLevels * level_tiles;
    float4 *xs = t.pos_sorted ? reinterpret_cast<float4 *>(t.pos_sorted) : nullptr;
    if (start_cell)   // batched: one chain with the build
        launch_after(leaf_tile_kernel<MODE>, dim3((unsigned)tiles), dim3(kLtThreads), leaf_tile_smem(), s, o,
                     t.leaf_cell, start_cell, t.perm, ws.xm, ws.ml, leaf_off, t.pend, n, xs,
                     long_queue(ws, n), ws.big_leaf, ws.info, g_wait_limit);
    else
        leaf_tile_kernel<MODE><<<(unsigned)tiles, kLtThreads, leaf_tile_smem(), s>>>(
            o, t.leaf_cell, start_cell, t.perm, ws.xm, ws.ml, leaf_off, t.pend, n, xs, long_queue(ws, n),
            ws.big_leaf, ws.info, g_wait_limit);
    ++g_launches;
    return cudaGetLastError();
}

template <int MODE>
cudaError_t moments_impl(tb_tree &t, Workspace &ws, cudaStream_t s) {
    TreeIn T{t.child_first, t.child_end, t.pfirst, t.pend, ws.big_leaf, t.parent};
    MomOut o{t.mass, t.com, t.com_lo, t.quad, t.aabb, t.mass64, t.com64, t.quad64};
    const int64_t n = t.n_particles;
    cudaError_t e = leaves_impl<MODE>(t, ws, nullptr, s);
    if (e != cudaSuccess) return e;
    mark(ws, "leaves", s);
    // every level in one cooperative launch of as many blocks as are resident
    // at once, never more than the tiles a level of at most n cells can have
    PermSrc src{ws.xm, t.perm};
    int d_hi = kDepthMax - 1, d_lo = 0;
    bool leaves = true;
    // a second buffer for the top levels where few blocks per SM are enough
    // (300,000 particles 155 us against 159; at 2,000,000 332 against 324)
    bool two = n <= kTwoBufferMax;
    const size_t smem = sizeof(LevelSmem) * (two ? 2 : 1);
    static std::atomic<int> resident[2][64];
    int64_t grid = 0;
    if ((e = resident_blocks(resident[two ? 1 : 0], reinterpret_cast<const void *>(upward_kernel<MODE>),
                             kLmThreads, smem, grid)) != cudaSuccess)
        return e;
    const int64_t most = (n + kLmMinTile - 1) / kLmMinTile;
    if (grid > most) grid = most;
    const int32_t *lq = long_queue(ws, n);
    int64_t lim = g_wait_limit;
    void *args[] = {&T, &o, &src, &lq, &ws.info, &d_hi, &d_lo, &leaves, &two, &lim};
    e = fault_cooperative()
            ? cudaErrorCooperativeLaunchTooLarge
            : cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(upward_kernel<MODE>),
                                          dim3((unsigned)grid), dim3(kLmThreads), args, smem, s);
    if (e == cudaSuccess) {
        ++g_launches;
    } else {
        // no cooperative launch here: the queued leaves, then one launch per level
        cudaGetLastError();
        for (int d = kDepthMax; d >= 0; --d) {
            upward_kernel<MODE><<<(unsigned)grid, kLmThreads, sizeof(LevelSmem), s>>>(
                T, o, src, lq, ws.info, d == kDepthMax ? -1 : d, d == kDepthMax ? -1 : d,
                d == kDepthMax, false, lim);
            ++g_launches;
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
        }
    }
    mark(ws, "moments", s);
    return cudaSuccess;
}

// xs[k] = xm[perm[k]]: the particles in key order, for the tree walk when
// the moments did not write them; every thread keeps four gathers in flight.
__global__ void __launch_bounds__(256)
    gather_records_kernel(const int32_t *__restrict__ perm, const float4 *__restrict__ xm,
                          float4 *__restrict__ xs, int64_t n) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t n4 = n / 4;
    const int4 *p4 = reinterpret_cast<const int4 *>(perm);
    for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < n4; g += stride) {
        const int4 id = __ldcs(p4 + g);
        const float4 a = __ldg(xm + id.x), b = __ldg(xm + id.y), c = __ldg(xm + id.z),
                     d = __ldg(xm + id.w);
        xs[4 * g] = a;
        xs[4 * g + 1] = b;
        xs[4 * g + 2] = c;
        xs[4 * g + 3] = d;
    }
    for (int64_t k = 4 * n4 + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += stride)
        xs[k] = __ldg(xm + perm[k]);
}

}  // namespace

cudaError_t launch_gather_records(const int32_t *perm, const float4 *xm, float4 *xs, int64_t n,
                                  cudaStream_t s) {
    int64_t g = (n / 4 + 255) / 256;
    if (g > 152 * 16) g = 152 * 16;
    if (g < 1) g = 1;
    gather_records_kernel<<<(unsigned)g, 256, 0, s>>>(perm, xm, xs, n);
    ++g_launches;
    return cudaGetLastError();
}

// The leaves of a batched build: the tiles of the whole key order, then the
// queued long ones.
template <int MODE>
static cudaError_t batched_leaves_impl(tb_tree &t, Workspace &ws, const int32_t *start_cell,
                                       cudaStream_t s) {
    cudaError_t e = leaves_impl<MODE>(t, ws, start_cell, s);
    if (e != cudaSuccess) return e;
    TreeIn T{t.child_first, t.child_end, t.pfirst, t.pend, ws.big_leaf, t.parent};
    MomOut o{t.mass, t.com, t.com_lo, t.quad, t.aabb, t.mass64, t.com64, t.quad64};
    launch_after(upward_kernel<MODE>, dim3(152), dim3(kLmThreads), sizeof(LevelSmem), s, T, o, PermSrc{ws.xm, t.perm}, long_queue(ws, t.n_particles), ws.info, -1, -1, true, false, g_wait_limit);
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_batched_leaves(tb_tree &t, Workspace &ws, int mode, const int32_t *start_cell,
                                  cudaStream_t s) {
    switch (mode) {
        case TB_MOM_FP32_COMP: return batched_leaves_impl<TB_MOM_FP32_COMP>(t, ws, start_cell, s);
        case TB_MOM_FP32_PLAIN: return batched_leaves_impl<TB_MOM_FP32_PLAIN>(t, ws, start_cell, s);
        case TB_MOM_FP64: return batched_leaves_impl<TB_MOM_FP64>(t, ws, start_cell, s);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_moments(tb_tree &t, Workspace &ws, int mode, cudaStream_t s) {
    switch (mode) {
        case TB_MOM_FP32_COMP: return moments_impl<TB_MOM_FP32_COMP>(t, ws, s);
        case TB_MOM_FP32_PLAIN: return moments_impl<TB_MOM_FP32_PLAIN>(t, ws, s);
        case TB_MOM_FP64: return moments_impl<TB_MOM_FP64>(t, ws, s);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_wait_selftest(int64_t limit, uint32_t *status, uint32_t *flag, cudaStream_t s) {
    wait_selftest_kernel<<<1, 1, 0, s>>>(limit, status, flag);
    ++g_launches;
    return cudaGetLastError();
}

}  // namespace tb
