// tb_sort.cu -- stable LSD radix sort of (key, original index) pairs
// (Sec. 2.3 step 2).
//
// The paper sorts on the CPU with parallel sorting by regular sampling; on
// the GPU the keys are sorted by ceil(40 / b) stable least-significant-digit
// passes of b bits, over their upper bits (bit 63 is always 1).  Each pass is one
// "onesweep" launch (Adinets & Merrill 2022):
//   - every block takes the next tile id from an atomic counter, so a block
//     only ever waits on tiles that blocks already running own;
//   - it ranks its tile's digits stably, warp by warp (ballot peer masks,
//     shared-memory counters), in tile order;
//   - it publishes its per-digit counts to a look-back array and walks back
//     over earlier tiles until it meets an inclusive prefix (decoupled
//     look-back); every wait is bounded and reports a timeout instead of
//     hanging;
//   - it orders the tile by digit in shared memory and writes keys and
//     indices out as runs of consecutive addresses.
// The passes order the keys by their upper ceil(40 / b) * b bits only; the runs
// of equal upper bits they leave (short in practice) are ordered by the low
// bits afterwards (tb_runs.cu).  Digit offsets of every pass come from the
// histograms taken while the keys were made.  Look-back words carry an epoch (build counter + pass) so that
// the array is never cleared between passes or builds.
#include "tb_device.cuh"

namespace tb {

namespace {

constexpr uint64_t kFlagAgg = 1ull << 62;
constexpr int kLookWindow = 4;
constexpr uint64_t kFlagIncl = 2ull << 62;

template <int RADIX_BITS, int THREADS, int ITEMS>
struct SortSmem {
    static constexpr int RADIX = 1 << RADIX_BITS;
    static constexpr int WARPS = THREADS / 32;
    static constexpr int TILE = THREADS * ITEMS;
    uint64_t keys[TILE];
    int32_t vals[TILE];
    uint32_t warp_hist[WARPS][RADIX + 1];
    uint32_t tile_off[RADIX + 1];
    uint32_t glob_base[RADIX];
    uint32_t scan_tmp[WARPS];
    uint32_t tile;
};

// Digit d's count over the tiles before `tile`: looks back, kLookWindow
// predecessors read per round so that one memory latency covers several
// tiles, until one that has published its inclusive prefix.  Every wait is
// bounded; one that runs out records a timeout (the count is then too small).
template <int RADIX>
__device__ __forceinline__ uint32_t look_back(const uint64_t *lookback, uint32_t tile, int d, uint64_t epoch,
                                              int64_t spin_limit, DevInfo *info) {
    uint32_t excl = 0;
    int64_t pred = (int64_t)tile - 1;
    int64_t iter = 0;
    for (;;) {
        uint64_t w[kLookWindow];
#pragma unroll
        for (int j = 0; j < kLookWindow; ++j)
            w[j] = (pred - j >= 0) ? ld_relaxed_u64(lookback + (pred - j) * RADIX + d) : 0ull;
        int adv = 0;
        bool found = false, blocked = false;
#pragma unroll
        for (int j = 0; j < kLookWindow; ++j) {
            if (found || blocked) continue;
            if (pred - j < 0 || ((w[j] >> 32) & 0x3fffffffu) != epoch || (w[j] >> 62) == 0) {
                blocked = true;
                continue;
            }
            excl += (uint32_t)w[j];
            adv = j + 1;
            if ((w[j] >> 62) == 2) found = true;
        }
        if (found) return excl;
        pred -= adv;
        if (adv == 0 && !poll_backoff(iter, spin_limit)) {
            flag_error(&info->status, kErrTimeout);
            return excl;
        }
    }
}

template <int RADIX_BITS, int THREADS, int ITEMS, bool FIRST>
__global__ void __launch_bounds__(THREADS, (THREADS <= 256 ? (ITEMS <= 8 ? 4 : 2) : (ITEMS <= 8 ? 2 : 1)))
    onesweep_kernel(const uint64_t *__restrict__ keys_in, const int32_t *__restrict__ vals_in,
                    uint64_t *__restrict__ keys_out, int32_t *__restrict__ vals_out, int64_t n,
                    int pass, int shift0, const uint32_t *__restrict__ digit_off, uint64_t *lookback,
                    DevInfo *info, int64_t spin_limit) {
    after_previous();
    using S = SortSmem<RADIX_BITS, THREADS, ITEMS>;
    constexpr int RADIX = S::RADIX;
    constexpr int WARPS = S::WARPS;
    constexpr int TILE = S::TILE;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    S &sm = *reinterpret_cast<S *>(smem_raw);

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int shift = shift0 + pass * RADIX_BITS;

    if (threadIdx.x == 0) sm.tile = atomicAdd(&info->sort_tile_ctr[pass], 1u);
    for (int i = threadIdx.x; i < WARPS * (RADIX + 1); i += THREADS)
        (&sm.warp_hist[0][0])[i] = 0;
    __syncthreads();
    const uint32_t tile = sm.tile;
    const int64_t tile_base = (int64_t)tile * TILE;
    const int valid = (int)min64(TILE, n - tile_base);

    // load (warp-striped: warp w owns 32*ITEMS consecutive elements)
    uint64_t key[ITEMS];
    int32_t val[ITEMS];
    uint32_t rank[ITEMS];
    const int wbase = warp * 32 * ITEMS;
    const bool full = valid == TILE;
    if (full) {
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            const int e = wbase + i * 32 + lane;
            key[i] = keys_in[tile_base + e];
            val[i] = FIRST ? (int32_t)(tile_base + e) : vals_in[tile_base + e];
        }
    } else {
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            const int e = wbase + i * 32 + lane;
            if (e < valid) {
                key[i] = keys_in[tile_base + e];
                val[i] = FIRST ? (int32_t)(tile_base + e) : vals_in[tile_base + e];
            } else {
                key[i] = 0;
                val[i] = 0;
            }
        }
    }

    // stable rank within the warp, in element order.  The lanes holding the
    // same digit are found with one ballot per digit bit (plus one for the
    // tail sentinel); the lowest of them adds the group's size to the warp's
    // digit counter with a shared-memory atomic, whose returned old value is
    // collected only after every item has been issued, so no item waits on
    // the one before.  A warp's atomics on one counter are applied in issue
    // order, which keeps equal digits in element order.
    const unsigned lt = lanemask_lt();
    uint32_t old_cnt[ITEMS], lead_rank[ITEMS];
    // a full tile needs no sentinel bit: RADIX_BITS ballots per item
    const int nbits = full ? RADIX_BITS : RADIX_BITS + 1;
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        const int e = wbase + i * 32 + lane;
        const uint32_t d = (full || e < valid) ? (uint32_t)((key[i] >> shift) & (RADIX - 1))
                                               : (uint32_t)RADIX;
        unsigned peers = 0xffffffffu;
#pragma unroll
        for (int b = 0; b <= RADIX_BITS; ++b) {
            if (b == RADIX_BITS && nbits == RADIX_BITS) break;
            const bool bit = (d >> b) & 1u;
            const unsigned v = __ballot_sync(0xffffffffu, bit);
            peers &= bit ? v : ~v;
        }
        const int leader = __ffs(peers) - 1;
        old_cnt[i] = (lane == leader) ? atomicAdd(&sm.warp_hist[warp][d], (uint32_t)__popc(peers)) : 0u;
        lead_rank[i] = (uint32_t)leader | ((uint32_t)__popc(peers & lt) << 8);
    }
#pragma unroll
    for (int i = 0; i < ITEMS; ++i)
        rank[i] = __shfl_sync(0xffffffffu, old_cnt[i], lead_rank[i] & 31u) + (lead_rank[i] >> 8);
    __syncthreads();

    // per-digit: offsets of each warp within the digit, tile digit counts
    uint32_t my_count[(RADIX + THREADS - 1) / THREADS];
#pragma unroll
    for (int r = 0; r < (RADIX + THREADS - 1) / THREADS; ++r) {
        int d = r * THREADS + threadIdx.x;
        uint32_t acc = 0;
        if (d < RADIX) {
            for (int w = 0; w < WARPS; ++w) {
                uint32_t c = sm.warp_hist[w][d];
                sm.warp_hist[w][d] = acc;
                acc += c;
            }
        }
        my_count[r] = acc;
    }
    // exclusive scan of the counts over digits
    if constexpr (RADIX <= THREADS) {
        // one digit per thread: a warp scan and one across the warps
        const uint32_t c = (threadIdx.x < RADIX) ? my_count[0] : 0u;
        uint32_t x = c;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, off);
            if (lane >= off) x += y;
        }
        if (lane == 31) sm.scan_tmp[warp] = x;
        __syncthreads();
        uint32_t wpre = 0;
        for (int w = 0; w < warp; ++w) wpre += sm.scan_tmp[w];
        if (threadIdx.x < RADIX) sm.tile_off[threadIdx.x] = wpre + x - c;
        if (threadIdx.x == 0) sm.tile_off[RADIX] = (uint32_t)valid;
    } else {
        // each thread holds a contiguous group of digits
        constexpr int PER = (RADIX + THREADS - 1) / THREADS;
        // regroup: thread t owns digits [t*PER, t*PER+PER) for the scan
        __syncthreads();
#pragma unroll
        for (int r = 0; r < PER; ++r) {
            int d = r * THREADS + threadIdx.x;
            if (d < RADIX) sm.tile_off[d] = my_count[r];
        }
        __syncthreads();
        uint32_t loc[PER];
        uint32_t sum = 0;
#pragma unroll
        for (int r = 0; r < PER; ++r) {
            int d = threadIdx.x * PER + r;
            loc[r] = (d < RADIX) ? sm.tile_off[d] : 0u;
            sum += loc[r];
        }
        uint32_t x = sum;
        for (int off = 1; off < 32; off <<= 1) {
            uint32_t y = __shfl_up_sync(0xffffffffu, x, off);
            if (lane >= off) x += y;
        }
        if (lane == 31) sm.scan_tmp[warp] = x;
        __syncthreads();
        uint32_t wpre = 0;
        for (int w = 0; w < warp; ++w) wpre += sm.scan_tmp[w];
        uint32_t run = wpre + x - sum;
        __syncthreads();
#pragma unroll
        for (int r = 0; r < PER; ++r) {
            int d = threadIdx.x * PER + r;
            if (d < RADIX) sm.tile_off[d] = run;
            run += loc[r];
        }
        if (threadIdx.x == 0) sm.tile_off[RADIX] = (uint32_t)valid;
    }
    __syncthreads();

    // publish this tile's digit counts (aggregate), then order the tile by
    // digit in shared memory while the predecessors finish theirs
    const uint64_t epoch = (uint64_t)((info->epoch + (uint32_t)pass) & 0x3fffffffu);
#pragma unroll
    for (int r = 0; r < (RADIX + THREADS - 1) / THREADS; ++r) {
        int d = r * THREADS + threadIdx.x;
        if (d >= RADIX) continue;
        uint64_t *slot = lookback + (int64_t)tile * RADIX + d;
        st_relaxed_u64(slot, (tile == 0 ? kFlagIncl : kFlagAgg) | (epoch << 32) | my_count[r]);
    }
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        int e = wbase + i * 32 + lane;
        if (e < valid) {
            uint32_t d = (uint32_t)((key[i] >> shift) & (RADIX - 1));
            uint32_t p = sm.tile_off[d] + sm.warp_hist[warp][d] + rank[i];
            sm.keys[p] = key[i];
            sm.vals[p] = val[i];
        }
    }

    // decoupled look-back, one digit per thread, kLookWindow predecessors
    // read per round so that one memory latency covers several tiles
#pragma unroll
    for (int r = 0; r < (RADIX + THREADS - 1) / THREADS; ++r) {
        int d = r * THREADS + threadIdx.x;
        if (d >= RADIX) continue;
        uint32_t excl = 0;
        if (tile > 0) {
            excl = look_back<RADIX>(lookback, tile, d, epoch, spin_limit, info);
            st_relaxed_u64(lookback + (int64_t)tile * RADIX + d,
                           kFlagIncl | (epoch << 32) | (excl + my_count[r]));
        }
        sm.glob_base[d] = digit_off[d] + excl - sm.tile_off[d];
    }
    __syncthreads();

    // write runs of equal digits to consecutive global addresses
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        int j = i * THREADS + threadIdx.x;
        if (j < valid) {
            uint64_t k = sm.keys[j];
            uint32_t d = (uint32_t)((k >> shift) & (RADIX - 1));
            uint64_t dst = (uint64_t)sm.glob_base[d] + (uint32_t)j;
            dst &= 0xffffffffull;
            if ((int64_t)dst < n) {
                keys_out[dst] = k;
                vals_out[dst] = sm.vals[j];
            } else {
                flag_error(&info->status, kErrTimeout);
            }
        }
    }
}

// The pass for 8-bit digits (the default), arranged for many keys per thread:
//   - keys go through shared memory and out first, then values through the same
//     memory, and the values are loaded only when the keys have left the
//     registers, so that a tile of 5376 keys (256 x 21) takes 52 KB, three to an
//     SM, at 80 registers (of which 112 to 124 bytes a thread spill; 512 x 14, two
//     to an SM at 64, spills 120 to 128);
//   - a key's place in the tile is kept in 16 bits, each warp's counters are
//     turned into places in the tile at once (one shared read per key), and a
//     full tile carries no bounds checks.
// What bounds it is latency: the warps wait on the tile's barriers and on shared
// memory, with 40% of the issue slots and a third of DRAM busy.  133
// instructions a key (172 before), 0.94 ms at 2^27 keys, 3.3 TB/s, where one thread-register tile of
// 512 x 8 pairs took 1.19; 142 us against 160 at 2^24.
template <int T, int ITEMS>
struct Sort8Smem {
    static constexpr int TILE = T * ITEMS;
    static constexpr int WARPS = T / 32;
    union {
        uint64_t keys[TILE];
        int32_t vals[TILE];
    };
    uint32_t warp_hist[WARPS][257];
    uint32_t cnt[256], loc[256], base[256];
    uint32_t carry[WARPS];
    uint32_t tile;
};

template <int T, int ITEMS, bool FIRST, bool FULL>
__device__ __forceinline__ void tile8(Sort8Smem<T, ITEMS> &sm, const uint64_t *__restrict__ keys_in,
                                          const int32_t *__restrict__ vals_in,
                                          uint64_t *__restrict__ keys_out, int32_t *__restrict__ vals_out,
                                          uint32_t n, uint32_t tile, int valid, int pass, int shift,
                                          const uint32_t *__restrict__ digit_off, uint64_t *lookback,
                                          DevInfo *info, int64_t spin_limit) {
    constexpr int TILE = Sort8Smem<T, ITEMS>::TILE, W = T / 32;
    constexpr int L = T / 256;   // lanes per digit when the tile's digits are counted
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int first = warp * 32 * ITEMS + lane;          // this thread's elements: first + 32 i
    const uint32_t tile_base = tile * (uint32_t)TILE;
    const unsigned lt = lanemask_lt();
    uint64_t key[ITEMS];
    uint32_t at[(ITEMS + 1) / 2] = {};   // rank in the warp's digit, then place in the tile (16 bits each)
    {
        const uint64_t *src = keys_in + tile_base + first;
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) key[i] = FULL || first + i * 32 < valid ? src[i * 32] : 0ull;
    }
    uint32_t *hist = sm.warp_hist[warp];
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        const bool in = FULL || first + i * 32 < valid;
        const uint32_t d = (uint32_t)(key[i] >> shift) & 255u;
        unsigned peers = 0xffffffffu;
        if (!FULL) {
            peers = __ballot_sync(0xffffffffu, in);
            if (!in) peers = 0;
        }
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            const bool bit = (d >> b) & 1u;
            const unsigned v = __ballot_sync(0xffffffffu, bit);
            peers &= bit ? v : ~v;
        }
        const unsigned below = peers & lt;               // the group's lowest lane has none
        uint32_t old = 0;
        if (in && below == 0) old = atomicAdd(hist + d, (uint32_t)__popc(peers));
        const uint32_t r = __shfl_sync(0xffffffffu, old, __ffs(peers) - 1) + (uint32_t)__popc(below);
        at[i / 2] = __byte_perm(at[i / 2], r, i & 1 ? 0x5410 : 0x3254);
    }
    __syncthreads();
    // the tile's count of each digit, L lanes a digit; where the digit starts
    // in the tile; each warp's first place in it
    {
        const int dg = threadIdx.x / L, part = threadIdx.x % L;
        uint32_t *col = &sm.warp_hist[part * (W / L)][dg];
        uint32_t c[W / L], sum = 0;
#pragma unroll
        for (int j = 0; j < W / L; ++j) {
            c[j] = col[j * 257];
            sum += c[j];
        }
        uint32_t before = 0, total = sum;
        if constexpr (L == 2) {
            const uint32_t other = __shfl_xor_sync(0xffffffffu, sum, 1);
            before = part ? other : 0u;
            total = sum + other;
        }
        uint32_t y = total;
#pragma unroll
        for (int off = L; off < 32; off <<= 1) {
            const uint32_t z = __shfl_up_sync(0xffffffffu, y, off);
            if (lane >= off) y += z;
        }
        if (lane == 31) sm.carry[warp] = y;
        __syncthreads();
        const uint32_t start =
            y - total + __reduce_add_sync(0xffffffffu, lane < warp ? sm.carry[lane] : 0u);
        uint32_t run = start + before;
#pragma unroll
        for (int j = 0; j < W / L; ++j) {
            col[j * 257] = run;
            run += c[j];
        }
        if (part == 0) {
            sm.loc[dg] = start;
            sm.cnt[dg] = total;
        }
    }
    __syncthreads();
    const uint64_t epoch = (uint64_t)((info->epoch + (uint32_t)pass) & 0x3fffffffu);
    const int d = threadIdx.x;
    uint64_t *slot = lookback + (int64_t)tile * 256 + d;
    uint32_t my = 0;
    if (d < 256) {
        my = sm.cnt[d];
        st_relaxed_u64(slot, (tile == 0 ? kFlagIncl : kFlagAgg) | (epoch << 32) | my);
    }
    // (a shift the compiler takes for another one, so that it forms the digits
    // again instead of keeping them in registers since the ranking)
    int again = shift;
    asm("" : "+r"(again));
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        const uint32_t p = hist[(uint32_t)(key[i] >> again) & 255u] + (at[i / 2] >> (i & 1 ? 16 : 0) & 0xffffu);
        at[i / 2] = __byte_perm(at[i / 2], p, i & 1 ? 0x5410 : 0x3254);
        if (FULL || first + i * 32 < valid) sm.keys[p] = key[i];
    }
    // the values on their way while the predecessors finish
    int32_t val[ITEMS];
    if (!FIRST) {
        const int32_t *src = vals_in + tile_base + first;
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) val[i] = FULL || first + i * 32 < valid ? src[i * 32] : 0;
    }
    if (d < 256) {
        uint32_t excl = 0;
        if (tile > 0) {
            excl = look_back<256>(lookback, tile, d, epoch, spin_limit, info);
            st_relaxed_u64(slot, kFlagIncl | (epoch << 32) | (excl + my));
        }
        sm.base[d] = digit_off[d] + excl - sm.loc[d];
    }
    __syncthreads();
    uint32_t dst[ITEMS];
    bool bad = false;
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        const int j = i * T + (int)threadIdx.x;
        dst[i] = 0xffffffffu;
        if (FULL || j < valid) {
            const uint64_t k = sm.keys[j];
            dst[i] = sm.base[(uint32_t)(k >> shift) & 255u] + (uint32_t)j;
            if (dst[i] < n) keys_out[dst[i]] = k;
            else bad = true;
        }
    }
    if (bad) flag_error(&info->status, kErrTimeout);
    __syncthreads();
#pragma unroll
    for (int i = 0; i < ITEMS; ++i)
        if (FULL || first + i * 32 < valid)
            sm.vals[at[i / 2] >> (i & 1 ? 16 : 0) & 0xffffu] = FIRST ? (int32_t)(tile_base + (uint32_t)(first + i * 32)) : val[i];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < ITEMS; ++i)
        if (dst[i] < n) vals_out[dst[i]] = sm.vals[i * T + (int)threadIdx.x];
}

template <int T, int ITEMS, bool FIRST>
__global__ void __launch_bounds__(T, T == 256 && ITEMS > 18 ? 3 : 1024 / T)
    onesweep8_kernel(const uint64_t *__restrict__ keys_in, const int32_t *__restrict__ vals_in,
                         uint64_t *__restrict__ keys_out, int32_t *__restrict__ vals_out, int64_t n,
                         int pass, int shift0, const uint32_t *__restrict__ digit_off,
                         uint64_t *lookback, DevInfo *info, int64_t spin_limit) {
    after_previous();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    using S = Sort8Smem<T, ITEMS>;
    S &sm = *reinterpret_cast<S *>(smem_raw);
    if (threadIdx.x == 0) sm.tile = atomicAdd(&info->sort_tile_ctr[pass], 1u);
    for (int i = threadIdx.x; i < S::WARPS * 257; i += T) (&sm.warp_hist[0][0])[i] = 0;
    __syncthreads();
    const uint32_t tile = sm.tile;
    const int valid = (int)min64(S::TILE, n - (int64_t)tile * S::TILE);
    if (valid == S::TILE)
        tile8<T, ITEMS, FIRST, true>(sm, keys_in, vals_in, keys_out, vals_out, (uint32_t)n, tile, valid, pass,
                                      shift0 + pass * 8, digit_off, lookback, info, spin_limit);
    else
        tile8<T, ITEMS, FIRST, false>(sm, keys_in, vals_in, keys_out, vals_out, (uint32_t)n, tile, valid, pass,
                                       shift0 + pass * 8, digit_off, lookback, info, spin_limit);
}

template <int B, int T, int I, bool FIRST>
constexpr auto pass_kernel() {
    if constexpr (B == 8) return &onesweep8_kernel<T, I, FIRST>;
    else return &onesweep_kernel<B, T, I, FIRST>;
}

template <int B, int T, int I>
cudaError_t run_passes(uint64_t *ka, uint64_t *kb, int32_t *pa, int32_t *pb, int64_t n,
                       Workspace &ws, const SortPlan &plan, uint64_t *&kout, int32_t *&pout,
                       cudaStream_t s) {
    auto first = pass_kernel<B, T, I, true>(), next = pass_kernel<B, T, I, false>();
    const size_t smem = B == 8 ? sizeof(Sort8Smem<T, I>) : sizeof(SortSmem<B, T, I>);
    static std::atomic<uint64_t> attr_done{0};
    cudaError_t e = once_on_device(attr_done, [&] {
        const cudaError_t a = allow_smem(first, smem, true);
        return a == cudaSuccess ? allow_smem(next, smem, true) : a;
    });
    if (e != cudaSuccess) return e;
    const int64_t tiles = (n + T * I - 1) / (T * I);
    // the unsorted keys are in `ka`; passes alternate ka -> kb -> ka ...
    uint64_t *src = ka, *dst = kb;
    int32_t *vsrc = pa, *vdst = pb;
    const int64_t spin = g_wait_limit;
    for (int p = 0; p < plan.passes; ++p) {
        launch_after(p == 0 ? first : next, dim3((unsigned)tiles), dim3(T), smem, s, 
            src, p == 0 ? nullptr : vsrc, dst, vdst, n, p, plan.shift0, ws.hist + p * (1 << B), ws.lookback,
            ws.info, spin);
        ++g_launches;
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        mark(ws, "sort_pass", s);
        uint64_t *t = src; src = dst; dst = t;
        int32_t *u = vsrc; vsrc = vdst; vdst = u;
    }
    kout = src;
    pout = vsrc;
    // finish the runs of equal upper bits; the other buffers are free scratch
    e = launch_runs(src, vsrc, dst, vdst, n, plan.shift0, ws.long_runs, ws, s);
    if (e != cudaSuccess) return e;
    if (plan.shift0 > 0) mark(ws, "sort_runs", s);
    return cudaSuccess;
}

}  // namespace

// Polls after which a look-back wait gives up (about 17 s with the back-off);
// tb_set_wait_limit lowers it to exercise the timeout path.
int64_t g_wait_limit = kDefaultWaitLimit;

// Compiled variants: digit bits, threads per tile, keys per thread.
static const SortCfg kVariants[] = {
    {8, 256, 16}, {8, 512, 16}, {8, 512, 12}, {8, 512, 8}, {8, 256, 8}, {8, 512, 14}, {8, 256, 21},
    {9, 256, 16}, {9, 512, 16}, {9, 512, 8}, {10, 256, 16}, {10, 512, 8}, {11, 256, 16},
};
static const int kNumVariants = sizeof(kVariants) / sizeof(kVariants[0]);

const SortCfg *sort_variant(int i) { return (i >= 0 && i < kNumVariants) ? &kVariants[i] : nullptr; }

// 8-bit digits, a pass at each size (us):
//   keys        80,000  400,000  10^6   2^22   8 10^6  12 10^6  2^24   2^27
//   256 x 8       10.3    14.4   22.8   53.9    91.8    130
//   512 x 8       12.3    13.6   18.9   46.0    82.1    117      160   1190
//   512 x 14      14.5    16.3   17.3   43.5    77.6    108      143   1025
//   256 x 21      15.7    15.4   20.4   49.4    81.6    109      142    937
// Few keys want small tiles, over more SMs; many keys want few look-backs and
// three blocks per SM.  Other digits: their first variant.
SortCfg default_sort_cfg(int radix_bits, int64_t n) {
    if (radix_bits == 8)
        return n <= kSmallTileMax ? SortCfg{8, 256, 8} : (n <= kMidTileMax ? SortCfg{8, 512, 14} : SortCfg{8, 256, 21});
    return first_sort_cfg(radix_bits);
}

// The first variant of a digit width: completes a named block or tile size.
SortCfg first_sort_cfg(int radix_bits) {
    for (int i = 0; i < kNumVariants; ++i)
        if (kVariants[i].radix_bits == radix_bits) return kVariants[i];
    return kVariants[0];
}

bool sort_cfg_valid(const SortCfg &c) {
    for (int i = 0; i < kNumVariants; ++i)
        if (kVariants[i].radix_bits == c.radix_bits && kVariants[i].threads == c.threads &&
            kVariants[i].items == c.items)
            return true;
    return false;
}

int64_t sort_tiles(const SortCfg &c, int64_t n) { return (n + c.tile() - 1) / c.tile(); }

cudaError_t load_sort_kernels() {
    // the default tile of every set tb_keys_sorted_noalloc takes
    cudaError_t e = load_kernel(onesweep8_kernel<256, 8, true>);
    return e == cudaSuccess ? load_kernel(onesweep8_kernel<256, 8, false>) : e;
}

SortPlan sort_plan(const SortCfg &c) {
    // global passes cover the upper ceil(40 / b) * b key bits; the runs of
    // equal upper bits are finished locally
    const int b = c.radix_bits;
    const int passes = (40 + b - 1) / b;
    return {passes, 63 - passes * b};
}

cudaError_t launch_sort(uint64_t *ka, uint64_t *kb, int32_t *pa, int32_t *pb, int64_t n,
                        Workspace &ws, const SortCfg &cfg, uint64_t *&kout, int32_t *&pout,
                        cudaStream_t s) {
    const SortPlan plan = sort_plan(cfg);
#define TB_SORT_CASE(B, T, I)                                             \
    if (cfg.radix_bits == B && cfg.threads == T && cfg.items == I)        \
        return run_passes<B, T, I>(ka, kb, pa, pb, n, ws, plan, kout, pout, s);
    TB_SORT_CASE(8, 256, 16)
    TB_SORT_CASE(8, 512, 16)
    TB_SORT_CASE(8, 512, 12)
    TB_SORT_CASE(8, 512, 8)
    TB_SORT_CASE(8, 256, 8)
    TB_SORT_CASE(8, 512, 14)
    TB_SORT_CASE(8, 256, 21)
    TB_SORT_CASE(9, 256, 16)
    TB_SORT_CASE(9, 512, 16)
    TB_SORT_CASE(9, 512, 8)
    TB_SORT_CASE(10, 256, 16)
    TB_SORT_CASE(10, 512, 8)
    TB_SORT_CASE(11, 256, 16)
#undef TB_SORT_CASE
    return cudaErrorInvalidValue;
}

}  // namespace tb
