// tb_cells.cu -- leaves and the remaining cells from the sorted keys
// (Sec. 2.3.1 Alg. 1, Sec. 2.3.2 Alg. 2, App. A), data-parallel.
//
// For sorted keys K and n = n_crit:
//   m_k = minDepth(k-1, k)  (m_0 = 0)                  -- where k leaves its predecessor's cells
//   c_i = min(21, minDepth(i, i+n)) for i+n < N, else 0 -- window [i, i+n] lies in a cell of
//                                                          depth < c_i, which then holds > n
//   L_k = max{ c_i : k-n <= i <= k }                    -- depth of the leaf holding k
// A depth-D cell holding k has more than n particles iff some window
// [i, i+n] containing k lies inside it, so L_k is the first depth at which
// k's cell holds n or fewer (or 21), which at a leaf start equals the
// D_k = max(minDepth(k-1,k), minDepth(k,k+n)) of App. A.  Particle k starts a
// cell at every depth d with m_k <= d <= L_k, and k starts a leaf iff
// m_k <= L_k.  Every cell is therefore (d, K_k >> (63 - 3d), first particle
// k) for exactly one k, which replaces the serial scans of Alg. 1 and the
// per-depth merges of Alg. 2 by one pass over the particles.
//
// Canonical order is level-major, key (= first particle) ascending within a
// level, so the index of cell (d, k) is level_offset[d] + P_d(k), P_d(k) the
// number of level-d starts before k: a 22-way prefix count, done in three
// launches over tiles of 1024 particles:
//   level_count_kernel : per tile, the cells started at each level and the
//                        leaves started (one warp ballot per level);
//   level_scan_kernel  : per level, prefix over tiles; the last block forms the
//                        level offsets, the cell count and the depth;
//   emit_starts_kernel : reads m and L back, lists the leaf starts, and writes
//                        every cell.
// Links follow from the same counts (P_d(k) before k's own starts):
//   index of (d, k)        = P_d(k);
//   parent of (d, k)       = (d-1, k) = P_{d-1}(k) if d > m_k, else the level-(d-1)
//                            cell holding k, started earlier: P_{d-1}(k) - 1;
//   child_first of (d, k)  = (d+1, k) = P_{d+1}(k) when d < L_k;
//   pend, child_end        = written by the leaf start k' that closes the cell:
//                            k' closes levels m_k' .. L_{k'-1} (the cells holding
//                            k'-1 but not k'), cell P_d(k') - 1, child_end
//                            P_{d+1}(k'); the last particle closes all.
// No cell is written twice and no pass over the cells is needed afterwards.
// L_k, a maximum over a window of n + 1 values of c, comes from a doubling
// table: M_1 = c, M_2q[i] = max(M_q[i], M_q[i+q]); with p the largest power of
// two <= n + 1, L_k = max(M_p[k-n], M_p[k-p+1]).
#include "tb_cells.cuh"

namespace tb {

namespace {

__global__ void __launch_bounds__(kLvThreads, 2)
    level_count_kernel(const uint64_t *__restrict__ skeys, int64_t n, int ncrit,
                       uint32_t *__restrict__ tile_cnt, int64_t n_tiles, uint16_t *__restrict__ ml) {
    after_previous();
    extern __shared__ __align__(16) unsigned char raw[];
    __shared__ TileShared ts;
    __shared__ uint32_t tot[kLevelFields];
    const int64_t t = blockIdx.x;
    const int64_t s = t * kLvTile, e = min64(n, s + kLvTile);
    const Front f = tile_front(skeys, 0, n, ncrit, s, e, raw, ts);
    // keep m and L of every particle for the emission
    if (f.k < e) ml[f.k] = (uint16_t)(f.m | (f.L << 8));
    field_totals(ts, tot);
    __syncthreads();
    if (threadIdx.x < kLevelFields) tile_cnt[(int64_t)threadIdx.x * n_tiles + t] = tot[threadIdx.x];
}

// One thread: the level offsets, counts and depth from the field totals; the
// record's counters cleared for what follows.
__device__ __forceinline__ void finish_levels(DevInfo *info, const uint32_t *tot, int64_t cell_cap) {
    int64_t off = 0;
    int dmax = 0;
    for (int d = 0; d < kLevels; ++d) {
        uint32_t c = tot[d];
        info->level_offset[d] = off;
        off += c;
        if (c) dmax = d;
    }
    info->level_offset[kLevels] = off;
    info->n_cells = off;
    info->n_leaves = tot[kLevels];
    info->max_depth = dmax;
    if (cell_cap > 0 && off > cell_cap) info->status |= kErrOverflow;
    info->misc_ctr[1] = 0;
    info->misc_ctr[2] = info->misc_ctr[5] = 0;   // the moments' leaf queues
}

// The same counts, four consecutive particles per thread, for n_crit in
// [kLcMinN, kLcMaxN] (count_tile4); a block of 256 threads takes one count tile.
// With at most kLcScanTiles tiles the last block to finish also forms the
// prefixes over the tiles, a warp per field, and saves the scan's launch (5 of
// 65 us at 3,001 particles).
constexpr int kLcThreads = kLvTile / 4;
constexpr int kLcScanTiles = 256;

__device__ __forceinline__ void scan_few_tiles(uint32_t *tile_cnt, int n_tiles, DevInfo *info,
                                               int64_t cell_cap) {
    constexpr int PER = kLcScanTiles / 32;
    __shared__ uint32_t s_tot[kLevelFields];
    const int lane = threadIdx.x & 31;
    for (int f = threadIdx.x >> 5; f < kLevelFields; f += kLcThreads / 32) {
        uint32_t *row = tile_cnt + (int64_t)f * n_tiles;
        uint32_t v[PER], sum = 0;
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            const int t = lane * PER + j;
            v[j] = t < n_tiles ? __ldcg(row + t) : 0u;
            sum += v[j];
        }
        uint32_t x = sum;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, off);
            if (lane >= off) x += y;
        }
        if (lane == 31) s_tot[f] = x;
        x -= sum;
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            const int t = lane * PER + j;
            if (t < n_tiles) row[t] = x;
            x += v[j];
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) finish_levels(info, s_tot, cell_cap);
}

__global__ void __launch_bounds__(kLcThreads, 6)
    level_count_fast_kernel(const uint64_t *__restrict__ skeys, int64_t n, int ncrit,
                            uint32_t *tile_cnt, int64_t n_tiles, uint16_t *__restrict__ ml, DevInfo *info,
                            int64_t cell_cap) {
    after_previous();
    extern __shared__ __align__(16) unsigned char raw[];
    __shared__ StartCounts sc;
    __shared__ bool s_last;
    for (int x = threadIdx.x; x <= kLevels; x += kLcThreads) sc.m[x] = sc.l[x] = 0;
    const int64_t t = blockIdx.x, s = t * kLvTile;
    count_tile4<kLcThreads>(skeys, 0, n, ncrit, s, min64(n, s + kLvTile), raw, sc, ml);
    __syncthreads();
    if (threadIdx.x < kLevelFields) tile_cnt[(int64_t)threadIdx.x * n_tiles + t] = sc.cells(threadIdx.x);
    if (n_tiles > kLcScanTiles) return;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(&info->misc_ctr[1], 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    scan_few_tiles(tile_cnt, (int)n_tiles, info, cell_cap);
}

// One block per field: exclusive prefix over tiles (in place); the last block
// to finish turns the field totals into level offsets.  The row is taken in
// chunks staged in shared memory (coalesced loads and stores), each thread
// scanning a contiguous stretch of a chunk.
constexpr int kScanThreads = 1024;
constexpr int kScanPer = 8;
constexpr int kScanChunk = kScanThreads * kScanPer;
static_assert(kScanPer == 8, "the scan moves each thread's eight counts as two uint4");

__global__ void __launch_bounds__(kScanThreads)
    level_scan_kernel(uint32_t *tile_cnt, int64_t n_tiles, DevInfo *info, int64_t cell_cap) {
    after_previous();
    const int f = blockIdx.x;
    uint32_t *row = tile_cnt + (int64_t)f * n_tiles;
    __shared__ __align__(16) uint32_t s_v[kScanChunk];
    __shared__ uint32_t s_w[kScanThreads / 32];
    __shared__ uint64_t s_carry;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) s_carry = 0;
    for (int64_t c0 = 0; c0 < n_tiles; c0 += kScanChunk) {
        const int len = (int)min64(kScanChunk, n_tiles - c0);
        for (int i = threadIdx.x; i < kScanChunk; i += kScanThreads) s_v[i] = i < len ? row[c0 + i] : 0u;
        __syncthreads();
        uint32_t v[kScanPer], sum = 0;
        {
            const uint4 *s4 = reinterpret_cast<const uint4 *>(s_v) + 2 * threadIdx.x;
            const uint4 a = s4[0], b = s4[1];
            v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
            v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
        }
#pragma unroll
        for (int j = 0; j < kScanPer; ++j) sum += v[j];
        uint32_t x = sum;
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, off);
            if (lane >= off) x += y;
        }
        if (lane == 31) s_w[warp] = x;
        __syncthreads();
        if (warp == 0) {
            const uint32_t w = s_w[lane];
            uint32_t z = w;
            for (int off = 1; off < 32; off <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, z, off);
                if (lane >= off) z += y;
            }
            s_w[lane] = z - w;
        }
        __syncthreads();
        // the per-field counts fit 32 bits (at most 2^31 particles)
        uint32_t run = (uint32_t)s_carry + s_w[warp] + x - sum;
        uint32_t o[kScanPer];
#pragma unroll
        for (int j = 0; j < kScanPer; ++j) { o[j] = run; run += v[j]; }
        {
            uint4 *s4 = reinterpret_cast<uint4 *>(s_v) + 2 * threadIdx.x;
            s4[0] = make_uint4(o[0], o[1], o[2], o[3]);
            s4[1] = make_uint4(o[4], o[5], o[6], o[7]);
        }
        __syncthreads();
        for (int i = threadIdx.x; i < len; i += kScanThreads) row[c0 + i] = s_v[i];
        if (threadIdx.x == kScanThreads - 1) s_carry = run;
        __syncthreads();
    }
    const uint64_t s_total = s_carry;
    __shared__ bool s_last;
    if (threadIdx.x == 0) {
        // totals land in a small array right after the per-tile rows
        tile_cnt[(int64_t)kLevelFields * n_tiles + f] = (uint32_t)s_total;
        __threadfence();
        s_last = (atomicAdd(&info->misc_ctr[1], 1u) == gridDim.x - 1);
    }
    __syncthreads();
    if (!s_last || threadIdx.x != 0) return;
    __threadfence();
    const uint32_t *tot = tile_cnt + (int64_t)kLevelFields * n_tiles;
    finish_levels(info, tot, cell_cap);
}

// Emission: one count tile per block (emit_tile in tb_cells.cuh).
constexpr int kEfThreads = 256;
static_assert(4 * kEfThreads == kLvTile, "a count tile per block, four particles per lane");

__global__ void __launch_bounds__(kEfThreads, 6)
    emit_starts_kernel(const uint64_t *__restrict__ skeys, const uint16_t *__restrict__ ml, int64_t n,
                       const uint32_t *__restrict__ tile_off, int64_t n_tiles, DevInfo *info_w,
                       EmitOut out) {
    after_previous();
    const DevInfo *info = info_w;
    if (info->status & (kErrOverflow | kErrNonFinite)) return;
    __shared__ EmitShared<kEfThreads> sm;
    const int lane = threadIdx.x & 31;
    // where the block's cells of level `lane` (its leaves) start
    uint32_t base = 0;
    if (lane < kLevelFields)
        base = (lane < kLevels ? (uint32_t)info->level_offset[lane] : 0u) +
               tile_off[(int64_t)lane * n_tiles + blockIdx.x];
    emit_tile<kEfThreads, false>(skeys, ml, 0, n, (int64_t)blockIdx.x * kLvTile, base,
                                 [&](int d) { return info->level_offset[d + 1]; }, out, sm, 0);
}

}  // namespace

int level_tile_size() { return kLvTile; }

cudaError_t launch_levels(const uint64_t *skeys, int64_t n, int ncrit, Workspace &ws,
                          cudaStream_t s) {
    const int64_t tiles = (n + kLvTile - 1) / kLvTile;
    const size_t smem = lv_smem_bytes(ncrit);
    static std::atomic<uint64_t> attr_done{0};
    cudaError_t err = once_on_device(attr_done, [] {
        const cudaError_t e = allow_smem(level_count_kernel, lv_smem_bytes(kMaxNcrit), true);
        return e == cudaSuccess ? allow_smem(level_count_fast_kernel, lc_smem_bytes<kLcThreads>(kLcMaxN), true) : e;
    });
    if (err != cudaSuccess) return err;
    if (ncrit >= kLcMinN && ncrit <= kLcMaxN) {
        launch_after(level_count_fast_kernel, dim3((unsigned)tiles), dim3(kLcThreads), lc_smem_bytes<kLcThreads>(ncrit), s, 
            skeys, n, ncrit, ws.level_cnt, tiles, ws.ml, ws.info, ws.cell_cap_request);
        if (tiles <= kLcScanTiles) {
            ++g_launches;
            return cudaGetLastError();
        }
    } else {
        launch_after(level_count_kernel, dim3((unsigned)tiles), dim3(kLvThreads), smem, s, skeys, n, ncrit, ws.level_cnt,
                                                                     tiles, ws.ml);
    }
    ++g_launches;
    err = cudaGetLastError();
    if (err != cudaSuccess) return err;
    launch_after(level_scan_kernel, dim3(kLevelFields), dim3(kScanThreads), 0, s, ws.level_cnt, tiles, ws.info,
                                                            ws.cell_cap_request);
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_emit(const uint64_t *skeys, int64_t n, int ncrit, Workspace &ws, tb_tree &t,
                        cudaStream_t s) {
    (void)ncrit;
    const int64_t tiles = (n + kLvTile - 1) / kLvTile;
    EmitOut o{t.ckey, t.level, t.parent, t.child_first, t.child_end, t.pfirst, t.pend,
              t.leaf_cell, nullptr};
    const int64_t blocks = (n + kLvTile - 1) / kLvTile;
    launch_after(emit_starts_kernel, dim3((unsigned)blocks), dim3(kEfThreads), 0, s, skeys, ws.ml, n, ws.level_cnt, tiles,
                                                               ws.info, o);
    ++g_launches;
    return cudaGetLastError();
}

}  // namespace tb
