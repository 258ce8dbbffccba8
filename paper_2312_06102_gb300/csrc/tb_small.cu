// tb_small.cu -- root cube, keys and sorted (key, index) pairs of a small set
// in one launch (Sec. 2.2; Sec. 2.3 steps 1 and 2).
//
// The launches of the general path (root, keys, five radix passes, two run
// steps) cost a small set 4 to 8 us each, nearly all of it latency.  tb_build
// with those and with this launch, us: 59 and 37 at 3,001 particles, 64 and 51 at
// 20,000, 63 and 57 at 32,768 (with five passes here too; the four taken now save
// another 2); from 50,000 on (64 and 70, with 4096 positions a block) the many SMs
// of the general passes win.  Here one cluster of up to 16
// blocks takes the whole set.  Block r owns positions [r P, (r + 1) P) of the
// current order, in registers while a pass ranks them:
//   1. particles to registers (records written out), bounding box by shuffles
//      and, across the blocks, distributed shared memory; every block forms
//      the same root cube; keys;
//   2. four stable 8-bit passes over the upper 32 key bits, as in the general
//      sort: ballot ranking within warps, digit counts of the block; a cluster
//      barrier; every block reads all blocks' counts and so knows where each
//      of its digits goes; the block orders its pairs by digit in shared
//      memory and stores them, runs of consecutive addresses, to the places'
//      owners' shared memory (the last pass: to global memory); a cluster
//      barrier.  A pass reads its pairs into registers before its first
//      barrier and stores after it, so the owners need one buffer;
//   3. runs of equal upper bits ordered in place by the low bits
//      (tb_runs.cuh), tiles shared out over the blocks.  A set with runs too
//      long for that and out of order (tight clumps) takes eight passes over
//      the whole key instead, over the order reached.
// Barriers are the cluster's own (barrier.cluster); nothing spins.
#include <cfloat>

#include "tb_runs.cuh"

namespace tb {

namespace {

constexpr int kSmThreads = 1024;
constexpr int kSmWarps = kSmThreads / 32;
constexpr int kSmBits = 8;
constexpr int kSmRadix = 1 << kSmBits;
constexpr int kSmPasses = 4;
constexpr int kSmShift0 = 63 - kSmPasses * kSmBits;
constexpr int kSmAllPasses = 8;   // of the whole key
constexpr int kSmMaxItems = 2;

template <int ITEMS>
struct SmallSmem {
    static constexpr int P = kSmThreads * ITEMS;   // positions per block
    uint64_t key[P];                               // this block's part of the current order
    uint64_t skey[P];                              // its pairs ordered by the pass's digit
    int32_t val[P];
    int32_t sval[P];
    uint32_t hist[kSmWarps][kSmRadix + 1];
    uint32_t cnt[2][kSmRadix];                     // this block's digit counts, by pass parity
    uint32_t base[kSmRadix];                       // where the digit goes, less loc
    uint32_t loc[kSmRadix];                        // where the digit starts in skey
    uint32_t carry[kSmWarps];
    float red[kSmWarps][8];
    float box[8];
};

__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// Address of this block's shared variable p in block `rank` of the cluster.
__device__ __forceinline__ uint32_t remote(const void *p, uint32_t rank) {
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
    return a;
}

__device__ __forceinline__ uint32_t ld_remote(uint32_t a) {
    uint32_t v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}

__device__ __forceinline__ void st_remote(uint32_t a, uint64_t v) {
    asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(a), "l"(v) : "memory");
}

__device__ __forceinline__ void st_remote(uint32_t a, int32_t v) {
    asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}

// The warp's bounding box from its lanes' (mn, mx, bad), in every lane.
__device__ __forceinline__ void warp_box(float mn[3], float mx[3], uint32_t &bad) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        for (int a = 0; a < 3; ++a) {
            mn[a] = fminf(mn[a], __shfl_xor_sync(0xffffffffu, mn[a], off));
            mx[a] = fmaxf(mx[a], __shfl_xor_sync(0xffffffffu, mx[a], off));
        }
        bad |= __shfl_xor_sync(0xffffffffu, bad, off);
    }
}

template <int ITEMS, bool HILBERT>
__global__ void __launch_bounds__(kSmThreads, 1)
    small_sort_kernel(const float *__restrict__ pos, const float *__restrict__ mass, float m_eq, int n,
                      uint64_t *pkey, int32_t *perm, float4 *__restrict__ xm, DevInfo *info,
                      bool pow2) {
    after_previous();
    using S = SmallSmem<ITEMS>;
    constexpr int P = S::P;
    extern __shared__ __align__(16) unsigned char sm_raw[];
    S &sm = *reinterpret_cast<S *>(sm_raw);
    __shared__ RootCube s_cube;
    __shared__ uint32_t s_long, s_desc, s_again;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t rank = cluster_rank(), blocks = gridDim.x;   // one cluster
    const int first = (int)rank * P;
    const int mine = max(0, min(P, n - first));
    const int wbase = warp * 32 * ITEMS;

    // 1. particles, bounding box, keys
    float x[ITEMS][3];
    {
        float mn[3] = {FLT_MAX, FLT_MAX, FLT_MAX}, mx[3] = {-FLT_MAX, -FLT_MAX, -FLT_MAX};
        uint32_t bad = 0;
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            const int e = wbase + i * 32 + lane;
            if (e < mine) {
                const int g = first + e;
                for (int a = 0; a < 3; ++a) x[i][a] = pos[3 * g + a];
                xm[g] = make_float4(x[i][0], x[i][1], x[i][2], mass ? mass[g] : m_eq);
                for (int a = 0; a < 3; ++a) {
                    bad |= !(fabsf(x[i][a]) <= FLT_MAX);
                    mn[a] = fminf(mn[a], x[i][a]);
                    mx[a] = fmaxf(mx[a], x[i][a]);
                }
            } else {
                for (int a = 0; a < 3; ++a) x[i][a] = 0.f;
            }
        }
        warp_box(mn, mx, bad);
        if (lane == 0) {
            for (int a = 0; a < 3; ++a) { sm.red[warp][a] = mn[a]; sm.red[warp][3 + a] = mx[a]; }
            sm.red[warp][6] = __uint_as_float(bad);
        }
        __syncthreads();
        if (warp == 0) {
            for (int a = 0; a < 3; ++a) { mn[a] = sm.red[lane][a]; mx[a] = sm.red[lane][3 + a]; }
            bad = __float_as_uint(sm.red[lane][6]);
            warp_box(mn, mx, bad);
            if (lane == 0) {
                for (int a = 0; a < 3; ++a) { sm.box[a] = mn[a]; sm.box[3 + a] = mx[a]; }
                sm.box[6] = __uint_as_float(bad);
            }
        }
        cluster_sync();
        if (warp == 0) {
            const uint32_t a0 = remote(sm.box, lane < blocks ? lane : rank);
            for (int a = 0; a < 3; ++a) {
                mn[a] = __uint_as_float(ld_remote(a0 + 4 * a));
                mx[a] = __uint_as_float(ld_remote(a0 + 12 + 4 * a));
            }
            bad = ld_remote(a0 + 24);
            warp_box(mn, mx, bad);
            if (lane == 0) {
                s_cube = root_cube(mn, mx, pow2);
                s_long = s_desc = 0;
                if (rank == 0) begin_build(info, s_cube, mx, bad != 0u);
            }
        }
        __syncthreads();
    }
    uint64_t key[ITEMS];
    int32_t val[ITEMS];
    {
        const RootCube &r = s_cube;
        const float lx = r.lo[0], ly = r.lo[1], lz = r.lo[2], shi = r.s_hi, slo = r.s_lo;
        const double sc = r.scale;
        const bool ex = r.exact_only, f32 = r.s_fp32;
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            const uint32_t qx = quantise(x[i][0], lx, shi, slo, sc, ex, f32),
                           qy = quantise(x[i][1], ly, shi, slo, sc, ex, f32),
                           qz = quantise(x[i][2], lz, shi, slo, sc, ex, f32);
            key[i] = HILBERT ? hilbert_key(qx, qy, qz) : morton_key(qx, qy, qz);
            val[i] = first + wbase + i * 32 + lane;
        }
    }

    // 2. passes
    const unsigned lt = lanemask_lt();
    const int tiles = (n + kRunTile - 1) / kRunTile;
    for (int passes = kSmPasses, shift0 = kSmShift0;; passes = kSmAllPasses, shift0 = 0) {
        for (int p = 0; p < passes; ++p) {
            const int shift = shift0 + p * kSmBits;
            if (p > 0) {
#pragma unroll
                for (int i = 0; i < ITEMS; ++i) {
                    const int e = wbase + i * 32 + lane;
                    key[i] = sm.key[e];
                    val[i] = sm.val[e];
                }
            }
            for (int i = threadIdx.x; i < kSmWarps * (kSmRadix + 1); i += kSmThreads) (&sm.hist[0][0])[i] = 0;
            __syncthreads();
            // stable ranks within the warp; positions past the set take no part
            uint32_t at[ITEMS];
#pragma unroll
            for (int i = 0; i < ITEMS; ++i) {
                const bool in = wbase + i * 32 + lane < mine;
                const uint32_t d = (uint32_t)(key[i] >> shift) & (kSmRadix - 1);
                unsigned peers = __ballot_sync(0xffffffffu, in);
                if (!in) peers = 0;
#pragma unroll
                for (int b = 0; b < kSmBits; ++b) {
                    const bool bit = (d >> b) & 1u;
                    const unsigned v = __ballot_sync(0xffffffffu, bit);
                    peers &= bit ? v : ~v;
                }
                const int leader = __ffs(peers) - 1;
                uint32_t old = 0;
                if (in && lane == leader) old = atomicAdd(&sm.hist[warp][d], (uint32_t)__popc(peers));
                at[i] = __shfl_sync(0xffffffffu, old, leader & 31) + (uint32_t)__popc(peers & lt);
            }
            __syncthreads();
            // each warp's offset within its digit, the block's count of the digit:
            // four lanes a digit, eight warps each
            const int dg = threadIdx.x >> 2, part = threadIdx.x & 3;
            {
                uint32_t c[kSmWarps / 4], sum = 0;
#pragma unroll
                for (int j = 0; j < kSmWarps / 4; ++j) {
                    c[j] = sm.hist[part * (kSmWarps / 4) + j][dg];
                    sum += c[j];
                }
                uint32_t y = sum;
#pragma unroll
                for (int off = 1; off < 4; off <<= 1) {
                    const uint32_t z = __shfl_up_sync(0xffffffffu, y, off, 4);
                    if (part >= off) y += z;
                }
                uint32_t run = y - sum;
#pragma unroll
                for (int j = 0; j < kSmWarps / 4; ++j) {
                    sm.hist[part * (kSmWarps / 4) + j][dg] = run;
                    run += c[j];
                }
                if (part == 3) sm.cnt[p & 1][dg] = y;
            }
            cluster_sync();
            // every block's count of the digit: those before this one's, and all
            {
                uint32_t tot = 0, pre = 0;
                for (uint32_t q = part; q < blocks; q += 4) {
                    const uint32_t v = ld_remote(remote(&sm.cnt[p & 1][dg], q));
                    tot += v;
                    if (q < rank) pre += v;
                }
#pragma unroll
                for (int off = 1; off < 4; off <<= 1) {
                    tot += __shfl_xor_sync(0xffffffffu, tot, off);
                    pre += __shfl_xor_sync(0xffffffffu, pre, off);
                }
                // prefixes over the digits of all blocks' counts (at most 2^15, low
                // 18 bits) and of this block's (at most 2^11, high 14 bits) at once
                const uint32_t own = sm.cnt[p & 1][dg], both = tot | (own << 18);
                uint32_t y = both;   // inclusive over the warp's eight digits
#pragma unroll
                for (int off = 4; off < 32; off <<= 1) {
                    const uint32_t z = __shfl_up_sync(0xffffffffu, y, off);
                    if (lane >= off) y += z;
                }
                if (lane == 31) sm.carry[warp] = y;
                __syncthreads();
                y += __reduce_add_sync(0xffffffffu, lane < warp ? sm.carry[lane] : 0u) - both;
                if (part == 0) {
                    sm.loc[dg] = y >> 18;
                    sm.base[dg] = (y & 0x3ffffu) + pre - (y >> 18);
                }
            }
            __syncthreads();
#pragma unroll
            for (int i = 0; i < ITEMS; ++i) {
                if (wbase + i * 32 + lane >= mine) continue;
                const uint32_t d = (uint32_t)(key[i] >> shift) & (kSmRadix - 1);
                const uint32_t e = sm.loc[d] + sm.hist[warp][d] + at[i];
                sm.skey[e] = key[i];
                sm.sval[e] = val[i];
            }
            __syncthreads();
#pragma unroll
            for (int i = 0; i < ITEMS; ++i) {
                const int j = i * kSmThreads + (int)threadIdx.x;
                if (j >= mine) continue;
                const uint64_t k = sm.skey[j];
                const uint32_t d = (uint32_t)(k >> shift) & (kSmRadix - 1);
                const uint32_t to = sm.base[d] + (uint32_t)j;
                if (p + 1 < passes) {
                    const uint32_t q = to / P, e = to % P;
                    st_remote(remote(&sm.key[e], q), k);
                    st_remote(remote(&sm.val[e], q), sm.sval[j]);
                } else {
                    pkey[to] = k;
                    perm[to] = sm.sval[j];
                }
            }
            cluster_sync();
        }

        if (passes == kSmAllPasses) return;

        // 3. runs of equal upper bits
        for (int t = rank; t < tiles; t += blocks) {
            const bool desc = run_tile<kSmThreads>(pkey, perm, 0, (int64_t)t * kRunTile, n, kSmShift0,
                                                   *reinterpret_cast<RunSmem *>(sm_raw),
                                                   [&](int64_t) { s_long = 1; });
            if (threadIdx.x == 0 && desc) s_desc = 1;
        }
        cluster_sync();
        // any block with a long run, and any descent: again, over the whole key
        if (warp == 0) {
            const uint32_t q = lane < blocks ? lane : rank;
            const uint32_t l = ld_remote(remote(&s_long, q)), d = ld_remote(remote(&s_desc, q));
            const bool again = __any_sync(0xffffffffu, l != 0) && __any_sync(0xffffffffu, d != 0);
            if (lane == 0) s_again = again ? 1u : 0u;
        }
        cluster_sync();   // no block leaves while another reads its flags
        if (!s_again) return;
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            const int e = wbase + i * 32 + lane;
            if (e < mine) {
                key[i] = __ldcg(reinterpret_cast<const unsigned long long *>(pkey) + first + e);
                val[i] = __ldcg(perm + first + e);
            }
        }
    }
}

template <int ITEMS>
constexpr size_t small_smem() {
    return sizeof(SmallSmem<ITEMS>) > sizeof(RunSmem) ? sizeof(SmallSmem<ITEMS>) : sizeof(RunSmem);
}

template <int ITEMS, bool H>
cudaError_t launch_small_t(const float *pos, const float *mass, int n, uint64_t *pkey, int32_t *perm,
                           Workspace &ws, bool ask, int *clusters, cudaStream_t s) {
    auto kern = small_sort_kernel<ITEMS, H>;
    const int blocks = (n + SmallSmem<ITEMS>::P - 1) / SmallSmem<ITEMS>::P;
    static std::atomic<uint64_t> attr_done{0};
    cudaError_t e = once_on_device(attr_done, [&] {
        const cudaError_t a = allow_smem(kern, small_smem<ITEMS>(), false);
        return a == cudaSuccess ? cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) : a;
    });
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = blocks;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(kSmThreads);
    cfg.dynamicSmemBytes = small_smem<ITEMS>();
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    if (ask) return cudaOccupancyMaxActiveClusters(clusters, kern, &cfg);
    const float m_eq = (float)(1.0 / (double)n);
    e = cudaLaunchKernelEx(&cfg, kern, pos, mass, m_eq, n, pkey, perm, ws.xm, ws.info,
                                       ws.root_pow2);
    if (e == cudaSuccess) ++g_launches;
    return e;
}

cudaError_t dispatch_small(const float *pos, const float *mass, int64_t n, int max_blocks, uint64_t *pkey,
                           int32_t *perm, Workspace &ws, int key_order, bool ask, int *clusters,
                           cudaStream_t s) {
    const bool h = key_order == TB_KEYS_HILBERT;
#define TB_SMALL(I)                                                                                     \
    if (n <= (int64_t)I * kSmThreads * max_blocks)                                                      \
        return h ? launch_small_t<I, true>(pos, mass, (int)n, pkey, perm, ws, ask, clusters, s) \
                 : launch_small_t<I, false>(pos, mass, (int)n, pkey, perm, ws, ask, clusters, s);
    TB_SMALL(1)
    TB_SMALL(2)
#undef TB_SMALL
    return cudaErrorInvalidValue;
}

// Blocks of the largest cluster the current device can hold: 16, else the
// portable 8; looked up once per device.
int small_blocks() {
    static std::atomic<int> known[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 8;
    int v = known[dev].load(std::memory_order_relaxed);
    if (v == 0) {
        Workspace none;
        int clusters = 0;
        const cudaError_t e =
            dispatch_small(nullptr, nullptr, (int64_t)16 * kSmThreads * kSmMaxItems, 16, nullptr, nullptr,
                           none, TB_KEYS_MORTON, true, &clusters, nullptr);
        if (e != cudaSuccess) cudaGetLastError();
        if (e == cudaErrorMemoryAllocation) return 8;   // asked again by the next call
        v = e == cudaSuccess && clusters > 0 ? 16 : 8;
        known[dev].store(v, std::memory_order_relaxed);
    }
    return v;
}

}  // namespace

// Largest set launch_small_sort takes on the current device.
int64_t small_sort_max() { return (int64_t)small_blocks() * kSmThreads * kSmMaxItems; }

cudaError_t load_small_kernels() {
    cudaError_t e = load_kernel(small_sort_kernel<1, false>);
    return e == cudaSuccess ? load_kernel(small_sort_kernel<2, false>) : e;
}

// Root cube (with the build record's start), records, sorted keys and
// permutation of 1 <= n <= small_sort_max() particles.
cudaError_t launch_small_sort(const float *pos, const float *mass, int64_t n, uint64_t *pkey, int32_t *perm,
                              Workspace &ws, int key_order, cudaStream_t s) {
    return dispatch_small(pos, mass, n, small_blocks(), pkey, perm, ws, key_order, false, nullptr, s);
}

}  // namespace tb
