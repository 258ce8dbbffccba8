// tb_batched.cu -- many independent trees in one call (tb_build_batched).
//
// Thousands of particle sets of uneven size each get their own tree (own
// root cube, keys, sort, cells and moments, exactly as tb_build + tb_moments
// would give for the set alone), with a fixed number of launches whatever the
// number of sets:
//   set_order_kernel    : sets ordered largest first (work-queue order);
//   batch_front_kernel  : persistent, one block of 256, 512 or 1024 threads per set
//                         taken from an atomic work queue: root cube, keys, (x, y, z, m)
//                         records and the digit histograms of every pass, then a
//                         stable LSD radix sort of the set inside the block (its
//                         tiles in order, so no look-back is needed), then the
//                         set's cell and leaf counts per level;
//   batch_scan_kernel   : cell and leaf offsets of every set (set order);
//   batch_emit_kernel   : persistent, one block per set: every cell with its
//                         links (the single-tree emission from the m_k and L_k
//                         the count stored, tile after tile with running
//                         counts);
//   leaf_tile_kernel    : every leaf, as in the single tree: tiles of the whole
//                         key order, whatever sets they hold;
//   batch_up_kernel     : persistent, one block per set: the other cells level
//                         by level, deepest first, with a block barrier
//                         between levels.
// The paper builds disjoint subtrees on dynamically scheduled threads
// (Sec. 2.3.3); here the unit of dynamic scheduling is a whole set.
#include <cfloat>

#include "tb_cells.cuh"
#include "tb_ctasort.cuh"
#include "tb_runs.cuh"
#include "tb_moments.cuh"

namespace tb {

namespace {

// front blocks: T threads per set, 1024 / T sets per SM at a time.  T = 512
// unless the sets are few and large, where a set's own time counts (300 sets
// of 4,000 to 65,536 particles: 1.28 ms with 1024 threads, 1.69 with 512; 600 of
// 1,000 to 30,000: 771 and 890 us; 4,096 of 256 to 65,536: 5.85 and 5.16 ms), or many
// and small, where the number of sets at a time does (1,000 sets of 32 to 700: 121
// us with 256 threads, 163 with 512).
constexpr int kBDefaultThreads = 512;
inline bool batch_few_large(int32_t S, int64_t n) { return S <= 608 && n >= int64_t(S) * 4096; }
inline bool batch_many_small(int32_t S, int64_t n) { return S > 304 && n <= int64_t(S) * 512; }
constexpr int kBRadixBits = kCtaRadixBits;
constexpr int kBRadix = kCtaRadix;
// the block sort orders the upper 40 key bits in five passes, or the upper 32
// in four; the runs of equal upper bits are then ordered in place
// (tb_runs.cuh), the long ones by the same block sort of their low bits, one
// after another.  Four passes for sets of up to 2^17 particles, unless many of
// their runs would be long (clumps), which fifth_pass tells.
constexpr int kBMaxPasses = 5;
constexpr int kBTopShift = 63 - 4 * kBRadixBits;   // above this the upper 32 bits
constexpr int64_t kBFourMax = int64_t(1) << 17;
constexpr int kBMomThreads = 256;
constexpr int kBigLeafSerial = 1 << 20;       // leaves above this are summed in FP64


struct BatchArgs {
    const float *pos;
    const float *mass;
    const int64_t *off;       // [S+1]
    const int32_t *order;     // [S]
    int32_t n_sets;
    int32_t ncrit;
    uint64_t *pkey;
    int32_t *perm;
    uint64_t *kalt;
    int32_t *palt;
    float4 *xm;
    float4 *xs;
    uint16_t *ml;             // [n] m_k | L_k << 8 of each sorted particle (count -> emit)
    uint32_t *set_cnt;        // [S][kLevelFields]
    int64_t *set_cell_off;    // [S+1]
    int64_t *set_leaf_off;    // [S+1]
    double *set_root;         // [S][4]
    uint32_t *queue;          // [8] work-queue tickets [0..2], grid barrier [4..5]
    DevInfo *info;
    int32_t root_pow2;        // each set's root side forced to a power of two
};

template <int T>
__host__ __device__ inline size_t batch_front_smem(int ncrit) {
    const bool fast = ncrit >= kLcMinN && ncrit <= kLcMaxN;
    const size_t a = sizeof(CtaSortSharedT<T>), b = fast ? lc_smem_bytes<T>(ncrit) : lv_smem_bytes<T>(ncrit);
    return (a > b ? a : b);
}

// Sets in descending size classes (floor(log2 size)), ascending index within
// a class: the largest sets are taken from the queues first.
// One block of up to 1024 threads (a multiple of 32).
__device__ void set_order_block(const int64_t *off, int32_t S, int32_t *order) {
    __shared__ uint32_t cls[34];
    if (threadIdx.x < 34) cls[threadIdx.x] = 0;
    __syncthreads();
    auto klass = [&](int s) {
        int64_t n = off[s + 1] - off[s];
        return n <= 0 ? 0 : 1 + (63 - __clzll((unsigned long long)n));   // 0 .. 32
    };
    for (int s = threadIdx.x; s < S; s += blockDim.x) atomicAdd(&cls[klass(s)], 1u);
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t run = 0;
        for (int c = 33; c >= 0; --c) { uint32_t v = cls[c]; cls[c] = run; run += v; }
    }
    __syncthreads();
    // stable within a class: chunks of 1024 sets in order; inside a chunk a
    // set's place is its class's running base, plus the sets of its class in
    // earlier warps, plus those in earlier lanes of its warp
    __shared__ uint32_t wc[32][34];
    __shared__ uint32_t tot[34];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const int nw = blockDim.x >> 5;
    for (int c0 = 0; c0 < S; c0 += blockDim.x) {
        for (int i = threadIdx.x; i < 32 * 34; i += blockDim.x) (&wc[0][0])[i] = 0;
        __syncthreads();
        const int s = c0 + (int)threadIdx.x;
        const int c = s < S ? klass(s) : -1;
        const unsigned peers = __match_any_sync(0xffffffffu, c);
        if (c >= 0 && lane == __ffs(peers) - 1) wc[warp][c] = (uint32_t)__popc(peers);
        __syncthreads();
        if (threadIdx.x < 34) {
            uint32_t r = 0;
            for (int w = 0; w < nw; ++w) { const uint32_t v = wc[w][threadIdx.x]; wc[w][threadIdx.x] = r; r += v; }
            tot[threadIdx.x] = r;
        }
        __syncthreads();
        if (c >= 0) order[cls[c] + wc[warp][c] + (uint32_t)__popc(peers & lt)] = s;
        __syncthreads();
        if (threadIdx.x < 34) cls[threadIdx.x] += tot[threadIdx.x];
        __syncthreads();
    }
}

__global__ void __launch_bounds__(1024) set_order_kernel(const int64_t *off, int32_t S,
                                                         int32_t *order, const DevInfo *info) {
    after_previous();
    if (info->status & kErrInvalid) return;
    set_order_block(off, S, order);
}

__device__ __forceinline__ int take_set(uint32_t *ticket, int32_t S, int *s_q) {
    if (threadIdx.x == 0) *s_q = (int)atomicAdd(ticket, 1u);
    __syncthreads();
    const int q = *s_q;
    __syncthreads();
    return q < S ? q : -1;
}

// Block-wide min / max / non-finite reduction of one set's positions.
__device__ void set_root_cube(const float *__restrict__ pos, int64_t o, int64_t ns, float *s_red,
                              uint32_t *s_bad) {
    float mn[3] = {FLT_MAX, FLT_MAX, FLT_MAX}, mx[3] = {-FLT_MAX, -FLT_MAX, -FLT_MAX};
    uint32_t bad = 0;
    for (int64_t i = o + threadIdx.x; i < o + ns; i += blockDim.x)
        for (int a = 0; a < 3; ++a) {
            const float x = pos[3 * i + a];
            bad |= !(fabsf(x) <= FLT_MAX);
            mn[a] = fminf(mn[a], x);
            mx[a] = fmaxf(mx[a], x);
        }
    for (int sh = 16; sh > 0; sh >>= 1) {
        for (int a = 0; a < 3; ++a) {
            mn[a] = fminf(mn[a], __shfl_xor_sync(0xffffffffu, mn[a], sh));
            mx[a] = fmaxf(mx[a], __shfl_xor_sync(0xffffffffu, mx[a], sh));
        }
        bad |= __shfl_xor_sync(0xffffffffu, bad, sh);
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) {
        for (int a = 0; a < 3; ++a) { s_red[warp * 6 + a] = mn[a]; s_red[warp * 6 + 3 + a] = mx[a]; }
        if (bad) atomicOr(s_bad, 1u);
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        float v = s_red[threadIdx.x];
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w)
            v = (threadIdx.x < 3) ? fminf(v, s_red[w * 6 + threadIdx.x])
                                  : fmaxf(v, s_red[w * 6 + threadIdx.x]);
        s_red[threadIdx.x] = v;   // warp 0's slots hold the result
    }
    __syncthreads();
}

// Whether many of a set's runs of equal upper 32 bits will be long: of more
// than kRunMax keys, each of which costs a block sort of its low bits (about 8 us,
// as much as a pass over four tiles of the sort).  If so, prepares a fifth pass
// before the four: its digit counts before theirs, and the keys where it starts
// from.  A long run brings one digit of every pass to kRunMax, which rules it out
// for most sets of up to 2^14 particles by the counts at hand.  Otherwise every
// step-th group of 32 keys, one key per counter at most, is counted by a hash of
// the upper 32 bits, in the place of the values: a long run brings its counter to
// kRunMax / step on average, and one other key beside it.  (Two more than that
// are asked for where keys are left out: at 2^17 keys 0.4% of the counters have
// them by chance, a fifth of those of the shortest long runs do.)  200 sets of 2^17
// particles in two cubes of 0.3% of the side each: 13.3 ms with four passes, 4.4
// with five; 4,096 sets without clumps pay 0.8% for the question.  All threads of
// the block, after a barrier; ends with one.
template <int T>
__device__ bool fifth_pass(CtaSortSharedT<T> &sm, uint64_t *keys, uint64_t *alt, int ns, bool staged) {
    constexpr int E = CtaSortSharedT<T>::TILE;
    uint32_t *count = reinterpret_cast<uint32_t *>(sm.vals);
    const int d = threadIdx.x;
    if (!__syncthreads_or(d < kBRadix && sm.hist[0][d] > kRunMax)) return false;
    const int step = ns <= E ? 1 : 1 << (32 - __clz((ns - 1) / E));
    for (int i = threadIdx.x; i < E; i += T) count[i] = 0;
    __syncthreads();
    for (int i = (d & ~31) * step + (d & 31); i < ns; i += T * step) {
        const uint64_t k = staged ? sm.keys[i] : keys[i];
        atomicAdd(count + (((uint32_t)(k >> kBTopShift) * 0x9e3779b1u) >> (__clz(E) + 1)), 1u);
    }
    __syncthreads();
    const uint32_t many = kRunMax / step + (step > 1 ? 4 : 2);
    bool run = false;
    for (int i = threadIdx.x; i < E; i += T) run |= count[i] >= many;
    // counted by the threads that find one, which are others for nearly each
    if (__syncthreads_count(run) <= ns / E / 4) return false;
    if (d < kBRadix) {
        for (int p = 4; p > 0; --p) sm.hist[p][d] = sm.hist[p - 1][d];
        sm.hist[0][d] = 0;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < ns; i += T) {
        const uint64_t k = staged ? sm.keys[i] : keys[i];
        if (!staged) alt[i] = k;
        atomicAdd(&sm.hist[0][(k >> (kBTopShift - kBRadixBits)) & (kBRadix - 1)], 1u);
    }
    __syncthreads();
    return true;
}

// Every set from work queue 0: root cube, keys, sort, counts.  `raw` is the
// block's dynamic shared memory (batch_front_smem<T> bytes).
template <int T>
__device__ void front_sets(const BatchArgs &A, unsigned char *raw) {
    static_assert(sizeof(RunSmem) <= sizeof(CtaSortSharedT<T>), "a run tile lies in the sort's shared memory");
    CtaSortSharedT<T> &sm = *reinterpret_cast<CtaSortSharedT<T> *>(raw);
    __shared__ TileSharedT<T> ts;
    __shared__ float s_red[(T / 32) * 6];
    __shared__ uint32_t s_bad, s_tot[kLevelFields], s_tile[kLevelFields];
    __shared__ float s_lo[3], s_shi, s_slo;
    __shared__ double s_scale;
    __shared__ bool s_exact, s_f32;
    __shared__ int s_q;
    __shared__ int s_nlong, s_desc, s_passes;
    __shared__ int64_t s_long[32];
    __shared__ unsigned long long s_end;
    __shared__ StartCounts s_sc;
    for (;;) {
        const int q = take_set(&A.queue[0], A.n_sets, &s_q);
        if (q < 0) return;
        const int set = A.order[q];
        const int64_t o = A.off[set], ns = A.off[set + 1] - o;
        if (ns <= 0) {
            if (threadIdx.x < kLevelFields) A.set_cnt[(int64_t)set * kLevelFields + threadIdx.x] = 0;
            if (threadIdx.x < 4) A.set_root[4 * (int64_t)set + threadIdx.x] = threadIdx.x == 3 ? 1.0 : 0.0;
            continue;
        }
        // ---- root cube (Sec. 2.2), as in root_kernel
        if (threadIdx.x == 0) s_bad = 0;
        __syncthreads();
        set_root_cube(A.pos, o, ns, s_red, &s_bad);
        if (threadIdx.x == 0) {
            const RootCube r = root_cube(s_red, s_red + 3, A.root_pow2 != 0);
            s_scale = r.scale;
            s_shi = r.s_hi;
            s_slo = r.s_lo;
            s_exact = r.exact_only;
            s_f32 = r.s_fp32;
            for (int a = 0; a < 3; ++a) {
                s_lo[a] = r.lo[a];
                A.set_root[4 * (int64_t)set + a] = (double)r.lo[a];
            }
            A.set_root[4 * (int64_t)set + 3] = r.side;
            if (s_bad) atomicOr(&A.info->status, kErrNonFinite);
        }
        const int passes0 = ns <= kBFourMax ? 4 : kBMaxPasses, shift00 = 63 - passes0 * kBRadixBits;
        if (threadIdx.x == 0) s_passes = passes0;
        for (int i = threadIdx.x; i < kBMaxPasses * kBRadix; i += blockDim.x) (&sm.hist[0][0])[i] = 0;
        __syncthreads();
        // ---- keys, records and every pass's digit histogram
        const bool staged = ns <= CtaSortSharedT<T>::TILE;
        {
            const float lx = s_lo[0], ly = s_lo[1], lz = s_lo[2], shi = s_shi, slo = s_slo;
            const double sc = s_scale;
            const bool ex = s_exact, f32 = s_f32;
            const float m_eq = (float)(1.0 / (double)ns);
            // unsorted keys go where pass 0 reads them, so that the last pass
            // ends in pkey (a set of one sort tile keeps them in shared memory)
            uint64_t *unsorted = passes0 & 1 ? A.kalt : A.pkey;
            for (int64_t i = o + threadIdx.x; i < o + ns; i += blockDim.x) {
                const float x = A.pos[3 * i], y = A.pos[3 * i + 1], z = A.pos[3 * i + 2];
                const uint64_t k = morton_key(quantise(x, lx, shi, slo, sc, ex, f32),
                                              quantise(y, ly, shi, slo, sc, ex, f32),
                                              quantise(z, lz, shi, slo, sc, ex, f32));
                if (staged) sm.keys[i - o] = k;
                else unsorted[i] = k;
                A.xm[i] = make_float4(x, y, z, A.mass ? A.mass[i] : m_eq);
                for (int p = 0; p < passes0; ++p)
                    atomicAdd(&sm.hist[p][(k >> (shift00 + p * kBRadixBits)) & (kBRadix - 1)], 1u);
            }
        }
        __syncthreads();
        if (passes0 == 4 && ns > kRunMax && fifth_pass<T>(sm, A.pkey + o, A.kalt + o, (int)ns, staged) && threadIdx.x == 0) s_passes = kBMaxPasses;
        __syncthreads();
        const int passes = s_passes, shift0 = 63 - passes * kBRadixBits;
        // ---- stable LSD sort of the set by its upper key bits (digit counts
        // taken above), then the runs of equal upper bits by the low bits
        if (passes & 1) cta_lsd_sort(A.kalt, A.palt, A.pkey, A.perm, o, ns, shift0, passes, true, staged, sm);
        else cta_lsd_sort(A.pkey, A.perm, A.kalt, A.palt, o, ns, shift0, passes, true, staged, sm);
        __syncthreads();
        for (int64_t t0 = o; t0 < o + ns; t0 += kRunTile) {
            if (threadIdx.x == 0) s_nlong = 0;
            __syncthreads();
            run_tile<T>(A.pkey, A.perm, o, t0, o + ns, shift0, *reinterpret_cast<RunSmem *>(raw),
                                [&](int64_t a) { s_long[atomicAdd(&s_nlong, 1)] = a; });
            const int nl = s_nlong;
            for (int j = 0; j < nl; ++j) {
                // a run of more than kRunMax keys (at most 16 start in a tile):
                // its end, then the block sort of its low bits, unless they are
                // in order (identical keys, as of particles on a lattice)
                const int64_t a = s_long[j];
                const uint64_t tp = A.pkey[a] >> shift0;
                if (threadIdx.x == 0) {
                    s_end = (unsigned long long)(o + ns);
                    s_desc = 0;
                }
                __syncthreads();
                for (int64_t base = a + 1; base < o + ns; base += blockDim.x) {
                    const int64_t p = base + threadIdx.x;
                    if (p < o + ns) {
                        const uint64_t k = A.pkey[p];
                        if ((k >> shift0) != tp) atomicMin(&s_end, (unsigned long long)p);
                        else if (k < A.pkey[p - 1]) s_desc = 1;
                    }
                    __syncthreads();
                    const bool done = s_end < (unsigned long long)(o + ns);
                    __syncthreads();
                    if (done) break;
                }
                if (s_desc) {
                    const int64_t len = (int64_t)s_end - a;
                    const int low_passes = (shift0 + kBRadixBits - 1) / kBRadixBits;
                    cta_histograms(A.pkey, a, len, 0, low_passes, sm);
                    const int np = cta_lsd_sort(A.pkey, A.perm, A.kalt, A.palt, a, len, 0, low_passes, false, false, sm);
                    if (np & 1)
                        for (int64_t p = a + threadIdx.x; p < a + len; p += blockDim.x) {
                            A.pkey[p] = A.kalt[p];
                            A.perm[p] = A.palt[p];
                        }
                }
                __syncthreads();
            }
        }
        // ---- cells and leaves started per level (the set is its own tree)
        if (A.ncrit >= kLcMinN && A.ncrit <= kLcMaxN) {
            // tiles of 4 T particles from a multiple of four on
            if (threadIdx.x <= kLevels) s_sc.m[threadIdx.x] = s_sc.l[threadIdx.x] = 0;
            for (int64_t s = o & ~int64_t(3); s < o + ns; s += 4 * T) {
                count_tile4<T>(A.pkey, o, o + ns, A.ncrit, s, min64(o + ns, s + 4 * T), raw, s_sc, A.ml);
                __syncthreads();
            }
            if (threadIdx.x < kLevelFields) s_tot[threadIdx.x] = s_sc.cells(threadIdx.x);
        } else {
            if (threadIdx.x < kLevelFields) s_tot[threadIdx.x] = 0;
            __syncthreads();
            for (int64_t s = o; s < o + ns; s += T) {
                const int64_t e = min64(o + ns, s + T);
                const Front f = tile_front<T>(A.pkey, o, o + ns, A.ncrit, s, e, raw, ts);
                if (f.k < e) A.ml[f.k] = (uint16_t)(f.m | (f.L << 8));
                field_totals(ts, s_tile);
                __syncthreads();
                if (threadIdx.x < kLevelFields) s_tot[threadIdx.x] += s_tile[threadIdx.x];
                __syncthreads();
            }
        }
        if (threadIdx.x < kLevelFields)
            A.set_cnt[(int64_t)set * kLevelFields + threadIdx.x] = s_tot[threadIdx.x];
        __syncthreads();
    }
}

template <int T>
__global__ void __launch_bounds__(T, 1024 / T) batch_front_kernel(BatchArgs A) {
    after_previous();
    if (A.info->status & kErrInvalid) return;
    extern __shared__ __align__(16) unsigned char raw[];
    front_sets<T>(A, raw);
}

// Cell and leaf offsets of the sets (in set order), totals and depth.
// One block of up to 1024 threads.
__device__ void batch_scan_block(const BatchArgs &A, int64_t cell_cap) {
    __shared__ int64_t s_c[32], s_l[32];
    __shared__ int s_dmax;
    const int S = A.n_sets;
    const int nt = blockDim.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int per = (S + nt - 1) / nt;
    const int lo = threadIdx.x * per, hi = min(S, lo + per);
    int64_t c = 0, l = 0;
    int dmax = 0;
    for (int s = lo; s < hi; ++s) {
        const uint32_t *r = A.set_cnt + (int64_t)s * kLevelFields;
#pragma unroll
        for (int d = 0; d < kLevels; ++d) {
            const uint32_t v = r[d];
            c += v;
            if (v) dmax = d;
        }
        l += r[kLevels];
    }
    // prefixes over the threads: within warps, then over the warps
    int64_t rc = c, rl = l;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int64_t y = __shfl_up_sync(0xffffffffu, rc, off), z = __shfl_up_sync(0xffffffffu, rl, off);
        if (lane >= off) { rc += y; rl += z; }
    }
    if (threadIdx.x == 0) s_dmax = 0;
    if (lane == 31) { s_c[warp] = rc; s_l[warp] = rl; }
    __syncthreads();
    dmax = __reduce_max_sync(0xffffffffu, dmax);
    if (lane == 0) atomicMax(&s_dmax, dmax);
    for (int w = 0; w < warp; ++w) { rc += s_c[w]; rl += s_l[w]; }
    if (threadIdx.x == nt - 1) {
        A.set_cell_off[S] = rc;
        A.set_leaf_off[S] = rl;
        A.info->n_cells = rc;
        A.info->n_leaves = (uint32_t)rl;
        for (int d = 0; d < kLevels; ++d) A.info->level_offset[d] = 0;
        A.info->level_offset[kLevels] = rc;
        if (cell_cap > 0 && rc > cell_cap) A.info->status |= kErrOverflow;
    }
    __syncthreads();
    rc -= c;
    rl -= l;
    for (int s = lo; s < hi; ++s) {
        A.set_cell_off[s] = rc;
        A.set_leaf_off[s] = rl;
        const uint32_t *r = A.set_cnt + (int64_t)s * kLevelFields;
        for (int d = 0; d < kLevels; ++d) rc += r[d];
        rl += r[kLevels];
    }
    if (threadIdx.x == 0) A.info->max_depth = s_dmax;
}

__global__ void __launch_bounds__(1024) batch_scan_kernel(BatchArgs A, int64_t cell_cap) {
    after_previous();
    if (A.info->status & kErrInvalid) return;
    batch_scan_block(A, cell_cap);
}

// Every cell of one set with its links and (GATHER, for moments_set) the
// set's particles in key order (tiles of 4 T particles from a multiple of four
// on; all T threads of the block).
template <int T, bool GATHER>
__device__ void emit_set(const BatchArgs &A, const EmitOut &out, int set, EmitShared<T> &sm) {
    __shared__ uint32_t s_lvl[kLevels + 1];   // the set's levels start (end) here
    const int64_t o = A.off[set], ns = A.off[set + 1] - o;
    if (ns <= 0) return;
    const int lane = threadIdx.x & 31;
    if (threadIdx.x < 32) {
        const uint32_t v = lane < kLevels ? A.set_cnt[(int64_t)set * kLevelFields + lane] : 0u;
        uint32_t x = v;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, off);
            if (lane >= off) x += y;
        }
        if (lane <= kLevels) s_lvl[lane] = (uint32_t)A.set_cell_off[set] + x - v;
    }
    __syncthreads();
    uint32_t base = 0;
    if (lane < kLevelFields) base = lane < kLevels ? s_lvl[lane] : (uint32_t)A.set_leaf_off[set];
    int parity = 0;
    for (int64_t s = o & ~int64_t(3); s < o + ns; s += 4 * T, parity ^= 1)
        base += emit_tile<T, !GATHER>(A.pkey, A.ml, o, o + ns, s, base,
                                   [&](int d) { return (int64_t)s_lvl[d + 1]; }, out, sm, parity);
    // the set's particles in key order, for its moments
    if constexpr (GATHER)
        for (int64_t k = o + threadIdx.x; k < o + ns; k += blockDim.x) A.xs[k] = A.xm[A.perm[k]];
    __syncthreads();
}

template <int T>
__global__ void __launch_bounds__(T, 1280 / T) batch_emit_kernel(BatchArgs A, EmitOut out) {
    after_previous();
    if (A.info->status & (kErrOverflow | kErrNonFinite | kErrInvalid)) return;
    __shared__ int s_q;
    __shared__ EmitShared<T> sm;
    for (;;) {
        const int q = take_set(&A.queue[1], A.n_sets, &s_q);
        if (q < 0) return;
        emit_set<T, false>(A, out, A.order[q], sm);
    }
}

// FP64 sum of a leaf too long for the FP32 routes (more than 2^20 members).
__device__ __noinline__ void leaf_sum_f64_serial(const MomOut &o, const float4 *xs, int64_t c,
                                                 int64_t pf, int64_t pe, bool has64) {
    const float4 r0 = xs[pf];
    const float ref[3] = {r0.x, r0.y, r0.z};
    float bb[6] = {r0.x, r0.y, r0.z, r0.x, r0.y, r0.z};
    AccD D;
    D.init();
    for (int64_t k = pf; k < pe; ++k) {
        const float4 v = xs[k];
        const float x[3] = {v.x, v.y, v.z};
        double dx[3];
        for (int a = 0; a < 3; ++a) {
            bb[a] = fminf(bb[a], x[a]);
            bb[3 + a] = fmaxf(bb[3 + a], x[a]);
            dx[a] = (double)x[a] - (double)ref[a];
        }
        D.add((double)v.w, dx);
    }
    finish_d(o, c, D, ref, bb, has64);
}

// The cells of one set above its leaves, level by level, deepest first (all
// threads of the block).  With AHEAD the next child's loads are issued before a
// child is added; the one-launch build, held to 64 registers by its front,
// spills less without (264 bytes, 616 with; 600 sets of 1,000 to 30,000 1.51 ms,
// 1.86 with).
template <int MODE, bool AHEAD>
__device__ void parents_set(const BatchArgs &A, const TreeIn &T, const MomOut &o, int set) {
    __shared__ int64_t s_lvl[kLevels + 1];
    {
        const int64_t ns = A.off[set + 1] - A.off[set];
        if (ns <= 0) return;
        if (threadIdx.x == 0) {
            int64_t r = A.set_cell_off[set];
            for (int d = 0; d < kLevels; ++d) {
                s_lvl[d] = r;
                r += A.set_cnt[(int64_t)set * kLevelFields + d];
            }
            s_lvl[kLevels] = r;
        }
        __syncthreads();
        for (int d = kDepthMax - 1; d >= 0; --d) {
            for (int64_t c = s_lvl[d] + threadIdx.x; c < s_lvl[d + 1]; c += blockDim.x)
                if (T.child_first[c] >= 0) combine_children<MODE>(T, o, c, cells_of<AHEAD>(o));
            __syncthreads();
        }
    }
}

// Moments of one set in the one-launch build: every leaf in key order, then
// the other cells.  Leaves are summed as the leaf tiles of the separate
// launches sum them -- short ones by a thread, the others (in the compensated
// mode those of more than kSplitLeaf, else those that do not fit their tile's
// span) by a warp -- so that both give the same bits up to leaves of 2048.
template <int MODE>
__device__ void moments_set(const BatchArgs &A, const TreeIn &T, const MomOut &o,
                            const int32_t *__restrict__ leaf_cell, int set, int64_t n_total) {
    const int lane = threadIdx.x & 31;
    if (A.off[set + 1] <= A.off[set]) return;
    const int64_t l0 = A.set_leaf_off[set], l1 = A.set_leaf_off[set + 1];
    for (int64_t j0 = l0 + threadIdx.x - lane; j0 < l1; j0 += blockDim.x) {
        int64_t c = 0, pf = 0, pe = 0;
        bool by_warp = false;
        if (j0 + lane < l1) {
            c = leaf_cell[j0 + lane];
            pf = T.pfirst[c];
            pe = T.pend[c];
            const int64_t k0 = pf & ~int64_t(kLtTile - 1);
            const bool staged = pe < k0 + kLtSpan || (pe == n_total && n_total <= k0 + kLtSpan);
            by_warp = pe - pf <= kBigLeafThread &&
                      (!staged || (MODE == TB_MOM_FP32_COMP && pe - pf > kSplitLeaf));
            if (pe - pf > kBigLeafSerial) leaf_sum_f64_serial(o, A.xs, c, pf, pe, MODE == TB_MOM_FP64);
            else if (!by_warp) leaf_sum<MODE>(o, A.xs, c, pf, pe);
        }
        for (unsigned b = __ballot_sync(0xffffffffu, by_warp); b; b &= b - 1) {
            const int w = __ffs(b) - 1;
            warp_leaf_sum<MODE>(o, (const float4 *)A.xs, __shfl_sync(0xffffffffu, c, w),
                                __shfl_sync(0xffffffffu, pf, w), __shfl_sync(0xffffffffu, pe, w));
        }
    }
    __syncthreads();
    parents_set<MODE, false>(A, T, o, set);
}

// The children's loads bound this: one block's levels follow one another, each
// a few dependent reads long, and few threads have a parent.
template <int MODE>
__global__ void __launch_bounds__(kBMomThreads, 3)
    batch_up_kernel(BatchArgs A, TreeIn T, MomOut o) {
    after_previous();
    if (A.info->status & (kErrOverflow | kErrNonFinite | kErrInvalid)) return;
    __shared__ int s_q;
    for (;;) {
        const int q = take_set(&A.queue[2], A.n_sets, &s_q);
        if (q < 0) return;
        parents_set<MODE, true>(A, T, o, A.order[q]);
    }
}

// The set offsets must partition [0, n_total): off[0] = 0, off[S] = n_total,
// non-decreasing.  Otherwise every batched kernel skips its work.
__device__ void set_check_grid(const int64_t *off, int32_t S, int64_t n_total, DevInfo *info) {
    bool bad = false;
    if (blockIdx.x == 0 && threadIdx.x == 0) bad = (off[0] != 0 || off[S] != n_total);
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < S;
         s += (int64_t)gridDim.x * blockDim.x)
        bad |= off[s + 1] < off[s] || off[s + 1] - off[s] > 2147483647LL;
    if (bad) atomicOr(&info->status, kErrInvalid);
}

__global__ void set_check_kernel(const int64_t *off, int32_t S, int64_t n_total, DevInfo *info) {
    after_previous();
    set_check_grid(off, S, n_total, info);
}

// A barrier across every block of a cooperative launch (all blocks are
// resident at once, so every block arrives).  bar[0] counts arrivals, bar[1]
// is the generation; the last block to arrive resets the count and opens the
// next generation.  The wait is bounded: one that runs out records a timeout
// and lets the block go on.
__device__ void grid_barrier(uint32_t *bar, int64_t limit, DevInfo *info) {
    __syncthreads();
    if (threadIdx.x == 0) {
        volatile uint32_t *gen = bar + 1;
        const uint32_t g = *gen;
        __threadfence();
        if (atomicAdd(&bar[0], 1u) == gridDim.x - 1) {
            bar[0] = 0;
            __threadfence();
            atomicAdd(&bar[1], 1u);
        } else {
            int64_t it = 0;
            while (*gen == g) {
                if (!poll_backoff(it, limit)) {
                    flag_error(&info->status, kErrTimeout);
                    break;
                }
            }
        }
        __threadfence();
    }
    __syncthreads();
}

// The whole batched build in one cooperative launch (fixed cell capacity):
// offsets checked, sets ordered, every set's front (keys, sort, counts), the
// offsets of all sets, then each set's cells and moments by the block that
// takes it -- phases separated by grid barriers.
template <int T, int MODE>
__global__ void __launch_bounds__(T, 1024 / T)
    batch_all_kernel(BatchArgs A, int32_t *order, EmitOut out, TreeIn Tr, MomOut o,
                     const int32_t *__restrict__ leaf_cell, int64_t n_total, int64_t cell_cap,
                     int64_t wait_limit) {
    extern __shared__ __align__(16) unsigned char raw[];
    uint32_t *bar = A.queue + 4;
    __shared__ int s_q;
    set_check_grid(A.off, A.n_sets, n_total, A.info);
    grid_barrier(bar, wait_limit, A.info);
    // the status words below were all written before a barrier: every block
    // reads the same values and takes the same branch
    if (*(volatile uint32_t *)&A.info->status & kErrInvalid) return;
    if (blockIdx.x == 0) set_order_block(A.off, A.n_sets, order);
    grid_barrier(bar, wait_limit, A.info);
    front_sets<T>(A, raw);
    grid_barrier(bar, wait_limit, A.info);
    if (blockIdx.x == 0) batch_scan_block(A, cell_cap);
    grid_barrier(bar, wait_limit, A.info);
    if (*(volatile uint32_t *)&A.info->status & (kErrOverflow | kErrNonFinite)) return;
    static_assert(sizeof(EmitShared<T>) <= sizeof(CtaSortSharedT<T>), "the emission's lists lie in the sort's shared memory");
    EmitShared<T> &em = *reinterpret_cast<EmitShared<T> *>(raw);
    for (;;) {
        const int q = take_set(&A.queue[1], A.n_sets, &s_q);
        if (q < 0) return;
        const int set = order[q];
        emit_set<T, true>(A, out, set, em);
        moments_set<MODE>(A, Tr, o, leaf_cell, set, n_total);
    }
}

}  // namespace

cudaError_t launch_set_check(const int64_t *off, int32_t S, int64_t n_total, Workspace &ws,
                             cudaStream_t s) {
    int grid = (S + 255) / 256;
    if (grid < 1) grid = 1;
    if (grid > 1024) grid = 1024;
    set_check_kernel<<<grid, 256, 0, s>>>(off, S, n_total, ws.info);
    ++g_launches;
    return cudaGetLastError();
}

namespace {

template <int T>
cudaError_t launch_batched_t(const BatchArgs &A, int32_t S, int ncrit, tb_tree &t, Workspace &ws,
                             int64_t cell_cap, int phase, int mode, cudaStream_t s) {
    cudaError_t e;
    static std::atomic<uint64_t> attr_done{0};
    if ((e = once_on_device(attr_done, [] {
             return allow_smem(batch_front_kernel<T>, batch_front_smem<T>(kMaxNcrit), true);
         })) != cudaSuccess)
        return e;
    int dev = 0, nsm = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    // persistent grids: as many blocks as fit at once (1024 / T front blocks
    // per SM), at most one per set
    auto fit = [&](int per_sm) { return S < per_sm * nsm ? (S > 0 ? S : 1) : per_sm * nsm; };
    if (phase == 0) {
        launch_after(set_order_kernel, dim3(1), dim3(1024), 0, s, A.off, S, ws.set_order, ws.info);
        ++g_launches;
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        launch_after(batch_front_kernel<T>, dim3(fit(1024 / T)), dim3(T), batch_front_smem<T>(ncrit), s, A);
        ++g_launches;
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        mark(ws, "batch_front", s);
        launch_after(batch_scan_kernel, dim3(1), dim3(1024), 0, s, A, cell_cap);
        ++g_launches;
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        mark(ws, "batch_scan", s);
        return cudaSuccess;
    }
    // the keys' second buffer is free by now
    int32_t *start_cell = reinterpret_cast<int32_t *>(ws.keys_alt);
    EmitOut out{t.ckey, t.level, t.parent, t.child_first, t.child_end, t.pfirst, t.pend,
                t.leaf_cell, start_cell};
    // blocks of 256 threads, 1,024 particles a tile, five sets per SM; a few
    // large sets, of many tiles, take an SM each, many small ones smaller
    // blocks.  With every particle's masks in tiles of 1,024 threads before,
    // building 4,096 sets took 4.71 ms, now 4.31; 300 sets 145 and 138 us;
    // 16 sets of up to 65,536 723 and 644; 100 sets of 1,000 to 2,000 92 and 93
    const bool small = batch_many_small(S, t.n_particles);
    if (batch_few_large(S, t.n_particles)) launch_after(batch_emit_kernel<1024>, dim3(fit(1)), dim3(1024), 0, s, A, out);
    else if (small) launch_after(batch_emit_kernel<128>, dim3(fit(10)), dim3(128), 0, s, A, out);
    else launch_after(batch_emit_kernel<256>, dim3(fit(5)), dim3(256), 0, s, A, out);
    ++g_launches;
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    mark(ws, "batch_emit", s);
    if ((e = launch_batched_leaves(t, ws, mode, start_cell, s)) != cudaSuccess) return e;
    TreeIn Tr{t.child_first, t.child_end, t.pfirst, t.pend, ws.big_leaf, t.parent};
    MomOut o{t.mass, t.com, t.com_lo, t.quad, t.aabb, t.mass64, t.com64, t.quad64};
    // (4,096 sets: 5.06 ms with 128 threads, 5.19 with 256; 1,000 sets of 1,000 to
    // 65,536: 2.14 and 2.00)
    const int up_threads = small ? 64 : (S > 1824 ? kBMomThreads / 2 : kBMomThreads);
    const int grid_mom = fit(3 * kBMomThreads / up_threads);
    switch (mode) {
        case TB_MOM_FP32_COMP:
            launch_after(batch_up_kernel<TB_MOM_FP32_COMP>, dim3(grid_mom), dim3(up_threads), 0, s, A, Tr, o);
            break;
        case TB_MOM_FP32_PLAIN:
            launch_after(batch_up_kernel<TB_MOM_FP32_PLAIN>, dim3(grid_mom), dim3(up_threads), 0, s, A, Tr, o);
            break;
        default:
            launch_after(batch_up_kernel<TB_MOM_FP64>, dim3(grid_mom), dim3(up_threads), 0, s, A, Tr, o);
            break;
    }
    ++g_launches;
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    mark(ws, "batch_moments", s);
    return cudaSuccess;
}

}  // namespace

template <int T, int MODE>
cudaError_t launch_batched_one_t(const BatchArgs &A, int32_t S, int ncrit, int64_t n_total,
                                 tb_tree &t, Workspace &ws, int64_t cell_cap, cudaStream_t s) {
    auto kern = batch_all_kernel<T, MODE>;
    const size_t smem = batch_front_smem<T>(ncrit);
    static std::atomic<uint64_t> attr_done{0};
    cudaError_t e = once_on_device(attr_done, [&] { return allow_smem(kern, batch_front_smem<T>(kMaxNcrit), true); });
    if (e != cudaSuccess) return e;
    int dev = 0, nsm = 152, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, T, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorCooperativeLaunchTooLarge;
    // every block resident at once (the grid barriers need it), at most one
    // block per set
    const int grid = S < per_sm * nsm ? (S > 0 ? S : 1) : per_sm * nsm;
    BatchArgs a = A;
    int32_t *order = ws.set_order;
    EmitOut out{t.ckey, t.level, t.parent, t.child_first, t.child_end, t.pfirst, t.pend,
                t.leaf_cell, nullptr};
    TreeIn Tr{t.child_first, t.child_end, t.pfirst, t.pend, ws.big_leaf, t.parent};
    MomOut o{t.mass, t.com, t.com_lo, t.quad, t.aabb, t.mass64, t.com64, t.quad64};
    const int32_t *leaf_cell = t.leaf_cell;
    int64_t nt = n_total, cap = cell_cap, lim = g_wait_limit;
    void *args[] = {&a, &order, &out, &Tr, &o, &leaf_cell, &nt, &cap, &lim};
    e = fault_cooperative() ? cudaErrorCooperativeLaunchTooLarge
                            : cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(kern), dim3(grid),
                                                          dim3(T), args, smem, s);
    if (e != cudaSuccess) return e;
    ++g_launches;
    mark(ws, "batch_all", s);
    return cudaSuccess;
}

bool batch_threads_valid(int threads) { return threads == 0 || threads == 512 || threads == 1024; }

cudaError_t launch_batched_one(const float *pos, const float *mass, const int64_t *off, int32_t S,
                               int64_t n_total, int ncrit, int threads, tb_tree &t, Workspace &ws,
                               int64_t cell_cap, int mode, cudaStream_t s) {
    BatchArgs A{pos, mass, off, ws.set_order, S, ncrit, t.pkey, t.perm, ws.keys_alt,
                ws.perm_alt, ws.xm, ws.xs, ws.ml, ws.set_cnt, t.set_cell_offset, ws.set_leaf_off,
                t.set_root, ws.set_ctr, ws.info, ws.root_pow2 ? 1 : 0};
    const int T = threads ? threads : kBDefaultThreads;
#define TB_ONE(TT, MM) \
    if (T == TT && mode == MM) return launch_batched_one_t<TT, MM>(A, S, ncrit, n_total, t, ws, cell_cap, s);
    TB_ONE(512, TB_MOM_FP32_COMP)
    TB_ONE(512, TB_MOM_FP32_PLAIN)
    TB_ONE(512, TB_MOM_FP64)
    TB_ONE(1024, TB_MOM_FP32_COMP)
    TB_ONE(1024, TB_MOM_FP32_PLAIN)
    TB_ONE(1024, TB_MOM_FP64)
#undef TB_ONE
    return cudaErrorInvalidValue;
}

cudaError_t launch_batched(const float *pos, const float *mass, const int64_t *off, int32_t S,
                           int ncrit, int threads, tb_tree &t, Workspace &ws, int64_t cell_cap,
                           int phase, int mode, cudaStream_t s) {
    BatchArgs A{pos, mass, off, ws.set_order, S, ncrit, t.pkey, t.perm, ws.keys_alt,
                ws.perm_alt, ws.xm, ws.xs, ws.ml, ws.set_cnt, t.set_cell_offset, ws.set_leaf_off,
                t.set_root, ws.set_ctr, ws.info, ws.root_pow2 ? 1 : 0};
    const int64_t n = t.n_particles;
    switch (threads ? threads
                    : (batch_few_large(S, n) ? 1024 : (batch_many_small(S, n) ? 256 : kBDefaultThreads))) {
        case 256: return launch_batched_t<256>(A, S, ncrit, t, ws, cell_cap, phase, mode, s);
        case 512: return launch_batched_t<512>(A, S, ncrit, t, ws, cell_cap, phase, mode, s);
        case 1024: return launch_batched_t<1024>(A, S, ncrit, t, ws, cell_cap, phase, mode, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace tb
