// tb_walk.cu -- gravity from the built tree (Sec. 2.1): the Barnes-Hut walk
// with the opening test l / d < theta of Eq. 1, monopole plus quadrupole, and
// Barnes' modified algorithm, in which the particles of one small cell share
// one interaction list.
//
//   walk_groups_kernel : the groups -- every cell holding at most n_group
//                        particles whose parent holds more (the root if it
//                        holds at most n_group), and every leaf holding more
//                        (only depth-21 leaves of one key can);
//   walk_kernel        : one warp per group (taken from an atomic ticket),
//                        32 particles at a time (a larger group
//                        is walked in chunks of 32, each with its own box).
//                        The warp walks the tree from the root, up to 32 cells
//                        at a time: a cell whose particle range meets the chunk's is
//                        always opened; any other cell is accepted when
//                        l < theta * d_min, d_min the distance from its centre
//                        of mass to the group's bounding box (so l / d < theta
//                        holds for every particle of the group); an opened leaf
//                        contributes its particles one by one.  Accepted cells
//                        and opened leaves' particles go to lists in shared
//                        memory, which are evaluated, eight entries a step, as
//                        they fill.
// Forces (G = 1): a softened point mass m (r^2 + eps^2)^(-3/2) r for every
// particle and cell; for a cell also the quadrupole term
//   T r / |r|^5 - (5/2) (r.T r) r / |r|^7,  T = 3 Q - tr(Q) I,
// with Q the cell's central second moment and r = x - COM (unsoftened).
// Offsets are taken as (x - com) - com_lo, exact to one rounding when the
// target and the centre are close.  The result is written in the caller's
// particle order.  A walk on a tree with profiling enabled also counts the
// interactions it evaluated (target-cell and target-particle pairs), read
// back by tb_walk_counts.
#include <cfloat>

#include "tb_device.cuh"

namespace tb {

namespace {

constexpr int kWalkWarps = 4;
constexpr int kWalkThreads = 32 * kWalkWarps;
constexpr int kWalkPerSm = 4;          // blocks resident per SM (registers and shared memory)
constexpr int kWalkBlocks = 152 * kWalkPerSm;
// cells waiting to be tested, per warp: the first kStackNear in shared memory,
// the rest in global memory.  A round takes at most 32 cells and adds at most
// 7 per cell, and only cells above depth 21 have
// children, so the stack stays below 21 * 256 + 1 entries
constexpr int kStackCap = 6144;
constexpr int kStackNear = 768;
constexpr int kCellCap = 40;           // accepted cells: under 8 left over and 32 of a round
constexpr int kSrcLeaf = 16;           // leaves of at most this many go to the source list
constexpr int kSrcCap = 640;           // sources: up to 128 waiting and 32 * kSrcLeaf of a round

struct WalkTree {
    const int32_t *child_first, *child_end, *pfirst, *pend;
    const uint8_t *level;
    const float *mass, *com, *com_lo, *quad, *aabb;
    const float4 *xs;               // particles in key order: x, y, z, m
    const int32_t *perm;
    double side;
    const float4 *rec;              // [C][4] per cell: com + m, com_lo, T xx xy xz yy, T yz zz
};

// Two FP32 values in one 64-bit register, and arithmetic on both at once
// (each half rounded as the scalar operation).
__device__ __forceinline__ uint64_t pack2(float a, float b) {
    uint64_t v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(a), "f"(b));
    return v;
}
__device__ __forceinline__ void unpack2(uint64_t v, float &a, float &b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t v;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(v) : "l"(a), "l"(b));
    return v;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t v;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(v) : "l"(a), "l"(b));
    return v;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t v;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(v) : "l"(a), "l"(b), "l"(c));
    return v;
}
__device__ __forceinline__ uint64_t dup2(float a) { return pack2(a, a); }
// 1 / sqrt.  With FULL for every argument; without it, the hardware's
// approximation alone (what rsqrtf rounds to), which takes a subnormal argument
// for 0.  launch_walk knows when no argument can be one; the steps that scale
// those cost a tenth of the walk (2^20 particles 1.98 and 2.19 ms).
template <bool FULL>
__device__ __forceinline__ uint64_t rsqrt2(uint64_t x) {
    float a, b;
    unpack2(x, a, b);
    if constexpr (FULL) {
        a = rsqrtf(a);
        b = rsqrtf(b);
    } else {
        asm("rsqrt.approx.ftz.f32 %0, %0;" : "+f"(a));
        asm("rsqrt.approx.ftz.f32 %0, %0;" : "+f"(b));
    }
    return pack2(a, b);
}

// One warp's lists.  A cell's row is its record's first four float4 (centre
// and mass, low centre, tensor) at a stride of five, which spreads eight rows
// over all banks.
struct WarpLists {
    float4 cell[kCellCap][5];
    int32_t src[kSrcCap];
    int32_t stack[kStackNear];
};

// The chunk's targets and their accelerations.  Lane 8 g + i evaluates entry
// i of each step's eight list entries for the targets t = 4 s + g, slots s =
// 0 .. 7, two slots to a packed register: an entry read from shared memory
// serves eight targets (one target per lane and entry after entry to all lanes
// held the walk at 63% of the shared memory's bandwidth), and the steps run
// over ceil(targets / 8) pairs only.
constexpr int kPairs = 4;
struct Chunk {
    uint64_t x[kPairs], y[kPairs], z[kPairs];
    uint64_t ax[kPairs], ay[kPairs], az[kPairs];
    int pairs;
};

// Steps of eight accepted cells, rows [from, to) of the list; to - from is a
// multiple of eight unless these are the last (missing rows are massless).
template <bool QUAD, bool FULL>
__device__ __forceinline__ void eval_cells(const WarpLists &W, int from, int to, float eps2, Chunk &C) {
    const int i = threadIdx.x & 7;
    const uint64_t E = dup2(eps2), K = dup2(-2.5f);
    for (int j = from; j < to; j += 8) {
        const bool in = j + i < to;
        const float4 *row = W.cell[in ? j + i : from];
        const float4 c0 = row[0], c1 = row[1];
        const uint64_t cx = dup2(-c0.x), cy = dup2(-c0.y), cz = dup2(-c0.z);
        const uint64_t lx = dup2(-c1.x), ly = dup2(-c1.y), lz = dup2(-c1.z);
        const uint64_t nm = dup2(in ? -c0.w : 0.f);
        uint64_t txx = 0, txy = 0, txz = 0, tyy = 0, tyz = 0, tzz = 0;
        if constexpr (QUAD) {
            const float4 t0 = row[2], t1 = row[3];
            txx = dup2(in ? t0.x : 0.f); txy = dup2(in ? t0.y : 0.f); txz = dup2(in ? t0.z : 0.f);
            tyy = dup2(in ? t0.w : 0.f); tyz = dup2(in ? t1.x : 0.f); tzz = dup2(in ? t1.y : 0.f);
        }
#pragma unroll
        for (int p = 0; p < kPairs; ++p) {
            if (p >= C.pairs) break;
            const uint64_t rx = add2(add2(C.x[p], cx), lx);
            const uint64_t ry = add2(add2(C.y[p], cy), ly);
            const uint64_t rz = add2(add2(C.z[p], cz), lz);
            const uint64_t r2 = fma2(rx, rx, fma2(ry, ry, mul2(rz, rz)));
            const uint64_t inv = rsqrt2<FULL>(add2(r2, E));
            uint64_t f = mul2(mul2(mul2(nm, inv), inv), inv);
            if constexpr (QUAD) {
                const uint64_t tx = fma2(txx, rx, fma2(txy, ry, mul2(txz, rz)));
                const uint64_t ty = fma2(txy, rx, fma2(tyy, ry, mul2(tyz, rz)));
                const uint64_t tz = fma2(txz, rx, fma2(tyz, ry, mul2(tzz, rz)));
                const uint64_t rtr = fma2(rx, tx, fma2(ry, ty, mul2(rz, tz)));
                const uint64_t ir = rsqrt2<FULL>(r2);
                const uint64_t ir2 = mul2(ir, ir);
                const uint64_t ir5 = mul2(mul2(ir2, ir2), ir);
                f = fma2(mul2(mul2(rtr, K), ir5), ir2, f);
                C.ax[p] = fma2(tx, ir5, C.ax[p]);
                C.ay[p] = fma2(ty, ir5, C.ay[p]);
                C.az[p] = fma2(tz, ir5, C.az[p]);
            }
            C.ax[p] = fma2(f, rx, C.ax[p]);
            C.ay[p] = fma2(f, ry, C.ay[p]);
            C.az[p] = fma2(f, rz, C.az[p]);
        }
    }
}

// One step of eight source particles; y is this lane's, eps2 its softening (a
// missing source has no mass and a softening of 1).  With SELF, `slot` is the
// slot of this lane's targets that is the source itself, or -1, and takes no
// force from it.
template <bool SELF, bool FULL>
__device__ __forceinline__ void eval_sources(float4 y, int slot, float eps2, Chunk &C) {
    const uint64_t E = dup2(eps2);
    const uint64_t sx = dup2(-y.x), sy = dup2(-y.y), sz = dup2(-y.z), nm = dup2(-y.w);
#pragma unroll
    for (int p = 0; p < kPairs; ++p) {
        if (p >= C.pairs) break;
        const uint64_t rx = add2(C.x[p], sx), ry = add2(C.y[p], sy), rz = add2(C.z[p], sz);
        const uint64_t inv = rsqrt2<FULL>(fma2(rx, rx, fma2(ry, ry, fma2(rz, rz, E))));
        uint64_t f = mul2(mul2(mul2(nm, inv), inv), inv);
        if constexpr (SELF) {
            float a, b;
            unpack2(f, a, b);
            f = pack2(slot == 2 * p ? 0.f : a, slot == 2 * p + 1 ? 0.f : b);
        }
        C.ax[p] = fma2(f, rx, C.ax[p]);
        C.ay[p] = fma2(f, ry, C.ay[p]);
        C.az[p] = fma2(f, rz, C.az[p]);
    }
}

// The source at sorted position q against the chunk [kb, ke).  When !in there is
// none: y is then some other source, and counts with no mass and a softening of
// 1, so that the distance is not 0 even if it is a target itself.
template <bool FULL>
__device__ __forceinline__ void eval_source(float4 y, int q, bool in, int kb, int ke, float eps2,
                                            Chunk &C) {
    if (!in) {
        y.w = 0.f;
        eps2 = 1.f;
    }
    const int t = q - kb;
    const bool mine = in && q >= kb && q < ke;
    if (__any_sync(0xffffffffu, mine))
        eval_sources<true, FULL>(y, mine && (t & 3) == (int)(threadIdx.x & 31) >> 3 ? t >> 2 : -1, eps2, C);
    else
        eval_sources<false, FULL>(y, -1, eps2, C);
}

// Steps of eight listed sources, entries [from, to); the next step's
// particles are loaded before this step's are used.
template <bool FULL>
__device__ __forceinline__ void eval_list(const WarpLists &W, const float4 *__restrict__ xs, int from, int to,
                                          int kb, int ke, float eps2, Chunk &C) {
    const int i = threadIdx.x & 7;
    int q = W.src[min(from + i, to - 1)];
    float4 y = xs[q];
    for (int j = from; j < to; j += 8) {
        const int qn = W.src[min(j + 8 + i, to - 1)];
        const float4 yn = xs[qn];
        eval_source<FULL>(y, q, j + i < to, kb, ke, eps2, C);
        q = qn;
        y = yn;
    }
}

// The sources [q0, q1) of one long leaf (unsigned: the last step may pass the
// largest position, 2^31 - 1).
template <bool FULL>
__device__ __forceinline__ void eval_range(const float4 *__restrict__ xs, int q0, int q1, int kb, int ke,
                                           float eps2, Chunk &C) {
    const uint32_t i = threadIdx.x & 7, end = (uint32_t)q1;
    for (uint32_t j = (uint32_t)q0; j < end; j += 8) {
        const int q = (int)min(j + i, end - 1);
        eval_source<FULL>(xs[q], q, j + i < end, kb, ke, eps2, C);
    }
}

// Per cell, kRec float4: the four the list evaluation reads (centre and
// mass; the centre's low part, with the cell's level in the last word; the
// traceless tensor T = 3 Q - tr(Q) I) and the links the traversal reads
// (pfirst, pend, child_first, child_end), so that a cell tested costs three
// 16-byte loads.
constexpr int kRec = 5;

__global__ void walk_pack_kernel(const float *__restrict__ mass, const float *__restrict__ com,
                                 const float *__restrict__ com_lo, const float *__restrict__ quad,
                                 const uint8_t *__restrict__ level, const int32_t *__restrict__ pfirst,
                                 const int32_t *__restrict__ pend, const int32_t *__restrict__ child_first,
                                 const int32_t *__restrict__ child_end, int64_t n_cells,
                                 float4 *__restrict__ rec) {
    after_previous();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < n_cells; c += stride) {
        const float *q = quad + 6 * c;
        const float tr = q[0] + q[3] + q[5];
        float4 *r = rec + kRec * c;
        r[0] = make_float4(com[3 * c], com[3 * c + 1], com[3 * c + 2], mass[c]);
        r[1] = make_float4(com_lo[3 * c], com_lo[3 * c + 1], com_lo[3 * c + 2],
                           __int_as_float((int)level[c]));
        r[2] = make_float4(3.f * q[0] - tr, 3.f * q[1], 3.f * q[2], 3.f * q[3] - tr);
        r[3] = make_float4(3.f * q[4], 3.f * q[5] - tr, 0.f, 0.f);
        reinterpret_cast<int4 *>(r)[4] = make_int4(pfirst[c], pend[c], child_first[c], child_end[c]);
    }
}

__global__ void walk_groups_kernel(const int32_t *__restrict__ parent, const int32_t *__restrict__ child_first,
                                   const int32_t *__restrict__ pfirst, const int32_t *__restrict__ pend,
                                   int64_t n_cells, int n_group, int32_t *groups, uint32_t *ctr) {
    after_previous();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < n_cells; c += stride) {
        const int64_t cnt = (int64_t)pend[c] - pfirst[c];
        const int32_t p = parent[c];
        const bool small = cnt <= n_group && (p < 0 || (int64_t)pend[p] - pfirst[p] > n_group);
        const bool big_leaf = child_first[c] < 0 && cnt > n_group;
        if (small || big_leaf) groups[atomicAdd(&ctr[0], 1u)] = (int32_t)c;
    }
}

template <bool QUAD, bool COUNT, bool FULL>
__global__ void __launch_bounds__(kWalkThreads, kWalkPerSm)
    walk_kernel(WalkTree T, const int32_t *__restrict__ groups, uint32_t *ctr, int32_t *stacks,
                float theta, float eps2, float *__restrict__ acc_out, DevInfo *info) {
    after_previous();
    if (info->status & (kErrOverflow | kErrNonFinite)) return;
    __shared__ WarpLists lists[kWalkWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    WarpLists &W = lists[warp];
    int32_t *far = stacks + ((int64_t)blockIdx.x * kWalkWarps + warp) * kStackCap;
    const uint32_t ngroups = *(volatile const uint32_t *)&ctr[0];
    const unsigned lt = lanemask_lt();
    const float side = (float)T.side, theta2 = theta * theta;
    // interactions evaluated by this warp (lane 0 counts): target x accepted
    // cell, and target x source particle (self excluded); added to the
    // walk's totals when the warp is done
    unsigned long long n_cell_int = 0, n_pp_int = 0;
    unsigned long long *totals = reinterpret_cast<unsigned long long *>(ctr + 2);
    for (;;) {
        uint32_t gi = 0;
        if (lane == 0) gi = atomicAdd(&ctr[1], 1u);
        gi = __shfl_sync(0xffffffffu, gi, 0);
        if (gi >= ngroups) {
            if (COUNT && lane == 0) {
                atomicAdd(&totals[0], n_cell_int);
                atomicAdd(&totals[1], n_pp_int);
            }
            return;
        }
        const int32_t g = groups[gi];
        const int gpf = T.pfirst[g], gpe = T.pend[g];
        for (int kb = gpf; kb < gpe; kb += min(32, gpe - kb)) {
            const int nt = min(32, gpe - kb), ke = kb + nt;
            // bounding box of the chunk
            float bmin[3], bmax[3];
            Chunk C;
            {
                const float4 x = T.xs[lane < nt ? kb + lane : kb];
                bmin[0] = bmax[0] = x.x;
                bmin[1] = bmax[1] = x.y;
                bmin[2] = bmax[2] = x.z;
                for (int off = 16; off > 0; off >>= 1)
                    for (int a = 0; a < 3; ++a) {
                        bmin[a] = fminf(bmin[a], __shfl_xor_sync(0xffffffffu, bmin[a], off));
                        bmax[a] = fmaxf(bmax[a], __shfl_xor_sync(0xffffffffu, bmax[a], off));
                    }
                // slot s of this lane: target 4 s + lane / 8 (the first, when
                // there is no such target)
                C.pairs = (nt + 7) / 8;
#pragma unroll
                for (int p = 0; p < kPairs; ++p) {
                    const int t0 = 8 * p + (lane >> 3), t1 = t0 + 4;
                    C.x[p] = pack2(__shfl_sync(0xffffffffu, x.x, t0), __shfl_sync(0xffffffffu, x.x, t1));
                    C.y[p] = pack2(__shfl_sync(0xffffffffu, x.y, t0), __shfl_sync(0xffffffffu, x.y, t1));
                    C.z[p] = pack2(__shfl_sync(0xffffffffu, x.z, t0), __shfl_sync(0xffffffffu, x.z, t1));
                    C.ax[p] = C.ay[p] = C.az[p] = 0;
                }
            }
            int sp = 1, ncell = 0, nsrc = 0;
            if (lane == 0) W.stack[0] = 0;
            __syncwarp();
            bool overflow = false;
            while (sp > 0) {
                // at most 32 cells, and room for 7 more stack entries per cell
                const int take = min(min(sp, 32), (kStackCap - sp) / 7);
                if (take == 0) {
                    overflow = true;
                    break;
                }
                int c = -1;
                if (lane < take) {
                    const int at = sp - 1 - lane;
                    c = at < kStackNear ? W.stack[at] : far[at];
                }
                sp -= take;
                float4 r0 = make_float4(0.f, 0.f, 0.f, 0.f), r1 = r0;
                int4 lk = make_int4(0, 0, 0, 0);        // pfirst, pend, child_first, child_end
                if (c >= 0) {
                    const float4 *rec = T.rec + kRec * (int64_t)c;
                    lk = reinterpret_cast<const int4 *>(rec)[4];
                    r0 = rec[0];
                    r1 = rec[1];
                }
                // what earlier rounds listed, while these loads are on their way:
                // whole steps from the lists' ends
                cp_async_wait_all();
                __syncwarp();
                if (ncell >= 8) {
                    eval_cells<QUAD, FULL>(W, ncell & 7, ncell, eps2, C);
                    ncell &= 7;
                }
                if (nsrc > kSrcCap - 32 * kSrcLeaf) {
                    eval_list<FULL>(W, T.xs, nsrc & 7, nsrc, kb, ke, eps2, C);
                    nsrc &= 7;
                }
                __syncwarp();
                int kind = 0;                           // 1 accept, 2 leaf, 3 open
                int nch = 0;
                const int c0 = lk.z;
                if (c >= 0) {
                    bool accept = false;
                    if (!(lk.x < ke && kb < lk.y)) {
                        const float l = side * __int_as_float((127 - __float_as_int(r1.w)) << 23);   // side 2^-level
                        const float cx[3] = {r0.x + r1.x, r0.y + r1.y, r0.z + r1.z};
                        float d2 = 0.f;
                        for (int a = 0; a < 3; ++a) {
                            const float u = fmaxf(fmaxf(bmin[a] - cx[a], cx[a] - bmax[a]), 0.f);
                            d2 = fmaf(u, u, d2);
                        }
                        accept = l * l < theta2 * d2;
                    }
                    if (accept) kind = 1;
                    else if (c0 < 0) kind = 2;
                    else { kind = 3; nch = lk.w - c0; }
                }
                const unsigned ba = __ballot_sync(0xffffffffu, kind == 1);
                if (kind == 1) {
                    float4 *row = W.cell[ncell + __popc(ba & lt)];
                    const float4 *rec = T.rec + kRec * (int64_t)c;
                    row[0] = r0;
                    row[1] = r1;
                    if constexpr (QUAD) {
                        cp_async16(row + 2, rec + 2);
                        cp_async16(row + 3, rec + 3);
                    }
                }
                ncell += __popc(ba);
                // prefixes of the children (low half) and of the listed sources
                const int cnt = kind == 2 ? lk.y - lk.x : 0;
                const int few = cnt <= kSrcLeaf ? cnt : 0;
                const int both = nch | (few << 16);
                int pos = both;
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, pos, off);
                    if (lane >= off) pos += y;
                }
                const int total = __shfl_sync(0xffffffffu, pos, 31);
                pos -= both;
                for (int j = 0; j < nch; ++j) {
                    const int at = sp + (pos & 0xffff) + j;
                    if (at < kStackNear) W.stack[at] = c0 + nch - 1 - j;
                    else far[at] = c0 + nch - 1 - j;
                }
                for (int j = 0; j < few; ++j) W.src[nsrc + (pos >> 16) + j] = lk.x + j;
                sp += total & 0xffff;
                nsrc += total >> 16;
                if (COUNT) {
                    long long srcs = cnt;
#pragma unroll
                    for (int off = 16; off > 0; off >>= 1) srcs += __shfl_xor_sync(0xffffffffu, srcs, off);
                    n_cell_int += (unsigned long long)(__popc(ba) * nt);
                    n_pp_int += (unsigned long long)(srcs * nt);
                }
                // longer leaves at once, one after another
                for (unsigned bl = __ballot_sync(0xffffffffu, cnt > kSrcLeaf); bl; bl &= bl - 1) {
                    const int w = __ffs(bl) - 1;
                    eval_range<FULL>(T.xs, __shfl_sync(0xffffffffu, lk.x, w), __shfl_sync(0xffffffffu, lk.y, w), kb,
                               ke, eps2, C);
                }
                __syncwarp();
            }
            if (overflow) {
                cp_async_wait_all();
                if (lane == 0) atomicOr(&info->status, kErrWalk);
                return;
            }
            if (COUNT) n_pp_int -= (unsigned long long)nt;   // own pairs
            cp_async_wait_all();
            __syncwarp();
            if (ncell) eval_cells<QUAD, FULL>(W, 0, ncell, eps2, C);
            if (nsrc) eval_list<FULL>(W, T.xs, 0, nsrc, kb, ke, eps2, C);
            __syncwarp();
            // the eight lanes' sums of each target; lane i of a group writes slot i
            float out[3] = {0.f, 0.f, 0.f};
#pragma unroll
            for (int p = 0; p < kPairs; ++p) {
                float v[6];
                unpack2(C.ax[p], v[0], v[3]);
                unpack2(C.ay[p], v[1], v[4]);
                unpack2(C.az[p], v[2], v[5]);
#pragma unroll
                for (int off = 1; off < 8; off <<= 1)
                    for (int a = 0; a < 6; ++a) v[a] += __shfl_xor_sync(0xffffffffu, v[a], off);
                for (int a = 0; a < 3; ++a) {
                    if ((lane & 7) == 2 * p) out[a] = v[a];
                    if ((lane & 7) == 2 * p + 1) out[a] = v[3 + a];
                }
            }
            const int t = 4 * (lane & 7) + (lane >> 3);
            if (t < nt) {
                const int64_t i = T.perm[kb + t];
                acc_out[3 * i] = out[0];
                acc_out[3 * i + 1] = out[1];
                acc_out[3 * i + 2] = out[2];
            }
        }
    }
}

}  // namespace

int64_t walk_buffer_words(int64_t n_cells) {
    return 4 * kRec * n_cells + 8 + n_cells + (int64_t)kWalkBlocks * kWalkWarps * kStackCap;
}

cudaError_t launch_walk(const tb_tree &t, Workspace &ws, float theta, float eps, int n_group,
                        int use_quad, float *acc, int32_t *buf, cudaStream_t s) {
    float4 *rec = reinterpret_cast<float4 *>(buf);   // first: 16-byte aligned
    uint32_t *ctr = reinterpret_cast<uint32_t *>(buf + 4 * kRec * t.n_cells);
    ws.walk_ctr = ctr;
    int32_t *groups = buf + 4 * kRec * t.n_cells + 8;
    int32_t *stacks = groups + t.n_cells;
    cudaError_t e = cudaMemsetAsync(ctr, 0, 8 * sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
    int64_t grid = (t.n_cells + 255) / 256;
    if (grid > 152 * 8) grid = 152 * 8;
    if (grid < 1) grid = 1;
    walk_groups_kernel<<<(unsigned)grid, 256, 0, s>>>(t.parent, t.child_first, t.pfirst, t.pend,
                                                      t.n_cells, n_group, groups, ctr);
    ++g_launches;
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    launch_after(walk_pack_kernel, dim3((unsigned)grid), dim3(256), 0, s, t.mass, t.com, t.com_lo, t.quad, t.level, t.pfirst,
                                                    t.pend, t.child_first, t.child_end, t.n_cells,
                                                    rec);
    ++g_launches;
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    WalkTree T{t.child_first, t.child_end, t.pfirst, t.pend, t.level, t.mass, t.com, t.com_lo,
               t.quad, t.aabb, ws.xs, t.perm, t.side, rec};
    // No argument of rsqrt2 is subnormal when eps^2 is not, for a softened
    // distance, and for the plain distance r of an accepted cell when the side
    // is at least theta 2^-39.  The cell has l < theta d and l >= side 2^-21; d
    // along its longest axis is at least d / sqrt(3); the centre's low part,
    // half a unit in the last place of the high part at most, takes at most half of
    // that away; so r^2 > l^2 / (12 theta^2) >= 2^-124 where 2^-126 is normal.
    const float eps2 = eps * eps;
    const bool full = !(eps2 >= FLT_MIN && t.side >= (double)theta * 0x1p-39);
    // the interaction counts cost about 15% of the walk: only profiled walks
    // take them
    auto pick = [&](auto plain, auto counting) { return ws.profile ? counting : plain; };
    auto kern = use_quad ? (full ? pick(walk_kernel<true, false, true>, walk_kernel<true, true, true>)
                                 : pick(walk_kernel<true, false, false>, walk_kernel<true, true, false>))
                         : (full ? pick(walk_kernel<false, false, true>, walk_kernel<false, true, true>)
                                 : pick(walk_kernel<false, false, false>, walk_kernel<false, true, false>));
    launch_after(kern, dim3(kWalkBlocks), dim3(kWalkThreads), 0, s, T, groups, ctr, stacks, theta, eps2, acc, ws.info);
    ++g_launches;
    return cudaGetLastError();
}

}  // namespace tb
