// tb_keys.cu -- root cell and particle keys (Sec. 2.2; Sec. 2.3 step 1).
//
// root_kernel : per-axis FP32 min / max of the positions and a non-finite
//               flag; the last block to finish derives the root cube
//               (corner lo, side L = largest extent, scale 2^21 / L) and
//               resets the per-build counters.
// keys_kernel : 21-bit quantisation per axis, bit interleave below a leading
//               1, and the digit histograms of every radix-sort pass (the
//               histogram of a digit does not depend on the order of the
//               keys, so all passes are counted in this one read).  The last
//               block turns the histograms into exclusive digit offsets.
//
// Both read the [n][3] FP32 positions four particles (three float4) per
// thread step when the array is 16-byte aligned.
#include <cfloat>
#include <cmath>

#include "tb_device.cuh"

namespace tb {

namespace {

constexpr int kRootThreads = 256;
constexpr int kKeysThreads = 256;

__device__ __forceinline__ bool finite_f(float x) { return fabsf(x) <= FLT_MAX; }

struct Box {
    float mn[3], mx[3];
    uint32_t bad;
    __device__ void init() {
        for (int a = 0; a < 3; ++a) { mn[a] = FLT_MAX; mx[a] = -FLT_MAX; }
        bad = 0;
    }
    __device__ void add(float x, int a) {
        bad |= !finite_f(x);
        mn[a] = fminf(mn[a], x);
        mx[a] = fmaxf(mx[a], x);
    }
};

__global__ void __launch_bounds__(kRootThreads) root_kernel(const float *__restrict__ pos, int64_t n,
                                                            bool vec, float *__restrict__ part,
                                                            DevInfo *info, uint32_t *hist,
                                                            int hist_len, bool pow2) {
    after_previous();
    Box b;
    b.init();
    const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int64_t done = 0;
    if (vec) {
        const float4 *p4 = reinterpret_cast<const float4 *>(pos);
        const int64_t groups = n / 4;
#pragma unroll 2
        for (int64_t g = tid; g < groups; g += stride) {
            float4 a = __ldcs(p4 + 3 * g), c = __ldcs(p4 + 3 * g + 1), d = __ldcs(p4 + 3 * g + 2);
            b.add(a.x, 0); b.add(a.y, 1); b.add(a.z, 2); b.add(a.w, 0);
            b.add(c.x, 1); b.add(c.y, 2); b.add(c.z, 0); b.add(c.w, 1);
            b.add(d.x, 2); b.add(d.y, 0); b.add(d.z, 1); b.add(d.w, 2);
        }
        done = groups * 4;
    }
    for (int64_t i = done + tid; i < n; i += stride)
        for (int a = 0; a < 3; ++a) b.add(pos[3 * i + a], a);

    // block reduction
    for (int off = 16; off > 0; off >>= 1) {
        for (int a = 0; a < 3; ++a) {
            b.mn[a] = fminf(b.mn[a], __shfl_xor_sync(0xffffffffu, b.mn[a], off));
            b.mx[a] = fmaxf(b.mx[a], __shfl_xor_sync(0xffffffffu, b.mx[a], off));
        }
        b.bad |= __shfl_xor_sync(0xffffffffu, b.bad, off);
    }
    __shared__ float s_red[kRootThreads / 32][8];
    __shared__ bool s_last;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) {
        for (int a = 0; a < 3; ++a) { s_red[warp][a] = b.mn[a]; s_red[warp][3 + a] = b.mx[a]; }
        s_red[warp][6] = __uint_as_float(b.bad);
    }
    __syncthreads();
    if (threadIdx.x < 7) {
        float v = s_red[0][threadIdx.x];
        for (int w = 1; w < kRootThreads / 32; ++w) {
            float u = s_red[w][threadIdx.x];
            if (threadIdx.x < 3) v = fminf(v, u);
            else if (threadIdx.x < 6) v = fmaxf(v, u);
            else v = __uint_as_float(__float_as_uint(v) | __float_as_uint(u));
        }
        part[blockIdx.x * 8 + threadIdx.x] = v;
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = (atomicAdd(&info->misc_ctr[0], 1u) == gridDim.x - 1);
    __syncthreads();
    if (!s_last) return;
    __threadfence();

    // last block: combine the per-block partials and derive the root cube
    // every thread folds a stride of the partials, then the block reduces
    {
        Box c;
        c.init();
        for (unsigned k = threadIdx.x; k < gridDim.x; k += blockDim.x) {
            const float4 lo = __ldcg(reinterpret_cast<const float4 *>(part + 8 * k));
            const float4 hi = __ldcg(reinterpret_cast<const float4 *>(part + 8 * k + 4));
            c.mn[0] = fminf(c.mn[0], lo.x); c.mn[1] = fminf(c.mn[1], lo.y); c.mn[2] = fminf(c.mn[2], lo.z);
            c.mx[0] = fmaxf(c.mx[0], lo.w); c.mx[1] = fmaxf(c.mx[1], hi.x); c.mx[2] = fmaxf(c.mx[2], hi.y);
            c.bad |= __float_as_uint(hi.z);
        }
        for (int off = 16; off > 0; off >>= 1) {
            for (int a = 0; a < 3; ++a) {
                c.mn[a] = fminf(c.mn[a], __shfl_xor_sync(0xffffffffu, c.mn[a], off));
                c.mx[a] = fmaxf(c.mx[a], __shfl_xor_sync(0xffffffffu, c.mx[a], off));
            }
            c.bad |= __shfl_xor_sync(0xffffffffu, c.bad, off);
        }
        __syncthreads();   // s_red's block partials were read above
        if (lane == 0) {
            for (int a = 0; a < 3; ++a) { s_red[warp][a] = c.mn[a]; s_red[warp][3 + a] = c.mx[a]; }
            s_red[warp][6] = __uint_as_float(c.bad);
        }
        __syncthreads();
        if (threadIdx.x < 7) {
            float v = s_red[0][threadIdx.x];
            for (int w = 1; w < kRootThreads / 32; ++w) {
                const float u = s_red[w][threadIdx.x];
                if (threadIdx.x < 3) v = fminf(v, u);
                else if (threadIdx.x < 6) v = fmaxf(v, u);
                else v = __uint_as_float(__float_as_uint(v) | __float_as_uint(u));
            }
            s_red[0][threadIdx.x] = v;
        }
    }
    for (int i = threadIdx.x; i < hist_len; i += blockDim.x) hist[i] = 0;
    __syncthreads();
    if (threadIdx.x == 0) {
        begin_build(info, root_cube(&s_red[0][0], &s_red[0][3], pow2), &s_red[0][3],
                    __float_as_uint(s_red[0][6]) != 0u);
        __threadfence();
        info->misc_ctr[0] = 0;
    }
}

template <int RADIX_BITS, bool HILBERT>
__global__ void __launch_bounds__(kKeysThreads, 6) keys_kernel(const float *__restrict__ pos,
                                                            const float *__restrict__ mass,
                                                            float m_eq, int64_t n, bool vec,
                                                            uint64_t *__restrict__ keys,
                                                            float4 *__restrict__ xm,
                                                            uint32_t *hist, int passes, int shift0,
                                                            DevInfo *info) {
    after_previous();
    constexpr int RADIX = 1 << RADIX_BITS;
    extern __shared__ uint32_t s_hist[];   // [passes][RADIX], then the Hilbert table
    uint16_t *tab = reinterpret_cast<uint16_t *>(s_hist + passes * RADIX);
    if constexpr (HILBERT) hilbert_table(tab);
    for (int i = threadIdx.x; i < passes * RADIX; i += blockDim.x) s_hist[i] = 0;
    __shared__ float s_lo[3];
    __shared__ float s_shi, s_slo;
    __shared__ double s_scale;
    __shared__ bool s_exact, s_f32, s_last;
    if (threadIdx.x == 0) {
        for (int a = 0; a < 3; ++a) s_lo[a] = info->lo[a];
        s_shi = info->s_hi;
        s_slo = info->s_lo;
        s_scale = info->scale;
        s_exact = info->exact_only != 0;
        s_f32 = info->s_fp32 != 0;
    }
    __syncthreads();
    const float lx = s_lo[0], ly = s_lo[1], lz = s_lo[2];
    const float shi = s_shi, slo = s_slo;
    const double sc = s_scale;
    const bool exact = s_exact, f32 = s_f32;

    auto count = [&](uint64_t k) {
        for (int p = 0; p < passes; ++p)
            atomicAdd(&s_hist[p * RADIX + (int)((k >> (shift0 + p * RADIX_BITS)) & (RADIX - 1))], 1u);
    };
    auto key_of = [&](float x, float y, float z) {
        const uint32_t qx = quantise(x, lx, shi, slo, sc, exact, f32),
                       qy = quantise(y, ly, shi, slo, sc, exact, f32),
                       qz = quantise(z, lz, shi, slo, sc, exact, f32);
        const uint64_t m = morton_key(qx, qy, qz);
        return HILBERT ? hilbert_of_morton(m, tab) : m;
    };

    const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int64_t done = 0;
    if (vec) {
        const float4 *p4 = reinterpret_cast<const float4 *>(pos);
        ulonglong2 *k2 = reinterpret_cast<ulonglong2 *>(keys);
        const int64_t groups = n / 4;
        const float4 *m4 = reinterpret_cast<const float4 *>(mass);
        for (int64_t g = tid; g < groups; g += stride) {
            float4 a = __ldcs(p4 + 3 * g), c = __ldcs(p4 + 3 * g + 1), d = __ldcs(p4 + 3 * g + 2);
            float4 w = mass ? __ldcs(m4 + g) : make_float4(m_eq, m_eq, m_eq, m_eq);
            uint64_t k0 = key_of(a.x, a.y, a.z);
            uint64_t k1 = key_of(a.w, c.x, c.y);
            uint64_t k2v = key_of(c.z, c.w, d.x);
            uint64_t k3 = key_of(d.y, d.z, d.w);
            k2[2 * g] = make_ulonglong2(k0, k1);
            k2[2 * g + 1] = make_ulonglong2(k2v, k3);
            xm[4 * g] = make_float4(a.x, a.y, a.z, w.x);
            xm[4 * g + 1] = make_float4(a.w, c.x, c.y, w.y);
            xm[4 * g + 2] = make_float4(c.z, c.w, d.x, w.z);
            xm[4 * g + 3] = make_float4(d.y, d.z, d.w, w.w);
            count(k0); count(k1); count(k2v); count(k3);
        }
        done = groups * 4;
    }
    for (int64_t i = done + tid; i < n; i += stride) {
        float x = pos[3 * i], y = pos[3 * i + 1], z = pos[3 * i + 2];
        uint64_t k = key_of(x, y, z);
        keys[i] = k;
        xm[i] = make_float4(x, y, z, mass ? mass[i] : m_eq);
        count(k);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < passes * RADIX; i += blockDim.x)
        if (s_hist[i]) atomicAdd(&hist[i], s_hist[i]);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = (atomicAdd(&info->misc_ctr[4], 1u) == gridDim.x - 1);
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // last block: counts -> exclusive offsets, a warp per pass, each lane a
    // run of digits (one pass after another, with block barriers, took 4 us
    // more: most of the kernel for a small set)
    const int lane = threadIdx.x & 31;
    for (int p = threadIdx.x >> 5; p < passes; p += kKeysThreads / 32) {
        constexpr int Q = RADIX / 128;   // uint4 per lane
        uint4 *row = reinterpret_cast<uint4 *>(hist + p * RADIX) + lane * Q;
        uint32_t sum = 0;
#pragma unroll 2
        for (int j = 0; j < Q; ++j) {
            const uint4 v = __ldcg(row + j);
            sum += v.x + v.y + v.z + v.w;
        }
        uint32_t x = sum;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, off);
            if (lane >= off) x += y;
        }
        x -= sum;
#pragma unroll 2
        for (int j = 0; j < Q; ++j) {
            const uint4 v = __ldcg(row + j);
            row[j] = make_uint4(x, x + v.x, x + v.x + v.y, x + v.x + v.y + v.z);
            x += v.x + v.y + v.z + v.w;
        }
    }
    if (threadIdx.x == 0) info->misc_ctr[4] = 0;
}

}  // namespace

int64_t bbox_grid() { return 152 * 4; }

cudaError_t launch_root(const float *pos, int64_t n, Workspace &ws, int hist_len, cudaStream_t s) {
    const bool vec = (reinterpret_cast<uintptr_t>(pos) & 15u) == 0;
    int64_t grid = bbox_grid();
    int64_t need = (n + 4 * kRootThreads - 1) / (4 * kRootThreads);
    if (need < grid) grid = need < 1 ? 1 : need;
    root_kernel<<<(unsigned)grid, kRootThreads, 0, s>>>(pos, n, vec, ws.bbox_part, ws.info, ws.hist,
                                                        hist_len, ws.root_pow2);
    ++g_launches;
    return cudaGetLastError();
}

template <int B, bool H>
static cudaError_t keys_impl(const float *pos, const float *mass, int64_t n, uint64_t *keys,
                             Workspace &ws, int passes, int shift0, cudaStream_t s) {
    const bool vec = (reinterpret_cast<uintptr_t>(pos) & 15u) == 0 &&
                     (reinterpret_cast<uintptr_t>(mass) & 15u) == 0 &&
                     (reinterpret_cast<uintptr_t>(keys) & 15u) == 0;
    const float m_eq = (float)(1.0 / (double)(n > 0 ? n : 1));
    size_t smem = sizeof(uint32_t) * passes * (1 << B) + (H ? sizeof(uint16_t) * kHilbertTab : 0);
    static std::atomic<uint64_t> attr_done{0};
    const cudaError_t e = once_on_device(attr_done, [] { return allow_smem(keys_kernel<B, H>, 64 * 1024, false); });
    if (e != cudaSuccess) return e;
    // six resident blocks per SM (42 registers), one wave
    int64_t grid = 152 * 6;
    int64_t need = (n + 4 * kKeysThreads - 1) / (4 * kKeysThreads);
    if (need < grid) grid = need < 1 ? 1 : need;
    launch_after(keys_kernel<B, H>, dim3((unsigned)grid), dim3(kKeysThreads), smem, s, pos, mass, m_eq, n, vec, keys, ws.xm,
                                                              ws.hist, passes, shift0, ws.info);
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_keys(const float *pos, const float *mass, int64_t n, uint64_t *keys,
                        Workspace &ws, const SortCfg &cfg, int key_order, cudaStream_t s) {
    const SortPlan plan = sort_plan(cfg);
    const int passes = plan.passes, shift0 = plan.shift0;
    const bool h = key_order == TB_KEYS_HILBERT;
    switch (cfg.radix_bits) {
        case 8: return h ? keys_impl<8, true>(pos, mass, n, keys, ws, passes, shift0, s)
                         : keys_impl<8, false>(pos, mass, n, keys, ws, passes, shift0, s);
        case 9: return h ? keys_impl<9, true>(pos, mass, n, keys, ws, passes, shift0, s)
                         : keys_impl<9, false>(pos, mass, n, keys, ws, passes, shift0, s);
        case 10: return h ? keys_impl<10, true>(pos, mass, n, keys, ws, passes, shift0, s)
                          : keys_impl<10, false>(pos, mass, n, keys, ws, passes, shift0, s);
        case 11: return h ? keys_impl<11, true>(pos, mass, n, keys, ws, passes, shift0, s)
                          : keys_impl<11, false>(pos, mass, n, keys, ws, passes, shift0, s);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t load_key_kernels() {
    cudaError_t e = load_kernel(root_kernel);
    return e == cudaSuccess ? load_kernel(keys_kernel<8, false>) : e;
}

// (x, y, z, m) of each particle in input order, for moment calls whose
// arrays differ from the ones the keys were made from.
__global__ void pack_kernel(const float *__restrict__ pos, const float *__restrict__ mass,
                            float m_eq, int64_t n, float4 *__restrict__ xm) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += stride)
        xm[i] = make_float4(pos[3 * i], pos[3 * i + 1], pos[3 * i + 2], mass ? mass[i] : m_eq);
}

cudaError_t launch_pack(const float *pos, const float *mass, int64_t n, float4 *xm,
                        cudaStream_t s) {
    const float m_eq = (float)(1.0 / (double)(n > 0 ? n : 1));
    int64_t grid = (n + 255) / 256;
    if (grid > 152 * 8) grid = 152 * 8;
    if (grid < 1) grid = 1;
    pack_kernel<<<(unsigned)grid, 256, 0, s>>>(pos, mass, m_eq, n, xm);
    ++g_launches;
    return cudaGetLastError();
}


}  // namespace tb
