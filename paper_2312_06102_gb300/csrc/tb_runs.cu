// tb_runs.cu -- the last step of the key sort (Sec. 2.3 step 2).
//
// The global radix passes order the (key, index) pairs stably by the upper
// bits of the key, key >> shift0.  What is left is to order every run of equal
// upper bits by the low shift0 bits, stably.  With 40 upper bits the runs of
// the tree workloads are short (most have one element; in a 2^27-particle
// clustered set about one in a million is longer than 128), so each run is
// finished where it lies:
//   run_sort_kernel  : per tile of 2048 positions (plus 128 beyond it), one
//                      bit per position marks where a run starts (a warp
//                      ballot per 32 positions); every run that starts in the
//                      tile and holds at most 128 keys is ordered in place,
//                      each member going to its rank by
//                      (low bits, position); longer runs are queued, and each
//                      tile notes whether any of its keys is smaller than its
//                      predecessor in the same run (a descent);
//   long_run_kernel  : each queued run that contains a descent is sorted by
//                      its low bits by one block with the block-local LSD sort
//                      (3 passes of 8 bits); runs without one (for instance
//                      identical keys) are already in order.
// The outcome equals a stable sort of the whole keys: equal upper bits stay
// in index order from the passes, and the run step orders them by the rest.
#include "tb_runs.cuh"

namespace tb {

namespace {

constexpr int kRunThreads = 256;

__global__ void __launch_bounds__(kRunThreads)
    run_sort_kernel(uint64_t *__restrict__ keys, int32_t *__restrict__ vals, int64_t n, int shift0,
                    RunBuffers rb, DevInfo *info) {
    after_previous();
    __shared__ RunSmem sm;
    const int64_t s = (int64_t)blockIdx.x * kRunTile;
    const bool desc = run_tile<kRunThreads>(keys, vals, 0, s, n, shift0, sm, [&](int64_t a) {
        rb.queue[atomicAdd(&info->misc_ctr[5], 1u)] = (int32_t)a;
    });
    if (threadIdx.x == 0) rb.desc[blockIdx.x] = desc ? 1 : 0;
}

__global__ void __launch_bounds__(kCtaThreads, 1)
    long_run_kernel(uint64_t *keys, int32_t *vals, uint64_t *alt_k, int32_t *alt_v, int64_t n,
                    int shift0, RunBuffers rb, DevInfo *info) {
    after_previous();
    // after a look-back that gave up the keys are not in order: the search for a
    // run's end could then take in another queued run, and two blocks would sort
    // the same keys, each with digit counts that no longer hold
    if (info->status & kErrTimeout) return;
    extern __shared__ __align__(16) unsigned char raw[];
    CtaSortShared &sm = *reinterpret_cast<CtaSortShared *>(raw);
    __shared__ uint32_t s_q;
    const uint32_t nq = *(volatile uint32_t *)&info->misc_ctr[5];
    for (;;) {
        if (threadIdx.x == 0) s_q = atomicAdd(&info->misc_ctr[6], 1u);
        __syncthreads();
        const uint32_t q = s_q;
        __syncthreads();
        if (q >= nq) return;
        sort_long_run<kCtaThreads>(keys, vals, alt_k, alt_v, n, shift0, rb.queue[q], rb.desc, sm);
    }
}

}  // namespace

cudaError_t launch_runs(uint64_t *keys, int32_t *vals, uint64_t *alt_k, int32_t *alt_v, int64_t n,
                        int shift0, int32_t *long_runs, Workspace &ws, cudaStream_t s) {
    const RunBuffers rb = run_buffers(long_runs, n);
    if (shift0 <= 0 || n <= 1) return cudaSuccess;
    if (shift0 > 32) return cudaErrorInvalidValue;   // the run step ranks the low bits as 32-bit words
    static std::atomic<uint64_t> attr_done{0};
    cudaError_t e = once_on_device(attr_done, [] { return allow_smem(long_run_kernel, sizeof(CtaSortShared), false); });
    if (e != cudaSuccess) return e;
    const int64_t tiles = (n + kRunTile - 1) / kRunTile;
    launch_after(run_sort_kernel, dim3((unsigned)tiles), dim3(kRunThreads), 0, s, keys, vals, n, shift0, rb, ws.info);
    ++g_launches;
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    launch_after(long_run_kernel, dim3(152), dim3(kCtaThreads), sizeof(CtaSortShared), s, keys, vals, alt_k, alt_v, n, shift0,
                                                                   rb, ws.info);
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t load_run_kernels() {
    cudaError_t e = load_kernel(run_sort_kernel);
    return e == cudaSuccess ? load_kernel(long_run_kernel) : e;
}

// int32 words for the queue and the tile flags of n keys
int64_t long_run_capacity(int64_t n) {
    return run_queue_cap(n) + (n / kRunTile + 1 + 3) / 4 + 1;
}

}  // namespace tb
