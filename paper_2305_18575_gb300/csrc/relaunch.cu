// relaunch.cu -- the relaunch of a search, shaped for throughput: it takes over
// the levels that outgrow the first launch, and continues or starts every
// search that launch cannot hold; and the rebuilding of the uniqueness table.
#include "launch.h"
#include "search.cuh"

namespace rei {

// Two CTAs of 16 warps an SM at 64 registers.  One of 128 registers for 2-word
// languages, whose tiles keep four candidates a lane with their table slots in
// registers (|ic| 36-42 to cost 20: 8.5 ms, with two CTAs, which spill into the
// L1, 8.8 ms; 1-word languages, bound by the L2, took 98.1 ms with one instead of
// 78.7, 4-word ones 4.87 ms instead of 3.73), and from 20 words on, where the warps'
// tiles leave room for one CTA an SM anyway (32 words to cost 12: 8.3 -> 7.0 ms; 8
// to 16 words 2.49 ms, with one CTA 2.74).
// The two CTAs may also be one of 32 warps: searches side by side take one an SM
// (solve_warps_max).
template <uint32_t WC>
__global__ void __launch_bounds__(WC == kWidest || WC == 2 ? kSolveThreads : 2 * kSolveThreads, 1)
    k_solve(const __grid_constant__ SolveJob J) {
    uint32_t bar_epoch = 0;
    solve_body<WC>(J, bar_epoch);
}

// the relaunch of a width
static const void *solve_kernel(uint32_t W) {
    return W == 1   ? (const void *)k_solve<1>
           : W == 2 ? (const void *)k_solve<2>
           : W == 4 ? (const void *)k_solve<4>
           : W < kWidest ? (const void *)k_solve<kWide>
                         : (const void *)k_solve<kWidest>;
}

// rebuild the uniqueness table after the cache grew (all entries are distinct)
__global__ void k_rehash(const __grid_constant__ SolveJob J, uint32_t count) {
    const uint32_t W = J.W;
    for (uint64_t k = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; k < count;
         k += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t *c = J.cs + k * W;
        if (J.exact) {
            J.used[k] = (uint32_t)exact_fill(J, exact_key(c, W), (uint32_t)k);
        } else {
            const uint64_t h = cs_hash(c, W, 1);
            const unsigned long long v = ((uint64_t)(uint32_t)(h >> 32) << 32) | (uint32_t)k;
            uint32_t p = probe_first(h, J.table_mask);
            while (atomicCAS(&J.table[p], kEmpty, v) != kEmpty) p = probe_next(p, (uint32_t)J.table_mask);
            J.used[k] = p;
        }
        if (J.seen) atomicOr(J.seen + (c[0] >> 5), 1u << (c[0] & 31u));
    }
}

cudaError_t launch_solve(const SolveJob *job, uint32_t grid, uint32_t threads, size_t smem,
                         cudaStream_t stream) {
    const void *fn = solve_kernel(job->W);
    cudaError_t e = prepare(fn);
    if (e != cudaSuccess) return e;
    void *args[] = {(void *)job};
    return cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(threads), args, smem, stream);
}

cudaError_t solve_occupancy(uint32_t W, uint32_t threads, size_t smem, int *blocks_per_sm) {
    return occupancy(solve_kernel(W), threads, smem, blocks_per_sm);
}

cudaError_t solve_smem_max(uint32_t W, size_t *bytes) { return smem_max_of(solve_kernel(W), bytes); }

uint32_t solve_warps_max(uint32_t W) { return (W == 2 || W >= kWidest ? 1 : 2) * kSolveThreads / 32; }

cudaError_t launch_rehash(const SolveJob *job, uint32_t count, uint32_t grid, cudaStream_t stream) {
    k_rehash<<<grid, 256, 0, stream>>>(*job, count);
    return cudaGetLastError();
}

}  // namespace rei
