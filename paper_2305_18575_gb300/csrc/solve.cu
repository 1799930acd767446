// solve.cu -- a problem staged and searched in one launch (the plain solve).
#include "launch.h"
#include "search.cuh"

namespace rei {

// chunk size for W-word languages (the host's rule for the plain launch)
__device__ __forceinline__ uint64_t auto_chunk(uint32_t W) {
    uint64_t c = (1ull << 28) / (4ull * W);
    if (c < (1ull << 16)) c = 1ull << 16;
    if (c > (1ull << 22)) c = 1ull << 22;
    return c;
}

// Stage (CTA 0, the strings and the staging scratch in its shared memory),
// size the search from the staged problem, then search, all in one launch.
// A problem whose staging or search the launch cannot hold (|ic| > 2048, a
// guide table beyond the pair buffer, shared memory) ends with ST_RESTAGE.
static_assert(sizeof(StageInfo) % 8 == 0 && offsetof(SolveState, launch) % 8 == 0, "state reset by 8-byte words");

// CTA 0's last step: the final state, tokens and staging report to the host
__device__ void state_out(const FuseArgs &F) {
    if (!F.host_out) return;
    __syncthreads();
    const unsigned long long *src = reinterpret_cast<const unsigned long long *>(F.tmpl.st);
    for (uint64_t i = threadIdx.x; i < F.out_words; i += blockDim.x) F.host_out[i] = ld_relaxed_u64(src + i);
    __threadfence_system();
}

__global__ void __launch_bounds__(kFusedThreads, 1) k_solve_fused(const __grid_constant__ FuseArgs F) {
    extern __shared__ __align__(16) uint8_t smem_raw[];
    __shared__ SolveJob J;
    __shared__ uint32_t s_go;
    SolveState *st = F.tmpl.st;
    uint32_t bar_epoch = 0;
#ifdef REI_TIMING
    const unsigned long long t_begin = globaltimer_ns();
    const long long c_begin = clock64();
#endif
    if (blockIdx.x == 0) {
        // this launch's state starts from zero (the state buffer holds the
        // previous launch's; the other CTAs read none of it before the release
        // below), and so does the level table
        {
            unsigned long long *w = reinterpret_cast<unsigned long long *>(st);
            for (uint32_t i = threadIdx.x; i < offsetof(SolveState, launch) / 8; i += blockDim.x) w[i] = 0;
            unsigned long long *si = reinterpret_cast<unsigned long long *>(F.sj.info);
            for (uint32_t i = threadIdx.x; i < sizeof(StageInfo) / 8; i += blockDim.x) si[i] = 0;
        }
        // (CTA 0 keeps the job in shared memory)
        {
            const unsigned long long *src = reinterpret_cast<const unsigned long long *>(&F.tmpl);
            unsigned long long *dst = reinterpret_cast<unsigned long long *>(&J);
            for (uint32_t i = threadIdx.x; i < sizeof(SolveJob) / 8; i += blockDim.x) dst[i] = src[i];
        }
        for (uint32_t c = threadIdx.x; c < F.tmpl.max_cost + 2; c += blockDim.x) {
            F.tmpl.lvl_start[c] = 0;
            F.tmpl.lvl_count[c] = 0;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            st->level = F.tmpl.cmin;
            st->found = kNone;
            st->partial_level = F.tmpl.max_cost + 1;
        }
        {
#ifdef REI_TIMING
            REI_TSPAN_BEGIN(t_sr);
#endif
            StageSmem M;
            stage_layout(kServeMaxIC, kServeMaxBytes, smem_raw, &M);
            stage_run(F.sj, M);
            __syncthreads();
            REI_TSPAN_END(st, t_sr, 22);
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            // (completed in place: copying the job through one thread's
            // registers took 3 us of every solve)
            const StageInfo I = *F.sj.info;
            SolveJob &j = J;
            bool ok = I.status == SE_OK;
            if (ok) {
                j.n = I.n;
                j.W = I.W;
                j.G = I.G;
                j.max_len = I.max_len;
                j.n_pos_set = I.n_pos_set;
                j.pos_eps = I.pos_eps;
                j.neg_eps = I.neg_eps;
                const uint32_t W = I.W;
                j.cap = umin64(F.mem_budget / (4ull * W + 28), 0x7FFF0000ull);
                j.exact = F.tmpl.exact && W <= 2 && I.n <= 62 ? 1u : 0u;
                j.seen = j.exact && W == 1 && I.n <= F.seen_bits ? F.seen : nullptr;
                j.direct = j.exact && W == 1 && (1ull << I.n) <= F.table_slots ? 1u : 0u;
                // (a slot per language: the table is as many words)
                if (j.direct) j.table_mask = (1ull << I.n) - 1;
                j.handover = F.handover;
                const uint64_t tmax = F.table_slots / 2;
                j.cache_alloc = umin64(umin64(j.cap, F.rows_alloc), umin64(F.cs_words / W, tmax / 2));
                uint64_t ch = F.chunk_opt ? F.chunk_opt : auto_chunk(W);
                ch = umin64(umin64(ch, 1ull << 24), umin64(F.tmp_words / W, F.pend_cap));
                j.chunk_max = umin64(ch, tmax - j.cache_alloc);
                // shared memory: guide table there if it fits, then the
                // largest shared-memory start that fits
                const uint32_t warps = blockDim.x / 32;
                j.gt_in_smem = search_smem_bytes(W, I.n, I.G, I.max_len, j.seg_cap, true, warps, 0) <= F.smem_cap;
                j.small_rows = 0;
                if (F.small_opt && W <= kSmallMaxW) {
                    uint32_t r = F.small_opt != 0xFFFFFFFFu ? F.small_opt : W <= 2 ? 4096u : W <= 4 ? 2048u : 1024u;
                    for (; r >= 256; r >>= 1)
                        if (search_smem_bytes(W, I.n, I.G, I.max_len, j.seg_cap, j.gt_in_smem, warps, r) <= F.smem_cap)
                            break;
                    if (r >= 256) j.small_rows = r;
                }
                ok = j.cache_alloc >= 1 && j.chunk_max >= 1 &&
                     search_smem_bytes(W, I.n, I.G, I.max_len, j.seg_cap, j.gt_in_smem, warps, j.small_rows) <=
                         F.smem_cap;
            }
            if (!ok) st->status = ST_RESTAGE;
            s_go = ok ? 1u : 0u;
        }
        __syncthreads();
        // the job for the other CTAs, written by every thread; then the
        // release: the job and the fresh state are in place
        {
            const unsigned long long *src = reinterpret_cast<const unsigned long long *>(&J);
            unsigned long long *dst = reinterpret_cast<unsigned long long *>(F.job);
            for (uint32_t i = threadIdx.x; i < sizeof(SolveJob) / 8; i += blockDim.x) dst[i] = src[i];
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            atomicExch(&st->launch, F.launch_id);
        }
        if (!s_go) {
            state_out(F);
            return;
        }
    } else {
        // the other CTAs wait for CTA 0's release of this launch (a stale id
        // in the state is always smaller: ids only grow), then take the job
        if (threadIdx.x == 0) {
            const unsigned long long t0 = globaltimer_ns();
            uint32_t nap = 64, go = 0;
            for (;;) {
                if (ld_acquire_u64(&st->launch) == F.launch_id) {
                    go = 1;
                    break;
                }
                if (globaltimer_ns() - t0 > kBarrierWaitNs) break;
                __nanosleep(nap);
                if (nap < REI_CMD_NAP) nap <<= 1;
            }
            __threadfence();
            if (go && ld_relaxed_u32(&st->status) != ST_RUNNING) go = 0;
            if (!go && ld_acquire_u64(&st->launch) != F.launch_id) {
                // (never released: the launch ends with an error for the host)
                atomicCAS(&st->err, 0u, 4u);
                atomicExch(&st->status, (uint32_t)ST_TIMEOUT);
            }
            s_go = go;
        }
        __syncthreads();
        if (!s_go) return;
        const unsigned long long *src = reinterpret_cast<const unsigned long long *>(F.job);
        unsigned long long *dst = reinterpret_cast<unsigned long long *>(&J);
        for (uint32_t i = threadIdx.x; i < sizeof(SolveJob) / 8; i += blockDim.x) dst[i] = ld_relaxed_u64(src + i);
        __syncthreads();
    }
#ifdef REI_TIMING
    if (blockIdx.x == 0 && threadIdx.x == 0) st->t_sub[10] = globaltimer_ns() - t_begin;
#endif
    solve_body<kAnyWidth>(J, bar_epoch);
#ifdef REI_TIMING
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        st->t_sub[11] = globaltimer_ns() - t_begin;
        st->t_sub[38] = (unsigned long long)(clock64() - c_begin);
    }
#endif
    if (blockIdx.x == 0) state_out(F);
}

cudaError_t launch_solve_fused(const FuseArgs *args, uint32_t grid, uint32_t threads, size_t smem,
                               cudaStream_t stream) {
    cudaError_t e = prepare((const void *)k_solve_fused);
    if (e != cudaSuccess) return e;
    void *args_[] = {(void *)args};
    return cudaLaunchCooperativeKernel((const void *)k_solve_fused, dim3(grid), dim3(threads), args_, smem, stream);
}

cudaError_t solve_fused_occupancy(uint32_t threads, size_t smem, int *blocks_per_sm) {
    return occupancy((const void *)k_solve_fused, threads, smem, blocks_per_sm);
}

// shared memory of a search CTA (the host's sizing)
size_t solve_smem_bytes(uint32_t W, uint32_t n, uint32_t G, uint32_t max_len, uint32_t seg_cap, bool gt_in_smem,
                        uint32_t warps, uint32_t small_rows) {
    return search_smem_bytes(W, n, G, max_len, seg_cap, gt_in_smem, warps, small_rows);
}

}  // namespace rei
