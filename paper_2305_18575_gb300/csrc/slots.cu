// slots.cu -- searches in memory slots: the batched form, the groups that
// continue its parked searches, and the served form.
#include "launch.h"
#include "search.cuh"

namespace rei {

// ---------------------------------------------------------------------------
// the batched search: one launch for many staged problems; every CTA takes
// problems from a queue and solves each one on its own (its own memory slot,
// no grid-wide synchronisation), with the same leader code as k_solve.

// a problem's search in memory slot `slot`: its cache, table, chunk
// workspace, level table, state and answer-walk stack (one CTA's share)
__device__ void bind_slot(SolveJob &J, const SlotMem &m, uint32_t slot) {
    const uint64_t so = slot;
    J.cs = m.cs + so * m.cs_words;
    J.bp_op = m.bp_op + so * m.rows;
    J.bp_l = m.bp_l + so * m.rows;
    J.bp_r = m.bp_r + so * m.rows;
    J.used = m.used + so * m.rows;
    J.cache_alloc = umin64(J.cap, m.cs_words / J.W < m.rows ? m.cs_words / J.W : m.rows);
    J.table = m.table + so * m.table_slots;
    J.table_mask = m.table_slots - 1;
    J.tmp = m.tmp + so * m.tmp_words;
    J.chunk_max = umin64(m.chunk, m.tmp_words / J.W);
    J.pending = m.pending + so * m.chunk;
    J.slotpos = m.slotpos + so * m.chunk;
    J.bitmap = m.bitmap + so * ((m.chunk + 31) / 32);
    J.blk = m.blk + so;
    J.lvl_start = m.lvl + so * 2 * (kMaxCost + 2);
    J.lvl_count = J.lvl_start + (kMaxCost + 2);
    J.st = m.state + so;
    J.tstack = m.tstack + so * 4 * (kMaxCost + 2);
    J.trace = nullptr;
}

// a slot search's report (thread 0)
__device__ void report_slot(const SolveJob &J, uint32_t status, uint32_t slot, unsigned long long ns, BatchOut &o) {
    const SolveState *st = J.st;
    o.status = status;
    o.cost = st->ans_cost;
    o.tree_len = st->tree_len;
    o.candidates = st->candidates;
    o.unique = st->unique_done;
    o.levels = st->level;
    for (int k = 0; k < 5; k++) o.cand_op[k] = st->cand_op[k];
    o.ns = ns;
    o.slot = slot;
    o.need_rows = status == ST_NEED_MEM ? st->need_rows : 0u;
}

// Solve the problem whose job (staged data, costs) is in shared memory J,
// in memory slot `slot`, on this CTA alone; the report goes to *out and the
// tree to J.tree.  Returns the search's status (every thread).  With
// ST_NEED_MEM (the time allowance ran out or the slot is too small) the slot
// keeps the cache rows, back-pointers, level table and state for the host to
// continue from; its survivor bitmap is emptied.  keep_table: its uniqueness
// table stays in the slot as well (the search continues there, or the host
// empties the table when it continues elsewhere); else it is emptied too.
__device__ uint32_t solve_in_slot(SolveJob &J, const SlotMem &m, uint32_t slot, BatchOut *out, uint8_t *smem_raw,
                              Plan *s_plan, uint32_t *s_red, uint64_t *s_tiles, unsigned long long *s_found,
                              uint32_t *s_marked, Lead *L, uint64_t yield_ns, bool keep_table) {
    const uint32_t tid = threadIdx.x;
    const unsigned long long t_start = globaltimer_ns();
    if (tid == 0) {
        J.yield_ns = yield_ns;
        J.t_start = t_start;
        bind_slot(J, m, slot);
        J.solo_tiles = 0xFFFFFFFFu;
        J.team_base = blockIdx.x;
        J.team_size = 1;
    }
    __syncthreads();
    SolveState *st = J.st;
    // fresh search state and level table for this problem
    for (uint32_t c = tid; c < 2 * (kMaxCost + 2); c += blockDim.x) J.lvl_start[c] = 0;
    if (tid == 0) {
        SolveState z{};
        z.status = ST_RUNNING;
        z.level = J.cmin;
        z.found = kNone;
        z.partial_level = J.max_cost + 1;
        *st = z;
    }
    __threadfence();
    __syncthreads();
    Shared S;
    uint32_t *wm;
    carve_shared(J, S, smem_raw, &wm);
    const Cta K{s_plan, s_red, s_tiles, s_found, s_marked, L, wm};
    uint32_t epoch = 0;
    lead_search<kAnyWidth, false>(J, st, S, K, false, epoch);
    const uint32_t status = st->status;
    if (status == ST_FOUND || status == ST_NOT_FOUND || status == ST_OOM) {
        clean_table(J, L->smode ? 0u : L->size, L->clean_marks, 1, 0);
    } else {
        // the search continues from the slot's rows and state (in the slot,
        // or on the whole GPU, where the table is rebuilt from the rows)
        if (!keep_table)
            for (uint64_t i = tid; i <= J.table_mask; i += blockDim.x) J.table[i] = kEmpty;
        for (uint64_t i = tid; i < (J.chunk_max + 31) / 32; i += blockDim.x) J.bitmap[i] = 0;
    }
    __syncthreads();
    if (tid == 0) report_slot(J, status, slot, globaltimer_ns() - t_start, *out);
    __syncthreads();
    return status;
}

__global__ void __launch_bounds__(256, 2) k_solve_batch(const BatchJob *jobs, const __grid_constant__ BatchArgs B) {
    extern __shared__ __align__(16) uint8_t smem_raw[];
    __shared__ Plan s_plan;
    __shared__ uint32_t s_red[32];
    __shared__ uint64_t s_tiles;
    __shared__ unsigned long long s_found;
    __shared__ uint32_t s_marked;
    __shared__ Lead L;
    __shared__ SolveJob J;
    __shared__ uint32_t s_prob;
    const uint32_t tid = threadIdx.x;
    for (;;) {
        if (tid == 0) s_prob = atomicAdd(B.queue, 1u);
        __syncthreads();
        const uint32_t pi = s_prob;
        __syncthreads();
        if (pi >= B.n) return;
        const BatchJob &bj = jobs[pi];
        if (tid == 0) {
            J = bj.job;
            J.tree = bj.tree;
        }
        __syncthreads();
        // a search left in this slot for the host to continue: the slot is
        // not reused, and this CTA takes no more problems (the host launches
        // again for any left in the queue)
        if (solve_in_slot(J, B.slot, blockIdx.x, bj.out, smem_raw, &s_plan, s_red, &s_tiles, &s_found, &s_marked,
                          &L, B.yield_ns, true) == ST_NEED_MEM)
            return;
    }
}

// ---------------------------------------------------------------------------
// searches a batch left in their slots at their time allowance, continued side
// by side: group g of G.group_ctas CTAs takes problem G.prob[g] in its slot and
// runs the plain search there (its first CTA leads, the others take the team
// chunks), with the slot's cache, uniqueness table and state as the batch CTA,
// or the group launch before, left them.  The leader writes the problem's report
// like a batch CTA.  A slot that a group has parked holds that launch's last
// command (to leave) and its barrier's arrivals: the leader resets them and then
// releases the others, which wait for its word (the host zeroes it in the copy
// that brings the groups, so it costs a batch nothing; the wait is bounded).
__global__ void __launch_bounds__(256, 2) k_solve_groups(const BatchJob *jobs, const __grid_constant__ GroupArgs G) {
    __shared__ SolveJob J;
    __shared__ unsigned long long s_t0;
    __shared__ uint32_t s_go;
    const uint32_t g = blockIdx.x / G.group_ctas;
    if (g >= G.groups) return;
    const uint32_t slot = G.slot_of[g];
    const BatchJob &bj = jobs[G.prob[g]];
    if (threadIdx.x == 0) {
        J = bj.job;
        J.tree = bj.tree;
        bind_slot(J, G.slot, slot);
        J.blk = G.blk + (uint64_t)g * G.group_ctas;
        J.plan = G.plan + (uint64_t)g * G.plan_stride;
        J.tmp = G.tmp + (uint64_t)g * G.tmp_words;
        J.pending = G.pending + (uint64_t)g * G.chunk;
        J.slotpos = G.slotpos + (uint64_t)g * G.chunk;
        J.bitmap = G.bitmap + (uint64_t)g * ((G.chunk + 31) / 32);
        // (new languages of a chunk and the cached ones keep the slot's
        // table at most half full)
        J.chunk_max = umin64(umin64(G.chunk, G.tmp_words / J.W), (J.table_mask + 1) / 2 - J.cache_alloc);
        J.team_base = g * G.group_ctas;
        J.team_size = G.group_ctas;
        J.yield_ns = G.yield_ns;
        J.solo_tiles = 64;
        J.small_rows = 0;
        J.handover = 0;
        s_t0 = globaltimer_ns();
        J.t_start = s_t0;
        // the leader continues the parked search
        SolveState *st = J.st;
        uint32_t go = 1;
        if (team_rank_of(J) == 0) {
            st->status = ST_RUNNING;
            st->need_rows = 0;
            st->marked = 0;
            st->bar_arrive = 0;
            st->cmd = 0;
            st->cmd_seq = 0;
            st->err = 0;
            __threadfence();
            atomicExch(&G.release[g], 1ull);
        } else {
            uint32_t nap = 64;
            while ((go = (uint32_t)ld_acquire_u64(&G.release[g])) == 0) {
                if (globaltimer_ns() - s_t0 > kBarrierWaitNs) break;
                __nanosleep(nap);
                if (nap < REI_CMD_NAP) nap <<= 1;
            }
            if (!go) {
                // (never released: the search ends with an error for the host)
                atomicCAS(&st->err, 0u, 4u);
                atomicExch(&st->status, (uint32_t)ST_TIMEOUT);
            }
        }
        s_go = go;
    }
    __syncthreads();
    if (!s_go) return;
    uint32_t epoch = 0;
    solve_body<kAnyWidth, false>(J, epoch);
    if (team_rank_of(J) == 0 && threadIdx.x == 0)
        report_slot(J, ld_relaxed_u32(&J.st->status), slot, globaltimer_ns() - s_t0, *bj.out);
}

// ---------------------------------------------------------------------------
// the served search: a persistent launch whose CTAs take requests from a ring
// in mapped host memory as the host publishes them, stage each one themselves
// (scratch in their slot), solve it, and write the answer and a completion
// word back to mapped memory.  A CTA that finds nothing to do for idle_ns, or
// sees the stop word, returns; the host relaunches when work arrives.

__device__ __forceinline__ unsigned long long ld_acquire_sys_u64(const volatile unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.acquire.sys.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__global__ void __launch_bounds__(256, 2) k_serve(const __grid_constant__ ServeArgs A) {
    extern __shared__ __align__(16) uint8_t smem_raw[];
    __shared__ Plan s_plan;
    __shared__ uint32_t s_red[32];
    __shared__ uint64_t s_tiles;
    __shared__ unsigned long long s_found;
    __shared__ uint32_t s_marked;
    __shared__ Lead L;
    __shared__ SolveJob J;
    __shared__ StageJob SJ;
    __shared__ unsigned long long s_job;
    const uint32_t tid = threadIdx.x;
    const uint32_t slot = blockIdx.x;
    for (;;) {
        if (tid == 0) {
            // claim the next published request, backing off while there is none
            const unsigned long long t0 = globaltimer_ns();
            uint32_t nap = 64;
            unsigned long long job = kNone;
            for (;;) {
                if (ld_acquire_sys_u64(A.stop)) break;
                const unsigned long long h = ld_relaxed_u64(A.head);
                const unsigned long long av = ld_acquire_sys_u64(A.avail);
                if (h < av) {
                    if (atomicCAS(A.head, h, h + 1) == h) {
                        job = h;
                        break;
                    }
                    continue;
                }
                __nanosleep(nap);
                if (nap < 2048) nap <<= 1;
                if (globaltimer_ns() - t0 > A.idle_ns) break;
            }
            s_job = job;
        }
        __syncthreads();
        const unsigned long long job = s_job;
        __syncthreads();
        if (job == kNone) return;
        const uint32_t r = (uint32_t)(job % A.ring_size);
        const ServeReq &q = A.ring[r];
        ServeOut &o = A.outs[r];
        // the entry is read only once it is whole: its sequence word names
        // this job and its sizes are in range (waited for at most 2 ms; a
        // request still incomplete then is answered as invalid, never read)
        if (tid == 0) {
            const unsigned long long t0 = globaltimer_ns();
            uint32_t ok = 0, tries = 0;
            for (;;) {
                if (ld_acquire_sys_u64(&q.seq) == job + 1) {
                    const uint32_t np = q.n_pos, nn = q.n_neg, ns = q.n_sym, tb = q.total_bytes;
                    if (np + nn <= kServeMaxStrings && np <= kServeMaxStrings && ns <= 256 && tb <= kServeMaxBytes &&
                        q.offs[np + nn] == tb && q.max_cost <= REI_MAX_COST) {
                        ok = 1;
                        break;
                    }
                }
                tries++;
                if (globaltimer_ns() - t0 > 2000000ull) break;
                __nanosleep(256);
            }
            if (tries) atomicAdd(A.head + 1, 1ull);
            if (!ok) atomicAdd(A.head + 2, 1ull);
            s_red[1] = ok;
        }
        __syncthreads();
        if (!s_red[1]) {
            if (tid == 0) {
                o.out = BatchOut{};
                o.out.status = ST_BAD;
                o.info = StageInfo{};
                __threadfence_system();
                *(volatile unsigned long long *)&o.done = job + 1;
                __threadfence_system();
            }
            __syncthreads();
            continue;
        }
        // the request's offsets into this slot's buffer, then staged by this CTA
        const uint32_t n_str = q.n_pos + q.n_neg;
        uint32_t *in_o = A.in_offs + (uint64_t)slot * (kServeMaxStrings + 1);
        for (uint32_t i = tid; i <= n_str; i += blockDim.x) in_o[i] = q.offs[i];
        if (tid == 0) {
            StageJob sj{};
            sj.bytes = q.bytes;  // copied once into shared memory by the staging
            sj.offs = in_o;
            sj.n_pos = q.n_pos;
            sj.n_neg = q.n_neg;
            for (uint32_t a = 0; a < q.n_sym; a++) sj.alphabet[a] = q.alphabet[a];
            sj.n_sym = q.n_sym;
            sj.total_bytes = q.total_bytes;
            sj.info = A.sinfo + slot;
            sj.word_start = A.word_start + (uint64_t)slot * kMaxIC;
            sj.word_len = A.word_len + (uint64_t)slot * kMaxIC;
            sj.len_start = A.len_start + (uint64_t)slot * (REI_MAX_STRLEN + 2);
            sj.gt_off = A.gt_off + (uint64_t)slot * (kMaxIC + 1);
            sj.gt_pair = A.gt_pair + (uint64_t)slot * A.pair_cap;
            sj.pair_cap = A.pair_cap;
            sj.pos_mask = A.pos + (uint64_t)slot * kMaxWords;
            sj.neg_mask = A.neg + (uint64_t)slot * kMaxWords;
            sj.leaf = A.leaf + (uint64_t)slot * kMaxWords * 256;
            SJ = sj;
        }
        __threadfence();
        __syncthreads();
        {
            // the staging scratch uses the shared memory the search carves later
            StageSmem M;
            stage_layout(kServeMaxIC, kServeMaxBytes, smem_raw, &M);
            stage_run(SJ, M);
        }
        __threadfence();
        __syncthreads();
        const StageInfo I = *SJ.info;
        __syncthreads();
        uint32_t verdict = 0;  // 0 solve, 1 invalid input, 2 too large for this launch
        // the job, built in shared memory (zeroed, the leaf table by every
        // thread, the rest by thread 0)
        if (tid == 0) {
            if (I.status == SE_PAIRS || I.status == SE_IC_LARGE) verdict = 2;
            else if (I.status != SE_OK) verdict = 1;
            s_red[0] = verdict;
        }
        for (uint32_t i = tid; i < sizeof(SolveJob) / 8; i += blockDim.x)
            reinterpret_cast<unsigned long long *>(&J)[i] = 0;
        __syncthreads();
        verdict = s_red[0];
        if (!verdict) {
            for (uint32_t a = tid; a < 256; a += blockDim.x) {
                J.leaf_cost[a] = q.leaf_cost[a];
                J.leaf_sym[a] = q.leaf_sym[a];
            }
            if (tid == 0) {
                SolveJob &j = J;
                j.n = I.n;
                j.W = I.W;
                j.G = I.G;
                j.n_sym = q.n_sym;
                j.max_len = I.max_len;
                j.gt_off = SJ.gt_off;
                j.gt_pair = SJ.gt_pair;
                j.len_start = SJ.len_start;
                j.pos_mask = SJ.pos_mask;
                j.neg_mask = SJ.neg_mask;
                j.leaf = SJ.leaf;
                j.leaf_stride = kMaxWords;
                j.n_pos_set = I.n_pos_set;
                j.pos_eps = I.pos_eps;
                j.neg_eps = I.neg_eps;
                j.cmin = q.cmin;
                j.c[0] = q.costs.c_sym;
                j.c[1] = q.costs.c_opt;
                j.c[2] = q.costs.c_star;
                j.c[3] = q.costs.c_cat;
                j.c[4] = q.costs.c_alt;
                j.max_cost = q.max_cost;
                j.max_errors = q.max_errors;
                j.flags = q.flags;
                const uint64_t per = 4ull * I.W + 28;
                j.cap = umin64(q.mem_budget / per, 0x7FFF0000ull);
                j.seg_cap = 2 * q.max_cost + 4;
                j.gt_in_smem = search_smem_bytes(I.W, I.n, I.G, I.max_len, j.seg_cap, true, blockDim.x / 32, 0) <=
                               A.smem_cap;
                if (search_smem_bytes(I.W, I.n, I.G, I.max_len, j.seg_cap, j.gt_in_smem, blockDim.x / 32, 0) >
                        A.smem_cap ||
                    I.W > A.slot.cs_words / A.slot.rows)
                    s_red[0] = 2;
                j.tree = o.tree;
            }
        }
        __syncthreads();
        verdict = s_red[0];
        __syncthreads();
        uint32_t status = ST_BAD;
        if (verdict == 0) {
            status = solve_in_slot(J, A.slot, slot, &o.out, smem_raw, &s_plan, s_red, &s_tiles, &s_found, &s_marked,
                                   &L, A.yield_ns, true);
            // a parked search's job, for its continuation (in its slot, or on
            // the whole GPU from the slot's rows)
            if (status == ST_NEED_MEM && threadIdx.x == 0) {
                BatchJob &pj = A.parked[slot];
                pj.job = J;
                pj.tree = o.tree;
                pj.out = &o.out;
            }
        } else if (tid == 0) {
            o.out.status = verdict == 1 ? ST_BAD : ST_NEED_MEM;
            o.out.slot = kNoSlot;  // (too large for a slot: never searched here)
        }
        if (tid == 0) {
            o.info = I;
            __threadfence_system();
            *(volatile unsigned long long *)&o.done = job + 1;
            __threadfence_system();
        }
        __syncthreads();
        // a search left in this slot for the host to continue: the CTA takes
        // no more requests, so the slot stays as it is until the host has
        // copied it (the host stops the launch before it does)
        if (status == ST_NEED_MEM) return;
    }
}

cudaError_t solve_batch_smem_max(size_t *bytes) { return smem_max_of((const void *)k_solve_batch, bytes); }

cudaError_t launch_solve_batch(const BatchJob *jobs_dev, const BatchArgs *args, uint32_t grid, uint32_t threads,
                               size_t smem, cudaStream_t stream) {
    cudaError_t e = prepare((const void *)k_solve_batch);
    if (e != cudaSuccess) return e;
    k_solve_batch<<<grid, threads, smem, stream>>>(jobs_dev, *args);
    return cudaGetLastError();
}

cudaError_t solve_batch_occupancy(uint32_t threads, size_t smem, int *blocks_per_sm) {
    return occupancy((const void *)k_solve_batch, threads, smem, blocks_per_sm);
}

cudaError_t launch_solve_groups(const BatchJob *jobs_dev, const GroupArgs *args, uint32_t grid, uint32_t threads,
                                size_t smem, cudaStream_t stream) {
    cudaError_t e = prepare((const void *)k_solve_groups);
    if (e != cudaSuccess) return e;
    void *args_[] = {(void *)&jobs_dev, (void *)args};
    return cudaLaunchCooperativeKernel((const void *)k_solve_groups, dim3(grid), dim3(threads), args_, smem, stream);
}

cudaError_t solve_groups_occupancy(uint32_t threads, size_t smem, int *blocks_per_sm) {
    return occupancy((const void *)k_solve_groups, threads, smem, blocks_per_sm);
}

cudaError_t solve_groups_smem_max(size_t *bytes) { return smem_max_of((const void *)k_solve_groups, bytes); }

cudaError_t launch_serve(const ServeArgs *args, uint32_t grid, uint32_t threads, size_t smem, cudaStream_t stream) {
    cudaError_t e = prepare((const void *)k_serve);
    if (e != cudaSuccess) return e;
    k_serve<<<grid, threads, smem, stream>>>(*args);
    return cudaGetLastError();
}

cudaError_t serve_occupancy(uint32_t threads, size_t smem, int *blocks_per_sm) {
    return occupancy((const void *)k_serve, threads, smem, blocks_per_sm);
}

}  // namespace rei
