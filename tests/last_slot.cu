// The last slots of a table of 2^32 slots (64 GiB): a language that would come to the
// last one, whose number stands for "not marked", takes the first, and its candidate is
// marked with that.
#include <cstdio>

#include "search.cuh"

using namespace rei;

struct Out {
    uint32_t q[6], err;
};

constexpr uint64_t kSlots = 1ull << 32;
constexpr int kKeys = 4;
// exact keys of slot 2^32 - 2, two at a time: the second comes to the last slot
__constant__ const unsigned long long g_keys[kKeys] = {0x3220c437f1207bf0ull, 0x23ff48196967f6eeull,
                                                       0x15ddcbfaec6b4decull, 0x7bc4fdc6e70d2eeull};
// 2-word languages whose fingerprints come to slot 2^32 - 1 (so 2^32 - 2 is their first)
__constant__ const uint32_t g_lang[2][2] = {{0x5dc1ea54u, 1u}, {0x91cd6784u, 1u}};

// the slots a search may probe here, emptied: 2 words at each end (all inside the table)
__device__ void empty_ends(unsigned long long *table, uint64_t words) {
    for (uint64_t i = 0; i < 4; i++) table[i] = table[words - 1 - i] = kEmpty;
    __threadfence();
}

__global__ void k_last_slot(unsigned long long *table, uint32_t *tmp, SolveState *st, Out *out) {
    if (threadIdx.x) return;
    __shared__ uint32_t masks[2];
    __shared__ unsigned long long found;
    masks[0] = masks[1] = 0xFFFFFFFFu;
    found = kNone;
    SolveJob J{};
    J.n = 62;
    J.W = 2;
    J.exact = 1;
    J.table = table;
    J.table_mask = kSlots - 1;
    J.tmp = tmp;
    J.cache_alloc = 1;
    J.chunk_max = 4;
    J.st = st;
    Shared S{};
    S.pos = S.neg = masks;
    TileCtx T{};
    T.J = &J;
    T.st = st;
    T.S = &S;
    T.W = 2;
    T.Ws = 3;
    T.n = 62;
    T.epoch = 1;
    T.dedup = true;
    T.found = &found;
    empty_ends(table, 2 * kSlots);
    for (int k = 0; k < 2; k++) {
        const uint32_t c[2] = {(uint32_t)g_keys[k], (uint32_t)(g_keys[k] >> 32)};
        out->q[k] = dedup_insert_exact<2>(T, c, k);
    }
    empty_ends(table, 2 * kSlots);
    Seg sg{};
    uint2 c[4] = {};
    for (int k = 0; k < 2; k++) c[k] = make_uint2((uint32_t)g_keys[2 + k], (uint32_t)(g_keys[2 + k] >> 32));
    uint32_t q[4] = {kNoMark, kNoMark, kNoMark, kNoMark};
    w2_finish<4>(T, sg, c, 0, 1, 3u, q);
    out->q[2] = q[0];
    out->q[3] = q[1];
    empty_ends(table, kSlots);
    J.exact = 0;
    for (int k = 0; k < 2; k++) {
        const uint32_t l[2] = {g_lang[k][0], g_lang[k][1]};
        out->q[4 + k] = dedup_insert<2>(T, l, k);
    }
    out->err = st->err;
}

int main() {
    size_t free_bytes = 0, all = 0;
    if (cudaMemGetInfo(&free_bytes, &all)) return 2;
    if (free_bytes < (size_t)80 << 30) {
        printf("too little memory\n");
        return 0;
    }
    unsigned long long *table;
    uint32_t *tmp;
    SolveState *st;
    Out *out, h;
    if (cudaMalloc(&table, 16 * kSlots) || cudaMalloc(&tmp, 256) || cudaMalloc(&st, sizeof(SolveState)) ||
        cudaMalloc(&out, sizeof(Out)) || cudaMemset(st, 0, sizeof(SolveState)) || cudaMemset(out, 0, sizeof(Out)))
        return 3;
    k_last_slot<<<1, 32>>>(table, tmp, st, out);
    if (cudaMemcpy(&h, out, sizeof h, cudaMemcpyDeviceToHost)) return 4;
    for (int k = 0; k < 6; k++) printf("%08x\n", h.q[k]);
    printf("err %u\n", h.err);
    return 0;
}
