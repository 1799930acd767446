// sizes.h -- sizes of a search's buffers, and the slots of its uniqueness table in
// the order they are probed (host and device).
#pragma once
#include <algorithm>
#include <cstddef>
#include <cstdint>

#ifdef __CUDACC__
#define REI_HD __host__ __device__ __forceinline__
#else
#define REI_HD inline
#endif

namespace rei {

inline uint64_t pow2_at_least(uint64_t x) {
    uint64_t p = 1;
    while (p < x) p <<= 1;
    return p;
}

// A table slot's number is held in 32 bits: with a marked candidate, in the list
// of slots a search empties, and in a candidate's registers.
constexpr uint64_t kMaxTableSlots = 1ull << 32;

// Bump carving of a fixed array.  A piece that does not fit ends it: the pieces after
// it are refused too, whatever their size, so that the last of several tells of all.
struct Carve {
    static constexpr size_t kAlign = 256;
    unsigned char *base;
    size_t used, cap;
    bool full = false;
    void *take(size_t bytes) {
        const size_t at = (used + kAlign - 1) & ~(kAlign - 1);
        full = full || at > cap || bytes > cap - at;
        if (full) return nullptr;
        used = at + bytes;
        return base + at;
    }
};

// Linear probing of a table of mask + 1 slots from hash h.  No candidate is marked
// with slot kNoMark, the last of the largest table: the number says that a candidate
// is not marked, and probing passes the slot over.  (A flag beside the slot instead
// cost searches of 8 to 16 words 2 %, medium ones 0.5 %.)
constexpr uint32_t kNoMark = 0xFFFFFFFFu;
REI_HD uint32_t probe_first(uint64_t h, uint64_t mask) {
    const uint32_t p = (uint32_t)(h & mask);
    return p < kNoMark - 1 ? p : kNoMark - 1;
}
REI_HD uint32_t probe_next(uint32_t p, uint32_t mask) {
    const uint32_t q = (p + 1) & mask;
    return q == kNoMark ? 0u : q;
}
// (fingerprint inserts of 8 to 16 words in the first launch: 0.5 % quicker than in 32 bits)
REI_HD uint64_t probe_next(uint64_t p, uint64_t mask) {
    const uint64_t q = (p + 1) & mask;
    return (uint32_t)q == kNoMark ? 0 : q;
}

// Slots of the uniqueness table of a search with room for `rows` languages of at
// most `cap`: at most half full with them and, once the cache cannot grow, a
// chunk of candidates that find no room.  It holds distinct languages, at most
// 2^n of them; direct: a slot for every language (1-word exact keys up to 2^26,
// never probed twice).  Bounded by the slots' numbers: 0x7FFF0000 languages and a
// chunk of 2^26 fill 52 % of 2^32 slots.
inline uint64_t table_slots(uint64_t rows, uint64_t cap, uint64_t chunk, uint32_t n, bool direct) {
    if (direct) return 1ull << n;
    uint64_t need = rows + (rows >= cap ? chunk : 0);
    if (n < 40) need = std::min<uint64_t>(need, 1ull << n);
    return std::min(kMaxTableSlots, pow2_at_least(std::max<uint64_t>(2 * need, 1024)));
}

}  // namespace rei
