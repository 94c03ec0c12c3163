// The dense pair-id table shared by the load (which fills it while it reads the edges) and
// the preprocessing (which tries a larger one otherwise, and numbers its pairs).
// An open-addressed table of 2^lg slots (linear probing from a multiplicative hash of the
// pair rank); slot value = rank + 1, 0 = empty.
#pragma once
#include <cstdlib>
#include <cstring>

#include "internal.cuh"

namespace folty {

// A longer probe sequence abandons the table: at the largest load that serves (1/2) a
// sequence of linear probing among random slots is this long with a probability below 1e-20.
// The slots of a multiplicative hash are not random: ranks in a bad progression only lose the
// table, not a result.
constexpr int PAIR_MAX_PROBE = 256;
constexpr uint64_t PAIR_HASH_MUL = 0x9E3779B97F4A7C15ull;  // 2^64 / golden ratio (Fibonacci hashing)
constexpr uint32_t PAIR_LOOP = 0x7fffffffu;  // slot word of a self-loop
constexpr uint32_t PAIR_DIR = 0x80000000u;   // direction bit of a slot word (tables hold < 2^31 slots)

__device__ __forceinline__ uint64_t pair_rank_of(int32_t x, int32_t y, int32_t n) {
    const uint64_t a = (uint64_t)min(x, y), b = (uint64_t)max(x, y);
    return a * (2 * (uint64_t)n - a - 1) / 2 + (b - a - 1);
}

// A table with more pairs than half its slots does not serve, and the insert stops as soon
// as that shows: the pairs placed in every 64th slot are counted, and 9/8 of the number they
// may reach (of slots from PAIR_COUNTED_LG on: 8192, eleven standard deviations of 90
// below it) abandons the table at a load of 0.56, where probe sequences are still short.
// Smaller tables hold 2 slots per edge and always serve. Against a first try of 2^19 slots,
// 6M edges of 3M pairs took 66.5 ms when every edge still walked 4096 steps of the full
// table, 0.8 ms when the first sequence of 256 steps ended the insert.
constexpr int PAIR_COUNTED = 64;
constexpr int PAIR_COUNTED_LG = 20;

// flags: [0] the table is abandoned, [1] distinct pairs (k_pair_table_compact),
// [PAIR_COUNT_AT] pairs placed in counted slots: additions to the line that every thread
// reads [0] from made the load of 70M edges take 1.2 ms instead of 0.8.
constexpr int PAIR_COUNT_AT = 64;
constexpr int PAIR_FLAGS = PAIR_COUNT_AT + 32;

// Whether the table is abandoned, on any thread: the edges still to come need no slot.
__device__ __forceinline__ bool pair_table_over(const int* flags) { return *(const volatile int*)flags != 0; }

// Places key in the empty slot h unless another thread was first; returns what the slot
// then holds.
__device__ __forceinline__ uint64_t pair_place(uint64_t* table, int lg, uint64_t h, uint64_t key, int* flags) {
    const unsigned long long old = atomicCAS((unsigned long long*)&table[h], 0ull, (unsigned long long)key);
    if (old != 0) return old;
    if ((h & (PAIR_COUNTED - 1)) == 0 && lg >= PAIR_COUNTED_LG) {
        const int most = (1 << lg) / 2 / PAIR_COUNTED;
        if (atomicAdd(flags + PAIR_COUNT_AT, 1) >= most + most / 8) atomicExch(flags, 1);
    }
    return key;
}

// Slot holding table value key (rank + 1), placing it in the first empty slot of its probe
// sequence when absent; -1 after PAIR_MAX_PROBE steps.
__device__ __forceinline__ int64_t pair_slot(uint64_t* table, int lg, uint64_t key, int* flags) {
    const uint64_t mask = (1ull << lg) - 1;
    uint64_t h = (key * PAIR_HASH_MUL) >> (64 - lg);
    for (int pr = 0; pr < PAIR_MAX_PROBE; pr++) {
        uint64_t cur = __ldcg(&table[h]);
        if (cur == 0) cur = pair_place(table, lg, h, key, flags);
        if (cur == key) return (int64_t)h;
        h = (h + 1) & mask;
    }
    return -1;
}

// Slot word of edge x -> y: its pair's slot and direction, PAIR_LOOP for a self-loop; a
// probe sequence that runs out abandons the table.
__device__ __forceinline__ uint32_t pair_slot_word(uint64_t* table, int lg, int32_t x, int32_t y, int32_t n,
                                                   int* flags) {
    if (x == y) return PAIR_LOOP;
    const int64_t sl = pair_slot(table, lg, pair_rank_of(x, y, n) + 1, flags);
    if (sl < 0) {
        atomicExch(flags, 1);
        return PAIR_LOOP;
    }
    return (uint32_t)sl | (x > y ? PAIR_DIR : 0u);
}

// log2 of the table's largest size for m edges (at least 2m slots, up to 2^23: 64 MB, in
// L2; tables of 2^26 slots lost to the full-key sort, 12.6 against 10.2 ms for 20M edges of
// 10M pairs) and of its first try: at least m / 12 slots (room for m / 24 distinct pairs at a
// load factor of 1/2, i.e. a mean multiplicity of 24 or more, as in the workloads' Zipf
// multiplicities), at most 2^22 slots (32 MB), and, as a table of up to 2^20 slots (8 MB)
// costs a few microseconds to clear and list, at least 2^20 or the largest size: graphs of
// up to 2^19 edges never need a second try.
inline int pair_table_lg_max(int64_t m) {
    int b = 0;
    for (uint64_t v = (uint64_t)(2 * m - 1); v; v >>= 1) b++;
    return b < 10 ? 10 : (b > 23 ? 23 : b);
}
inline int pair_table_lg_first(int64_t m) {
    int b = 0;
    for (uint64_t v = (uint64_t)((m + 11) / 12); v; v >>= 1) b++;
    b = b < PAIR_COUNTED_LG ? PAIR_COUNTED_LG : (b > 22 ? 22 : b);
    return pair_table_lg_max(m) < b ? pair_table_lg_max(m) : b;
}

// The occupied slots of a table as (rank, slot) lists (at most cap entries), their number
// added to *cnt.
void enqueue_pair_list(const uint64_t* table, int lg, uint64_t* rank, uint32_t* slot, int* cnt, int cap, cudaStream_t s);

// The dense-id path is off when FOLTY_PAIR_SORT=keys (the full-key sort then runs).
inline bool pair_table_forced_off() {
    const char* env = std::getenv("FOLTY_PAIR_SORT");
    return env && std::strcmp(env, "keys") == 0;
}

}  // namespace folty
