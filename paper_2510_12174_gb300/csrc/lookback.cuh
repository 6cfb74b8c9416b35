// The walk of a decoupled look-back over published chunk counts, free of
// device-only code so that its waiting can be tested on the host.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define UNIGS_HD __host__ __device__ __forceinline__
#else
#define UNIGS_HD inline
#endif

namespace unigs {

// Counts the polls of a walk that saw nothing new since its last step: the
// limit is on the wait for one word, however long the walk.
struct PollLimit {
    uint32_t limit, polls;
    UNIGS_HD explicit PollLimit(uint32_t limit_) : limit(limit_), polls(0u) {}
    // After a poll; true: give up.
    UNIGS_HD bool give_up(bool advanced) {
        polls = advanced ? 0u : polls + 1u;
        return polls > limit;
    }
};

// Sum of the counts of chunks [0, chunk).  load(p) is the word of chunk p:
// (epoch << 2 | state) << 32 | count, state 1: the chunk's own count, 2: its
// inclusive prefix; any other epoch: not written yet.  Reads WIDE predecessors
// at a time: one memory latency per step, where one at a time a full first
// wave of chunks would pay a latency per chunk.  Returns false when the wait
// for a word gave up.
template <int WIDE, typename Load>
UNIGS_HD bool look_back_walk(const Load& load, int64_t chunk, uint32_t epoch, uint32_t limit,
                             uint32_t* sum_out) {
    uint32_t sum = 0;
    PollLimit wait(limit);
    int64_t p = chunk - 1;
    while (p >= 0) {
        unsigned long long v[WIDE];
#pragma unroll
        for (int j = 0; j < WIDE; ++j) v[j] = p - j >= 0 ? load(p - j) : 0ull;
        int used = 0;
        bool open = true, found = false;
#pragma unroll
        for (int j = 0; j < WIDE; ++j) {
            const uint32_t tag = (uint32_t)(v[j] >> 32);
            open = open && !found && p - j >= 0 && (tag >> 2) == epoch && (tag & 3u) != 0u;
            if (open) {
                sum += (uint32_t)v[j];
                found = (tag & 3u) == 2u;
                ++used;
            }
        }
        if (found) break;
        p -= used;
        if (wait.give_up(used > 0)) return false;
    }
    *sum_out = sum;
    return true;
}

}  // namespace unigs
