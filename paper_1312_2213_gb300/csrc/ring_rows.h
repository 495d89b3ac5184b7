// ring_rows.h -- the row counters of the producer/consumer rings (plain C++, for host and device).
// Every role of a block counts the rows it has handed over or taken: row k uses ring slot k mod RD in
// phase (k / RD) mod 2.  The counter is 32 bits wide and a launch may run any 64-bit number of sweeps,
// so a chunk of sweeps between two flushes holds at most kMaxChunkRows rows, and behind each chunk the
// counters start again at the same slot and phase.
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define MUCA_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define MUCA_HOST_DEVICE inline
#endif

namespace muca {

constexpr int64_t kMaxChunkRows = int64_t(1) << 30;

// Sweeps of a chunk: at most `cap` (what the block's counters hold, or the caller asked for), the
// launch's own and kMaxChunkRows rows of an L x L lattice; at least one.
MUCA_HOST_DEVICE int chunk_sweeps(uint64_t cap, int64_t sweeps, int L)
{
    int64_t n = kMaxChunkRows / L;
    if (cap < (uint64_t)n) n = (int64_t)cap;
    if (sweeps < n) n = sweeps;
    return n < 1 ? 1 : (int)n;
}

// Takes whole turns of a ring of `depth` slots (two phases) off the counter k, and with it off `drop`,
// the row of a hand-over to leave out (negative: none, or passed).
MUCA_HOST_DEVICE void rebase_rows(int &k, int &drop, int depth)
{
    const int base = k - k % (2 * depth);
    k -= base;
    drop = drop >= base ? drop - base : -1;
}

}  // namespace muca
