// A thread's work counters: 32 bits each, emptied into the launch's 64-bit counters.
#pragma once

#ifdef __CUDACC__
#define WC_FN __host__ __device__ __forceinline__
#else
#define WC_FN static inline
#endif

namespace skirt {

// Adds the crossings of one traversal (below 2^31 + 2^30: a line crosses fewer cells
// than the grid holds, below 2^31, and an octree's bound is smaller still) to c.
// True when c is large enough to be emptied before it takes the next: at most
// 2^30 - 1 stay, so that no sum passes 2^32 however long a packet lives.
WC_FN bool count_add(unsigned& c, unsigned n)
{
    c += n;
    return (c >> 30) != 0u;
}

// Whether one packet can make so many crossings that its counters have to be emptied
// before its end: those of max_events events, each with a deposit, a search and a
// peel-off per instrument along lines of at most `line` cells, on top of the 2^30 - 1
// that may stay from the packets before.
inline bool counts_within_packet(int max_events, int ninstr, unsigned long long line)
{
    const unsigned long long events = (unsigned long long)(max_events > 0 ? max_events : 0) + 1ull;
    return events * (unsigned long long)(ninstr + 2) >= ((1ull << 32) - (1ull << 30)) / (line > 0 ? line : 1ull);
}

}  // namespace skirt
