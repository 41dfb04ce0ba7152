// Packets a thread takes from the work queue per refill (host code, no CUDA).
#pragma once

namespace skirt {

// What was asked for, to the letter (a caller who sets it measures what is set: the
// autotuner does).  By default (asked <= 0) four, but no more than leaves every
// thread eight refills: fewer starve the launch's end, or, below a refill per
// thread, most of the launch.  1e5 packets in the sphere took 1.68 ms by fours and
// take 1.00 ms one by one, 3e5 on an octree 12.6 and 7.8 ms; where there is work for
// many refills, single packets cost more in queue traffic (2e6 dust packets 14.9 ms
// against 13.8 ms by twos).
inline int queue_chunk(int asked, unsigned long long packets, unsigned long long threads)
{
    if (asked > 0) return asked;
    const unsigned long long fair = threads ? packets / (8ull * threads) : 0ull;
    return fair >= 4 ? 4 : (fair > 0 ? (int)fair : 1);
}

}  // namespace skirt
