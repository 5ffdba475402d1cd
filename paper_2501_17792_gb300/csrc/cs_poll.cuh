// cs_poll.cuh -- the host's wait for words a kernel writes to pinned memory
// (host code only; no CUDA in it).
#pragma once
#include <stdint.h>

namespace cs {

enum class Arrival { kThere = 0, kMissing = 1, kFailed = 2 };

// Waits until *flag is seq: polled, at most `polls` times, then through
// `sync`, which waits for the stream (false: it failed) and after which the
// flag must be there.
template <class Sync>
Arrival wait_for(const uint32_t *flag, uint32_t seq, int polls, Sync sync) {
    const auto there = [=] { return __atomic_load_n(flag, __ATOMIC_ACQUIRE) == seq; };
    for (int i = 0; i < polls; ++i)
        if (there()) return Arrival::kThere;
    if (!sync()) return Arrival::kFailed;
    return there() ? Arrival::kThere : Arrival::kMissing;
}

}  // namespace cs
