// bh_wait.h -- the limits of a bounded device wait (plain C++, no CUDA headers).
#pragma once

#ifdef __CUDACC__
#define BH_WAIT_FN __host__ __device__ __forceinline__
#else
#define BH_WAIT_FN inline
#endif

namespace bh {

constexpr int kWsSpinLimit = 1 << 22;                       // polls
constexpr unsigned long long kWsTimeoutNs = 1000000000ull;  // on the global timer ...
constexpr int kWsLatePolls = 1 << 16;                       // ... and then this many polls more

// A wait polls while its poll is below `end`, at most kWsSpinLimit times.  Once
// a second has passed on the global timer that many polls more remain: the
// timer also goes on while the GPU runs another process or is stopped in a
// debugger, when the warp waited for stands still as well, but polls are only
// made while both run (a millisecond of them at least, for work of
// microseconds).  A running sum of the time between polls instead cost 3% of the
// walk of clumpy 100003.
struct WaitLimit {
    unsigned long long t0;
    int end;
    BH_WAIT_FN explicit WaitLimit(unsigned long long now) : t0(now), end(kWsSpinLimit) {}
    BH_WAIT_FN void look(int poll, unsigned long long now)
    {
        if (now - t0 > kWsTimeoutNs && end == kWsSpinLimit && poll + kWsLatePolls < end) end = poll + kWsLatePolls;
    }
};

}  // namespace bh
