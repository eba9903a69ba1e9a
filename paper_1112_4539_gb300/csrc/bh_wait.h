// bh_wait.h -- the time limit of a bounded device wait (plain C++, no CUDA headers).
#pragma once

#ifdef __CUDACC__
#define BH_WAIT_FN __host__ __device__ __forceinline__
#else
#define BH_WAIT_FN inline
#endif

namespace bh {

constexpr int kWsSpinLimit = 1 << 22;                       // polls
constexpr unsigned long long kWsTimeoutNs = 1000000000ull;  // running time
constexpr unsigned long long kWsStepNs = 20000000ull;

// Running time of a wait, from the clock readings of its polls.  The global
// timer also goes on while the GPU runs another process or is stopped in a
// debugger, when the warp waited for stands still as well: of the time
// between two readings at most kWsStepNs counts, so that such a stop, however
// long, uses up 2% of the limit.  Readings are 64 polls apart, far closer.
struct WaitClock {
    unsigned long long last, spent;
    BH_WAIT_FN explicit WaitClock(unsigned long long now) : last(now), spent(0) {}
    BH_WAIT_FN bool over(unsigned long long now)
    {
        const unsigned long long step = now - last;
        last = now;
        spent += step < kWsStepNs ? step : kWsStepNs;
        return spent > kWsTimeoutNs;
    }
};

}  // namespace bh
