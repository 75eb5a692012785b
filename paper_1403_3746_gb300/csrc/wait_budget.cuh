// Budget of a bounded device wait, in clock cycles of polling.
#pragma once

namespace lbm {

// A poll counts for the cycles since the last one, but for no more than kMostPerPoll (8 ms): a kernel
// that is switched out in the middle of a wait (another process's time slice) finds a long gap when it
// resumes, and would take the clock alone for a copy that never lands.
struct WaitBudget {
    static constexpr long long kMostPerPoll = 1LL << 24;
    long long last, left;
    __host__ __device__ WaitBudget(long long now, long long budget) : last(now), left(budget) {}
    __host__ __device__ bool spent(long long now) {
        const long long gap = now - last;
        last = now;
        left -= gap < kMostPerPoll ? gap : kMostPerPoll;
        return left < 0;
    }
};

}  // namespace lbm
