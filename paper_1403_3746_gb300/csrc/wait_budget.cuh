// Budget of a bounded device wait, in clock cycles of polling.
#pragma once

namespace lbm {

// A poll counts for the cycles since the last one, but for no more than kMostPerPoll (8 ms): a kernel
// that is switched out in the middle of a wait (another process's time slice) finds a long gap when it
// resumes, and would take the clock alone for a copy that never lands.
// The clock's low 32 bits are enough: a gap counts for its remainder at most.
struct WaitBudget {
    static constexpr unsigned kMostPerPoll = 1u << 24;
    unsigned last;
    long long left;
    __host__ __device__ WaitBudget(unsigned now, long long budget) : last(now), left(budget) {}
    __host__ __device__ bool spent(unsigned now) {
        const unsigned gap = now - last;
        last = now;
        left -= gap < kMostPerPoll ? gap : kMostPerPoll;
        return left < 0;
    }
};

}  // namespace lbm
