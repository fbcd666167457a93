// The clock of a bounded device-side wait (host and device, so that it can be
// checked on the host).
#pragma once

#if defined(__CUDACC__)
#define LBIB_WAIT_HD __host__ __device__ __forceinline__
#else
#define LBIB_WAIT_HD inline
#endif

namespace lbib {

// Nanoseconds that a waiting thread has spent, from readings of the global timer.
// The timer also runs while the GPU is held by something else (another process, a
// debugger): two readings that lie further apart than GAP_NS count as that much, so
// a wait gives up for the time it has waited and not for the time it was held.
struct WaitClock {
    static constexpr unsigned long long GAP_NS = 10000000ull;
    unsigned long long last, spent;
    LBIB_WAIT_HD void start(unsigned long long now) {
        last = now;
        spent = 0;
    }
    LBIB_WAIT_HD bool over(unsigned long long now, unsigned long long bound_ns) {
        const unsigned long long d = now - last;
        last = now;
        spent += d < GAP_NS ? d : GAP_NS;
        return spent > bound_ns;
    }
};

}  // namespace lbib
