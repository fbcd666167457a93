// Host driver for csrc/bounded_wait.h: the time, in ms of the readings, at which a
// wait bounded by 10 s gives up, read every 0.7 ms, every 40 us, and with one gap of an
// hour; and that one with gaps of 9 s or 30 s does not within 9.8 s of its own (-1).
#include <cstdio>

#include "bounded_wait.h"

using lbib::WaitClock;

static double gives_up(double every_ms, double gap_at_ms, double gap_ms, double until_ms) {
    WaitClock c;
    unsigned long long t = 123456789ull;
    const unsigned long long bound = 10000000000ull, start = t;
    c.start(t);
    for (bool held = false;;) {
        t += (unsigned long long)(every_ms * 1e6);
        const double ms = (double)(t - start) / 1e6;
        if (!held && gap_ms > 0.0 && ms > gap_at_ms) {
            t += (unsigned long long)(gap_ms * 1e6);
            held = true;
        }
        if (c.over(t, bound)) return (double)(t - start) / 1e6;
        if (until_ms > 0.0 && ms > until_ms) return -1.0;
    }
}

int main() {
    std::printf("%.3f\n", gives_up(0.7, 0, 0, 0));
    std::printf("%.3f\n", gives_up(0.04, 0, 0, 0));
    std::printf("%.3f\n", gives_up(0.7, 5000, 3600e3, 0));
    std::printf("%.3f\n", gives_up(0.7, 100, 9000, 18900));
    std::printf("%.3f\n", gives_up(0.7, 100, 30000, 39800));
    return 0;
}
