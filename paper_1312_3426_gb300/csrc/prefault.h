// Page faults of a read-out's destination beside the wait for the device (host only).
#pragma once

#include <sys/mman.h>
#include <unistd.h>

#include <algorithm>
#include <cstddef>
#include <cstdint>
#include <exception>
#include <thread>

namespace lbib {

// Faults the pages of a large read-out's destination in beside the wait for
// the device: a fresh array costs more in page faults than the copy takes
// (400 MB: 16.5 ms with the copy, 3.6 without).  Contents stay, only whole pages
// inside the range are touched, and where it is refused the copy faults.  A
// destination that is there already is left alone: the threads took 60 us of a
// read-out of 9.4 MB into the same array as before (0.184 -> 0.128 ms without) and
// the walk over its pages 1.2 ms of one of 403 MB (3.85 -> 2.65).
class Prefault {
   public:
    Prefault(void *p, size_t bytes) {
        if (!p || bytes < MIN_BYTES || resident(p, bytes)) return;
        const Pages r(p, bytes);
        const size_t part = ((r.end - r.begin + THREADS - 1) / THREADS + r.size - 1) / r.size * r.size;
        for (int i = 0; i < THREADS && r.begin + i * part < r.end; ++i) {
            const size_t lo = r.begin + i * part, n = std::min(part, r.end - lo);
            try {
                th_[i] = std::thread([lo, n] { madvise((void *)lo, n, 23 /* MADV_POPULATE_WRITE */); });
            } catch (const std::exception &) {
                return;  // no thread to be had
            }
        }
    }
    ~Prefault() { join(); }
    void join() {
        for (std::thread &t : th_)
            if (t.joinable()) t.join();
    }
    // Whether the pages of the range are there, by a few of them spread over it.
    static bool resident(const void *p, size_t bytes) {
        const Pages r(p, bytes);
        if (r.end <= r.begin) return true;
        const size_t n = (r.end - r.begin) / r.size;
        for (size_t i = 0; i < SAMPLES; ++i) {
            unsigned char in = 0;
            if (mincore((void *)(r.begin + (n - 1) * i / (SAMPLES - 1) * r.size), r.size, &in) != 0 || !(in & 1)) return false;
        }
        return true;
    }
    static constexpr size_t MIN_BYTES = 8 << 20;

   private:
    struct Pages {  // the whole pages of a range
        size_t size, begin, end;
        Pages(const void *p, size_t bytes) : size((size_t)sysconf(_SC_PAGESIZE)) {
            begin = ((size_t)p + size - 1) / size * size;
            end = ((size_t)p + bytes) / size * size;
        }
    };
    static constexpr size_t SAMPLES = 16;
    static constexpr int THREADS = 4;
    std::thread th_[THREADS];
};

}  // namespace lbib
