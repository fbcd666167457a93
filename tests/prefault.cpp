// Host driver for csrc/prefault.h: what counts as there already (a fresh range, one with
// a few pages touched, all of it, one whose middle is fresh again, one without a whole
// page), and that the contents stay.
#include <cstdio>
#include <cstring>

#include "prefault.h"

int main() {
    const size_t bytes = 3 * lbib::Prefault::MIN_BYTES + 12345, third = lbib::Prefault::MIN_BYTES;
    char *p = (char *)mmap(nullptr, bytes, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS, -1, 0);
    if (p == MAP_FAILED) return 2;
    std::printf("fresh %d\n", lbib::Prefault::resident(p + 17, bytes - 17));
    p[0] = 1, p[bytes - 1] = 2, p[bytes / 2] = 3;
    std::printf("ends %d\n", lbib::Prefault::resident(p + 17, bytes - 17));
    { lbib::Prefault f(p + 17, bytes - 17); }
    std::printf("contents %d\n", p[0] == 1 && p[bytes - 1] == 2 && p[bytes / 2] == 3 && p[5000] == 0);
    std::memset(p, 1, bytes);
    std::printf("touched %d\n", lbib::Prefault::resident(p + 17, bytes - 17));
    madvise(p + third, third, MADV_DONTNEED);
    std::printf("middle %d\n", lbib::Prefault::resident(p + 17, bytes - 17));
    std::printf("small %d\n", lbib::Prefault::resident(p + 17, 100));
    return 0;
}
