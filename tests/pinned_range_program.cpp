/* pinned_view on a made-up address space: argv[1] lists the page-locked spans as host:device:bytes,...,
 * argv[2] and argv[3] are the range's first address and length. Prints the device address, 0 = none. */
#include <cstdio>
#include <cstdlib>

#include "../paper_2301_13062_b200/csrc/pinned_range.h"

int main(int, char **argv) {
    const char *spans = argv[1];
    const size_t at = strtoull(argv[2], nullptr, 10), bytes = strtoull(argv[3], nullptr, 10);
    void *view = cp::pinned_view(reinterpret_cast<void *>(at), bytes, [&](char *q, cp::PinnedSpan &s) {
        const size_t a = reinterpret_cast<size_t>(q);
        for (const char *c = spans; *c;) {
            char *e;
            const size_t host = strtoull(c, &e, 10), device = strtoull(e + 1, &e, 10), size = strtoull(e + 1, &e, 10);
            if (a >= host && a < host + size) {
                s = cp::PinnedSpan{reinterpret_cast<char *>(device + (a - host)), host + size - a};
                return true;
            }
            c = *e ? e + 1 : e;
        }
        return false;
    });
    printf("%zu\n", reinterpret_cast<size_t>(view));
    return 0;
}
