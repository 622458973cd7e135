// The set limit: a set counts for the sum of its parts as listed here, and is
// taken up to 2^32 - 1 bytes.  Prints "ok".
#include <cstdio>

#include "rk_limit.h"

using rk::SetParts;

static int fail(const char *what, unsigned long long got, unsigned long long want) {
    std::printf("%s: %llu, expected %llu\n", what, got, want);
    return 1;
}

int main() {
    // 3 patterns of 5, 8 and 8 bytes, two prefixes; a map of 16 slots, every
    // other part below 256 bytes
    const SetParts small{3, 24, 2, 3, 8, 2, 8, 0, 0, 0};
    if (rk::set_bytes(small) != 12 * 256) return fail("small", rk::set_bytes(small), 12 * 256);
    // 9,000,000 patterns of 128 bytes with as many prefixes, sampled
    const SetParts many{9000000, 1152000000, 9000000, 9000000, 1u << 25, 1, 128, 1u << 27,
                        65536, 0};
    const unsigned long long want = 536870912ull + 36000256 + 1280 + 536871168 + 36000256 +
                                    1152000256 + 72000256 + 36000256 + 256 + 1073742080 + 65792 +
                                    256;
    if (rk::set_bytes(many) != want) return fail("many", rk::set_bytes(many), want);
    if (!rk::set_fits(many)) return fail("many fit", 0, 1);
    // the last set of 4096-byte patterns that is taken, and the next
    SetParts edge{0, 0, 0, 0, 1u << 21, 1, 4096, 0, 0, 0};
    unsigned long long last = 0;
    for (unsigned long long k = 1000000; k < 1048576; ++k) {
        edge.patterns = edge.prefixes = edge.runs = k;
        edge.packed = 4096 * k;
        if (!rk::set_fits(edge)) break;
        last = k;
    }
    const unsigned long long per = 4096 + 4 + 4 + 8 + 4, rest = (1ull << 25) + (1ull << 25);
    if (last < (0xFFFFFFFFull - rest - 36864) / per || last > (0xFFFFFFFFull - rest) / per)
        return fail("edge", last, (0xFFFFFFFFull - rest) / per);
    std::puts("ok");
    return 0;
}
