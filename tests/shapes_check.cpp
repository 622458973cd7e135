// The autotuner's pick of launch shapes: never more than asked for, the shape in
// use among them, the rest distinct and in order.  Prints "ok".
#include <cstdio>

#include "rk_shapes.h"

int main() {
    for (int n = 0; n < 40; ++n) {
        std::vector<int> cand;
        for (int i = 0; i < n; ++i) cand.push_back(i);
        for (unsigned most = 0; most < 45; ++most) {
            const std::vector<int> p = rk::pick_shapes(cand, most, -7);
            const size_t want = most && most < (unsigned)n + 1 ? most : n + 1;
            if (p.size() != want || p.back() != -7) {
                std::printf("n %d most %u: %zu shapes\n", n, most, p.size());
                return 1;
            }
            for (size_t i = 0; i + 1 < p.size(); ++i)
                if (p[i] < 0 || p[i] >= n || (i && p[i] <= p[i - 1])) {
                    std::printf("n %d most %u: shape %zu\n", n, most, i);
                    return 1;
                }
        }
    }
    std::puts("ok");
    return 0;
}
