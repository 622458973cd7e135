// The launch shapes a batch's autotuner times.  Host code only (no CUDA), so it
// is tested on its own.
#pragma once

#include <cstddef>
#include <cstdint>
#include <vector>

namespace rk {

// At most `most` (0: no limit) of the candidates, evenly spread over their list,
// the last place kept for the shape in use.
template <class Shape>
std::vector<Shape> pick_shapes(const std::vector<Shape> &candidates, uint32_t most,
                               const Shape &in_use) {
    std::vector<Shape> pick;
    const size_t n = candidates.size(), room = most ? most - 1 : n;
    if (n <= room) {
        pick = candidates;
    } else {
        for (size_t i = 0; i < room; ++i) pick.push_back(candidates[i * n / room]);
    }
    pick.push_back(in_use);
    return pick;
}

}  // namespace rk
