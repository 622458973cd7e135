// The largest pattern set a table takes.  Host code only (no CUDA), so it is
// tested on its own.
#pragma once

#include <cstdint>

namespace rk {

// The parts of a set's table.
struct SetParts {
    uint64_t patterns, packed;   // their number, and bytes with each rounded up to 8
    uint64_t prefixes, runs;     // distinct prefixes, and pairs of prefix and length
    uint64_t hash_slots;         // of the lengths' hash tables
    uint64_t lengths, max_len;   // distinct lengths, the longest
    uint64_t sample_slots;       // sample map (0: none)
    uint64_t sample_filter_bytes, role_filter_bytes;  // bit sets (0: none)
};

// Bytes the set counts for: every part at 256 bytes' alignment, the prefix map
// with at least one slot in two free, a run as its length alone.  What a table
// takes may be more (a sparser map, runs that name their pattern), by at most 12
// bytes a pattern and 32 MiB; the limit is on the set, so that a faster layout
// refuses no set that a smaller one took.
inline uint64_t set_bytes(const SetParts &s) {
    const auto part = [](uint64_t n) { return (n + 255) / 256 * 256; };
    uint64_t map = 16;
    while (map < 2 * s.prefixes) map *= 2;
    return part(16 * map) + part(4 * s.runs + 4) + part(8 * (s.max_len + 1)) +
           part(16 * s.hash_slots + 16) + part(4 * s.patterns + 4) + part(s.packed + 16) +
           part(8 * s.patterns + 8) + part(4 * s.patterns + 4) + part(4 * s.lengths + 4) +
           part(8 * s.sample_slots + 8) + part(s.sample_filter_bytes + 16) +
           part(s.role_filter_bytes + 16);
}

inline bool set_fits(const SetParts &s) { return set_bytes(s) <= 0xFFFFFFFFull; }  // 4 GiB

}  // namespace rk
