// solve_plan.h -- sizes of the solve's launches: host arithmetic only, no CUDA.
#pragma once

#include <algorithm>

namespace ovl {

// bytes of one shared-memory body slot: with the inverse mass and inertia, or without
constexpr int solve_slot_bytes(bool masses) { return masses ? 32 : 24; }

// a CTA's slots and its zero slot
constexpr long long solve_smem_bytes(long long slots, bool masses) { return (slots + 1) * solve_slot_bytes(masses); }

// the dynamic shared memory a CTA of the launch with the masses asks for:
// slots, the impulses of its rows (12 B each, padded to 16) and `stage` bytes,
// as far as the budget goes.  64-bit: a worker may have more rows than 32-bit bytes.
inline int solve_dynamic_bytes(int budget, long long slots, long long rows, long long stage) {
    return (int)std::min<long long>(budget, solve_smem_bytes(slots, true) + 12 * rows + 16 + stage);
}

// Rows a CTA of a worker's group of C makes room for: its even share, plus a
// quarter (and a little) for uneven owners.
inline long long solve_cta_rows(long long np, int C) { return C == 1 ? np : (long long)(1.25 * np / C) + 64; }

// the most of them over P workers, worker p's rows being [start[p], start[p + 1])
inline long long solve_most_rows(const int *start, int P, int C) {
    long long most = 0;
    for (int p = 0; p < P; ++p) most = std::max(most, solve_cta_rows((long long)start[p + 1] - start[p], C));
    return most;
}

}  // namespace ovl
