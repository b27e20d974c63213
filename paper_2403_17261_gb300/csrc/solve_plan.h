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

}  // namespace ovl
