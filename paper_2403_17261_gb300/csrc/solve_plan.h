// solve_plan.h -- sizes of the solve's launches: host arithmetic only, no CUDA.
#pragma once

#include <algorithm>

namespace ovl {

constexpr int SOLVE_THREADS = 512;   // most threads of a CTA

// bytes of one shared-memory body slot: with the inverse mass and inertia, or without
constexpr int solve_slot_bytes(bool masses) { return masses ? 32 : 24; }

// a CTA's slots and its zero slot
constexpr long long solve_smem_bytes(long long slots, bool masses) { return (slots + 1) * solve_slot_bytes(masses); }

// Dynamic shared memory a CTA may use with one resident CTA per SM (of the
// `optin` bytes a block may have) or two (of the SM's `per_sm`, less 1 KB that
// the system takes per block), beside its static memory: 1.8 KB of row-bucket
// offsets and reductions without the masses, 2.2 KB with them.
inline int solve_smem_budget(int optin, int per_sm, int ctas_per_sm, bool masses) {
    const int fixed = masses ? 2560 : 2048;
    return ctas_per_sm == 1 ? optin - fixed : per_sm / 2 - 1024 - fixed;
}

// body slots of that memory, less the CTA's zero slot
inline int solve_slot_capacity(int optin, int per_sm, int ctas_per_sm, bool masses) {
    return std::max(0, solve_smem_budget(optin, per_sm, ctas_per_sm, masses) / solve_slot_bytes(masses) - 1);
}

// Rows a CTA of a worker's group of C makes room for: its even share, plus a
// quarter (and a little) for uneven owners.
inline long long solve_cta_rows(long long np, int C) { return C == 1 ? np : (long long)(1.25 * np / C) + 64; }

// Shared memory a CTA of the launch with the masses wants for a worker of nb
// bodies and np rows: slots and the impulses of its rows (12 B each, padded to
// 16), or the slots alone when an even share of the impulses already exceeds
// the budget: what no impulses will fill is better left to the L1 cache, which
// holds row records (30,000 spheres of mixed radii, 8 workers of 75,000 rows:
// 1.66 ms with the whole budget, 1.50 without; 100,000, 2.36 and 2.15).
// 64-bit: a worker may have more rows than 32-bit bytes.
inline long long solve_worker_room(int nb, long long np, int C, long long budget) {
    const long long slots = solve_smem_bytes((nb + C - 1) / C, true);
    return slots + (slots + 12 * (np / C) > budget ? 0 : 12 * solve_cta_rows(np, C) + 16);
}

// The most of it over P workers, bodies and rows of worker p from b[p] and
// q[p] on.  The worker with the most bodies is seldom the one with the most
// rows (a chain has one row per body, a pile three), so the maximum is taken
// over workers, not over bodies and rows apart.
inline long long solve_most_room(const int *b, const int *q, int P, int C, long long budget) {
    long long most = 0;
    for (int p = 0; p < P; ++p)
        most = std::max(most, solve_worker_room(b[p + 1] - b[p], (long long)q[p + 1] - q[p], C, budget));
    return most;
}

// the dynamic shared memory of that launch: the room and `stage` bytes, as far as the budget goes
inline int solve_dynamic_bytes(int budget, long long room, long long stage) {
    return (int)std::min<long long>(budget, room + stage);
}

// Whether a launch of one row per thread whose slots fit with the masses takes
// the kernel that keeps them and the impulses in shared memory (k_solve_m).
// Its 91 to 124 registers leave an SM 512 / threads CTAs; the kernel without
// them has 64 and leaves twice as many, if its slots fit that often and there
// are CTAs enough.  The launch gives the masses up only where the other kernel
// runs twice as many CTAs at once: a row costs it about 15 % more.  (Solves,
// ms, with and without: 1200 small workers with 256 threads 0.54 and 0.30,
// with 512 threads 0.99 and 0.53, two CTAs each 3.66 and 2.52; 64 workers of
// eight 512-thread CTAs 2.43 and 1.50, larger ones 4.55 and 3.83; of eight
// 256-thread CTAs, two or three of which share an SM, 3.55 and 3.87.)
inline bool solve_takes_masses(int threads, long long ctas, int sms, int per_sm, long long slots) {
    const long long other = std::min<long long>(std::max(1, 1024 / threads),
                                                std::max(1ll, per_sm / (solve_smem_bytes(slots, false) + 3072)));
    return 2 * std::max(1, 512 / threads) > std::min(other, (ctas + sms - 1) / sms);
}

// How many of a worker's rows are full rows (a box end), as its launch takes
// them.  The kernel for workers of boxes (FULL_MOST) copies the full row of a
// thread's first row of a colour to shared memory ahead of use, which leaves a
// CTA half the threads: 256 rows of a colour in one pass.  It pays where seven
// in ten rows are full, or a quarter in a worker of up to 1000 bodies (a colour
// holds a body once, so about bodies / 2.6 rows).  Other workers with full rows
// (FULL_FEW) keep the spheres' CTAs.  (Solves of piles with boxes, ms, as
// FULL_FEW and as FULL_MOST: 8 workers of about 1600 bodies, 2 % of them boxes,
// 0.71 and 0.96, 20 % 1.25 and 1.54, 75 % 2.46 and 1.89; 8 of 450, 20 %, 1.09
// and 0.77; 8 of 800, 20 %, 1.06 and 0.95.)
enum { FULL_NONE, FULL_FEW, FULL_MOST };
inline int solve_full_kind(long long full, long long rows, int bodies) {
    if (full == 0) return FULL_NONE;
    return 10 * full >= 7 * rows || (4 * full >= rows && bodies <= 1000) ? FULL_MOST : FULL_FEW;
}

// Rows as the growth of a worker's CTAs counts them, in rows of a pile (three
// per body, 13 colours).  Where few are full, such a row, read straight from
// global memory, costs as much as six plain ones; below 2500 rows a worker has
// too few to share.  (One and four CTAs per worker, a sixth of the rows full:
// 2200 rows 0.53 and 0.61 ms, 2800 0.66 and 0.61, 4300 0.87 and 0.63; spheres
// cross at 5000.)  Where joints outnumber contacts the colours are few, about
// 2.9 per row and body, so a worker has more rows in each (a chain, one CTA and
// four: 1100 rows 0.13 and 0.15 ms, 2200 0.21 and 0.15, 4400 0.39 and 0.18).
// Contacts alone do not say so: the fullest body sets the colours.
inline double solve_grow_rows(long long full, long long rows, int bodies, bool jointed) {
    const int kind = solve_full_kind(full, rows, bodies);
    if (kind == FULL_MOST) return (double)rows;
    const double plain = kind == FULL_FEW && rows >= 2500 ? rows + 5.0 * full : (double)rows;
    return jointed && rows > 0 ? plain * std::max(1.0, 13.5 / 2.9 * bodies / rows) : plain;
}

// Rows a thread takes at once in a colour: with the masses one (k_solve_m), the
// kernels with full rows that read the masses two, else what the shape asks for.
inline int solve_rows_at_once(bool masses, int full, int rows_per_thread) {
    return masses ? 1 : (full != FULL_NONE ? 2 : rows_per_thread);
}

// Threads of a CTA that keeps the masses of a worker of boxes: at most 256
// (its 155 to 226 registers leave no more), and 128 where it is to share its SM
// with another, which 256 leave neither the registers nor, for the two stages
// of full rows (512 B per thread), the shared memory.  (Solves of box batches,
// ms, with 256 and 128 threads: 400 small workers 1.56 and 0.86, 192 of 2500
// rows 3.87 and 1.88, 320 of 4200 6.97 and 4.90.)
inline int solve_box_threads(int threads, int ctas_per_sm) { return std::min(threads, ctas_per_sm == 1 ? 256 : 128); }

}  // namespace ovl
