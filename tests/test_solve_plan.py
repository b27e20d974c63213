"""Sizes of the solve's launches (csrc/solve_plan.h), host arithmetic that
needs no GPU."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

EXPORTS = r"""
#include "csrc/solve_plan.h"
extern "C" {
int dynamic_bytes(int budget, long long slots, long long rows, long long stage) {
    return ovl::solve_dynamic_bytes(budget, ovl::solve_worker_room((int)slots, rows, 1, 1ll << 62), stage);
}
int takes_masses(int threads, long long ctas, int sms, int per_sm, long long slots) {
    return ovl::solve_takes_masses(threads, ctas, sms, per_sm, slots);
}
int full_kind(long long full, long long rows, int bodies) { return ovl::solve_full_kind(full, rows, bodies); }
double grow_rows(long long full, long long rows, int bodies, int jointed) { return ovl::solve_grow_rows(full, rows, bodies, jointed); }
int box_threads(int threads, int ctas_per_sm) { return ovl::solve_box_threads(threads, ctas_per_sm); }
int slot_capacity(int optin, int per_sm, int ctas, int masses) { return ovl::solve_slot_capacity(optin, per_sm, ctas, masses); }
long long most_room(const int *b, const int *q, int P, int C) { return ovl::solve_most_room(b, q, P, C, 1ll << 62); }
long long worker_room(int nb, long long np, int C, long long budget) { return ovl::solve_worker_room(nb, np, C, budget); }
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("needs g++")
    d = tmp_path_factory.mktemp("plan")
    src, so = d / "plan.cpp", d / "plan.so"
    src.write_text(EXPORTS)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I",
                           os.path.join(ROOT, "paper_2403_17261_gb300"), str(src), "-o", str(so)])
    lib = ctypes.CDLL(str(so))
    L = ctypes.c_longlong
    lib.dynamic_bytes.argtypes = [ctypes.c_int, L, L, L]
    lib.full_kind.argtypes = [L, L, ctypes.c_int]
    lib.grow_rows.argtypes = [L, L, ctypes.c_int, ctypes.c_int]
    lib.grow_rows.restype = ctypes.c_double
    lib.takes_masses.argtypes = [ctypes.c_int, L, ctypes.c_int, ctypes.c_int, L]
    lib.worker_room.argtypes = [ctypes.c_int, L, ctypes.c_int, L]
    lib.worker_room.restype = L
    lib.most_room.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int, ctypes.c_int]
    lib.most_room.restype = L
    return lib


@pytest.mark.parametrize("rows", [178_956_971, 200_000_000, 1 << 31])
def test_rows_beyond_32_bit_bytes_take_the_budget(plan, rows):
    """12 B per row of that many rows are more than 2^31"""
    assert plan.dynamic_bytes(220_000, 1000, rows, 0) == 220_000


def test_small_launches_take_what_they_need(plan):
    assert plan.dynamic_bytes(220_000, 99, 200, 0) == 100 * 32 + 200 * 12 + 16
    assert plan.dynamic_bytes(220_000, 99, 200, 65536) == 100 * 32 + 200 * 12 + 16 + 65536


def _starts(counts):
    return (ctypes.c_int * (len(counts) + 1))(*[sum(counts[:i]) for i in range(len(counts) + 1)])


def _room(plan, bodies, rows, C):
    return plan.most_room(_starts(bodies), _starts(rows), len(rows), C)


@pytest.mark.parametrize("rows,C,want", [
    ([10], 1, 10),
    ([10, 490, 10], 1, 490),                # the largest worker's rows, not the sum
    ([10, 490, 10], 4, 153 + 64),
    ([300] * 600, 1, 300),
    ([0, 0], 2, 64),
])
def test_uniform_launch_makes_room_for_its_largest_worker(plan, rows, C, want):
    assert _room(plan, [0] * len(rows), rows, C) == 32 + 12 * want + 16


@pytest.mark.parametrize("bodies,rows,C,want", [
    ([974, 300], [300, 1900], 1, (974 + 1) * 32 + 12 * 300 + 16),       # not 974 bodies with 1900 rows
    ([300, 200], [300, 1900], 1, (200 + 1) * 32 + 12 * 1900 + 16),
    ([301, 10], [100, 20], 2, (151 + 1) * 32 + 12 * (62 + 64) + 16),
])
def test_room_is_one_workers(plan, bodies, rows, C, want):
    assert _room(plan, bodies, rows, C) == want


def test_no_workers_want_no_room(plan):
    assert plan.most_room(_starts([]), _starts([]), 0, 1) == 0


@pytest.mark.parametrize("ctas,masses,static", [(1, 0, 1808), (2, 0, 1808), (1, 1, 2192), (2, 1, 2192)])
def test_slots_fill_the_shared_memory(plan, ctas, masses, static):
    """static: the kernels' own (ptxas -v).  One more KB of slots would not fit beside it."""
    optin, per_sm, system = 232448, 233472, 1024
    slot = 32 if masses else 24
    used = (plan.slot_capacity(optin, per_sm, ctas, masses) + 1) * slot + static
    most = optin if ctas == 1 else per_sm // 2 - system
    assert used <= most
    assert used + 1024 > most
    # the layout without the masses gives nothing to the other kernel's tables
    assert masses or used + 256 > most - 15


@pytest.mark.parametrize("threads,ctas,slots,masses", [
    (512, 152, 200, 1),          # every CTA has an SM of its own
    (512, 153, 200, 0),          # two per SM: the registers leave one
    (512, 153, 4600, 0),
    (512, 153, 8000, 1),         # but the slots leave one too
    (256, 1200, 200, 0),
    (256, 512, 3500, 1),         # two per SM, by registers and by slots
    (256, 512, 2500, 1),         # two and three
    (256, 512, 2000, 0),         # two and four
    (128, 152 * 7, 200, 1),
    (128, 152 * 7 + 1, 200, 0),
    (32, 152 * 16, 20, 1),
    (1024, 100, 200, 1),
])
def test_ctas_that_share_an_sm_find_registers(plan, threads, ctas, slots, masses):
    assert plan.takes_masses(threads, ctas, 152, 233472, slots) == masses


@pytest.mark.parametrize("threads,ctas,want", [(512, 1, 256), (256, 1, 256), (96, 1, 96), (256, 2, 128), (512, 2, 128), (64, 2, 64)])
def test_box_ctas_leave_room_for_their_stages(plan, threads, ctas, want):
    """two CTAs per SM: 128 threads, whose two stages of 16 records take 64 KB of the half SM's 110"""
    assert plan.box_threads(threads, ctas) == want
    assert 2 * 16 * 16 * want < (232448 if ctas == 1 else 233472 // 2 - 3584)


@pytest.mark.parametrize("full,rows,bodies,kind", [
    (0, 40_000, 14_000, 0),       # no box end: the spheres' kernel
    (1, 40_000, 14_000, 1),       # one box does not change its worker's launch
    (2000, 40_000, 14_000, 1),
    (28_000, 40_000, 14_000, 2),
    (250, 1000, 300, 2),
    (249, 1000, 300, 1),
    (250, 1000, 1001, 1),
    (4200, 4200, 170, 2),         # the building
])
def test_full_rows_of_a_worker(plan, full, rows, bodies, kind):
    assert plan.full_kind(full, rows, bodies) == kind


@pytest.mark.parametrize("full,rows,bodies,jointed,want", [
    (0, 5000, 1700, 0, 5000.0),
    (500, 3000, 1100, 0, 5500.0),
    (500, 2400, 1100, 0, 2400.0),
    (4200, 4200, 170, 0, 4200.0),
    (4200, 4200, 170, 1, 4200.0),
    (0, 2200, 1250, 0, 2200.0),               # few rows per body, but the fullest body sets the colours
    (0, 2200, 1250, 1, 13.5 / 2.9 * 1250),    # a chain: five colours where a pile has 13
    (0, 60_000, 10_000, 1, 60_000.0),
    (0, 0, 0, 1, 0.0),
])
def test_rows_in_the_growth(plan, full, rows, bodies, jointed, want):
    assert plan.grow_rows(full, rows, bodies, jointed) == pytest.approx(want, rel=1e-12)


@pytest.mark.parametrize("nb,np,C,fits", [(1000, 16000, 1, True), (1000, 17000, 1, False), (7500, 75000, 4, False),
                                          (7500, 56000, 4, True), (7183, 0, 1, True), (7184, 0, 1, False)])
def test_no_room_for_impulses_that_do_not_fit(plan, nb, np, C, fits):
    """an even share beyond the budget leaves the rest of the shared memory to the L1 cache"""
    slots = ((nb + C - 1) // C + 1) * 32
    rows = np if C == 1 else int(1.25 * np / C) + 64
    assert plan.worker_room(nb, np, C, 229888) == slots + (12 * rows + 16 if fits else 0)
