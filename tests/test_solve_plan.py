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
    return ovl::solve_dynamic_bytes(budget, slots, rows, stage);
}
long long most_rows(const int *start, int P, int C) { return ovl::solve_most_rows(start, P, C); }
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
    lib.most_rows.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int]
    lib.most_rows.restype = L
    return lib


@pytest.mark.parametrize("rows", [178_956_971, 200_000_000, 1 << 31])
def test_rows_beyond_32_bit_bytes_take_the_budget(plan, rows):
    """12 B per row of that many rows are more than 2^31"""
    assert plan.dynamic_bytes(220_000, 1000, rows, 0) == 220_000


def test_small_launches_take_what_they_need(plan):
    assert plan.dynamic_bytes(220_000, 99, 200, 0) == 100 * 32 + 200 * 12 + 16
    assert plan.dynamic_bytes(220_000, 99, 200, 65536) == 100 * 32 + 200 * 12 + 16 + 65536


@pytest.mark.parametrize("rows,C,want", [
    ([10], 1, 10),
    ([10, 490, 10], 1, 490),                # the largest worker's rows, not the sum
    ([10, 490, 10], 4, 153 + 64),
    ([300] * 600, 1, 300),
    ([0, 0], 2, 64),
    ([], 1, 0),
])
def test_uniform_launch_makes_room_for_its_largest_worker(plan, rows, C, want):
    start = (ctypes.c_int * (len(rows) + 1))(*[sum(rows[:i]) for i in range(len(rows) + 1)])
    assert plan.most_rows(start, len(rows), C) == want
