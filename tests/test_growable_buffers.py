"""A growable buffer whose reallocation fails holds nothing: a later request
may not be answered with the memory that was freed to make room.  The CUDA
calls are fakes, so this needs no GPU."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include <cstdio>
#include <cstdlib>
#include <set>
#include "csrc/common.cuh"

static std::set<void *> live;
static int failures;          // calls from now on that fail
static cudaError_t take(void **p, size_t n) {
    if (failures) { --failures; return cudaErrorMemoryAllocation; }
    live.insert(*p = std::malloc(n));
    return cudaSuccess;
}
static cudaError_t give(void *p) {
    if (!live.erase(p)) return cudaErrorInvalidValue;   // freed twice
    std::free(p);
    return cudaSuccess;
}
extern "C" {
cudaError_t cudaMalloc(void **p, size_t n) { return take(p, n); }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { return take(p, n); }
cudaError_t cudaFree(void *p) { return give(p); }
cudaError_t cudaFreeHost(void *p) { return give(p); }
}

template <class B>
int check() {
    B b;
    b.ensure(100);
    failures = 1;
    bool refused = false;
    try { b.ensure(100000); } catch (const ovl::CudaError &) { refused = true; }
    if (!refused) return 1;
    b.ensure(10);                       // within what was freed
    if (!live.count(b.p)) return 2;
    b.release();
    return live.empty() ? 0 : 3;
}

int main() {
    const int d = check<ovl::DBuf<int>>(), h = check<ovl::HBuf<int>>();
    std::printf("%d %d\n", d, h);
    return d || h;
}
"""


def test_failed_growth_leaves_an_empty_buffer(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if not shutil.which("g++") or not os.path.exists(os.path.join(inc, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    src, exe = tmp_path / "h.cpp", tmp_path / "h"
    src.write_text(HARNESS)
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2403_17261_gb300"), "-I", inc,
                        str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.split() == ["0", "0"], r.stdout + r.stderr
