"""Arithmetic that kernels and host code share through csrc/layout.h, compiled for the host and checked there."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2411_10666_b200", "csrc")
SOURCE = """
#include "layout.h"
extern "C" int64_t grid_index(uint32_t block, uint32_t threads, uint32_t thread) { return (int64_t)sam_grid_index(block, threads, thread); }
extern "C" int64_t grid_size(uint32_t blocks, uint32_t threads) { return (int64_t)sam_grid_size(blocks, threads); }
extern "C" uint64_t path_max() { return SAM_PATH_MAX; }
// pointer jumping over the chain 0 -> 1 -> ... -> n, one state after the other in the order given
extern "C" void path_pass(uint64_t* path, const int64_t* order, int64_t n) {
    for (int64_t k = 0; k < n; k++) {
        const int64_t s = order[k];
        const uint32_t steps = (uint32_t)path[s];
        if (steps == 0 || steps >= SAM_PATH_MAX) continue;
        const uint64_t q = path[path[s] >> 32];
        if ((uint32_t)q != 0) path[s] = sam_path_join(path[s], q);
    }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("layout")
    src, out = str(d / "layout_test.cpp"), str(d / "layout_test.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.check_call([os.environ.get("NVCC", "nvcc"), "-O1", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", CSRC, "-o", out, src])
    L = ctypes.CDLL(out)
    L.path_max.restype = ctypes.c_uint64
    L.grid_index.restype = L.grid_size.restype = ctypes.c_int64
    return L


@pytest.mark.parametrize("order", ["up", "down", "mixed"])
def test_a_path_never_has_more_steps_than_a_tree_entry_holds(lib, order):
    """A passage of more than 65536 tokens that occurs twice: whatever the order in which states are taken, steps stay within
    the 16 bits beside an entry's flags, no path becomes empty, and a path below the bound ends where it says."""
    n, most = 200_000, lib.path_max()
    path = np.array([(s + 1) << 32 | 1 for s in range(n)] + [n << 32], dtype=np.uint64)
    visit = np.arange(n, dtype=np.int64)
    if order == "down":
        visit = visit[::-1].copy()
    elif order == "mixed":
        np.random.default_rng(1).shuffle(visit)
    for _ in range(7):
        lib.path_pass(path.ctypes.data_as(ctypes.c_void_p), visit.ctypes.data_as(ctypes.c_void_p), ctypes.c_int64(n))
    steps, end = (path & 0xFFFFFFFF).astype(np.int64)[:n], (path >> 32).astype(np.int64)[:n]
    left = n - np.arange(n)
    assert most < 1 << 16 and (steps >= np.minimum(left, 128)).all() and (steps <= most).all()
    exact = steps < most
    assert np.array_equal(end[exact], np.arange(n)[exact] + steps[exact]) and (steps[exact] <= left[exact]).all()


def test_thread_numbers_at_the_largest_batch(lib):
    """2^24 slots, a block of 128 threads each, clear the batch: thread numbers and the grid's size pass 2^31."""
    slots, threads = 1 << 24, 128
    assert lib.grid_size(slots, threads) == slots * threads == 1 << 31
    assert lib.grid_index(slots - 1, threads, threads - 1) == (1 << 31) - 1
