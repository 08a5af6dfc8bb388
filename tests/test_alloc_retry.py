"""Allocations that fail give the library's unused pool memory back and try again
(csrc/retry.cuh, compiled for the host with fakes of the calls)."""
import ctypes as C
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2304_12465_gb300", "csrc")
HARNESS = r"""
#include "retry.cuh"
// `fails` calls of the allocator fail with 2; *log counts calls and trims
extern "C" int run(int fails, int have_pool, int *log) {
  return krr::alloc_or_trim(0, [&] { return log[0]++ < fails ? 2 : 0; },
                            [&] { ++log[1]; return have_pool != 0; });
}
"""


@pytest.mark.parametrize("fails,pool,want,calls,trims", [
    (0, 1, 0, 1, 0),    # nothing to mend
    (1, 1, 0, 2, 1),    # the pool held the memory
    (2, 1, 2, 2, 1),    # really out of memory: one retry
    (1, 0, 2, 1, 1),    # no pool: the first error stands
])
def test_one_retry_after_the_trim(tmp_path, fails, pool, want, calls, trims):
    (tmp_path / "h.cpp").write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", f"-I{CSRC}", str(tmp_path / "h.cpp"),
                    "-o", str(tmp_path / "h.so")], check=True)
    log = (C.c_int * 2)()
    assert C.CDLL(str(tmp_path / "h.so")).run(fails, pool, log) == want
    assert list(log) == [calls, trims]


def test_persistent_allocations_take_it():
    """Every device allocation of the library goes through the two functions that
    trim; the raw calls stand in them alone."""
    raw = {}
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        n = text.count("cudaMalloc(") + text.count("cudaMallocAsync(") + \
            text.count("cudaMallocFromPoolAsync(")
        if n:
            raw[name] = n
    assert raw == {"abi.cu": 3}
