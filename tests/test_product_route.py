"""Kernel choice of a float32 product (csrc/route.cuh, compiled for the host).

Whatever path the process asks for, the chosen kernel has operands; the asked
one is taken where it has them.  Points that carry tcgen05 operands alone and
a path changed after their preparation are the case that used to launch the FMA
kernel on NULL pointers.
"""
import ctypes as C
import itertools
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2304_12465_gb300", "csrc")
TCGEN05, FMA, MMA_SYNC, NONE = 0, 1, 2, -1


@pytest.fixture(scope="module")
def route(tmp_path_factory):
    d = tmp_path_factory.mktemp("route")
    (d / "h.cpp").write_text('#include "route.cuh"\nextern "C" int route(int p, int t, int m, int f)'
                             "{ return krr::product_route(p, t, m, f); }")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", f"-I{CSRC}", str(d / "h.cpp"), "-o",
                    str(d / "h.so")], check=True)
    return C.CDLL(str(d / "h.so")).route


@pytest.mark.parametrize("path", [TCGEN05, FMA, MMA_SYNC])
def test_the_chosen_kernel_has_operands(route, path):
    for tc5, mma, fma in itertools.product([0, 1], repeat=3):
        have = {TCGEN05: tc5, MMA_SYNC: mma, FMA: fma}
        got = route(path, tc5, mma, fma)
        assert have[got] if any(have.values()) else got == NONE
        if have[path]:
            assert got == path


def test_path_changed_after_the_preparation(route):
    assert [route(p, 1, 0, 0) for p in (TCGEN05, FMA, MMA_SYNC)] == [TCGEN05] * 3
    assert route(TCGEN05, 0, 1, 1) == MMA_SYNC     # points beyond the tcgen05 split
    assert route(MMA_SYNC, 1, 0, 1) == FMA
