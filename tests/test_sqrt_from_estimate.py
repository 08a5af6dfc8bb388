"""Square root and inverse from a float32 estimate (csrc/rsqrt.cuh, on the host).

For estimates off by up to 2^-21 (the device's float32 reciprocal square root: 2
units of its last place, and the rounding of the argument) the root is within 0.51
units of the last place, so at most one neighbour from the correctly rounded one,
and the inverse within 2^-53 (rounding) + 2^-54 (e) + 2^-58 of it.
"""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2304_12465_gb300", "csrc")
HARNESS = r"""
#include "rsqrt.cuh"
extern "C" void run(int n, const double *p, const double *y, double *d, double *r) {
  for (int i = 0; i < n; ++i) krr::sqrt_from_estimate(p[i], y[i], d + i, r + i);
}
"""


@pytest.mark.parametrize("exponents", [(-100, 100), (-2, 2)])   # the whole range, around 1
def test_against_the_library(tmp_path, exponents):
    (tmp_path / "h.cpp").write_text(HARNESS)
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-std=c++17", "-shared", "-fPIC",
                    f"-I{CSRC}", str(tmp_path / "h.cpp"), "-o", str(tmp_path / "h.so")], check=True)
    run = C.CDLL(str(tmp_path / "h.so")).run
    rng = np.random.default_rng(6)
    n = 200_000
    p = np.ldexp(1 + rng.random(n), rng.integers(*exponents, n).astype(np.int32))
    p[:8] = [1.0, 2.0, 4.0, 1 + 2.0 ** -52, 1 - 2.0 ** -53, 4 - 2.0 ** -51, 1e-30, 1e30]
    off = rng.uniform(-1, 1, n) * 2.0 ** -21
    off[: n // 4] = np.sign(off[: n // 4]) * 2.0 ** -21
    off[n // 4: n // 2] = 0
    y = ((1 + off) / np.sqrt(p)).astype(np.float64)
    d, r = np.empty(n), np.empty(n)
    ptr = lambda a: a.ctypes.data_as(C.POINTER(C.c_double))
    run(n, ptr(p), ptr(y), ptr(d), ptr(r))
    root = np.sqrt(p.astype(np.longdouble))
    assert np.all(np.abs(d - root) <= 0.51 * np.spacing(np.sqrt(p)))
    assert np.all(np.abs(d - np.sqrt(p)) <= np.spacing(np.sqrt(p)))
    assert np.all(np.abs(r * root - 1) <= 1.5 * 2.0 ** -53 + 2.0 ** -58)
