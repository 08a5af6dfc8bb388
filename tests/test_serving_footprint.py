"""The serving engine's admission estimate charges the residual product's
scratch by the shape that the product takes (host only).

The symmetric product holds nt (nt + 1) M RT float64 sums for nt tiles of RT
points and serves up to four right-hand sides and 4 GiB; other shapes hold a
few sums a row (at most 3648 / (N / 256) + 1 splits), far below 1 GiB here.
"""
import ctypes as C

import pytest

import paper_2304_12465_gb300 as K

GIB = 2.0 ** 30


def footprint(N, d, m, k=1):
    lib = K.load()
    b = C.c_double()
    assert lib.krr_server_footprint(N, d, m, k, C.byref(b)) == 0
    return b.value


# everything else a request holds: 1.05 (32 N M split sums of the float32
# product, 8 N d points and 4.6 times that prepared, 52 N m vectors, 60 N) + 16 MiB
def others(N, d, m):
    M = 1 << (m - 1).bit_length()
    return 1.05 * N * (32 * 4 * M + 45 * d + 64 * 2 + 60 * m + 60) + 2 ** 24


@pytest.mark.parametrize("N,m", [(100_000, 5), (100_000, 16), (300_000, 16), (1_000_000, 4),
                                 (1_000_000, 16), (400_000, 4), (2000, 4)])
def test_no_symmetric_scratch_where_it_is_not_taken(N, m):
    M = 1 << (m - 1).bit_length()
    splits = 1.05 * min(3648 / (N / 256) + 2, N / 32 + 1) * M * N * 8
    assert footprint(N, 8, m) <= others(N, 8, m) + splits


@pytest.mark.parametrize("N,m,RT", [(2560, 4, 128), (200_000, 4, 1024), (300_000, 1, 1024)])
def test_symmetric_scratch_is_charged(N, m, RT):
    M = 1 << (m - 1).bit_length()
    nt = -(-N // RT)
    scratch = nt * (nt + 1) * M * RT * 8
    assert scratch <= 4 * GIB
    assert footprint(N, 8, m) >= scratch
