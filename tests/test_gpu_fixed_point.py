"""GPU parity of the fixed-point float64 products and kernel columns.

Kernel entries are read out with unit right-hand sides and compared with the
oracle's float64 entries.  Tolerance: the oracle rounds every difference,
square, sum and the exponent E (at most (d + 6) E units of 2^-53), the fixed
point its coordinates (2 sqrt(d E) units at the largest accepted range, d
2^(e - 5) for Laplace) and both the result (4 units).  Point sets beyond the
accepted range, or with a non-finite value, take the float64 kernels and must
agree to the same bound.
"""
import numpy as np
import pytest

import oracle as O
from gpu_common import require_gpu, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def K():
    return require_gpu()


def bound(ref, d):
    with np.errstate(divide="ignore"):
        E = np.where(ref > 0, -np.log(np.maximum(ref, 1e-307)), 0.0)
    return 2.0 ** -53 * ref * (6 + (d + 8) * E + 2 * np.sqrt(d * E) + d) + 2.0 ** -1020


@pytest.mark.parametrize("kern", [O.GAUSSIAN, O.LAPLACE_L1, O.MATERN52])
@pytest.mark.parametrize("N,d,m,spread,sigma", [
    (1, 1, 1, 1.0, 1.0),            # one point: the smallest range
    (31, 3, 2, 1.0, 2.0),           # one ragged tile
    (257, 8, 16, 1.0, 0.7),         # one row past a tile
    (1000, 16, 5, 3.0, 1.0),        # two rows a thread, ragged columns
    (513, 17, 3, 1.0, 0.5),         # one row a thread
    (300, 32, 1, 1.0, 8.0),
    (300, 4, 4, 1e3, 1.0),          # beyond the accepted range: float64 kernels
    (300, 4, 4, 1e-9, 1.0),         # all points nearly equal
])
def test_entries(K, kern, N, d, m, spread, sigma):
    rng = np.random.default_rng(N + d)
    X = spread * rng.standard_normal((N, d)) + 7.0
    if N > 4:
        X[1] = X[0]
        X[3] = X[2] + 1e-7 * rng.standard_normal(d)
    cols = rng.permutation(N)[:min(m, N)]
    V = np.zeros((m, N))
    for c, j in enumerate(cols):
        V[c, j] = 1.0
    got = K.krr_kmatvec(to_dev(X), kern, sigma, 0.0, to_dev(V), prec="fp64").cpu().numpy()
    ref = O.kernel_block(X, kern, sigma, None, cols.astype(np.int64)).T
    assert np.all(np.abs(got[:len(cols)] - ref) <= bound(ref, d))
    # rectangular, with rows the column set's range does not cover
    T = spread * 1.5 * rng.standard_normal((97, d)) + 7.0
    got = K.krr_predict(to_dev(X), kern, sigma, to_dev(V), to_dev(T), prec="fp64").cpu().numpy()
    XT = np.vstack([X, T])
    ref = O.kernel_block(XT, kern, sigma, np.arange(N, N + 97), cols.astype(np.int64)).T
    assert np.all(np.abs(got[:len(cols)] - ref) <= bound(ref, d))


@pytest.mark.parametrize("kern", [O.GAUSSIAN, O.LAPLACE_L1, O.MATERN52])
def test_non_finite_points_reach_the_result(K, kern):
    rng = np.random.default_rng(3)
    X = rng.standard_normal((200, 5))
    X[17, 2] = np.nan
    X[44, 0] = np.inf
    got = K.krr_kmatvec(to_dev(X), kern, 1.0, 0.5, to_dev(rng.standard_normal((2, 200))),
                        prec="fp64").cpu().numpy()
    assert np.all(np.isnan(got[:, 17]))
    assert np.all(np.isnan(got))      # every row meets the NaN point


@pytest.mark.parametrize("N", [700, 4096])
def test_reduction_of_many_splits(K, N):
    rng = np.random.default_rng(N)
    X, V = rng.standard_normal((N, 6)), rng.standard_normal((3, N))
    got = K.krr_kmatvec(to_dev(X), 0, 1.0, 0.3, to_dev(V), prec="fp64").cpu().numpy()
    ref = O.kmatvec(X, 0, 1.0, 0.3, V)
    scale = O.kmatvec(X, 0, 1.0, 0.3, np.abs(V))
    assert np.all(np.abs(got - ref) <= (N + 64) * 2.0 ** -53 * scale)
