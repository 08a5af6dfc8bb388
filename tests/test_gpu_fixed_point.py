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


# --------------------------------------------- symmetric and float-float products
# Sizes around the symmetric kernel's limits: 20 tiles of 128 points (2432 and
# 2433), ragged last tiles, the step to wider tiles, one to four right-hand
# sides (five take the rectangular kernel), one point past 16 coordinates.
# Float64: |error| <= (N + 64) 2^-53 sum |a v| as above with the entries' own
# bound; float-float: 2^-44 sum |a v| for the entries (d 2^(2 e - 56) and 2^-46
# of their value) plus N 2^-47 sum |a v| for the sums' low parts.
SYM = [(2432, 8, 1), (2433, 8, 2), (2500, 3, 4), (3001, 17, 3), (2700, 32, 1), (17950, 4, 1),
       (3000, 8, 5)]


@pytest.mark.parametrize("prec", ["fp64", "ff"])
@pytest.mark.parametrize("kern", [O.GAUSSIAN, O.LAPLACE_L1, O.MATERN52])
@pytest.mark.parametrize("N,d,m", SYM)
def test_symmetric_product(K, prec, kern, N, d, m):
    if N > 4000 and kern != O.GAUSSIAN:
        pytest.skip("one kernel at the larger size")
    rng = np.random.default_rng(N + d + m)
    X, V = rng.standard_normal((N, d)), rng.standard_normal((m, N))
    X[5] = X[4]
    X[N - 1] = X[0] + 1e-8
    sigma = 1.0 + d / 8.0
    rows = np.unique(np.concatenate([[0, 4, 5, N - 1], rng.integers(0, N, 400)]))
    got = K.krr_kmatvec(to_dev(X), kern, sigma, 0.25, to_dev(V), prec=prec).cpu().numpy()[:, rows]
    ref = O.kmatvec(X, kern, sigma, 0.25, V, rows)
    scale = O.kmatvec(X, kern, sigma, 0.25, np.abs(V), rows)
    eps = (N + 64) * 2.0 ** -53 if prec == "fp64" else 2.0 ** -44 + N * 2.0 ** -47
    assert np.all(np.abs(got - ref) <= eps * scale)


@pytest.mark.parametrize("kern", [O.GAUSSIAN, O.LAPLACE_L1, O.MATERN52])
def test_float_float_beyond_the_range(K, kern):
    """Points too spread for the fixed-point float-float product take the
    float-float kernels, to the same bound."""
    rng = np.random.default_rng(1)
    N = 2600
    X, V = 300.0 * rng.standard_normal((N, 5)), rng.standard_normal((2, N))
    X[:50] = X[50:100] + rng.standard_normal((50, 5))
    got = K.krr_kmatvec(to_dev(X), kern, 1.0, 0.25, to_dev(V), prec="ff").cpu().numpy()
    ref = O.kmatvec(X, kern, 1.0, 0.25, V)
    scale = O.kmatvec(X, kern, 1.0, 0.25, np.abs(V))
    # beyond the float-float coordinates' own 2^-48 |x| = 2^-39: dE <= 2 |d| 2^-39 sqrt(d)
    assert np.all(np.abs(got - ref) <= 2.0 ** -34 * scale)
