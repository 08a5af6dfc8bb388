"""Accuracy of the factor where it is nearly sparse.

Points far apart in units of sigma: F is 1 at its pivots and small elsewhere, and
an update subtracts products of small rows from small entries.  The reference
repeats Alg. 3's recursion on the same pivots in long double.  Every entry is
rounded at 2^-53 of itself a few times, and the products by digits are off by about
2^-57 of their rows' norms, so the Frobenius norm of the error stays within two
units of 2^-53 of the factor's (float64 sums: half a unit; digits without the rows'
own scales: four).
"""
import numpy as np
import pytest

import oracle as O
from gpu_common import require_gpu, to_dev

pytestmark = pytest.mark.gpu
LD = np.longdouble


def columns(kern, X, S, sigma):
    out = np.empty((len(S), len(X)), dtype=LD)
    for a, i in enumerate(S):
        t = X - X[i]
        if kern == O.LAPLACE_L1:
            out[a] = np.exp(-np.abs(t).sum(1) / sigma)
            continue
        r2 = (t * t).sum(1)
        q = np.sqrt(5 * r2) / sigma
        out[a] = np.exp(-r2 / (2 * sigma * sigma)) if kern == O.GAUSSIAN else (1 + q + q * q / 3) * np.exp(-q)
    return out


@pytest.mark.parametrize("kern,d,sigma", [(O.LAPLACE_L1, 8, 0.5), (O.MATERN52, 24, 0.7),
                                          (O.GAUSSIAN, 16, 0.6)])
@pytest.mark.parametrize("N,k,B", [(900, 150, 15), (400, 190, 95), (130, 40, 1)])
def test_nearly_sparse_factor(kern, d, sigma, N, k, B):
    K = require_gpu()
    X = np.random.default_rng(N + d).standard_normal((N, d))
    f = K.krr_rpcholesky(to_dev(X), kern, sigma, k, B, 3)
    F, S, D = f.export()
    f.free()
    G = columns(kern, X.astype(LD), S, LD(sigma))
    for j in range(len(S)):
        G[j] /= np.sqrt(G[j, S[j]])
        G[j + 1:] -= G[j][S[j + 1:]][:, None] * G[j][None, :]
        G[j, S[:j]] = 0
    assert np.sqrt(((F - G) ** 2).sum() / (G ** 2).sum()) <= 2 * 2.0 ** -53
    rest = np.setdiff1d(np.arange(N), S)
    assert np.max(np.abs(D - (1 - (G ** 2).sum(0)))[rest]) <= 16 * 2.0 ** -53
