"""Float64 Laplace entries of near pairs at the widest accepted range.

In units of 2^-53 of the value, root mean square: the result's rounding 0.29, E's
at 2^-54 0.2, and the coordinates', which are kept to 2^-(60 - e): sqrt(d / 6) ln 2
2^(e - 7).  1.25 times their root sum of squares bounds some 700 entries; two bits
less in the coordinates make the last term four times as large.
"""
import decimal

import numpy as np
import pytest

import oracle as O
from gpu_common import require_gpu, to_dev
from test_fixed_point import exact

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [1, 4, 8, 9, 16, 17, 24, 25, 32])
@pytest.mark.parametrize("e", [1, 4, 5])
def test_near_pairs(d, e):
    K = require_gpu()
    decimal.getcontext().prec = 50
    rng = np.random.default_rng(d)
    sigma = 1 / np.log(2) / (2.0 ** e * (1 - 1e-3))
    base = rng.uniform(-0.9, 0.9, (8, d))
    rows = [base]
    for E in np.geomspace(2.0 ** -40, 2.0 ** -4, 90):
        t = rng.standard_normal((8, d))
        rows.append(base + E * np.log(2) * sigma * t / np.abs(t).sum(1, keepdims=True))
    X = np.concatenate(rows + [-np.ones((1, d)), np.ones((1, d))])
    V = np.zeros((8, len(X)))
    V[np.arange(8), np.arange(8)] = 1.0
    got = K.krr_kmatvec(to_dev(X), O.LAPLACE_L1, sigma, 0.0, to_dev(V), prec="fp64").cpu().numpy()
    err = []
    for g in range(len(rows)):
        for c in range(8):
            _, want = exact(O.LAPLACE_L1, X[8 * g + c], X[c], sigma)
            err.append(float((decimal.Decimal(got[c, 8 * g + c]) - want) / want) * 2.0 ** 53)
            if g == 0:
                assert err[-1] == 0.0
    rms = np.sqrt(0.29 ** 2 + 0.2 ** 2 + d / 6 * (np.log(2) * 2.0 ** (e - 7)) ** 2)
    assert np.sqrt(np.mean(np.square(err[8:]))) <= 1.25 * rms
