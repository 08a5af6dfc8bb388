"""Entries of the float-float products, read out with unit right-hand sides,
against 50-digit arithmetic.

Derivation, in units of 2^-53 (Gaussian and Laplace; the value is at most 1):
49 bits of the mantissa give 8, the roundings of E and of the low bits 1, the
coordinates (rounded to 2^-(53 - e), Laplace 2^-(58 - e)) 2 sqrt(d E) 2^e, Laplace
d 2^(e - 5).  From E = 2^-8 on the squares of the low limbs enter by their mean:
a squared difference of low limbs uniform over 2^25 values has a standard
deviation of 0.197 2^50, so the sum of d of them, worth ln 2 2^(2 e - 3) a
coordinate, has 0.137 sqrt(d) 2^(2 e - 3); six of them bound an entry and 1.5
the root mean square of the entries around one distance (a mean left out or
taken over padded coordinates too shifts all of them by 0.115 2^(2 e - 3) a
coordinate).  Equal points give exactly 1.  Matern: 2^-44, the float-float
square root, exponential and polynomial.
"""
import decimal

import numpy as np
import pytest

import oracle as O
from gpu_common import require_gpu, to_dev
from test_fixed_point import exact

pytestmark = pytest.mark.gpu
DISTANCES = [2.0 ** -60, 2.0 ** -40, 2.0 ** -24, 2.0 ** -16, 2.0 ** -10, 2.0 ** -6, 2.0 ** -2, 2.0]
SCALE = {O.GAUSSIAN: 1 / np.sqrt(2 * np.log(2)), O.LAPLACE_L1: 1 / np.log(2), O.MATERN52: np.sqrt(5)}


def planted(rng, kern, d, e, reps):
    """Eight base points; copies of them; points at each distance in E (Matern: q^2)."""
    sigma = SCALE[kern] / (2.0 ** e * (1 - 1e-3))
    base = rng.uniform(-0.7, 0.7, (8, d))
    groups = [base, base.copy()]
    for E in DISTANCES:
        r = {O.GAUSSIAN: np.sqrt(2 * np.log(2) * E), O.LAPLACE_L1: np.log(2) * E,
             O.MATERN52: np.sqrt(E / 5)}[kern] * sigma
        for _ in range(reps):
            t = rng.standard_normal((8, d))
            t /= np.abs(t).sum(1, keepdims=True) if kern == O.LAPLACE_L1 else \
                np.linalg.norm(t, axis=1, keepdims=True)
            groups.append(base + r * t)
    return np.clip(np.concatenate(groups), -1, 1), sigma


@pytest.mark.parametrize("N,cols", [(0, 8), (2600, 4)])   # rectangular, symmetric
@pytest.mark.parametrize("kern,e", [(O.GAUSSIAN, 1), (O.GAUSSIAN, 3), (O.GAUSSIAN, 4),
                                    (O.LAPLACE_L1, 5), (O.MATERN52, 2), (O.MATERN52, 5)])
@pytest.mark.parametrize("d", [1, 5, 32])
def test_entries(d, kern, e, N, cols):
    K = require_gpu()
    decimal.getcontext().prec = 50
    rng = np.random.default_rng(100 * d + e)
    reps = 6
    X, sigma = planted(rng, kern, d, e, reps)
    n = len(X)
    X = np.concatenate([X, -np.ones((1, d)), np.ones((1, d)), rng.uniform(-1, 1, (max(0, N - n - 2), d))])
    V = np.zeros((cols, len(X)))
    V[np.arange(cols), np.arange(cols)] = 1.0
    got = K.krr_kmatvec(to_dev(X), kern, sigma, 0.0, to_dev(V), prec="ff").cpu().numpy()
    for g in range(n // 8):
        err, lim, E = [], [], 0.0
        for c in range(cols):
            E, want = exact(kern, X[8 * g + c], X[c], sigma)
            err.append(float(abs(decimal.Decimal(got[c, 8 * g + c]) - want)) * 2.0 ** 53)
            E = float(E) / np.log(2)
            lim.append({O.GAUSSIAN: 9 + 2 * np.sqrt(d * E) * 2.0 ** e,
                        O.LAPLACE_L1: 9 + d * 2.0 ** (e - 5), O.MATERN52: 512}[kern])
        err, lim = np.array(err), np.array(lim)
        if g < 2:
            assert np.all(err == 0), ("equal points", g, err)
        elif kern == O.GAUSSIAN and E >= 2.0 ** -8:
            dev = 0.137 * np.sqrt(d) * 2.0 ** (2 * e - 3)
            assert np.all(err <= lim + 6 * dev), (g, E, err)
        else:
            assert np.all(err <= lim), (g, E, err)
    if kern == O.GAUSSIAN:      # around E = 2^-2
        g0 = 2 + DISTANCES.index(2.0 ** -2) * reps
        err, E = [], 0.0
        for g in range(g0, g0 + reps):
            for c in range(cols):
                E, want = exact(kern, X[8 * g + c], X[c], sigma)
                err.append(float(decimal.Decimal(got[c, 8 * g + c]) - want) * 2.0 ** 53)
        dev = 0.137 * np.sqrt(d) * 2.0 ** (2 * e - 3)
        assert np.sqrt(np.mean(np.square(err))) <= 9 + 2 * np.sqrt(d) * 2.0 ** (e - 1) / 2 + 1.5 * dev


@pytest.mark.parametrize("kern", [O.GAUSSIAN, O.LAPLACE_L1])
def test_small_entries(kern):
    """Down to 2^-148 both floats count: the mantissa's 2^-49, E = 2 sqrt(E) 2^3
    (Gaussian, e = 3) or 4 (Laplace, e <= 7) units of 2^-53 times ln 2, and the
    two roundings to subnormal floats, 2^-150 each."""
    K = require_gpu()
    decimal.getcontext().prec = 50
    E = np.linspace(90, 148, 117)
    x = {O.GAUSSIAN: np.sqrt(2 * np.log(2) * E), O.LAPLACE_L1: np.log(2) * E}[kern]
    X = np.concatenate([[0.0], x])[:, None]
    V = np.zeros((1, len(X)))
    V[0, 0] = 1.0
    got = K.krr_kmatvec(to_dev(X), kern, 1.0, 0.0, to_dev(V), prec="ff").cpu().numpy()[0]
    for i in range(1, len(X)):
        _, want = exact(kern, X[i], X[0], 1.0)
        rel = (17 + (16 * np.sqrt(E[i - 1]) if kern == O.GAUSSIAN else 4)) * 2.0 ** -53
        lim = decimal.Decimal(rel) * want + decimal.Decimal(2) ** -149
        assert abs(decimal.Decimal(got[i]) - want) <= lim, (E[i - 1], got[i])
