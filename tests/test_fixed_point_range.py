"""Fixed-point Matern values of the farthest pairs (csrc/kfix.cuh, on the host).

From d = 31 on, points of the accepted range reach q = 128 sqrt(d) > 709.8,
where q log2 e passes the 10 integer bits that E has.  Near opposite corners
the value must follow exp(-q) to test_fixed_point's bound while it is at least
2^-1000 = 9.3e-302, lie between 0 and 1e-301 beyond, and be 0 from E = 1022 on.
"""
import decimal

import numpy as np
import pytest

from test_fixed_point import exact, lib  # noqa: F401


@pytest.mark.parametrize("d", [31, 32])
def test_matern_near_the_end_of_the_exponent(lib, d):  # noqa: F811
    decimal.getcontext().prec = 50
    five = decimal.Decimal(5).sqrt()
    seen = 0
    for q in np.concatenate([np.arange(660.0, 725.0, 0.25), [708.38, 708.39, 708.4, 709.78, 709.79]]):
        y = q / (2 * np.sqrt(d))              # scaled corners +-y
        if y >= 64 * (1 - 1e-6):
            continue
        scale = five / (five / decimal.Decimal(float(y)))
        s_hi = float(scale)
        s_lo = float(scale - decimal.Decimal(s_hi))
        x = np.ones(d)
        x[::3] = -1.0
        sigma = float(five / decimal.Decimal(float(y)))
        got = lib.entry(2, d, 6, x, -x, np.zeros(d), s_hi, s_lo)
        E, want = exact(2, x, -x, sigma)
        if want < decimal.Decimal(2) ** -1000:
            assert 0.0 <= got <= 1e-301, (q, got)
            if q >= 708.4:
                assert got == 0.0, (q, got)
                seen += 1
        else:
            units = 6 + 2 * float(E) + 4 * np.sqrt(d)
            assert abs(decimal.Decimal(got) - want) <= decimal.Decimal(units * 2.0 ** -53) * want
    assert seen >= (10 if d == 31 else 50)
