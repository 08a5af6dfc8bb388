"""Fixed-point kernel values (csrc/kfix.cuh), compiled for the host.

Entries of each kernel function, over every range exponent the fixed-point
products accept, against 50-digit arithmetic and next to the float64 formulas
of the general path.

Derivation: a coordinate is rounded to 2^-(58 - e) (half a unit of 2^-(57 - e))
of its scaled value, |y| < 2^e.  With e <= 4 a difference is off by at most
2^-53, so E = sum d^2 by at most 2 sqrt(d E) 2^-53 (Gaussian), q by sqrt(d)
2^(e - 57) (Matern), E by d 2^(e - 58) (Laplace).  E is then rounded at 2^-55,
2^-E and the result at 2^-53 relative.  The Matern value adds the roundings of
r^2, q, the polynomial and the product: at most q + 4 units.
"""
import ctypes as C
import decimal
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2304_12465_gb300", "csrc")

HARNESS = r"""
#include "kfix.cuh"
using namespace krr;
extern "C" double entry(int kern, int d, int e, const double *x, const double *y,
                        const double *ctr, double s_hi, double s_lo) {
  const int q = kern == 1 ? 58 - e : 57 - e, r = kern == 1 ? 4 - e : 30 - 2 * e;
  int64_t S1 = 0, S2 = 0; uint64_t S3 = 0, S = 0;
  for (int k = 0; k < d; ++k) {
    const int64_t a = fix_coord(x[k], ctr[k], s_hi, s_lo, q), b = fix_coord(y[k], ctr[k], s_hi, s_lo, q);
    const int64_t D = a - b;
    S += (uint64_t)(D < 0 ? -D : D);
    int32_t ah, al, bh, bl;
    fix_limbs(a, kFixLimb, &ah, &al);
    fix_limbs(b, kFixLimb, &bh, &bl);
    const int64_t dh = (int64_t)ah - bh, dl = (int64_t)al - bl;
    if (dh != (int32_t)dh || dl != (int32_t)dl) return -1.0;
    S1 += dh * dh; S2 += dh * dl; S3 += (uint64_t)(dl * dl);
  }
  if (kern == 1) return fix_exp2(fix_exponent_l1(S, r), kFixExp2Tab);
  if (kern == 2) return fix_matern(S1, S2, S3, ldexp(1.0, 30 - 2 * q), kFixExp2Tab);
  const int64_t s1_max = e == 1 ? INT64_MAX : (int64_t)((1022ull << 54) >> (28 - r));
  return fix_exp2(fix_exponent(S1, S2, S3, r, s1_max), kFixExp2Tab);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("kfix")
    src, so = d / "h.cpp", d / "h.so"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-std=c++17", "-shared", "-fPIC",
                    f"-I{CSRC}", str(src), "-o", str(so)], check=True)
    L = C.CDLL(str(so))
    L.entry.restype = C.c_double
    p = np.ctypeslib.ndpointer(np.float64)
    L.entry.argtypes = [C.c_int, C.c_int, C.c_int, p, p, p, C.c_double, C.c_double]
    return L


def exact(kern, x, y, sigma):
    D = decimal.Decimal
    diff = [D(float(a)) - D(float(b)) for a, b in zip(x, y)]
    s = D(float(sigma))
    if kern == 1:
        E = sum(abs(t) for t in diff) / s
        return E, (-E).exp()
    r2 = sum(t * t for t in diff)
    if kern == 0:
        E = r2 / (2 * s * s)
        return E, (-E).exp()
    q = (5 * r2).sqrt() / s
    return q, (1 + q + q * q / 3) * (-q).exp()


def float64(kern, x, y, sigma):
    t = x - y
    if kern == 1:
        return float(np.exp(-np.abs(t).sum() / sigma))
    s = float((t * t).sum())
    if kern == 0:
        return float(np.exp(-s / (2.0 * sigma * sigma)))
    q = np.sqrt(5.0 * s) / sigma
    return float((1.0 + q + q * q / 3.0) * np.exp(-q))


@pytest.mark.parametrize("kern,emin,emax", [(0, 1, 4), (1, 1, 5), (2, 1, 6)])
@pytest.mark.parametrize("d", [1, 5, 32])
def test_entries(lib, kern, emin, emax, d):
    decimal.getcontext().prec = 50
    rng = np.random.default_rng(100 * kern + d)
    unit = {0: decimal.Decimal(2).ln(), 1: decimal.Decimal(2).ln(), 2: decimal.Decimal(5)}[kern]
    for e in range(emin, emax + 1):
        # sigma so that the scaled half-range of points in [-1, 1] is just below 2^e
        base = {0: (1 / (2 * unit)).sqrt(), 1: 1 / unit, 2: unit.sqrt()}[kern]
        sigma = float(base) / (2.0 ** e * (1 - 1e-6))
        scale = base / decimal.Decimal(sigma)
        s_hi = float(scale)
        s_lo = float(scale - decimal.Decimal(s_hi))
        ctr = np.zeros(d)
        for it in range(60):
            x = rng.uniform(-1, 1, d)
            # near, typical and opposite pairs
            y = [x + 1e-6 * rng.standard_normal(d), rng.uniform(-1, 1, d),
                 x + 2.0 ** -e * rng.uniform(-1, 1, d) / np.sqrt(d), -np.sign(x), x.copy()][it % 5]
            if it % 5 == 3:
                x = np.sign(x)
            y = np.clip(y, -1, 1)
            E, want = exact(kern, x, y, sigma)
            got = lib.entry(kern, d, e, x, y, ctr, s_hi, s_lo)
            err = abs(decimal.Decimal(got) - want)
            if want < decimal.Decimal(2) ** -1020:
                assert 0 <= got <= 2.0 ** -1019
                continue
            E = float(E)
            units = {0: 1.5 + 2 * np.sqrt(d * E) * 2.0 ** (e - 4), 1: 1.5 + d * 2.0 ** (e - 5),
                     2: 6 + 2 * E + np.sqrt(d) * 2.0 ** (e - 4)}[kern]
            assert err <= decimal.Decimal(units * 2.0 ** -53) * want, (e, it, E, got, want)
            # and against the float64 formula: never worse than it by more
            # than two units of the last place
            ref = abs(decimal.Decimal(float64(kern, x, y, sigma)) - want)
            assert err <= ref + decimal.Decimal(2.0 ** -52), (e, it, E, got, want)
