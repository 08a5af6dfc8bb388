"""How right-hand sides and kernel settings are grouped into launches.

The batched product takes up to four settings of one kernel type per launch,
in any order of the types; the square tcgen05 product takes 13 to 16
right-hand sides in one launch.  Both meet the float32 product bound
|Y - Y_oracle| <= 2e-5 (A|V| + lambda|V|) of the other float32 paths at the
edges of their groups and tiles.
"""
import numpy as np
import pytest

import oracle as O
from gpu_common import f32_product_bound, require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def K():
    return require_gpu()


G, L, M = O.GAUSSIAN, O.LAPLACE_L1, O.MATERN52


@pytest.mark.parametrize("N,d,ms", [(1, 1, 1), (65, 8, 2), (1023, 4, 2), (1025, 9, 1),
                                    (1500, 32, 2)])
@pytest.mark.parametrize("kerns", [[L], [G, M, L, G], [M, G, M, M, L, M, M, M],
                                   [G, G, G, G, G, L, L]])
def test_batched_product_groups(K, N, d, ms, kerns):
    rng = np.random.default_rng(N + 10 * d + len(kerns))
    X = 1.5 * rng.standard_normal((N, d)) / np.sqrt(d)
    S = len(kerns)
    sigmas = rng.uniform(0.4, 3.0, S)
    lams = rng.uniform(1e-3, 1.0, S * ms)
    V = rng.standard_normal((S * ms, N))
    got = K.krr_kmatvec_batched(X, kerns, sigmas, lams, V)
    for q in range(S):
        for c in range(q * ms, (q + 1) * ms):
            ref = O.kmatvec(X, kerns[q], sigmas[q], lams[c], V[c])
            bound = f32_product_bound(X, kerns[q], sigmas[q], lams[c], V[c][None])
            assert np.all(np.abs(got[c] - ref[0]) <= 2e-5 * bound[0]), (q, c)


@pytest.mark.parametrize("variant", [0, 8])
@pytest.mark.parametrize("kern", [G, M])
@pytest.mark.parametrize("N,d,m", [(1, 4, 16), (127, 16, 13), (257, 17, 16), (1031, 27, 15),
                                   (2049, 32, 12), (4099, 3, 14)])
def test_sixteen_right_hand_sides(K, kern, variant, N, d, m):
    rng = np.random.default_rng(N + d + m + kern)
    X, V = rng.standard_normal((N, d)), rng.standard_normal((m, N))
    V[m // 2] *= 1e20
    V[m - 1] = 0.0
    try:
        K.krr_set_product_variant(variant)
        got = K.krr_kmatvec(X, kern, 1.1, 0.5, V, prec="mixed")
    finally:
        K.krr_set_product_variant(0)
    ref = O.kmatvec(X, kern, 1.1, 0.5, V)
    bound = f32_product_bound(X, kern, 1.1, 0.5, V)
    assert np.all(np.abs(got - ref) <= 2e-5 * bound)
    assert np.all(got[m - 1] == 0.0)
