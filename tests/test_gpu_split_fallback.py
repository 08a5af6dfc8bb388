"""Calls whose points do not fit the tcgen05 product's split.

One point far out sends a call to another kernel after its operands were
prepared.  The discarded product must cost nothing: the product kernels of such
a call take at most 1.2 times those of the same call with that kernel asked for
(a discarded product adds 0.2 to 0.5 of it at these sizes), the result is that
call's, and the operands are not prepared a second time.
"""
import numpy as np
import pytest

import oracle as O
from gpu_common import require_gpu, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def K():
    K = require_gpu()
    yield K
    K.krr_set_product_path(0)


def product_ms(K, path, call):
    K.krr_set_product_path(path)
    try:
        times, launches, out = [], [], None
        for _ in range(6):
            before = K.krr_launch_count()
            K.krr_set_profiling(True)
            out = call()
            times.append(K.krr_profile_collect(0)[0])
            K.krr_set_profiling(False)
            launches.append(K.krr_launch_count() - before)
        return min(times), min(launches), out.cpu().numpy()
    finally:
        K.krr_set_profiling(False)
        K.krr_set_product_path(0)


@pytest.mark.parametrize("far,path", [(1e3, 2), (1e6, 1)])   # mma.sync, FMA
@pytest.mark.parametrize("kern", [O.GAUSSIAN, O.MATERN52])
def test_discarded_product_costs_nothing(K, kern, far, path):
    rng = np.random.default_rng(4)
    N = 50_000
    X, V = rng.standard_normal((N, 16)), to_dev(rng.standard_normal((4, N)))
    X[N // 2, 0] = far
    X = to_dev(X)
    call = lambda: K.krr_kmatvec(X, kern, 1.0, 0.5, V, prec="mixed")
    t0, n0, ref = product_ms(K, path, call)
    t1, n1, got = product_ms(K, 0, call)
    np.testing.assert_array_equal(got, ref)
    assert t1 <= 1.2 * t0
    # beside that call's launches: the means (2), the operands once, the
    # right-hand sides, the empty product and its sum
    assert n1 <= n0 + 6


@pytest.mark.parametrize("m", [1, 3, 8, 11, 16])
@pytest.mark.parametrize("N", [2, 300, 5000])
def test_results_of_the_fallback(K, N, m):
    """Row blocks summed by one CTA and by many, one launch and two: the same
    bits as with the FMA kernel asked for."""
    rng = np.random.default_rng(N + m)
    X, V = rng.standard_normal((N, 5)), to_dev(rng.standard_normal((m, N)))
    T = rng.standard_normal((77, 5))
    T[3] = 2e6
    far = X.copy()
    far[N // 2, 1] = 2e6
    for call in (lambda: K.krr_predict(to_dev(X), 0, 1.0, V, to_dev(T), prec="mixed"),
                 lambda: K.krr_kmatvec(to_dev(far), 0, 1.0, 0.25, V, prec="mixed")):
        K.krr_set_product_path(1)
        ref = call().cpu().numpy()
        K.krr_set_product_path(0)
        np.testing.assert_array_equal(call().cpu().numpy(), ref)
