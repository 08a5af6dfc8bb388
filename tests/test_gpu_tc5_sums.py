"""Float32 sums of the tcgen05 product with up to two right-hand sides.

Equal points make every kernel value exactly 1, so a product is its sums.  The
right-hand sides lie in [3/4, 1) as multiples of 2^-20: chains of 16 stay below
16 and are exact; the two chains of 32 columns are added with a rounding of at
most 2^-20 (below 32), the two sums of a 64-column share with one of at most
2^-19 (below 64): 2^-18 in all.  Chains of 32 round another 16 times each by up
to 2^-20, about 2^-18 in the root mean square, and pass the bound for about a
third of the columns.
"""
import numpy as np
import pytest

from gpu_common import require_gpu, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kern", [0, 2])
@pytest.mark.parametrize("m", [1, 2])
def test_short_chains(kern, m):
    K = require_gpu()
    rng = np.random.default_rng(m)
    X = to_dev(np.zeros((64, 5)))
    for _ in range(20):
        V = rng.integers(3 << 18, 1 << 20, (m, 64)) * 2.0 ** -20
        got = K.krr_kmatvec(X, kern, 1.0, 0.0, to_dev(V), prec="mixed").cpu().numpy()
        assert np.all(np.abs(got - V.sum(1)[:, None]) <= 2.0 ** -18)
