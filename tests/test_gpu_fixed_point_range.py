"""Float64 Matern products of the farthest pairs on the GPU.

Points in {0, 1}^32 with their complements: opposite pairs have q = sqrt(160) /
sigma between 705 and 723, where kappa lies below 1e-300.  Unit right-hand sides
read the entries out; everything else about them is test_gpu_fixed_point's bound.
"""
import numpy as np
import pytest

import oracle as O
from gpu_common import require_gpu, to_dev
from test_gpu_fixed_point import bound

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sigma", [0.0175, 0.0176, 0.0177, 0.0178, 0.0179])
@pytest.mark.parametrize("N", [40, 2600])   # a tile; the symmetric product
def test_complementary_corners(N, sigma):
    K = require_gpu()
    rng = np.random.default_rng(N)
    half = rng.integers(0, 2, (N // 2, 32)).astype(float)
    X = np.vstack([half, 1.0 - half])
    X[0], X[1] = 0.0, 1.0
    V = np.zeros((2, N))
    V[0, 0], V[1, 5] = 1.0, 1.0
    ref = O.kernel_block(X, O.MATERN52, sigma, None, np.array([0, 5])).T
    got = K.krr_kmatvec(to_dev(X), O.MATERN52, sigma, 0.0, to_dev(V), prec="fp64").cpu().numpy()
    assert np.all(np.abs(got - ref) <= bound(ref, 32) + 1e-300)
    got = K.krr_predict(to_dev(X), O.MATERN52, sigma, to_dev(V), to_dev(X), prec="fp64").cpu().numpy()
    assert np.all(np.abs(got - ref) <= bound(ref, 32) + 1e-300)
