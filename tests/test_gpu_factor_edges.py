"""GPU parity of the factorization at the sizes where its kernels change shape.

Blocks around the groups of the triangular solve (20 columns), the column
tiles of the product by digits (8, 16, 32, 64, 112 columns) and its chunks of
128 terms; point counts around its 64-row tiles; cores around the 32-wide
diagonal blocks of the Cholesky factorisation and the doubling of the inverse.
Pivots are identical to the oracle's and F agrees to rounding (entries of size
<= 1: atol 1e-10, as in test_gpu_rpcholesky.py); the preconditioner agrees with
the dense formula on the exported factor to 1e-10 of the result, cond(core)
being at most about N / mu-shift = 1e4 here.
"""
import numpy as np
import pytest

import oracle as O
from gpu_common import require_gpu, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def K():
    return require_gpu()


@pytest.mark.parametrize("N,k,B", [
    (64, 17, 1), (63, 40, 20), (65, 42, 21), (129, 90, 41), (300, 200, 100), (300, 240, 112),
    (513, 260, 128), (513, 300, 113), (1000, 127, 8), (1000, 129, 9), (777, 400, 64),
])
def test_block_and_tile_edges(K, N, k, B):
    rng = np.random.default_rng(N + B)
    X = rng.standard_normal((N, 6))
    ref = O.rpcholesky(X, O.MATERN52, 0.8, k, B, 5)
    f = K.krr_rpcholesky(X, O.MATERN52, 0.8, k, B, 5)
    F, S, D = f.export()
    np.testing.assert_array_equal(S, ref.S)
    np.testing.assert_allclose(F, ref.F, atol=1e-10, rtol=0)
    np.testing.assert_allclose(D, ref.dres, atol=1e-10, rtol=0)
    f.free()


def test_dropped_candidates_inside_a_block(K):
    """Twins and near-twins in one block: the kept columns of G are not
    contiguous and the groups of the solve skip the dropped ones."""
    rng = np.random.default_rng(8)
    base = rng.standard_normal((30, 3))
    X = np.vstack([base, base, base + 1e-9 * rng.standard_normal((30, 3))])
    ref = O.rpcholesky(X, O.GAUSSIAN, 0.7, 90, 90, 2)
    f = K.krr_rpcholesky(X, O.GAUSSIAN, 0.7, 90, 90, 2)
    F, S, D = f.export()
    assert f.rank == ref.rank < 60
    np.testing.assert_array_equal(S, ref.S)
    np.testing.assert_allclose(F, ref.F, atol=1e-9, rtol=0)
    f.free()


@pytest.mark.parametrize("rank", [1, 31, 32, 33, 64, 65, 96, 129, 257])
def test_core_edges(K, rank):
    rng = np.random.default_rng(rank)
    N, mu = 600, 1e-4
    X = rng.standard_normal((N, 4))
    f = K.krr_rpcholesky(X, O.LAPLACE_L1, 1.0, rank, 0, 3)
    F, _, _ = f.export()
    lam = mu * N
    R = rng.standard_normal((3, N))
    core = F @ F.T + lam * np.eye(F.shape[0])
    ref = (R - (F.T @ np.linalg.solve(core, F @ R.T)).T) / lam
    got = K.krr_precond_apply(f, mu, to_dev(R), prec="fp64").cpu().numpy()
    assert np.linalg.norm(got - ref) <= 1e-10 * np.linalg.norm(ref)
    f.free()


@pytest.mark.parametrize("N,nd", [(5000, 1024), (3, 1024), (600_001, 33)])
def test_many_draws(K, N, nd):
    d = np.random.default_rng(N).random(N)
    np.testing.assert_array_equal(K.krr_rpc_sample(d, 11, 4, nd), O.rpc_sample(d, 11, 4, nd))


@pytest.mark.parametrize("N,k,B", [
    (127, 64, 16), (128, 96, 33), (385, 225, 32), (640, 352, 65), (1025, 672, 128), (1153, 810, 90),
])
def test_digit_product_edges(K, N, k, B):
    """128-row tiles, column groups of 16 to 64 and two groups, and the
    read-outs of the accumulators after 160 and 640 terms."""
    rng = np.random.default_rng(N + B)
    X = rng.standard_normal((N, 6))
    ref = O.rpcholesky(X, O.MATERN52, 0.8, k, B, 9)
    f = K.krr_rpcholesky(X, O.MATERN52, 0.8, k, B, 9)
    F, S, D = f.export()
    np.testing.assert_array_equal(S, ref.S)
    np.testing.assert_allclose(F, ref.F, atol=1e-10, rtol=0)
    np.testing.assert_allclose(D, ref.dres, atol=1e-10, rtol=0)
    f.free()
