"""Float fold-ins whose products leave the float range on the way, and FP32-hard data.

Tolerance: each component of a row within 16 units of 2^-24 of the dense FP64 solve (the
rounding of the residual, of the right-hand side of its correction and of the triangular
solves with a factor whose off-diagonal part hardly couples the components)."""
import numpy as np
import pytest

import paper_1410_5209_gb300 as tf

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1410_5209_gb300 import build
    build.build()


def solve(A, other, x, lam):
    h = np.ones((len(x), A[0].shape[1]))
    for t, a in enumerate(A[1:]):
        h = h * a.astype(np.float64)[other[:, t]]
    return np.linalg.solve(h.T @ h + lam * np.eye(h.shape[1]), h.T @ x.astype(np.float64))


def check(A, other, x, lam, tol=16 * 2.0 ** -24):
    f = tf.Factorization(np.zeros((1, len(A)), np.int32), np.ones(1), [len(a) for a in A],
                         A[0].shape[1], dtype=tf.F32)
    for n, a in enumerate(A):
        f.set_factors(n, a)
    lam = float(np.float32(lam))
    ref = solve(A, other, x, lam)
    got = f.foldin(0, other, x, lam)
    assert np.all(np.abs(got - ref) <= tol * np.abs(ref)), np.max(np.abs(got - ref) / np.abs(ref))


@pytest.mark.parametrize("K", [5, 31, 40, 100])
@pytest.mark.parametrize("m", [1, 40, 700])
def test_products_that_underflow_on_the_way(K, m):
    """Order 4: a column of 1e-30, 1e-30 and 1e30 has products of 1e-30, which FP32 products
    lose; beside it columns of ordinary size.  lambda far above the Gram matrix."""
    rng = np.random.default_rng(K + m)
    A = [np.zeros((3, K), np.float32)] + [rng.uniform(0.5, 1.0, (20, K)).astype(np.float32)
                                          for _ in range(3)]
    for a, scale in zip(A[1:], (1e-30, 1e-30, 1e30)):
        a[:, K // 2] *= np.float32(scale)
    other = rng.integers(0, 20, (m, 3)).astype(np.int32)
    check(A, other, rng.uniform(0.5, 1.0, m).astype(np.float32), 1e6 * m)


@pytest.mark.parametrize("K", [3, 100])
def test_collapsed_columns_and_tiny_values(K):
    """Order 3 and 2, columns of 1e-14 and zeros (whose components are exact zeros)."""
    rng = np.random.default_rng(K)
    for N in (2, 3):
        A = [np.zeros((3, K), np.float32)] + [rng.uniform(0.5, 1.0, (20, K)).astype(np.float32)
                                              for _ in range(N - 1)]
        A[1][:, 1] *= np.float32(1e-14)
        A[1][:, 2] = 0
        other = rng.integers(0, 20, (300, N - 1)).astype(np.int32)
        x = rng.uniform(0.5, 1.0, 300).astype(np.float32)
        check(A, other, x, 1e5)
        check(A, other, (x * np.float32(1e-18)).astype(np.float32), 1e5)
