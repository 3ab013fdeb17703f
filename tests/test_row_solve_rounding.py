"""Row solves whose every quotient is exact: rows whose entries each touch one column, so that
B is diagonal with the squares of integers, lambda = 0 and the solution are integers.  A
division, and whatever rounds as one, returns exactly them."""
import numpy as np
import pytest

import paper_1410_5209_gb300 as tf

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1410_5209_gb300 import build
    build.build()


def diagonal_rows(C, rows, top, rng):
    """Coordinates, values, factors: row i meets, for each column c, the row (c, m) of mode 1,
    which is m in column c and zero elsewhere; values k m for a wanted k."""
    m = rng.integers(1, top, (rows, C))
    k = rng.integers(-top, top, (rows, C))
    col = np.broadcast_to(np.arange(C), (rows, C))
    coords = np.stack([np.repeat(np.arange(rows), C), (col * top + m).ravel(),
                       np.zeros(rows * C, int)], 1).astype(np.int32)
    B = np.zeros((C * top, C))
    B[np.arange(C * top), np.arange(C * top) // top] = np.arange(C * top) % top
    return coords, (k * m).ravel().astype(float), [np.zeros((rows, C)), B, np.ones((1, C))], m, k


@pytest.mark.parametrize("dtype,top", [(tf.F64, 5000), (tf.F32, 200)])
@pytest.mark.parametrize("C", [1, 2, 3, 4, 5, 6, 8, 10, 12, 16])
def test_exact_quotients(C, dtype, top):
    coords, x, A, m, k = diagonal_rows(C, 2000, top, np.random.default_rng(C))
    f = tf.Factorization(coords, x, [len(a) for a in A], C, dtype=dtype)
    for n in range(3):
        f.set_factors(n, A[n])
    f.sweep(C, 0.0, 1, np.arange(C, dtype=np.int32))
    assert np.array_equal(f.factors(0).astype(np.float64), k)
    if dtype == tf.F64:  # the products with a rounded inverse are not all exact
        inv = 1.0 / m
        assert (k * m * m * inv * inv != k).any()
