"""The loss's regulariser alone (a tensor of zeros under a zero first factor has no data term).

Tolerance, FP32 values: 2^-42 for squares summed eight at a time in pairs of floats (the square
of eight times 2^-24) plus 2^-53 for each of the at most 300 sums of doubles behind them."""
import numpy as np
import pytest

import paper_1410_5209_gb300 as tf

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1410_5209_gb300 import build
    build.build()


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("rows,K", [(300, 2000), (300, 7), (5000, 9), (1, 2001)])
@pytest.mark.parametrize("scale", [1.1, 0.9, 3e-20, 2e18])
def test_sum_of_squares(rows, K, weighted, scale):
    """Equal values (whose rounding errors all point one way) beside a few others, also where
    single squares leave the float range."""
    rng = np.random.default_rng(rows + K)
    A = [np.zeros((rows, K), np.float32), np.full((rows, K), scale, np.float32),
         (rng.standard_normal((3, K)) * scale).astype(np.float32)]
    coords = np.stack([np.arange(rows), np.arange(rows), np.arange(rows) % 3], 1)
    f = tf.Factorization(coords.astype(np.int32), np.zeros(rows), [rows, rows, 3], K)
    for n in range(3):
        f.set_factors(n, A[n])
    ref = np.longdouble(0)
    for n in (1, 2):
        w = np.bincount(coords[:, n], minlength=len(A[n])) if weighted else np.ones(len(A[n]))
        ref += ((A[n].astype(np.longdouble) ** 2).sum(1) * w).sum()
    got, rmse = f.loss(1.0, weighted=weighted)
    assert rmse == 0
    assert abs(got - ref) <= (2.0 ** -42 + 300 * 2.0 ** -53) * ref
