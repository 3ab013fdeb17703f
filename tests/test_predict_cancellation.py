"""FP32 predictions whose terms cancel, vanish or underflow.

Tolerance: half a unit in the last place of the result (2^-24 relative, 1% slack for the
reference's own rounding) plus (K / 8 + N + 4) 2^-53 of the sum of the terms' magnitudes, what
N - 1 FP64 products a term and their sum over eight lanes lose at worst."""
import numpy as np
import pytest

import paper_1410_5209_gb300 as tf

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1410_5209_gb300 import build
    build.build()


def context(A):
    f = tf.Factorization(np.zeros((1, len(A)), np.int32), np.ones(1), [len(a) for a in A],
                         A[0].shape[1], dtype=tf.F32)
    for n, a in enumerate(A):
        f.set_factors(n, a)
    return f


def terms(A, c):
    t = np.ones((len(c), A[0].shape[1]), np.longdouble)
    for n, a in enumerate(A):
        t = t * a.astype(np.longdouble)[c[:, n]]
    return t


@pytest.mark.parametrize("N,K", [(2, 6), (3, 3), (3, 33), (3, 100), (3, 132), (5, 12)])
def test_cancelling_terms(N, K):
    """The first mode's last column makes each row of it cancel against one row of every other
    mode, to 2^-24 of its terms: what is left is rounding that only products and sums of more
    than 48 bits keep."""
    rng = np.random.default_rng(10 * N + K)
    rows = 400
    A = [rng.standard_normal((rows, K)).astype(np.float32) for _ in range(N)]
    c = np.repeat(np.arange(rows, dtype=np.int32)[:, None], N, 1)
    t = terms(A, c)
    rest = terms(A[1:], c[:, 1:])[:, -1]
    A[0][:, -1] = (-t[:, :-1].sum(1) / rest).astype(np.float32)
    t = terms(A, c)
    ref, mag = t.sum(1), np.abs(t).sum(1)
    assert np.median(np.abs(ref) / mag) < 2.0 ** -24
    got = context(A).predict(c)
    bound = 1.01 * 2.0 ** -24 * np.abs(ref) + (K / 8 + N + 4) * 2.0 ** -53 * mag
    assert np.all(np.abs(got - ref) <= bound)


@pytest.mark.parametrize("K", [7, 100])
def test_zero_rows_and_terms_below_the_float_range(K):
    """Terms with a zero factor beside huge ones are exact zeros; terms of 2^-150 are not: their
    sum is a subnormal float."""
    A = [np.ones((4, K), np.float32) for _ in range(3)]
    A[0][0] = 0
    A[1][0] = 3e38
    A[0][1, ::2] = 0
    A[1][1, 1::2] = 0
    A[0][2], A[1][2], A[2][2] = 2.0 ** -50, 2.0 ** -50, -(2.0 ** -50)
    A[0][3, 0] = 0
    A[1][3, 0] = np.inf
    f = context(A)
    got = f.predict(np.array([[0, 0, 0], [1, 1, 0], [2, 2, 2], [3, 3, 0], [1, 2, 2]], np.int32))
    assert got[0] == 0 and got[1] == 0
    assert got[2] == np.float32(-K * 2.0 ** -150)
    assert np.isnan(got[3])
    assert got[4] == np.float32(-(K // 2) * 2.0 ** -100)
