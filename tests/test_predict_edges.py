"""Prediction at the edges of its vector loads and of the float range.

Tolerances: a value in FP64 within 1e-13 of the sum of its terms' magnitudes; in FP32 within
half a unit in the last place (2^-24 relative, 1% slack for the reference's own rounding)
plus 2^-40 of that sum, which covers products and sums held to about 48 bits."""
import numpy as np
import pytest

import paper_1410_5209_gb300 as tf

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1410_5209_gb300 import build
    build.build()


def model(dims, K, dtype, seed, scale=None):
    rng = np.random.default_rng(seed)
    npdt = np.float64 if dtype == tf.F64 else np.float32
    A = [(rng.standard_normal((d, K)) * (scale or K ** (-1.0 / (2 * len(dims))))).astype(npdt)
         for d in dims]
    f = tf.Factorization(np.zeros((1, len(dims)), np.int32), np.ones(1), dims, K, dtype=dtype)
    for n, a in enumerate(A):
        f.set_factors(n, a)
    return f, A, rng


def check_values(f, A, c):
    t = np.ones((len(c), A[0].shape[1]), np.longdouble)
    for n, a in enumerate(A):
        t = t * a.astype(np.longdouble)[c[:, n]]
    ref, mag = t.sum(1), np.abs(t).sum(1)
    got = f.predict(c)
    if f.dtype == tf.F64:
        bound = 1e-13 * mag
    else:
        bound = 1.01 * 2.0 ** -24 * np.abs(ref) + 2.0 ** -40 * mag + 2.0 ** -149
    assert np.all(np.abs(got - ref) <= bound)


@pytest.mark.parametrize("dtype", [tf.F64, tf.F32])
@pytest.mark.parametrize("N,K", [(1, 5), (2, 8), (3, 1), (3, 4), (3, 33), (3, 36), (3, 100),
                                 (3, 130), (5, 12), (8, 7)])
def test_predict_edges(N, K, dtype):
    dims = [20 + n for n in range(N)]
    f, A, rng = model(dims, K, dtype, 7 * N + K)
    for m in (1, 31, 33, 500):
        check_values(f, A, np.stack([rng.integers(0, d, m) for d in dims], 1).astype(np.int32))


@pytest.mark.parametrize("K", [3, 100])
def test_predict_outside_the_float_pair_range(K):
    """Products that overflow or underflow FP32 on the way, zero rows, infinities and NaN."""
    f, A, rng = model([6, 5, 4], K, tf.F32, 3)
    A[0][1] *= 1e30
    A[1][1] *= 1e25
    A[2][1] *= 1e-35
    A[1][2] *= 1e-30
    A[2][2] *= 1e-12
    A[0][3] = 0
    for n in range(3):
        f.set_factors(n, A[n])
    c = np.stack(np.meshgrid(range(4), range(3), range(3), indexing="ij"), -1).reshape(-1, 3)
    c = c.astype(np.int32)
    keep = [e for e in c if not (e[0] == 1 and e[1] == 1 and e[2] != 1)]  # beyond FP32 itself
    check_values(f, A, np.array(keep, np.int32))
    A[0][4, 0], A[0][5, 0] = np.inf, np.nan
    f.set_factors(0, A[0])
    got = f.predict(np.array([[4, 0, 0], [5, 0, 0], [2, 0, 0]], np.int32))
    assert np.isinf(got[0]) and np.isnan(got[1]) and np.isfinite(got[2])
