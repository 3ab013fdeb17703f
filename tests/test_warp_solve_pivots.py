"""Warp solves of 17 to 63 columns: square roots, inverses and quotients of single pivots.

Rows whose entries each touch one column have a diagonal B; values and factors of eight
significant bits make B and c exact in every pass.  Tolerance: 4.5 units of 2^-24, what a
rounded square root, its two rounded quotients and half a unit of slack allow."""
import numpy as np
import pytest

import paper_1410_5209_gb300 as tf

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1410_5209_gb300 import build
    build.build()


def short(rng, shape, lo, hi):
    """Numbers of eight significant bits and either sign, exponents lo .. hi."""
    return (rng.integers(128, 256, shape) * rng.choice([-1.0, 1.0], shape) *
            2.0 ** (rng.integers(lo, hi + 1, shape) - 7))


@pytest.mark.parametrize("C", [17, 23, 24, 31, 32, 39, 40, 47, 48, 55, 56, 63])
@pytest.mark.parametrize("lo,hi,lam", [(-60, 62, 0.0),    # pivots of 2^-120 .. 2^126
                                       (-33, -28, 0.0),   # both sides of 2^-60
                                       (58, 62, 0.0),     # both sides of 2^120
                                       (-4, 4, 0.37)])    # pivots of 24 bits
def test_pivots_over_the_float_range(C, lo, hi, lam):
    rng = np.random.default_rng([C, hi + 64])
    rows = 200
    h, v = short(rng, (rows, C), lo, hi), short(rng, (rows, C), -2, 2)
    n = rows * C
    coords = np.stack([np.repeat(np.arange(rows), C), np.arange(n), np.zeros(n, int)], 1)
    A1 = np.zeros((n, C), np.float32)
    A1[np.arange(n), np.arange(n) % C] = h.ravel()
    f = tf.Factorization(coords.astype(np.int32), v.ravel().astype(np.float32), (rows, n, 1), C)
    for k, a in enumerate((np.zeros((rows, C)), A1, np.ones((1, C)))):
        f.set_factors(k, a)
    f.sweep(C, lam, 1, np.arange(C, dtype=np.int32))
    pivot = ((h * h).astype(np.float32) + np.float32(lam)).astype(np.float64)
    ref = h * v / pivot
    err = np.abs(f.factors(0).astype(np.float64) - ref) / np.abs(ref)
    assert err.max() <= 4.5 * 2.0 ** -24, err.max() * 2 ** 24
