"""Fold-in (K < 128) at the edges of its tiles and blocks.

Tolerance: a row within 1e-9 (FP64) and 1e-5 (FP32) of a dense FP64 solve from the same
numbers."""
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


def dense(A, mode, other, x, lam):
    h = np.ones((len(x), A[0].shape[1]))
    for t, l in enumerate(l for l in range(len(A)) if l != mode):
        h = h * A[l].astype(np.float64)[other[:, t]]
    return np.linalg.solve(h.T @ h + lam * np.eye(h.shape[1]), h.T @ x.astype(np.float64))


@pytest.mark.parametrize("dtype,tol", [(tf.F64, 1e-9), (tf.F32, 1e-5)])
@pytest.mark.parametrize("K", [1, 7, 16, 17, 31, 32, 48, 63, 64, 100, 127])
def test_foldin_edges(K, dtype, tol):
    """Every tile width, panel remainder and vector / scalar row load, requests around the
    blocks of 64 and 256 entries, the three orders; in a batch and alone, bit for bit."""
    for N, mode in ((3, 1), (2, 0), (4, 2)):
        dims = [40, 60, 50, 30][:N]
        f, A, rng = model(dims, K, dtype, 10 * K + N)
        reqs = []
        for m in ((1, 31, 64, 65, 300, 1024, 1025) if N == 3 else (1, 70, 1500)):
            other = np.stack([rng.integers(0, dims[l], m) for l in range(N) if l != mode], 1)
            reqs.append((other.astype(np.int32), rng.standard_normal(m).astype(f.npdt)))
        rows, status = f.foldin_batch(mode, reqs, 0.8)
        assert not status.any()
        for row, (other, x) in zip(rows, reqs):
            ref = dense(A, mode, other, x, 0.8)
            assert np.linalg.norm(row - ref) <= tol * np.linalg.norm(ref)
            assert np.array_equal(row, f.foldin(mode, other, x, 0.8))


def test_foldin_flags_only_the_bad_requests():
    """A bad index in a later block and a singular system leave their neighbours alone."""
    f, A, rng = model([40, 60, 50], 33, tf.F32, 5)
    good = (rng.integers(0, 50, (700, 2)).astype(np.int32), rng.standard_normal(700))
    bad = (good[0].copy(), good[1])
    bad[0][650, 1] = 50
    few = (good[0][:5], good[1][:5])
    none = (good[0][:0], good[1][:0])
    rows, status = f.foldin_batch(0, [good, bad, none, good], 0.0)
    assert list(status) == [0, 1, 2, 0] and not rows[1:3].any()
    assert np.array_equal(rows[0], rows[3])
    rows, status = f.foldin_batch(0, [few, none], 0.5)
    assert list(status) == [0, 0] and not rows[1].any()
    assert np.linalg.norm(rows[0] - dense(A, 0, *few, 0.5)) <= 1e-5 * np.linalg.norm(rows[0])
