"""Device memory of fold-in batches: bounded whatever the number of requests, rows the same as
alone."""
import numpy as np
import pytest

import paper_1410_5209_gb300 as tf

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1410_5209_gb300 import build
    build.build()


@pytest.mark.parametrize("dtype", [tf.F32, tf.F64])
def test_batch_scratch_is_bounded(dtype):
    rng = np.random.default_rng(1)
    dims, K, n = (10, 300, 200), 100, 700
    f = tf.Factorization(np.zeros((1, 3), np.int32), np.ones(1), dims, K, dtype=dtype)
    for k, d in enumerate(dims):
        f.set_factors(k, rng.standard_normal((d, K)) * 0.5)
    reqs = []
    for r in range(n):
        m = 0 if r == 5 else int(rng.integers(900, 1025)) if r != 400 else 60_000
        other = np.stack([rng.integers(0, 300, m), rng.integers(0, 200, m)], 1)
        reqs.append((other.astype(np.int32), rng.standard_normal(m).astype(f.npdt)))
    reqs[300][0][17, 1] = 200  # out of range
    f.foldin(0, *reqs[0], 0.5)
    tf.pool_trim()
    before = tf.pool_usage(reset_high=True)[0]
    rows, status = f.foldin_batch(0, reqs, 0.5)
    grown = tf.pool_usage()[1] - before
    size = np.dtype(f.npdt).itemsize
    inputs = sum(len(x) for _, x in reqs) * (8 + size) + n * K * size
    # 64 MiB of scratch, or what the largest request takes: 235 blocks of 91 tiles of 8 x 8
    # values; inputs and rows, block tables, and the pool's rounding of five buffers to 2 MiB
    assert grown <= max(64 << 20, 235 * 91 * 64 * size + (1 << 20)) + inputs + (14 << 20)
    assert list(np.flatnonzero(status)) == [300] and status[300] == 1
    for r in (0, 5, 150, 299, 301, 399, 400, 401, 699):
        assert np.array_equal(rows[r], f.foldin(0, *reqs[r], 0.5)) or len(reqs[r][1]) == 0
    assert not rows[5].any()
