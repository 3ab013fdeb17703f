"""Which mode pass a float three-way tensor takes by default: the lean pass caches rows that
have at least as many entries as there are blocks to copy them, and runs where such rows serve
a quarter of the gathers or where a tensor is small.

Tolerance: 2e-4 normwise in the factors after two sweeps, the FP32 bar of the other passes."""
import numpy as np
import pytest

import oracle
import paper_1410_5209_gb300 as tf
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1410_5209_gb300 import build
    build.build()


def rel(a, b):
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))


@pytest.mark.parametrize("dims,nnz,lean", [((700, 700, 700), 70_000, False),  # 100 a row
                                           ((300, 300, 300), 70_000, True),   # 233 a row
                                           ((3000, 3000, 3000), 40_000, True)])  # small
@pytest.mark.parametrize("C", [4, 10])
def test_rows_with_few_entries_take_the_staged_pass(dims, nnz, lean, C):
    p = synth.small(7 + C, dims, nnz, 4, C + 3)
    c, x = p.numpy()
    x = x.astype(np.float32).astype(np.float64)
    A = [a.numpy().astype(np.float32).astype(np.float64) for a in p.init_factors()]
    f = tf.Factorization(c, x, p.dims, p.K, dtype=tf.F32)
    for n in range(3):
        f.set_factors(n, A[n])
    t = oracle.Tensor(c, x, p.dims)
    r = oracle.residual(t, A)
    for s in range(2):
        order = p.column_order(s, C)
        f.sweep(C, 0.2, 1, order)
        oracle.sals_sweep(t, A, r, C, 0.2, 1, order)
        assert bool(f.counters()["pass_path"] & 8) == lean
    for n in range(3):
        assert rel(f.factors(n).astype(np.float64), A[n]) < 2e-4
    _, rmse = f.loss(0.2)
    _, ref = oracle.loss(t, r, A, 0.2)
    assert abs(rmse - ref) <= 1e-3 * ref
