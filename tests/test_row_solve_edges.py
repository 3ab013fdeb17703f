"""Row solves of the narrow passes (rows of one, few and many partial slots) and slice packs.

FP64 against the oracle within 1e-9: only summation orders and roundings differ."""
import numpy as np
import pytest
import torch

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


@pytest.mark.parametrize("C", [1, 2, 4, 5, 8, 10, 12, 16])
@pytest.mark.parametrize("P", [1, 40, 3000])
def test_rows_of_every_slot_count(C, P):
    """A heavy row beside light, single and empty ones: with 3,000 bins (items of at most four
    entries) rows of 1 to 4 slots, of 5 to 64 and of several units of 64, two sweeps so that
    the units' counters are used again; uneven last split (K = 2 C + 1)."""
    rng = np.random.default_rng(C)
    dims, K = (37, 150, 40), 2 * C + 1
    row = np.repeat(np.arange(37), [0, 1, 2, 4, 5, 8, 9, 16, 17, 20, 21, 40, 100, 256, 257, 300,
                                    520, 1030] + [150] * 19)
    cell = np.concatenate([rng.choice(150 * 40, n, replace=False) for n in np.bincount(row)])
    coords = np.stack([row, cell // 40, cell % 40], 1).astype(np.int32)
    x = rng.standard_normal(len(row))
    A = [np.zeros((dims[0], K))] + [rng.standard_normal((d, K)) * 0.5 for d in dims[1:]]
    f = tf.Factorization(coords, x, dims, K, dtype=tf.F64)
    f.set_schedule(P=P)
    for n in range(3):
        f.set_factors(n, A[n])
    t = oracle.Tensor(coords, x, dims)
    r = oracle.residual(t, A)
    for s in range(2):
        order = rng.permutation(K).astype(np.int32)
        f.sweep(C, 0.3, 1, order)
        oracle.sals_sweep(t, A, r, C, 0.3, 1, order)
    for n in range(3):
        assert rel(f.factors(n), A[n]) < 1e-9
    assert rel(f.residual(), r) < 1e-9
    assert f.counters()["singular_rows"] == 0
