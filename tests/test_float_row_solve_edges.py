"""Float row solves of the narrow passes over rows of one, few and many partial slots, plain,
refined and with the FP64 fallback: runs of 32 single-slot rows whose first slot takes every
residue of the 16-byte vectors they are copied in, after 0 to 3 split rows.

Tolerances: a first row update sees the oracle's very inputs and is held to the FP32 bar of
1e-5 normwise, the factors after two sweeps to 2e-4."""
import numpy as np
import pytest

import oracle
import paper_1410_5209_gb300 as tf

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1410_5209_gb300 import build
    build.build()


def rel(a, b):
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))


@pytest.mark.parametrize("C", [1, 2, 3, 4, 5, 6, 8, 10, 12, 16])
@pytest.mark.parametrize("P", [1, 40, 2500])
@pytest.mark.parametrize("options", [None, (True, 0.0), (True, 1.5)])
def test_rows_of_every_slot_count(C, P, options):
    """With 2,500 bins (items of at most four entries) rows of 2, 3, 5 to 60 and more than 64
    slots between runs of single ones; uneven last split (K = 2 C + 1)."""
    rng = np.random.default_rng(C)
    counts = []
    for split in ([], [7], [9, 12], [30, 5, 300], [8, 1100, 100, 61]):
        counts += split + list(rng.integers(1, 5, 70))
    dims, K = (len(counts), 150, 40), 2 * C + 1
    row = np.repeat(np.arange(dims[0]), counts)
    cell = np.concatenate([rng.choice(150 * 40, n, replace=False) for n in counts])
    coords = np.stack([row, cell // 40, cell % 40], 1).astype(np.int32)
    x = rng.standard_normal(len(row)).astype(np.float32).astype(np.float64)
    A = [np.zeros((dims[0], K))]
    A += [(rng.standard_normal((d, K)) * 0.5).astype(np.float32).astype(np.float64) for d in dims[1:]]
    f = tf.Factorization(coords, x, dims, K, dtype=tf.F32)
    f.set_schedule(P=P)
    if options:
        f.set_solve(*options)
    for n in range(3):
        f.set_factors(n, A[n])
    t = oracle.Tensor(coords, x, dims)
    r = oracle.residual(t, A)
    for s in range(2):
        order = rng.permutation(K).astype(np.int32)
        f.sweep(C, 0.3, 1, order)
        oracle.sals_sweep(t, A, r, C, 0.3, 1, order)
        if s == 0:
            S = order[:C]
            assert rel(f.factors(0)[:, S].astype(np.float64), A[0][:, S]) <= 1e-5
    for n in range(3):
        assert rel(f.factors(n).astype(np.float64), A[n]) < 2e-4
    assert f.counters()["singular_rows"] == 0
    assert bool(f.fp64_rows()) == bool(options and options[1] and C > 1)
