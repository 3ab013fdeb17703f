"""Float passes and solves of 17 to 63 columns (register operands on the tensor cores, warp
solves in registers) at the edges of their chunks, steps and slots.

Tolerances: a first-split row update sees the oracle's very inputs and is held to the FP32 bar
of 1e-5 normwise; whole sweeps to 1e-3 in training RMSE and, as rounding travels through the
later modes and splits, 2e-4 in the factors; the residual copies to 1e-4 of a recomputation."""
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


def make(p, P):
    c, x = p.numpy()
    x = x.astype(np.float32).astype(np.float64)
    A = [a.numpy().astype(np.float32).astype(np.float64) for a in p.init_factors()]
    f = tf.Factorization(c, x, p.dims, p.K, dtype=tf.F32)
    if P:
        f.set_schedule(P=P)
    for n in range(p.N):
        f.set_factors(n, A[n])
    return f, oracle.Tensor(c, x, p.dims), A


def rel(a, b):
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))


@pytest.mark.parametrize("C", [17, 20, 28, 31, 32, 33, 52, 60, 63])
@pytest.mark.parametrize("P", [0, 1, 2000])
def test_row_update_and_sweeps(C, P):
    """Every chunk count, column C of H' first and last in a chunk, partial steps of 8, rows of
    one and of many items; two modes of unequal length with empty rows; a last split of five
    columns after full ones, weighted lambda and two inner iterations."""
    p = synth.small(300 + C, (211, 90, 61), 9_001, 5, C + 5, modes=["zipf", "uniform", "uniform"])
    f, t, A = make(p, P)
    r = oracle.residual(t, A)
    order = p.column_order(0, C)
    f.sweep(C, 0.5, 1, order)
    assert f.counters()["pass_path"] & 4
    oracle.sals_sweep(t, A, r, C, 0.5, 1, order)
    S = order[:C]
    assert rel(f.factors(0)[:, S].astype(np.float64), A[0][:, S]) <= 1e-5
    order = p.column_order(1, C)
    f.sweep(C, 0.2, 2, order, weighted=True)
    oracle.sals_sweep(t, A, r, C, 0.2, 2, order, weighted=True)
    for n in range(3):
        assert rel(f.factors(n).astype(np.float64), A[n]) < 2e-4
    _, rmse = f.loss(0.2)
    _, ref = oracle.loss(t, r, A, 0.2)
    assert abs(rmse - ref) <= 1e-3 * ref
    got = oracle.residual(t, [f.factors(n).astype(np.float64) for n in range(3)])
    assert rel(f.residual().astype(np.float64), got) < 1e-4


def test_singular_rows_and_empty_tensor():
    """lambda = 0: empty rows have no system and stay as they are; a tensor without entries
    solves to zero with lambda > 0."""
    rng = np.random.default_rng(2)
    cell = rng.choice(40 * 30, 900, replace=False)
    coords = np.stack([rng.integers(0, 3, 900) * 2, cell // 30, cell % 30], 1).astype(np.int32)
    f = tf.Factorization(coords, rng.standard_normal(900).astype(np.float32), (7, 40, 30), 20)
    A0 = np.full((7, 20), 0.25, np.float32)
    f.set_factors(0, A0)
    f.sweep(20, 0.0, 1)
    assert f.counters()["singular_rows"] >= 4
    assert np.array_equal(f.factors(0)[1::2], A0[1::2]) and not np.array_equal(f.factors(0)[0], A0[0])
    g = tf.Factorization(np.zeros((0, 3), np.int32), np.zeros(0), (5, 4, 3), 40)
    g.sweep(20, 1.0, 1)
    assert not g.factors(1).any() and g.loss(1.0) == (0.0, 0.0)
