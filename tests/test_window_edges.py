"""The pass over five-way tensors stages a step's indices and residuals as the 16-byte vectors
that cover them: items that start and end anywhere in a vector, and at the arrays' end.  Four-way
tensors run the generic form, which copies value by value."""
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


@pytest.mark.parametrize("dtype,tol", [(tf.F64, 1e-9), (tf.F32, 1e-4)])
@pytest.mark.parametrize("dims", [(61, 37, 300, 5), (61, 37, 300, 5, 40)])
@pytest.mark.parametrize("nnz,P", [(1, 0), (33, 0), (5_001, 1), (5_003, 0), (5_006, 700)])
def test_items_anywhere(dtype, tol, dims, nnz, P):
    """Two sweeps in subsets of 3, 1 columns against the oracle, the loss included.  FP64 1e-9;
    FP32 1e-4: rounding units of 6e-8 times systems whose condition (lambda 1, up to a few
    hundred entries a row) stays below 1e3, with the first sweep's error going through the
    second."""
    p = synth.small(71, dims, nnz, 3, 4, modes=["zipf"] + ["uniform"] * (len(dims) - 1))
    c, x = p.numpy()
    A = [a.numpy() for a in p.init_factors()]
    if dtype == tf.F32:
        x = x.astype(np.float32).astype(np.float64)
        A = [a.astype(np.float32).astype(np.float64) for a in A]
    f = tf.Factorization(c, x, p.dims, 4, dtype=dtype)
    if P:
        f.set_schedule(P=P)
    for n in range(len(dims)):
        f.set_factors(n, A[n])
    t = oracle.Tensor(c, x, p.dims)
    r = oracle.residual(t, A)
    for _ in range(2):
        f.sweep(3, 1.0, 2, order=np.arange(4))
        oracle.sals_sweep(t, A, r, 3, 1.0, 2, np.arange(4))
    for n in range(len(dims)):
        got = f.factors(n).astype(np.float64)
        assert np.linalg.norm(got - A[n]) <= tol * np.linalg.norm(A[n])
    assert np.linalg.norm(f.residual() - r) <= tol * max(np.linalg.norm(r), np.linalg.norm(x))
    assert abs(f.loss(0.0)[0] - float(r @ r)) <= 4 * tol * float(x @ x)
