"""The one-column pass of three-way tensors and the loss's sums at the edges of their steps and
ranges."""
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


@pytest.mark.parametrize("dtype,tol", [(tf.F64, 1e-9), (tf.F32, 2e-5)])
@pytest.mark.parametrize("P", [0, 1, 700])
def test_cdtf_pass(dtype, tol, P):
    """C = 1 against the oracle: items of 1 to many steps of 32 and of 128 entries, empty rows,
    three columns of which the second and third refresh R-hat, two inner iterations.  FP64
    1e-9; FP32 2e-5 in the factors (sums of FP32 products over up to 400 entries a row, three
    columns deep: a few hundred rounding units of 6e-8)."""
    p = synth.small(61, (90, 37, 500), 7_003, 3, 3, modes=["zipf", "uniform", "uniform"])
    c, x = p.numpy()
    A = [a.numpy() for a in p.init_factors()]
    if dtype == tf.F32:
        x = x.astype(np.float32).astype(np.float64)
        A = [a.astype(np.float32).astype(np.float64) for a in A]
    f = tf.Factorization(c, x, p.dims, 3, dtype=dtype)
    if P:
        f.set_schedule(P=P)
    for n in range(3):
        f.set_factors(n, A[n])
    t = oracle.Tensor(c, x, p.dims)
    r = oracle.residual(t, A)
    for _ in range(2):
        f.sweep(1, 0.3, 2)
        oracle.sals_sweep(t, A, r, 1, 0.3, 2, np.arange(3))
    for n in range(3):
        got = f.factors(n).astype(np.float64)
        assert np.linalg.norm(got - A[n]) <= tol * np.linalg.norm(A[n])
    assert np.linalg.norm(f.residual() - r) <= tol * np.linalg.norm(r)


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("scale", [1.0, 1e-20, 1e18])
def test_regulariser_over_the_float_range(scale, weighted):
    """lambda ||A||^2 of factors around 1, and where squares leave the float range (FP64 form):
    1e-12 of a long double sum."""
    rng = np.random.default_rng(3)
    dims, K = (300, 50, 7), 33
    coords = np.stack([np.arange(40), np.arange(40), np.arange(40) % 7], 1).astype(np.int32)
    f = tf.Factorization(coords, np.zeros(40), dims, K, dtype=tf.F32)
    A = [np.zeros((dims[0], K), np.float32)] + [
        (rng.standard_normal((d, K)) * scale).astype(np.float32) for d in dims[1:]]
    for n in range(3):
        f.set_factors(n, A[n])
    loss, rmse = f.loss(0.7, weighted=weighted)
    ref = sum(((a.astype(np.longdouble) ** 2).sum(1)
               * (np.bincount(coords[:, n], minlength=dims[n]) if weighted else 1)).sum()
              for n, a in enumerate(A))
    assert rmse == 0.0 and abs(loss - 0.7 * float(ref)) <= 1e-12 * 0.7 * float(ref)
