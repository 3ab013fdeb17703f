"""Which of the two launches of a wide pass works (float, 17 to 63 columns): the one with
register operands where every column's products stay in 2^-80 .. 2^60 or are zero, the block-wide
one otherwise.  The counts come from the device (pass_path bit 4: register operands, bit 0:
SIMT, bit 2 alone: tcgen05).

Tolerances: a first row update sees the very inputs of a dense FP64 solve and is held to the
FP32 bar of 1e-5 normwise, a later mode's to 2e-4 of the block-wide pass; what only block-wide
passes formed is bit for bit that of a context that asks for them."""
import numpy as np
import pytest

import paper_1410_5209_gb300 as tf
import synth

pytestmark = pytest.mark.gpu

REGISTER, SIMT, TCGEN05 = 16, 1, 4


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1410_5209_gb300 import build
    build.build()


DIMS, NNZ = (60, 90, 41), 9000


def problem(C, K=None):
    """Coordinates, values, factors: a zero first mode, others with a largest value of exactly 1
    in every column."""
    p = synth.small(20 + C, DIMS, NNZ, 5, K or C)
    coords, x = p.numpy()
    rng = np.random.default_rng(C)
    A = [np.zeros((DIMS[0], K or C), np.float32)]
    for d in DIMS[1:]:
        a = rng.uniform(0.1, 1.0, (d, K or C)) * rng.choice([-1.0, 1.0], (d, K or C))
        a[0] = 1.0
        A.append(a.astype(np.float32))
    return coords, x.astype(np.float32), A


def context(coords, x, A, P=0, path=0):
    f = tf.Factorization(coords, x, DIMS, A[0].shape[1], dtype=tf.F32)
    if P:
        f.set_schedule(P=P)
    if path:
        f.set_kernel_path(path)
    for n in range(3):
        f.set_factors(n, A[n])
    return f


def block_path(C):
    return 1 if C <= 31 else 2  # SIMT for 32-wide tiles, tcgen05 beyond


def block_bit(C):
    return SIMT if C <= 31 else TCGEN05


def row_update(coords, x, A, lam):
    """The first mode's rows, FP64."""
    h = A[1].astype(np.float64)[coords[:, 1]] * A[2].astype(np.float64)[coords[:, 2]]
    out = np.zeros(A[0].shape)
    for i in range(len(out)):
        e = coords[:, 0] == i
        out[i] = np.linalg.solve(h[e].T @ h[e] + lam * np.eye(h.shape[1]),
                                 h[e].T @ x[e].astype(np.float64))
    return out


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("P", [0, 1, 2000])
@pytest.mark.parametrize("C", [17, 20, 31, 32, 50, 63])
def test_products_on_both_sides_of_the_range(C, P):
    coords, x, A = problem(C)
    order = np.arange(C, dtype=np.int32)
    for power, register in ((-80, True), (-81, False), (59, True), (60, False)):
        B = [A[0], A[1] * np.float32(2.0 ** (power // 2)), A[2] * np.float32(2.0 ** (power - power // 2))]
        f, g = context(coords, x, B, P), context(coords, x, B, P, block_path(C))
        for h in (f, g):
            h.sweep(C, 1.0, 1, order)
        path = f.counters()["pass_path"]
        assert rel(f.factors(0), row_update(coords, x, B, 1.0)) <= 1e-5
        assert np.array_equal(f.factors(0), g.factors(0)) == (not register)
        if power == -81:  # the new first factor is as small, and so every later product
            assert path == block_bit(C)
        elif power == 60:  # the new first factor is as small as the others are large
            assert path == block_bit(C) | REGISTER | 4
        else:
            assert path & REGISTER


@pytest.mark.parametrize("C", [20, 31, 40, 63])
def test_one_column_out_of_range(C):
    """A collapsed column beside healthy ones takes every pass to the block-wide one, a NaN
    those that read it (the rows that meet it stay as they are); a zero column changes nothing."""
    coords, x, A = problem(C)
    order = np.arange(C, dtype=np.int32)
    for column in ("collapsed", "nan", "zero"):
        B = [A[0], A[1].copy(), A[2]]
        if column == "collapsed":
            B[1][:, C // 2] *= np.float32(2.0 ** -118)
        elif column == "nan":
            B[1][5, C // 2] = np.nan
        else:
            B[1][:, C // 2] = 0
        f, g = context(coords, x, B), context(coords, x, B, path=block_path(C))
        f.sweep(C, 1.0, 1, order)
        g.sweep(C, 1.0, 1, order)
        path = f.counters()["pass_path"]
        assert g.counters()["pass_path"] == block_bit(C)
        if column == "collapsed":
            assert path == block_bit(C)
            for n in range(3):
                assert np.array_equal(f.factors(n), g.factors(n))
            ref = row_update(coords, x, B, 1.0)
            assert rel(f.factors(0)[:, C // 2], ref[:, C // 2]) <= 1e-5
            continue
        if column == "nan":
            assert path == block_bit(C) | REGISTER | 4
            assert np.array_equal(f.factors(0), g.factors(0))
            meets = np.zeros(DIMS[0], bool)
            meets[coords[coords[:, 1] == 5, 0]] = True
            assert meets.any() and not f.factors(0)[meets].any() and f.factors(0)[~meets].all()
            assert f.counters()["singular_rows"] == g.counters()["singular_rows"]
        else:
            assert path == REGISTER | 4
        for n in range(3):
            a, b = f.factors(n), g.factors(n)
            assert np.array_equal(np.isnan(a), np.isnan(b))
            assert rel(np.nan_to_num(a), np.nan_to_num(b)) < 2e-4


@pytest.mark.parametrize("C,K", [(20, 45), (40, 85)])
def test_modes_that_enter_and_leave(C, K):
    """Products of 2^-100 against values of 2^40: the first mode's pass is out of range and its
    solve brings the second's into it; several splits, two inner iterations, eager and replayed
    as a graph: the same bits."""
    import torch
    coords, x, A = problem(C, K)
    x = x * np.float32(2.0 ** 40)
    B = [A[0], A[1] * np.float32(2.0 ** -100), A[2]]
    out = []
    for graphs in (False, True):
        f = context(coords, x, B)
        if graphs:
            stream = torch.cuda.Stream()
            f.set_stream(stream)
            f.set_graphs(True)
        f.sweep(C, 1.0, 1, np.arange(K, dtype=np.int32))
        first = f.counters()["pass_path"]
        assert first == block_bit(C) | REGISTER | 4
        seen = []
        for s in range(4):
            order = np.random.default_rng(s).permutation(K).astype(np.int32)
            f.sweep(C, 1.0, 2, order)
            seen.append(f.counters()["pass_path"])
        out.append((seen, [f.factors(n) for n in range(3)], f.loss(1.0)))
        if graphs:
            assert f.graph_info()["replays"] >= 3
        f.close()
    assert out[0][0] == out[1][0] and out[0][2] == out[1][2]
    for a, b in zip(out[0][1], out[1][1]):
        assert np.isfinite(a).all() and np.array_equal(a, b)
