"""Workloads by which the speed of this framework is followed, through its public calls.

Each case is a dict of plain values; ``prepare`` makes from it what a user's program has in
hand (a tensor, the context that holds it, initial factors, requests), ``run`` is one pass of
that program, ``work`` what the pass cannot do without and ``exact`` its result in 64 bits from
plain torch.  Kinds of case:

  sweep    outer SALS / CDTF iterations over a resident tensor, the loss after them, and the
           factors copied back
  batch    the same over many small independent tensors held as one block-diagonal tensor,
           sweeps replayed as CUDA graphs
  fit      a whole job from host arrays: layout build, sweeps, loss, factors back, release
  foldin   new rows against frozen factors, one request or a batch of them
  predict  model values at held-out coordinates

Tensors are drawn like the rating-shaped data that the method is made for: coordinates distinct,
each mode's rows uniform or Zipf(1.1)-skewed, values from a low-rank CP model plus noise.
"""
import math

import numpy as np
import torch

import paper_1410_5209_gb300 as tf

DEV = "cuda"
RANK, NOISE = 10, 0.1
ZIPF = 1.1


# ------------------------------------------------------------------------------- the cases

def listed():
    return [
        # The reference setting in double precision: a small uniform tensor, five sweeps.  A pass
        # is a few hundred short launches, so latency counts.
        dict(name="sweep_f64_small", kind="sweep", dims="1000,1000,100", nnz=100_000, K=10, C=5,
             lam=1.0, sweeps=5, T_in=1, skew=False, weighted=False, dtype="f64"),
        # The headline: a large skewed three-way tensor, ten-column subsets.
        dict(name="sweep_skewed_c10", kind="sweep", dims="100000,100000,1000", nnz=100_000_000,
             K=100, C=10, lam=0.1, sweeps=2, T_in=1, skew=True, weighted=False, dtype="f32"),
        # CDTF: one column at a time, on a mid-sized skewed tensor of odd lengths.
        dict(name="sweep_cdtf", kind="sweep", dims="30011,20021,503", nnz=10_000_003, K=20, C=1,
             lam=0.1, sweeps=1, T_in=1, skew=True, weighted=False, dtype="f32"),
        # Subsets just past the narrow kernels, weighted lambda, two inner iterations.
        dict(name="sweep_c20_weighted", kind="sweep", dims="30011,20021,503", nnz=5_000_001,
             K=40, C=20, lam=0.1, sweeps=1, T_in=2, skew=True, weighted=True, dtype="f32"),
        # Wide subsets: two halves of K = 100.
        dict(name="sweep_c50", kind="sweep", dims="50021,40009,701", nnz=10_000_019, K=100, C=50,
             lam=0.1, sweeps=1, T_in=1, skew=True, weighted=False, dtype="f32"),
        # Five modes of a million rows, uniform: slices larger than the L2, coordinates too wide
        # for one 64-bit key.
        dict(name="sweep_5way", kind="sweep", dims="1000000,1000000,1000000,1000000,1000000",
             nnz=20_000_000, K=20, C=10, lam=1.0, sweeps=1, T_in=1, skew=False, weighted=False,
             dtype="f32"),
        # Hundreds of small tensors at once.
        dict(name="batch_small_tensors", kind="batch", count=256, lo_dim=50, hi_dim=5000,
             lo_nnz=1000, hi_nnz=1_000_000, K=16, C=4, lam=0.1, sweeps=3),
        # A small job as a serving process takes it: plain host arrays in, factors out.
        dict(name="fit_small_job", kind="fit", dims="700,3001,151", nnz=60_000, K=16, C=4,
             lam=0.1, sweeps=5, skew=False, pinned=False),
        # A large job end to end, from page-locked host arrays.
        dict(name="fit_large_job", kind="fit", dims="100000,100000,1000", nnz=30_000_000, K=20,
             C=10, lam=0.1, sweeps=1, skew=True, pinned=True),
        # One new user's row against a rank-100 model: an interactive request.
        dict(name="foldin_one", kind="foldin", dims="100000,100000,1000", K=100, lam=0.1,
             requests=1, lo_m=317, hi_m=317),
        # The requests that a loaded server finds waiting, of 10 to 10,000 entries each.
        dict(name="foldin_batch", kind="foldin", dims="100000,100000,1000", K=100, lam=0.1,
             requests=256, lo_m=10, hi_m=10_000),
        # Held-out error of the rank-100 model on device-resident test coordinates.
        dict(name="predict_heldout", kind="predict", dims="100000,100000,1000", K=100,
             m=3_000_017, dtype="f32"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["narrow", "narrow", "narrow", "wide", "order", "f64", "batch", "fit",
                       "foldin", "foldin", "predict"])
    K = rng.choice([8, 10, 16, 20, 33, 50, 64, 100])
    lam = rng.choice([0.1, 0.3, 1.0])
    if kind in ("narrow", "wide", "order", "f64"):
        N = rng.choice([2, 4, 5]) if kind == "order" else 3
        C = min(K, rng.choice([1, 2, 3, 4, 5, 8, 10, 10, 12, 15, 16]))
        nnz = _log(rng, 20_000, 20_000_000)
        if kind == "wide":
            K = rng.choice([33, 40, 64, 100])
            C = rng.randint(17, min(K, 100))
            nnz = _log(rng, 20_000, 10_000_000)
        if kind == "f64":
            nnz = _log(rng, 10_000, 1_000_000)
        if kind == "order":
            C = min(K, rng.choice([1, 4, 5, 10]))
        skew = rng.random() < 0.6
        dims = [_log(rng, 300 if N > 2 else 3000, 60_000 if N == 3 else 200_000) for _ in range(N)]
        if N == 3:
            dims[2] = _log(rng, 100, 3000)
        nnz = min(nnz, _cells(dims) // 40)
        return dict(kind="sweep", dims=",".join(map(str, dims)), nnz=nnz, K=K, C=C, lam=lam,
                    sweeps=1 if nnz > 1_000_000 else rng.choice([1, 2]),
                    T_in=2 if rng.random() < 0.2 else 1, skew=skew,
                    weighted=rng.random() < 0.25, dtype="f64" if kind == "f64" else "f32")
    if kind == "batch":
        return dict(kind="batch", count=_log(rng, 16, 400), lo_dim=50, hi_dim=5000, lo_nnz=1000,
                    hi_nnz=_log(rng, 100_000, 1_000_000), K=16, C=rng.choice([2, 4, 5, 8]),
                    lam=lam, sweeps=3)
    if kind == "fit":
        dims = [_log(rng, 50, 50_000), _log(rng, 50, 50_000), _log(rng, 50, 1000)]
        return dict(kind="fit", dims=",".join(map(str, dims)),
                    nnz=min(_log(rng, 1000, 20_000_000), _cells(dims) // 40), K=16,
                    C=rng.choice([4, 8, 10]), lam=lam, sweeps=2, skew=rng.random() < 0.5,
                    pinned=rng.random() < 0.5)
    if kind == "foldin":
        lo = _log(rng, 5, 300)
        return dict(kind="foldin", dims="100000,100000,1000",
                    K=rng.choice([10, 20, 31, 50, 64, 100, 127]), lam=lam,
                    requests=1 if rng.random() < 0.4 else _log(rng, 2, 400), lo_m=lo,
                    hi_m=_log(rng, lo, 10_000))
    return dict(kind="predict", dims="100000,100000,1000", K=rng.choice([10, 25, 50, 64, 100]),
                m=_log(rng, 1000, 4_000_000), dtype=rng.choice(["f32", "f32", "f64"]))


# ------------------------------------------------------------------------------- inputs

def _cells(dims):
    p = 1
    for d in dims:
        p *= d
    return p


def _dims(case):
    return [int(d) for d in case["dims"].split(",")]


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) * 7919 + 11)


def _torch_type(case):
    return torch.float64 if case.get("dtype") == "f64" else torch.float32


def _index(g, n, d, skew, shuffle=None):
    """n indices in 0..d-1, uniform or Zipf; shuffle: generator that maps Zipf ranks to rows."""
    u = torch.rand(n, generator=g, device=DEV, dtype=torch.float64)
    if not skew:
        return (u * d).long().clamp_(max=d - 1)
    cdf = torch.arange(1, d + 1, device=DEV, dtype=torch.float64).pow_(-ZIPF).cumsum_(0)
    rank = torch.searchsorted(cdf, u.mul_(cdf[-1])).clamp_(max=d - 1)
    return torch.randperm(d, generator=shuffle or g, device=DEV)[rank]


def _coords(g, dims, nnz, skew):
    """nnz distinct coordinates in random order; skew: all modes but the last are Zipf."""
    N = len(dims)
    lead = N  # modes whose packed index fits 62 bits; the tuples differ in these already
    while _cells(dims[:lead]) >= 2 ** 62:
        lead -= 1
    got, need = None, nnz
    while True:
        n = int(need * 1.2) + 64
        h = _gen(g.initial_seed())  # every round maps ranks to the same rows
        key = torch.zeros(n, dtype=torch.int64, device=DEV)
        for m in range(lead):
            key.mul_(dims[m]).add_(_index(g, n, dims[m], skew and m < N - 1, h))
        got = torch.unique(key if got is None else torch.cat([got, key]))
        del key
        if got.numel() >= nnz:
            break
        need = max(nnz - got.numel(), nnz // 8)
    got = got[torch.randperm(got.numel(), generator=g, device=DEV)[:nnz]]
    out = torch.empty((nnz, N), dtype=torch.int32, device=DEV)
    for m in reversed(range(lead)):
        out[:, m] = got % dims[m]
        got = got // dims[m]
    for m in range(lead, N):
        out[:, m] = _index(g, nnz, dims[m], False)
    return out


def _truth(g, dims, rank=RANK):
    std = rank ** (-1.0 / (2 * len(dims)))
    return [torch.randn((d, rank), generator=g, device=DEV) * std for d in dims]


def _values(g, coords, truth, dtype):
    out = torch.empty(coords.shape[0], device=DEV, dtype=dtype)
    for s in range(0, out.numel(), 1 << 24):
        c = coords[s:s + (1 << 24)].long()
        p = truth[0][c[:, 0]]
        for n in range(1, len(truth)):
            p = p * truth[n][c[:, n]]
        out[s:s + (1 << 24)] = p.sum(1)
    return out.add_(torch.randn(out.numel(), generator=g, device=DEV, dtype=dtype), alpha=NOISE)


def _initial(g, dims, K, dtype):
    """Algorithm 1's start: the first mode zero, the others normal."""
    std = K ** (-1.0 / (2 * len(dims)))
    return [torch.zeros((dims[0], K), dtype=dtype, device=DEV)] + [
        (torch.randn((d, K), generator=g, device=DEV) * std).to(dtype) for d in dims[1:]]


def _tensor(case, seed):
    """dims, coords, values, initial factors and the sweeps' column orders of a case."""
    g = _gen(seed)
    if case["kind"] == "batch":
        dims, coords = _block_diagonal(case, g)
    else:
        dims = _dims(case)
        coords = _coords(g, dims, case["nnz"], case["skew"])
    x = _values(g, coords, _truth(g, dims), _torch_type(case))
    A = _initial(g, dims, case["K"], _torch_type(case))
    r = np.random.RandomState(seed % (1 << 31))
    K = case["K"]
    orders = [(np.arange(K) if case["C"] == 1 else r.permutation(K)).astype(np.int32)
              for _ in range(case["sweeps"])]
    return dims, coords, x, A, orders


def _block_diagonal(case, g):
    """Independent tensors side by side, lengths and entry counts log-uniform.  The case alone
    fixes the lengths; the seed draws the entries."""
    n = case["count"]
    u = np.random.RandomState(n).rand(n, 4)
    lo, hi = math.log(case["lo_dim"]), math.log(case["hi_dim"])
    dims = torch.from_numpy(np.exp(lo + u[:, :3] * (hi - lo)).astype(np.int64)).to(DEV)
    lo, hi = math.log(case["lo_nnz"]), math.log(case["hi_nnz"])
    nnz = torch.from_numpy(np.exp(lo + u[:, 3] * (hi - lo)).astype(np.int64)).to(DEV)
    nnz = torch.minimum(nnz, dims.prod(1) // 2)
    which = torch.repeat_interleave(torch.arange(n, device=DEV), nnz)
    total = dims.sum(0)
    first = dims.cumsum(0) - dims
    key = torch.zeros(which.numel(), dtype=torch.int64, device=DEV)
    for m in range(3):
        r = torch.rand(which.numel(), generator=g, device=DEV, dtype=torch.float64)
        d = dims[which, m]
        i = torch.minimum((r * d).long(), d - 1) + first[which, m]
        key = key * total[m] + i
    key = torch.unique(key)  # a cell drawn twice is one entry
    key = key[torch.randperm(key.numel(), generator=g, device=DEV)]
    out = torch.empty((key.numel(), 3), dtype=torch.int32, device=DEV)
    for m in (2, 1, 0):
        out[:, m] = key % total[m]
        key = key // total[m]
    return [int(d) for d in total], out


def _requests(case, seed):
    """Fold-in requests: slices of the first mode, distinct entries, Zipf second mode."""
    g = _gen(seed)
    dims, K = _dims(case), case["K"]
    A = [torch.randn((d, K), generator=g, device=DEV) * K ** (-1.0 / 6) for d in dims]
    n = case["requests"]
    u = torch.rand(n, generator=g, device=DEV, dtype=torch.float64)
    lo, hi = math.log(case["lo_m"]), math.log(case["hi_m"] + 1)
    m = torch.exp(lo + u * (hi - lo)).long().clamp_(case["lo_m"], case["hi_m"])
    which = torch.repeat_interleave(torch.arange(n, device=DEV), m)
    j, k = _index(g, which.numel(), dims[1], True), _index(g, which.numel(), dims[2], False)
    key = torch.unique((which * dims[1] + j) * dims[2] + k)
    other = torch.stack([key // dims[2] % dims[1], key % dims[2]], 1)
    which = key // (dims[1] * dims[2])
    row = torch.randn((n, K), generator=g, device=DEV) * K ** (-1.0 / 6)
    x = (row[which] * A[1][other[:, 0]] * A[2][other[:, 1]]).sum(1)
    x += NOISE * torch.randn(x.numel(), generator=g, device=DEV)
    count = torch.bincount(which, minlength=n)
    return dims, A, other.to(torch.int32), x, which, count


# ------------------------------------------------------------------------------- the contract

def prepare(case, seed):
    kind = case["kind"]
    if kind in ("sweep", "batch"):
        dims, coords, x, A, orders = _tensor(case, seed)
        stream = torch.cuda.Stream() if kind == "batch" else None
        torch.cuda.synchronize()
        f = tf.Factorization(coords, x, dims, case["K"], seed=1, device_input=True,
                             dtype=tf.F64 if case.get("dtype") == "f64" else tf.F32,
                             stream=stream.cuda_stream if stream else None)
        for n, a in enumerate(A):
            f.set_factors(n, a.cpu().numpy())
        if kind == "batch":
            f.set_graphs(True)
        return dict(case=case, f=f, orders=orders, stream=stream)
    if kind == "fit":
        g = _gen(seed)
        dims = _dims(case)
        coords = _coords(g, dims, case["nnz"], case["skew"])
        x = _values(g, coords, _truth(g, dims), torch.float32)
        host = []
        for t in (coords, x):
            h = torch.empty(t.shape, dtype=t.dtype, pin_memory=case["pinned"])
            host.append(h.copy_(t))
        return dict(case=case, dims=dims, hold=host, coords=host[0].numpy(),
                    x=host[1].numpy(), seed=seed % 1000)
    if kind == "foldin":
        dims, A, other, x, which, count = _requests(case, seed)
        f = _model(dims, A, tf.F32, seed)
        other, x, ends = other.cpu().numpy(), x.cpu().numpy(), np.cumsum(count.cpu().numpy())
        reqs = [(other[a:b].copy(), x[a:b].copy()) for a, b in zip([0, *ends[:-1]], ends)]
        return dict(case=case, f=f, reqs=reqs)
    if kind == "predict":
        g = _gen(seed)
        dims, K, t = _dims(case), case["K"], _torch_type(case)
        A = [(torch.randn((d, K), generator=g, device=DEV) * K ** (-1.0 / 6)).to(t) for d in dims]
        f = _model(dims, A, tf.F64 if t == torch.float64 else tf.F32, seed)
        return dict(case=case, f=f, coords=_heldout(g, dims, case["m"]))
    raise ValueError(kind)


def _heldout(g, dims, m):
    return torch.stack([_index(g, m, d, n < len(dims) - 1) for n, d in enumerate(dims)],
                       1).to(torch.int32)


def _model(dims, A, dtype, seed):
    """A context that holds given factors (its own tensor is small: only the factors count)."""
    g = _gen(seed + 1)
    coords = _coords(g, dims, 10_000, False)
    x = torch.randn(10_000, generator=g, device=DEV, dtype=A[0].dtype)
    f = tf.Factorization(coords, x, dims, A[0].shape[1], seed=1, dtype=dtype, device_input=True)
    for n, a in enumerate(A):
        f.set_factors(n, a.cpu().numpy())
    return f


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("sweep", "batch"):
        f = state["f"]
        for order in state["orders"]:
            f.sweep(case["C"], case["lam"], T_in=case.get("T_in", 1), order=order,
                    weighted=case.get("weighted", False))
        loss, rmse = f.loss(case["lam"], weighted=case.get("weighted", False))
        return {"factors": [f.factors(n) for n in range(f.N)], "loss": loss, "rmse": rmse}
    if kind == "fit":
        with tf.Factorization(state["coords"], state["x"], state["dims"], case["K"],
                              seed=state["seed"]) as f:
            for _ in range(case["sweeps"]):
                f.sweep(case["C"], case["lam"])
            loss, rmse = f.loss(case["lam"])
            return {"factors": [f.factors(n) for n in range(f.N)], "loss": loss, "rmse": rmse}
    if kind == "foldin":
        if len(state["reqs"]) == 1:
            return {"rows": state["f"].foldin(0, *state["reqs"][0], case["lam"])}
        rows, status = state["f"].foldin_batch(0, state["reqs"], case["lam"])
        return {"rows": rows, "status": status}
    return {"values": state["f"].predict(state["coords"])}


def work(case):
    kind, K = case["kind"], case["K"]
    if kind == "foldin":
        lo, hi = case["lo_m"], case["hi_m"]
        each = (lo + hi) / 2 if hi < 1.5 * lo else (hi - lo) / math.log(hi / lo)
        m = case["requests"] * each
        return {"bytes": m * (12 + 8 * K) + case["requests"] * 4 * K,
                "flops": m * (K * (K + 1) + 3 * K) + case["requests"] * K ** 3 / 3}
    es = 8 if case.get("dtype") == "f64" else 4
    if kind == "predict":
        N = len(_dims(case))
        rows = sum(min(d, case["m"]) for d in _dims(case))
        return {"bytes": case["m"] * (4 * N + es) + rows * K * es, "flops": case["m"] * K * N}
    # per split and inner iteration every mode's pass reads the other modes' indices and the
    # residual, and the residual is written once per split; plus the factors, read and written
    if kind == "batch":
        N, lo, hi = 3, case["lo_nnz"], case["hi_nnz"]
        nnz = case["count"] * (hi - lo) / math.log(hi / lo)
        rows = 3 * case["count"] * (case["hi_dim"] - case["lo_dim"]) / math.log(
            case["hi_dim"] / case["lo_dim"])
    else:
        N, nnz, rows = len(_dims(case)), case["nnz"], sum(_dims(case))
    C, T = case["C"], case.get("T_in", 1)
    splits = -(-K // C) * case["sweeps"]
    stream = splits * nnz * (T * N * (4 * (N - 1) + es) + es)
    factors = case["sweeps"] * 2 * rows * K * es
    entry = T * N * (C * (C + 1) + (N - 1) * C + 2 * C) + 4 * C * N
    return {"bytes": stream + factors + (nnz * (4 * N + es) if kind == "fit" else 0),
            "flops": splits * (nnz * entry + rows * T * C ** 3 / 3)}


# ------------------------------------------------------------------------------- in 64 bits

def exact(case, seed):
    kind = case["kind"]
    if kind == "foldin":
        dims, A, other, x, which, count = _requests(case, seed)
        A = [a.double() for a in A]
        rows, at = [], 0
        for m in count.tolist():
            o, v = other[at:at + m].long(), x[at:at + m].double()
            h = A[1][o[:, 0]] * A[2][o[:, 1]]
            B = h.T @ h + case["lam"] * torch.eye(h.shape[1], device=DEV, dtype=torch.float64)
            rows.append(torch.cholesky_solve((h.T @ v)[:, None], torch.linalg.cholesky(B))[:, 0])
            at += m
        rows = torch.stack(rows)
        if len(rows) == 1:
            return {"rows": rows[0]}
        return {"rows": rows, "status": None}
    if kind == "predict":
        g = _gen(seed)
        dims, K, t = _dims(case), case["K"], _torch_type(case)
        A = [(torch.randn((d, K), generator=g, device=DEV) * K ** (-1.0 / 6)).to(t).double()
             for d in dims]
        coords = _heldout(g, dims, case["m"])
        out = torch.empty(case["m"], device=DEV, dtype=torch.float64)
        for s in range(0, case["m"], 1 << 20):
            c = coords[s:s + (1 << 20)].long()
            p = A[0][c[:, 0]]
            for n in range(1, len(dims)):
                p = p * A[n][c[:, n]]
            out[s:s + (1 << 20)] = p.sum(1)
        return {"values": out}
    if kind == "fit":
        return None  # starts from the library's own random factors
    if kind == "sweep" and case["nnz"] * -(-case["K"] // case["C"]) > 500_000_000:
        return None  # minutes of work in 64 bits
    dims, coords, x, A, orders = _tensor(case, seed)
    return _sals64(dims, coords, x.double(), [a.double() for a in A], orders, case)


SEG = 32  # entries per padded segment


def _sals64(dims, coords, R, A, orders, case):
    """Algorithm 1 in doubles: Gram matrices by padded segments of a mode's sorted entries."""
    N, C, lam = len(dims), case["C"], case["lam"]
    weighted = case.get("weighted", False)
    modes = []
    for n in range(N):
        perm = torch.argsort(coords[:, n], stable=True)
        count = torch.bincount(coords[:, n].long(), minlength=dims[n])
        segs = (count + SEG - 1) // SEG
        row = torch.repeat_interleave(torch.arange(dims[n], device=DEV), segs)
        k = torch.arange(row.numel(), device=DEV) - (segs.cumsum(0) - segs)[row]
        begin = (count.cumsum(0) - count)[row] + SEG * k
        length = torch.minimum(count[row] - SEG * k, torch.tensor(SEG, device=DEV))
        modes.append((perm, count, row, begin, length))
    lanes = torch.arange(SEG, device=DEV)

    def model(S):
        out = torch.empty_like(R)
        for s in range(0, R.numel(), 1 << 22):
            c = coords[s:s + (1 << 22)].long()
            p = A[0][:, S][c[:, 0]]
            for n in range(1, N):
                p = p * A[n][:, S][c[:, n]]
            out[s:s + (1 << 22)] = p.sum(1)
        return out

    def update(n, S, rhat):
        perm, count, row, begin, length = modes[n]
        c = S.numel()
        G = torch.zeros((dims[n], c + 1, c + 1), device=DEV, dtype=torch.float64)
        step = max(1, (1 << 24) // (SEG * (c + 1)) * 4)
        for s in range(0, row.numel(), step):
            b, ln, rw = begin[s:s + step], length[s:s + step], row[s:s + step]
            live = lanes < ln[:, None]
            e = perm[torch.where(live, b[:, None] + lanes, b[:, None])]
            h = live[..., None].double()
            for m in range(N):
                if m != n:
                    h = h * A[m][:, S][coords[:, m][e].long()]
            H = torch.cat([h, (rhat[e] * live)[..., None]], 2)
            G.index_add_(0, rw, H.transpose(1, 2) @ H)
        w = lam * count.double() if weighted else torch.full_like(count, lam, dtype=torch.float64)
        ok = w > 0
        B = G[:, :c, :c] + torch.where(ok, w, 1.0)[:, None, None] * torch.eye(
            c, device=DEV, dtype=torch.float64)
        for s in range(0, dims[n], 1 << 17):
            L = torch.linalg.cholesky(B[s:s + (1 << 17)])
            new = torch.cholesky_solve(G[s:s + (1 << 17), :c, c:], L)[..., 0]
            old = A[n][s:s + (1 << 17)][:, S]
            A[n][s:s + (1 << 17), S] = torch.where(ok[s:s + (1 << 17), None], new, old)

    R = R - model(torch.arange(case["K"], device=DEV))
    for order in orders:
        for s in range(0, case["K"], C):
            S = torch.from_numpy(order[s:s + C].astype(np.int64)).to(DEV)
            rhat = R + model(S)
            for _ in range(case.get("T_in", 1)):
                for n in range(N):
                    update(n, S, rhat)
            R = rhat - model(S)
    sq = float((R * R).sum())
    reg = sum(float(((a * a).sum(1) * (modes[n][1].double() if weighted else 1.0)).sum())
              for n, a in enumerate(A))
    return {"factors": [a.clone() for a in A], "loss": sq + lam * reg,
            "rmse": math.sqrt(sq / R.numel())}
