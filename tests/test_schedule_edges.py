"""LPT schedules (host) against a plain heap: equal item by item, whichever way the loads are
kept (ring of buckets; heap for items too long for it)."""
import heapq

import numpy as np
import pytest

import paper_1410_5209_gb300 as tf

ITEM_COST = 32


def reference(off, P, cap):
    nnz = off[-1]
    cap = cap or max(1, -(-nnz // P))
    jobs = []
    for row, (b, e) in enumerate(zip(off, off[1:])):
        n = int(e - b)
        k = max(1, -(-n // cap))
        for c in range(k):
            length = n // k + (1 if c < n % k else 0)
            jobs.append((int(b), length, row, len(jobs)))
            b += length
    heap = [(0, p) for p in range(P)]
    bins = [[] for _ in range(P)]
    for job in sorted(jobs, key=lambda j: (-j[1], j[3])):
        load, p = heapq.heappop(heap)
        bins[p].append(job + (p,))
        heapq.heappush(heap, (load + job[1] + ITEM_COST, p))
    return [j for b in bins for j in b], np.cumsum([0] + [len(b) for b in bins])


@pytest.mark.parametrize("kind", ["ties", "zipf", "empty rows", "one row", "long items"])
@pytest.mark.parametrize("P", [1, 7, 64, 1000, 4099])
def test_lpt_equals_the_heap(kind, P):
    """Equal lengths by the thousand (whole buckets move on together), skewed rows split into
    chunks, rows without entries, a single row, and items longer than the ring of buckets
    holds (cap 3,000,000)."""
    rng = np.random.default_rng(P)
    cap = 0
    if kind == "ties":
        lens = rng.integers(18, 22, 6_000)
    elif kind == "zipf":
        lens = (40_000 / np.arange(1, 3_001) ** 1.1).astype(np.int64)
        rng.shuffle(lens)
    elif kind == "empty rows":
        lens = rng.integers(0, 3, 2_500) * rng.integers(0, 2, 2_500)
    elif kind == "one row":
        lens = np.array([12_345])
    else:
        lens, cap = rng.integers(0, 5_000_000, 300), 3_000_000
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    items, slots, ptr = tf.plan_mode(off, P, cap=cap)
    ref, ref_ptr = reference(off, P, cap)
    assert slots == len(ref) and np.array_equal(ptr, ref_ptr)
    got = np.stack([items[k] for k in ("begin", "len", "row", "slot", "bin")], 1)
    assert np.array_equal(got, np.array(ref, np.int64))
