"""Row schedules of rows longer than 32 bits: chunks that fit are planned, items that do not
are refused."""
import numpy as np
import pytest

import paper_1410_5209_gb300 as tf


def test_long_row_in_chunks_below_a_cap_beyond_32_bits():
    off = np.array([0, 3_000_000_000, 3_000_000_005], np.int64)
    plan = tf.plan_mode(off, 2, cap=2_500_000_000)
    items = plan[0]
    rows = {}
    for begin, length, row, *_ in items:
        rows.setdefault(int(row), []).append((int(begin), int(length)))
    assert sorted(rows[0]) == [(0, 1_500_000_000), (1_500_000_000, 1_500_000_000)]
    assert rows[1] == [(3_000_000_000, 5)]


@pytest.mark.parametrize("length,cap,policy", [(2_500_000_000, 3_000_000_000, tf.SCHED_LPT),
                                               (6_000_000_000, 5_000_000_000, tf.SCHED_LPT),
                                               (2 ** 31, 1000, tf.SCHED_GREEDY)])
def test_items_beyond_32_bits_are_refused(length, cap, policy):
    with pytest.raises(Exception):
        tf.plan_mode(np.array([0, length], np.int64), 2, cap=cap, policy=policy)
