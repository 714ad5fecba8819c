"""The cell method's exclusive-neighbour counters, which lanes add to one by one
when a batch of row segments holds members of several cells and together when it
holds one cell's: lists in which both kinds of batch follow each other.  GPU
only."""
import numpy as np
import pytest

import oracle
import synthetic as syn
from gpu_helpers import oracle_dense

pytestmark = pytest.mark.gpu


def _mixed_and_long_rows(groups, singles, long_row):
    """A hub whose list repeats `singles` members of short rows, their arcs to the
    hub cycling through the three codes, and one member with `long_row` pendant
    neighbours of all codes: segments of many members, then of one."""
    src, dst = [], []

    def arc(a, b, code):
        if code & 1:
            src.append(a)
            dst.append(b)
        if code & 2:
            src.append(b)
            dst.append(a)

    nxt = 1
    for g in range(groups):
        members = list(range(nxt, nxt + singles + 1))
        nxt += singles + 1
        for i, y in enumerate(members):
            arc(0, y, 1 + (i + g) % 3)
            for _ in range(long_row if i == singles else 1 + i % 3):
                arc(y, nxt, 1 + nxt % 3)
                nxt += 1
        for a, b in zip(members, members[1:]):  # arcs inside the list
            if (a + g) % 4 == 0:
                arc(a, b, 1 + (a + b) % 3)
    return syn.csr_from_arcs(nxt, src, dst)


@pytest.mark.parametrize("k,groups,singles,long_row", [
    (3, 6, 37, 300), (4, 4, 33, 290), (5, 2, 20, 60), (6, 1, 38, 8)])
def test_single_and_mixed_batches_follow_each_other(lib, k, groups, singles, long_row):
    lib.load_library()
    t = lib.table_build(k)
    g = _mixed_and_long_rows(groups, singles, long_row)
    want = oracle_dense(oracle.count(g, k)[0], t.class_masks())
    dg = lib.graph_from(g)
    for wpb in (0, 1):
        got = lib.to_numpy_u64(lib.count_tuned(dg, t, warps_per_block=wpb,
                                               method=lib.METHOD_CELLS))
        assert lib.count_stats(dg)[1] == 0
        np.testing.assert_array_equal(got, want)
    # equal graphs (no swaps), so many that at k = 5 and 6 their lists are kept: a
    # member brought by the last choice is then taken from its neighbours' counts
    R = 600 if k == 5 else 200
    b = lib.Batch(dg, t, R, 0)
    assert b.launch_info()["keeps_lists"] == (k >= 5)
    h = lib.to_numpy_u64(b.run(np.arange(1, R + 1, dtype=np.uint64))[0])
    assert b.error() == 0
    for r in range(R + 1):
        np.testing.assert_array_equal(h[r], want)
    b.free()
    t.free()
