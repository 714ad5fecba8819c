"""The cell method on both sides of its layout switches, with the layout that the
launch reports asserted: graph copy and relation words in shared memory, words
only, neither; and kept lists that have to give up, in batches that keep lists.
GPU only."""
import numpy as np
import pytest

import oracle
import synthetic as syn
from gpu_helpers import oracle_dense

pytestmark = pytest.mark.gpu

COPY, WORDS, NEITHER = (True, True), (False, True), (False, False)


@pytest.mark.parametrize("k,n,m,dmax,layout", [
    (3, 3500, 7000, 60, COPY), (3, 4096, 8192, 60, WORDS),
    (3, 12000, 24000, 60, WORDS), (3, 13000, 26000, 60, NEITHER),
    (4, 3500, 7000, 60, COPY), (4, 4096, 8192, 60, WORDS),
    (4, 12000, 24000, 60, WORDS), (4, 12500, 25000, 60, NEITHER),
    (5, 2500, 4500, 20, COPY), (5, 3200, 5500, 20, WORDS),
    (5, 8000, 14000, 20, WORDS), (5, 10000, 18000, 20, NEITHER),
    (6, 1600, 1900, 9, COPY), (6, 2600, 3000, 9, WORDS), (6, 6500, 7500, 9, NEITHER)])
def test_both_sides_of_a_layout_switch(lib, k, n, m, dmax, layout):
    lib.load_library()
    t = lib.table_build(k)
    g = syn.chung_lu_digraph(n, m, 2.4, dmax, 0.1, 9)
    dg = lib.graph_from(g)
    info = lib.launch_info(dg, k)
    assert (info["graph_in_smem"], info["words_in_smem"]) == layout, info
    want = oracle_dense(oracle.count(g, k)[0], t.class_masks())
    np.testing.assert_array_equal(lib.count_host(dg, t), want)
    dg.free()
    t.free()


def _two_hubs(leaves, arcs, seed):
    """Two hubs, not adjacent, one arc between either and every leaf, and arcs among
    the leaves.  Hubs are numbered first: the second is in the lists of the first's
    leaves, never before them."""
    rng = np.random.default_rng(seed)
    key = set()
    for h in (0, 1):
        for u in range(2, 2 + leaves):
            key.add((h, u) if rng.integers(2) else (u, h))
    while arcs:
        a, b = (int(x) for x in rng.integers(2, 2 + leaves, 2))
        if a != b and (a, b) not in key and (b, a) not in key:
            key.add((a, b))
            arcs -= 1
    a = np.array(sorted(key))
    return syn.csr_from_arcs(2 + leaves, a[:, 0], a[:, 1])


@pytest.mark.parametrize("leaves,R", [(1020, 8), (1023, 8), (1023, 7), (1023, 6), (1024, 8),
                                      (1060, 8)])
def test_rows_at_the_limit_of_kept_counts(lib, leaves, R):
    """A kept list's counts hold rows of up to 1,023 entries; with a longer row in
    it (the second hub's, in the list below the first hub and a leaf) the sets
    read all rows."""
    lib.load_library()
    t = lib.table_build(5)
    g = _two_hubs(leaves, 200, leaves)
    dg = lib.graph_from(g)
    assert dg.max_degree == leaves
    want = lib.to_numpy_u64(lib.count_tuned(dg, t, method=lib.METHOD_ENUMERATE))
    assert lib.count_stats(dg)[1] == 0
    b = lib.Batch(dg, t, R, 0)  # no swaps: the same graph R + 1 times
    assert b.launch_info()["keeps_lists"] == (R >= 7)  # from 8 graphs on
    h = lib.to_numpy_u64(b.run(np.arange(1, R + 1, dtype=np.uint64))[0])
    assert b.error() == 0
    for r in range(R + 1):
        np.testing.assert_array_equal(h[r], want)
    b.free()
    dg.free()
    t.free()


@pytest.mark.parametrize("k,n,p,R", [(5, 90, 0.3, 31), (6, 64, 0.4, 7)])
def test_lists_of_more_arcs_than_are_kept(lib, k, n, p, R):
    """Dense graphs: lists with more than the 1,024 arcs that fit."""
    lib.load_library()
    t = lib.table_build(k)
    g = syn.random_small_digraph(n, p, 0.3, 8)
    dg = lib.graph_from(g)
    want = lib.to_numpy_u64(lib.count_tuned(dg, t, method=lib.METHOD_ENUMERATE))
    b = lib.Batch(dg, t, R, 0)
    assert b.launch_info()["keeps_lists"]
    h = lib.to_numpy_u64(b.run(np.arange(1, R + 1, dtype=np.uint64))[0])
    assert b.error() == 0
    for r in range(R + 1):
        np.testing.assert_array_equal(h[r], want)
    b.free()
    dg.free()
    t.free()


@pytest.mark.parametrize("k,n,m,dmax,R,keeps", [
    (5, 900, 5000, None, 7, False), (5, 900, 5000, None, 15, True),   # sets per item
    (5, 700, 3000, None, 15, False), (5, 700, 3000, None, 31, True),
    (5, 700, 3000, 20, 63, False),                                    # degrees
    (6, 300, 1100, 40, 15, False), (6, 300, 1100, 40, 31, True),
    (6, 300, 1100, 25, 63, False)])
def test_both_sides_of_the_rule_for_keeping_lists(lib, k, n, m, dmax, R, keeps):
    """Every row against the single count of the same null graph, which reads the
    rows each time, and one against per-subgraph classification."""
    lib.load_library()
    t = lib.table_build(k)
    g = syn.chung_lu_digraph(n, m, 2.2 if k == 5 else 2.4, dmax, 0.1, 5)
    dg = lib.graph_from(g)
    b = lib.Batch(dg, t, R, 2 * g.m)
    assert b.launch_info()["keeps_lists"] == keeps
    h = lib.to_numpy_u64(b.run(np.arange(1, R + 1, dtype=np.uint64))[0])
    assert b.error() == 0
    for r in range(R + 1):
        one = dg if r == 0 else lib.randomize(dg, r, 2 * g.m)
        np.testing.assert_array_equal(
            h[r], lib.to_numpy_u64(lib.count_tuned(one, t, method=lib.METHOD_CELLS)))
    np.testing.assert_array_equal(
        h[R], lib.to_numpy_u64(lib.count_tuned(one, t, method=lib.METHOD_ENUMERATE)))
    b.free()
    dg.free()
    t.free()
