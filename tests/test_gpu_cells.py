"""The cell method where its branches change: more distinct cells than it
numbers, rows longer than a lane's segments, hubs, lists that fill batches
exactly, against per-subgraph classification of the same graph (itself checked
against the oracle elsewhere).  GPU only."""
import numpy as np
import pytest

import oracle
import synthetic as syn
from gpu_helpers import oracle_dense

pytestmark = pytest.mark.gpu


def _hub(n, d, m, seed):
    """A vertex adjacent to d others (ids on both sides of it) in a sparse background."""
    rng = np.random.default_rng(seed)
    hub = n // 3
    others = rng.choice(np.delete(np.arange(n), hub), d, replace=False)
    key = {(hub, int(o)) if i % 3 else (int(o), hub) for i, o in enumerate(others)}
    while len(key) < d + m:
        a, b = (int(x) for x in rng.integers(0, n, 2))
        if a != b and a != hub and b != hub:
            key.add((a, b))
    a = np.array(sorted(key))
    return syn.csr_from_arcs(n, a[:, 0], a[:, 1])


GRAPHS = {
    "dense100": lambda: syn.random_small_digraph(100, 0.35, 0.4, 3),   # > 64 cells at k = 6
    "dense64": lambda: syn.random_small_digraph(64, 0.5, 0.2, 4),
    "complete33": lambda: syn.complete_digraph(33),                    # lists of 32 and fewer
    "hub": lambda: _hub(700, 260, 900, 5),
    "hub_rows": lambda: _hub(400, 97, 1500, 6),
    "power": lambda: syn.chung_lu_digraph(500, 2200, 2.1, None, 0.2, 7),
}


@pytest.mark.parametrize("k,name", [(k, g) for g in GRAPHS for k in (3, 4, 5, 6)
                                    if not (k == 6 and g in ("hub", "power"))])
def test_cells_equal_per_subgraph_counts(lib, k, name):
    lib.load_library()
    t = lib.table_build(k)
    dg = lib.graph_from(GRAPHS[name]())
    want = lib.to_numpy_u64(lib.count_tuned(dg, t, method=lib.METHOD_ENUMERATE))
    assert lib.count_stats(dg)[1] == 0
    for wpb in (0, 3):
        got = lib.to_numpy_u64(lib.count_tuned(dg, t, warps_per_block=wpb,
                                               method=lib.METHOD_CELLS))
        assert lib.count_stats(dg)[1] == 0
        np.testing.assert_array_equal(got, want)
    t.free()


@pytest.mark.parametrize("k", [3, 4, 5, 6])
def test_per_subgraph_counts_equal_oracle(lib, k):
    """The per-subgraph method asked for by name (calls without a tuning take
    the faster method for their k and size)."""
    lib.load_library()
    t = lib.table_build(k)
    for g in (syn.random_small_digraph(24, 0.18, 0.3, k),
              syn.chung_lu_digraph(150, 500, 2.2, None, 0.15, k)):
        dg = lib.graph_from(g)
        h = lib.to_numpy_u64(lib.count_tuned(dg, t, method=lib.METHOD_ENUMERATE))
        assert lib.count_stats(dg)[1] == 0
        np.testing.assert_array_equal(h, oracle_dense(oracle.count(g, k)[0], t.class_masks()))
    t.free()


@pytest.mark.parametrize("n", [4096, 16383, 16384, 16385])
def test_large_graphs_equal_oracle(lib, n):
    """Sizes around the 16-bit graph copy's limit (2^14 vertices)."""
    lib.load_library()
    t = lib.table_build(4)
    g = syn.chung_lu_digraph(n, 2 * n, 2.4, 60, 0.1, 9)
    want = oracle_dense(oracle.count(g, 4)[0], t.class_masks())
    np.testing.assert_array_equal(lib.count_host(lib.graph_from(g), t), want)
    t.free()


@pytest.mark.parametrize("k", [4, 5, 6])
def test_one_branch_holds_the_work(lib, k):
    """A path into a hub: one branch, and one of its choices, hold nearly all of
    the work, so it is cut and handed over at every level (third at k = 6)."""
    lib.load_library()
    t = lib.table_build(k)
    leaves = {4: 400, 5: 120, 6: 60}[k]
    src = [0, 1, 2] + [3] * leaves
    dst = [1, 2, 3] + list(range(4, 4 + leaves))
    g = syn.csr_from_arcs(4 + leaves, src, dst)
    want = oracle_dense(oracle.count(g, k)[0], t.class_masks())
    for perm in (np.arange(g.n), np.arange(g.n)[::-1]):
        dg = lib.graph_from(syn.relabel(g, perm))
        for _ in range(3):
            np.testing.assert_array_equal(lib.count_host(dg, t), want)
    t.free()


def _batch_equals_single_counts(lib, g, k, R):
    t = lib.table_build(k)
    dg = lib.graph_from(g)
    b = lib.Batch(dg, t, R, 2 * g.m)
    seeds = np.arange(3, 3 + R, dtype=np.uint64)
    h = lib.to_numpy_u64(b.run(seeds)[0])
    assert b.error() == 0
    for r in range(R + 1):
        one = dg if r == 0 else lib.randomize(dg, int(seeds[r - 1]), 2 * g.m)
        np.testing.assert_array_equal(
            h[r], lib.to_numpy_u64(lib.count_tuned(one, t, method=lib.METHOD_CELLS)))
        assert lib.count_stats(one)[1] == 0
    b.free()
    t.free()


@pytest.mark.parametrize("k,d", [(5, 58), (5, 70), (5, 90), (6, 38), (6, 50)])
def test_kept_lists_equal_single_counts(lib, k, d):
    """Batches of 8 graphs and more share the kept arcs of a list (largest degrees
    around and above the line); one graph's count reads the rows each time."""
    lib.load_library()
    _batch_equals_single_counts(lib, _hub(160 if k == 6 else 260, d, 400, d), k, 8)


@pytest.mark.parametrize("name", ["dense", "hub1100", "dense_hub"])
def test_kept_lists_that_do_not_fit(lib, name):
    """More arcs than a list keeps, a row too long for its counts, both in part."""
    lib.load_library()
    g = {"dense": lambda: syn.random_small_digraph(90, 0.3, 0.3, 8),
         "hub1100": lambda: _hub(1500, 1100, 1500, 9),
         "dense_hub": lambda: syn.disjoint_union(syn.random_small_digraph(75, 0.35, 0.5, 2),
                                                 _hub(200, 80, 300, 3))}[name]()
    _batch_equals_single_counts(lib, g, 5, 8)


@pytest.mark.parametrize("k", [3, 5, 6])
def test_smaller_plans_between_a_batch_and_its_run(lib, k):
    """Plans of one kernel with different shared-memory sizes, the largest made
    first and run last."""
    lib.load_library()
    t = lib.table_build(k)
    large = lib.graph_from(syn.chung_lu_digraph(400, 1200, 2.3, 40, 0.1, k))
    small = lib.graph_from(syn.chung_lu_digraph(60, 150, 2.3, 20, 0.1, k))
    want = lib.count_host(large, t)
    b = lib.Batch(large, t, 2, 100)
    bs = lib.Batch(small, t, 2, 100)
    seeds = np.array([1, 2], dtype=np.uint64)
    ws = lib.count_host(small, t)
    np.testing.assert_array_equal(lib.to_numpy_u64(b.run(seeds)[0])[0], want)
    np.testing.assert_array_equal(lib.to_numpy_u64(bs.run(seeds)[0])[0], ws)
    assert b.error() == 0 and bs.error() == 0
    b.free()
    bs.free()
    t.free()
