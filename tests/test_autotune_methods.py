"""The autotuner against the automatic launch, which counts by cells: what it
returns names its method, and is never slower than passing no tuning."""
import numpy as np
import pytest

import synthetic as syn
from paper_1804_09741_gb300 import METHOD_CELLS, METHOD_ENUMERATE, autotune


def test_cached_entries_without_a_method_are_per_subgraph():
    p = autotune.TuneParams(**{"warps_per_block": 16, "split_scale": 0.5, "stack_cap": 0, "ms": 1.0})
    t = p.tuning()
    assert (t.warps_per_block, t.split_scale, t.method) == (16, 0.5, METHOD_ENUMERATE)


def test_tuning_keeps_the_method():
    assert autotune.TuneParams(32, 1.0, 0, method=int(METHOD_CELLS)).tuning().method == METHOD_CELLS
    assert autotune.TuneParams(method=None).tuning() is None
    for m in (METHOD_ENUMERATE, METHOD_CELLS):
        assert {c.method for c in autotune.candidates(100, 5, m)} == {int(m)}


def test_cached_batch_entry_of_a_method_keeps_it(tmp_path):
    """Entries of earlier caches carry the method in their key only."""
    g = syn.chung_lu_digraph(300, 1000, 2.2, None, 0.1, 12)
    path = str(tmp_path / "c.json")
    old = {"warps_per_block": 32, "split_scale": 0.5, "stack_cap": 0, "ms": 1.0}

    class Table:
        k, compact = 5, False
    for m in (METHOD_ENUMERATE, METHOD_CELLS):
        autotune.save_cache({autotune.degree_profile(g, 5) + f"-batch-m{int(m)}": old}, path)
        p = autotune.tune_batch(None, Table, g, 1, method=m, cache_path=path)
        assert p.tuning().method == m


@pytest.mark.gpu
@pytest.mark.parametrize("compact", [False, True])
def test_tuned_launch_is_not_slower_than_the_automatic_one(lib, tmp_path, compact):
    lib.load_library()
    k = 6 if compact else 5
    t = lib.table_build(k, compact=compact)
    g = syn.workload_graph("nullmodel_k6" if compact else "nullmodel_k5")
    dg = lib.graph_from(g)
    path = str(tmp_path / "t.json")
    p = autotune.tune(dg, t, graph=g, reps=3, cache_path=path)
    # per-subgraph launches take twice the time of cells on these graphs
    assert p.method is None or p.method == METHOD_CELLS
    assert autotune.tune(dg, t, graph=g, cache_path=path) == p
    seeds = np.arange(1, 4, dtype=np.uint64)
    pb = autotune.tune_batch(dg, t, g, g.m, probe_nulls=3, cache_path=path)
    assert (pb.tuning() is None) if compact else (pb.tuning().method == METHOD_CELLS)
    h0 = lib.to_numpy_u64(lib.Batch(dg, t, 3, g.m).run(seeds)[0])
    h1 = lib.to_numpy_u64(lib.Batch(dg, t, 3, g.m, pb.tuning()).run(seeds)[0])
    np.testing.assert_array_equal(h0, h1)
    t.free()
