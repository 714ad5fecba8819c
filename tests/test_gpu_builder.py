"""The graph builder where its branches change: rows of 32 entries and fewer sit in
registers, longer ones go through bitmaps; sorted rows are uploaded in place,
unsorted ones are sorted on the device, which also finds self-loops and duplicate
arcs.  GPU only."""
import numpy as np
import pytest

import oracle
import synthetic as syn
from gpu_helpers import oracle_dense

pytestmark = pytest.mark.gpu


def _rows(n, d, seed, both=False):
    """Vertex 0 with d out-neighbours (and the reverse arcs), a ring behind it."""
    rng = np.random.default_rng(seed)
    out = np.sort(rng.choice(np.arange(1, n), d, replace=False))
    src, dst = [np.zeros(d, np.int64)], [out]
    if both:
        src.append(out[::2])
        dst.append(np.zeros(out[::2].size, np.int64))
    ring = np.arange(1, n)
    src.append(ring)
    dst.append(np.roll(ring, -1))
    return syn.csr_from_arcs(n, np.concatenate(src), np.concatenate(dst))


def _shuffled(g, seed):
    rng = np.random.default_rng(seed)
    col = np.array(g.col, np.int32)
    for v in range(g.n):
        rng.shuffle(col[g.row_ptr[v]:g.row_ptr[v + 1]])
    return col


@pytest.mark.parametrize("n,d", [(60, 31), (60, 32), (60, 33), (700, 64), (4000, 2500),
                                 (65535, 40000)])
@pytest.mark.parametrize("both", [False, True])
def test_unsorted_rows(lib, n, d, both):
    lib.load_library()
    t = lib.table_build(3)
    g = _rows(n, d, d, both)
    dg = lib.graph_load_csr(n, g.row_ptr, _shuffled(g, 1))
    rp, col = dg.copy_csr()
    np.testing.assert_array_equal(rp, g.row_ptr)
    np.testing.assert_array_equal(col, g.col)
    want = lib.count_host(lib.graph_from(g), t)
    np.testing.assert_array_equal(lib.count_host(dg, t), want)
    if d <= 2500:
        np.testing.assert_array_equal(want, oracle_dense(oracle.count(g, 3)[0], t.class_masks()))
        np.testing.assert_array_equal(
            lib.count_roots(dg, t, 0, 1) + lib.count_roots(dg, t, 1, n), want)
    dg.free()
    t.free()


@pytest.mark.parametrize("n,d", [(60, 20), (60, 32), (60, 33), (4000, 2500)])
@pytest.mark.parametrize("order", ["sorted", "shuffled"])
@pytest.mark.parametrize("fault", ["duplicate", "selfloop"])
def test_faulty_rows_are_refused(lib, n, d, order, fault):
    """The same arc twice, or a self-loop, in a long row: MT_EINVAL, and the next
    load is fine."""
    lib.load_library()
    g = _rows(n, d, d)
    row = list(g.col[: g.row_ptr[1]])
    row.append(row[d // 2] if fault == "duplicate" else 0)
    row = np.sort(row)
    if order == "shuffled":
        np.random.default_rng(2).shuffle(row)
    rp = np.array(g.row_ptr, np.int32)
    rp[1:] += 1
    col = np.concatenate([row, g.col[g.row_ptr[1]:]])
    with pytest.raises(lib.MotifsError) as err:
        lib.graph_load_csr(n, rp, col)
    assert err.value.status == lib.MT_EINVAL
    ok = lib.graph_from(g)
    assert (ok.n, ok.m) == (g.n, g.m)
    ok.free()


def test_more_null_graphs_than_a_grid_dimension(lib):
    """65,600 null graphs of a graph smaller than k: built in parts, nothing to
    count."""
    lib.load_library()
    t = lib.table_build(4)
    dg = lib.graph_load_csr(3, [0, 1, 2, 3], [1, 2, 0])
    R = 65600
    b = lib.Batch(dg, t, R, 2)
    h, z = b.run(np.arange(R, dtype=np.uint64))
    assert not h.any() and not z.any()
    assert b.error() == 0
    b.free()
    dg.free()
    t.free()
