"""Counts captured into CUDA graphs: replays give the count again, after other
counts of the handle have moved on to more scratch and other graphs have come
and gone, and also when the first count of a root range is the captured one.  GPU
only."""
import numpy as np
import pytest

import synthetic as syn

pytestmark = pytest.mark.gpu


def capture(call):
    import torch
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call()
    return graph


def replay(lib, graph, out):
    import torch
    out.fill_(-1)
    graph.replay()
    torch.cuda.synchronize()
    return lib.to_numpy_u64(out)


def churn(lib, t):
    """Other handles take and give back pool memory."""
    for i in range(6):
        g = syn.chung_lu_digraph(900 + 50 * i, 4000, 2.3, 60, 0.1, i)
        lib.count_host(lib.graph_from(g), t)


@pytest.mark.parametrize("k", [3, 4, 5, 6])
@pytest.mark.parametrize("method", ["automatic", "enumerate"])
def test_captured_count_replays(lib, k, method):
    import torch
    lib.load_library()
    t, t6 = lib.table_build(k), lib.table_build(6, compact=True)
    g = syn.chung_lu_digraph(200, 560, 2.3, 30, 0.15, k)
    dg = lib.graph_from(g)
    out = torch.empty(t.num_classes, dtype=torch.int64, device="cuda")

    def count():
        if method == "automatic":
            lib.count(dg, t, out)
        else:
            lib.count_tuned(dg, t, out=out, method=lib.METHOD_ENUMERATE)
    count()
    want = lib.to_numpy_u64(out).copy()
    graph = capture(count)
    np.testing.assert_array_equal(replay(lib, graph, out), want)
    lib.count(dg, t6)  # needs more scratch for k < 6
    churn(lib, t)
    np.testing.assert_array_equal(replay(lib, graph, out), want)
    np.testing.assert_array_equal(lib.count_host(dg, t), want)
    np.testing.assert_array_equal(replay(lib, graph, out), want)
    del graph
    dg.free()
    t.free()
    t6.free()


def test_first_root_range_is_captured(lib):
    import torch
    lib.load_library()
    t = lib.table_build(4)
    g = syn.chung_lu_digraph(400, 1500, 2.3, 60, 0.15, 3)
    want = lib.count_roots(lib.graph_from(g), t, 50, 260)
    dg = lib.graph_from(g)
    full = lib.count_host(dg, t)  # allocates the scratch
    out = torch.empty(t.num_classes, dtype=torch.int64, device="cuda")

    def count():
        stream = torch.cuda.current_stream().cuda_stream
        st = lib.load_library().mt_count_roots(dg.handle, t.handle, 50, 260, out.data_ptr(), stream)
        assert st == lib.MT_OK
    graph = capture(count)
    np.testing.assert_array_equal(replay(lib, graph, out), want)
    np.testing.assert_array_equal(lib.count_host(dg, t), full)
    np.testing.assert_array_equal(lib.count_roots(dg, t, 50, 260), want)
    np.testing.assert_array_equal(lib.count_roots(dg, t, 0, 50) + want +
                                  lib.count_roots(dg, t, 260, 400), full)
    np.testing.assert_array_equal(replay(lib, graph, out), want)
    del graph
    dg.free()
    t.free()


def test_first_count_under_capture_is_refused(lib):
    """Scratch outlives a launch, so a captured count does not allocate it."""
    import torch
    lib.load_library()
    t = lib.table_build(3)
    dg = lib.graph_from(syn.chung_lu_digraph(100, 300, 2.3, 30, 0.15, 1))
    out = torch.empty(t.num_classes, dtype=torch.int64, device="cuda")
    status = []

    def count():
        stream = torch.cuda.current_stream().cuda_stream
        status.append(lib.load_library().mt_count(dg.handle, t.handle, out.data_ptr(), stream))
        out.fill_(7)
    graph = capture(count)
    assert status == [lib.MT_ECUDA]
    assert (replay(lib, graph, out) == 7).all()  # the refused call added nothing
    want = lib.count_host(dg, t)
    assert int(want.sum()) > 0
    dg.free()
    t.free()
