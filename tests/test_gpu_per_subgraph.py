"""Per-subgraph classification (METHOD_ENUMERATE) asked for by name in the
layouts and tail passes it has of its own: candidate stacks and relation words in
global memory, the packed passes over short lists and both groupings of the
k = 6 tail, and compact tables.  Calls without a tuning use the cell method, so
none of them gets here.  GPU only."""
from math import comb

import numpy as np
import pytest

import oracle
import synthetic as syn
from gpu_helpers import oracle_dense

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tables(lib):
    lib.load_library()
    out = {}

    def get(k, compact=False):
        if (k, compact) not in out:
            out[k, compact] = lib.table_build(k, compact=compact)
        return out[k, compact]
    yield get
    for t in out.values():
        t.free()


def per_subgraph(lib, dg, t, **tuning):
    h = lib.to_numpy_u64(lib.count_tuned(dg, t, method=lib.METHOD_ENUMERATE, **tuning))
    assert lib.count_stats(dg)[1] == 0
    return h


@pytest.mark.parametrize("k,n,m", [(6, 26, 34), (6, 40, 70), (6, 24, 60), (5, 40, 90)])
def test_short_lists_equal_oracle(lib, tables, k, n, m):
    """Lists of up to 16 candidates, which several choices share a pass over."""
    t = tables(k)
    for seed in (1, 2, 3):
        g = syn.uniform_digraph(n, m, seed)
        want = oracle_dense(oracle.count(g, k)[0], t.class_masks())
        np.testing.assert_array_equal(per_subgraph(lib, lib.graph_from(g), t), want)


def _star(d, both):
    leaves = np.arange(1, d + 1)
    zero = np.zeros(d, np.int64)
    return syn.csr_from_arcs(d + 1, np.concatenate([zero, leaves]) if both else zero,
                             np.concatenate([leaves, zero]) if both else leaves)


@pytest.mark.parametrize("k,d,both", [(3, 4000, False), (4, 4000, False), (4, 4000, True),
                                      (5, 1000, False), (6, 300, True)])
def test_stacks_in_global_memory(lib, tables, k, d, both):
    """A star's C(d, k - 1) sets, all of one class."""
    t = tables(k)
    one, sets = oracle.count(_star(k - 1, both), k)
    assert sets == 1
    want = oracle_dense({next(iter(one)): comb(d, k - 1)}, t.class_masks())
    np.testing.assert_array_equal(per_subgraph(lib, lib.graph_from(_star(d, both)), t), want)


@pytest.mark.parametrize("k,m,dmax", [(3, 60000, 60), (4, 40000, 30), (5, 30000, 12)])
def test_words_in_global_memory(lib, tables, k, m, dmax):
    """n = 20,000: 16 warps' relation words do not fit shared memory."""
    t = tables(k)
    g = syn.chung_lu_digraph(20000, m, 2.5, dmax, 0.1, k)
    dg = lib.graph_from(g)
    assert not lib.launch_info(dg, k)["words_in_smem"]
    want = oracle_dense(oracle.count(g, k)[0], t.class_masks())
    np.testing.assert_array_equal(per_subgraph(lib, dg, t), want)


@pytest.mark.parametrize("seed", [0, 1, 2])
def test_compact_table(lib, tables, seed):
    g = syn.random_small_digraph([14, 22, 30][seed], [0.3, 0.15, 0.1][seed], 0.3, 40 + seed)
    t = tables(6, True)
    dg = lib.graph_from(g)
    want = oracle_dense(oracle.count(g, 6)[0], t.class_masks())
    np.testing.assert_array_equal(per_subgraph(lib, dg, t), want)
    np.testing.assert_array_equal(per_subgraph(lib, dg, t, warps_per_block=2), want)


@pytest.mark.parametrize("compact", [False, True])
@pytest.mark.parametrize("R", [3, 63])
def test_k6_batches(lib, tables, R, compact):
    """At most 3 blocks per graph (one match for all choices of a group) and more
    (three choices per match): every row against the cell method's, three of them
    against the oracle's count of the oracle's null graph."""
    g = syn.chung_lu_digraph(60, 130, 2.3, None, 0.1, 106)
    t = tables(6, compact)
    dg = lib.graph_from(g)
    blocks = lib.launch_info(dg, 6)["blocks"]
    assert (blocks <= 3 * (R + 1)) == (R == 63)
    seeds = np.arange(1, R + 1, dtype=np.uint64)
    b = lib.Batch(dg, t, R, 10 * g.m, lib.make_tuning(method=lib.METHOD_ENUMERATE))
    h = lib.to_numpy_u64(b.run(seeds)[0]).copy()
    assert b.error() == 0
    cells = lib.Batch(dg, t, R, 10 * g.m)
    np.testing.assert_array_equal(h, lib.to_numpy_u64(cells.run(seeds)[0]))
    roots = np.arange(g.n)
    for r in (0, 1, R):
        gr = g if r == 0 else syn.Graph(g.n, *oracle.randomize(g, r, 10 * g.m)[:2])
        np.testing.assert_array_equal(
            h[r], oracle_dense(oracle.count_roots_split(gr, 6, roots)[0], t.class_masks()))
    b.free()
    cells.free()


@pytest.mark.parametrize("k", [3, 4, 5])
def test_batches(lib, tables, k):
    g = syn.chung_lu_digraph(140, 440, 2.3, None, 0.1, 200 + k)
    t = tables(k)
    dg = lib.graph_from(g)
    for null_model, make in ((lib.NULL_ARC_SWAP, oracle.randomize),
                             (lib.NULL_DYAD_SWAP, oracle.randomize_dyads)):
        b = lib.Batch(dg, t, 4, 10 * g.m, lib.make_tuning(method=lib.METHOD_ENUMERATE),
                      null_model=null_model)
        h = lib.to_numpy_u64(b.run(np.arange(1, 5, dtype=np.uint64))[0])
        assert b.error() == 0
        for r in range(5):
            gr = g if r == 0 else syn.Graph(g.n, *make(g, r, 10 * g.m)[:2])
            np.testing.assert_array_equal(h[r], oracle_dense(oracle.count(gr, k)[0],
                                                             t.class_masks()))
        b.free()


def test_server_by_name(lib, tables):
    """Rounds of per-subgraph launches, over all k and with a compact table."""
    from paper_1804_09741_gb300.server import Server, run_stream
    ts = {3: tables(3), 4: tables(4), 5: tables(5), 6: tables(6, True)}
    reqs = [(k, syn.chung_lu_digraph(n, 3 * n, 2.3, 25, 0.2, 10 * k + n))
            for k in (3, 4, 5, 6) for n in ([40, 200, 600] if k < 6 else [30, 60, 110])]
    srv = Server(ts, memory_budget=2 << 30, max_slots=6, round_cost=2e6,
                 method=lib.METHOD_ENUMERATE)
    out, _, _ = run_stream(srv, reqs)
    for (k, g), (st, hist, status) in zip(reqs, out):
        assert st == 2, status
        np.testing.assert_array_equal(hist, per_subgraph(lib, lib.graph_from(g), ts[k]))
    assert srv.used_bytes() == 0
    srv.free()


@pytest.mark.parametrize("name", ["uniform_k3", "chunglu_k4", "nullmodel_k5", "nullmodel_k6"])
def test_workload_graphs(lib, tables, name):
    """The four workload graphs, hubs and rows of many batches among them: the
    cell method's histogram, and at k = 3 and 4 the oracle's."""
    k = syn.WORKLOADS[name]["k"]
    g = syn.workload_graph(name)
    t = tables(k)
    dg = lib.graph_from(g)
    got = per_subgraph(lib, dg, t)
    np.testing.assert_array_equal(got, lib.count_host(dg, t))
    if k <= 4:
        np.testing.assert_array_equal(got, oracle_dense(oracle.count(g, k)[0], t.class_masks()))
