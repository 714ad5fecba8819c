"""Orders that the library's host code has to keep and that one GPU cannot show:
which device a free waits for, what a captured count may hold, when a pool may
be trimmed, what a server's budget is charged.  The library's objects are linked
with a CUDA runtime that runs no kernel and logs the calls (fake_cudart/), so
nothing here needs a GPU."""
import ctypes
import os
import re
import shutil
import subprocess

import numpy as np
import pytest

import paper_1804_09741_gb300 as mt
from paper_1804_09741_gb300 import build as b

HERE = os.path.dirname(os.path.abspath(__file__))
CUDA = os.path.dirname(os.path.dirname(b.NVCC))
STREAM = 0x5000  # any non-null stream


class Fake:
    def __init__(self, path):
        self.lib = ctypes.CDLL(path)
        for name, (res, args) in mt.SIGNATURES.items():
            fn = getattr(self.lib, name)
            fn.restype, fn.argtypes = res, args
        self.lib.fake_log.restype = ctypes.c_char_p
        self.lib.fake_alloc.restype = ctypes.c_void_p
        self.lib.fake_alloc.argtypes = [ctypes.c_size_t]
        self.lib.fake_free.argtypes = [ctypes.c_void_p]
        self.lib.fake_set_capturing.argtypes = [ctypes.c_void_p]
        self.lib.fake_poke.argtypes = [ctypes.c_size_t, ctypes.c_size_t, ctypes.c_uint32]
        self.lib.fake_allocations.restype = ctypes.c_size_t

    def __getattr__(self, name):
        return getattr(self.lib, name)

    def log(self):
        """[(call, current device, pointer)] since the last log()."""
        out = [(m[1], int(m[2]), m[3]) for m in
               re.finditer(r"(.*) dev=(\d+) ptr=(\S+)\n", self.lib.fake_log().decode())]
        self.lib.fake_clear()
        return out

    def graph(self, n, rp, col):
        rp, col = np.array(rp, np.int32), np.array(col, np.int32)
        h = ctypes.c_void_p()
        self.fake_poke(16, 0, 2 * len(col))  # what the build found: undirected entries
        assert self.mt_graph_load_csr(n, int(rp[-1]), rp.ctypes.data, col.ctypes.data, None,
                                      ctypes.byref(h)) == mt.MT_OK
        return h.value

    def table(self, k):
        h = ctypes.c_void_p()
        self.fake_poke(4, 0, mt.NUM_CLASSES[k])  # the number of classes it found
        assert self.mt_table_build(k, None, ctypes.byref(h)) == mt.MT_OK
        return h.value


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None or not os.path.exists(os.path.join(CUDA, "include", "cuda_runtime_api.h")):
        pytest.skip("no host compiler or CUDA headers")
    objects = [os.path.join(b.BUILD, os.path.basename(src)[:-3] + ".o") for src in b._sources()]
    if not b.up_to_date() or not all(os.path.exists(o) for o in objects):
        if not os.path.exists(b.NVCC):
            pytest.skip("nvcc not available to build the library")
        b.build(force=True)
    out = str(tmp_path_factory.mktemp("fake") / "libmotifs_fake.so")
    # -Bsymbolic: the library's calls go to this runtime, whatever else is loaded
    subprocess.check_call([gxx, "-std=c++17", "-O1", "-fPIC", "-shared", "-Wl,-Bsymbolic",
                           "-I", os.path.join(CUDA, "include"),
                           os.path.join(HERE, "fake_cudart", "cudart.cc"),
                           *objects, "-o", out])
    return Fake(out)


PATH = (4, [0, 1, 2, 3, 3], [1, 2, 3])  # 0 -> 1 -> 2 -> 3


def calls(log, *names):
    return [e for e in log if e[0] in names]


def test_graph_free_waits_for_the_graphs_device(fake):
    """Counts may still run on the graph's device, which need not be the current
    one: it is waited for before its memory goes back to the pool."""
    fake.cudaSetDevice(1)
    g = fake.graph(*PATH)
    fake.cudaSetDevice(0)
    fake.log()
    assert fake.mt_graph_free(g) == mt.MT_OK
    log = calls(fake.log(), "sync", "free_async")
    frees = [i for i, e in enumerate(log) if e[0] == "free_async"]
    assert frees and all(log[i][1] == 1 for i in frees)
    assert ("sync", 1) in [e[:2] for e in log[:frees[0]]]
    dev = ctypes.c_int()
    fake.cudaGetDevice(ctypes.byref(dev))
    assert dev.value == 0


def test_set_workspace_waits_for_the_graphs_device(fake):
    fake.cudaSetDevice(1)
    g, t = fake.graph(*PATH), fake.table(3)
    hist = fake.fake_alloc(8 * 13)
    assert fake.mt_count(g, t, hist, None) == mt.MT_OK  # scratch on device 1
    fake.cudaSetDevice(0)
    fake.log()
    assert fake.mt_set_workspace(g, None, 0) == mt.MT_OK
    log = calls(fake.log(), "sync", "free_async")
    assert [e[:2] for e in log] == [("sync", 1), ("free_async", 1)]
    dev = ctypes.c_int()
    fake.cudaGetDevice(ctypes.byref(dev))
    assert dev.value == 0
    fake.mt_graph_free(g)
    fake.mt_table_free(t)
    fake.fake_free(hist)


def test_pools_are_trimmed_after_their_frees_have_run(fake):
    """Memory freed in stream order is the pool's only once the stream gets there:
    with its last handle a device is waited for before its pool is trimmed, and no
    other device is."""
    fake.cudaSetDevice(1)
    g1, g2, t1 = fake.graph(*PATH), fake.graph(*PATH), fake.table(3)
    fake.cudaSetDevice(0)
    g0 = fake.graph(*PATH)

    def freed(free, handle):
        fake.log()
        assert free(handle) == mt.MT_OK
        log = calls(fake.log(), "sync", "free_async", "trim")
        return [e[:2] for e in log]
    assert "trim" not in [e[0] for e in freed(fake.mt_graph_free, g1)]
    for free, last, device in ((fake.mt_graph_free, g0, 0), (fake.mt_graph_free, g2, None),
                               (fake.mt_table_free, t1, 1)):
        log = freed(free, last)
        if device is None:
            assert "trim" not in [e[0] for e in log]
            continue
        assert log[-2:] == [("sync", device), ("trim", device)]
        assert {d for _, d in log} == {device}
    dev = ctypes.c_int()
    fake.cudaGetDevice(ctypes.byref(dev))
    assert dev.value == 0


def test_captured_count_holds_no_host_memory_and_keeps_its_scratch(fake):
    """What a captured count uploads is read at every replay, so it uploads nothing
    from the host; and the scratch it uses stays, whatever later counts need."""
    g, t3, t4 = fake.graph(*PATH), fake.table(3), fake.table(4)
    hist = fake.fake_alloc(8 * 199)
    assert fake.mt_count(g, t3, hist, STREAM) == mt.MT_OK
    fake.fake_set_capturing(STREAM)
    fake.log()
    assert fake.mt_count(g, t3, hist, STREAM) == mt.MT_OK
    assert fake.mt_count_roots(g, t3, 1, 3, hist, STREAM) == mt.MT_OK
    log = fake.log()
    assert not calls(log, "captured_upload")
    assert not calls(log, "malloc", "free_async", "sync", "sync_stream")
    # nothing is allocated under capture
    assert fake.mt_count(g, t4, hist, STREAM) == mt.MT_ECUDA
    fake.fake_set_capturing(None)
    fake.log()
    assert fake.mt_count(g, t4, hist, STREAM) == mt.MT_OK  # moves on to more scratch
    log = fake.log()
    assert calls(log, "malloc") and not calls(log, "free_async")
    assert fake.mt_set_workspace(g, None, 0) == mt.MT_OK  # gives that back, not the captured one
    assert len(calls(fake.log(), "free_async")) == 1
    fake.mt_graph_free(g)
    assert len(calls(fake.log(), "free_async")) == 2  # the arrays and the captured scratch
    fake.mt_table_free(t3)
    fake.mt_table_free(t4)
    fake.fake_free(hist)


class FakeServer:
    def __init__(self, fake, tables, budget, slots=8):
        self.fake = fake
        h = ctypes.c_void_p()
        ts = [tables.get(k) for k in (3, 4, 5, 6)]
        assert fake.mt_server_create(*ts, budget, slots, 1e9, ctypes.byref(h)) == mt.MT_OK
        self.h = h.value

    def submit(self, k, n, rp, col):
        rp, col = np.array(rp, np.int32), np.array(col, np.int32)
        rid = ctypes.c_uint64()
        assert self.fake.mt_server_submit(self.h, k, n, int(rp[-1]), rp.ctypes.data,
                                          col.ctypes.data, ctypes.byref(rid)) == mt.MT_OK
        return rid.value

    def step(self):
        assert self.fake.mt_server_step(self.h, None, None, None) == mt.MT_OK

    def state(self, rid):
        """(state, status) without taking the result."""
        st = ctypes.c_int32()
        status = self.fake.mt_server_result(self.h, rid, ctypes.byref(st), None, None)
        return st.value, status

    def used(self):
        u = ctypes.c_size_t()
        assert self.fake.mt_server_used_bytes(self.h, ctypes.byref(u)) == mt.MT_OK
        return u.value

    def free(self):
        self.fake.mt_server_free(self.h)


def _used_by_one(fake, tables, k):
    s = FakeServer(fake, tables, 1 << 40)
    s.submit(k, *PATH)
    s.step()
    used = s.used()
    s.free()
    return used


@pytest.mark.parametrize("good_first", [False, True])
def test_failed_load_leaves_no_charge(fake, good_first):
    """A duplicate arc is found on the device, after the request and its k's
    scratch have been charged: both charges go with it, and requests of another k
    are admitted under a budget that holds one k's scratch at a time."""
    tables = {k: fake.table(k) for k in (3, 4)}
    one = {k: _used_by_one(fake, tables, k) for k in (3, 4)}
    s = FakeServer(fake, tables, max(one.values()) + 4096)
    if good_first:  # after rounds have run, too
        rid = s.submit(3, *PATH)
        for _ in range(3):
            s.step()
        assert s.state(rid) == (2, mt.MT_OK)
    fake.fake_poke(16, 8, 2)  # the next build finds a duplicate arc
    bad = s.submit(3, 4, [0, 2, 2, 2, 2], [1, 1])
    for _ in range(2):
        s.step()
    assert s.state(bad)[1] == mt.MT_EINVAL
    assert s.used() == 0
    good = s.submit(4, *PATH)
    for _ in range(4):
        s.step()
    assert s.state(good) == (2, mt.MT_OK)
    assert s.used() == 0
    s.free()
    for t in tables.values():
        fake.mt_table_free(t)


def test_failed_load_beside_a_good_one_is_charged_no_more(fake):
    """Of two requests of one k admitted together the failed one's share of the
    scratch is given back at once."""
    tables = {3: fake.table(3)}
    one = _used_by_one(fake, tables, 3)
    s = FakeServer(fake, tables, 1 << 40)
    fake.fake_poke(16, 8, 2)
    big = 400
    bad = s.submit(3, big + 1, [0] + [big] * (big + 1), list(range(1, big)) + [1])
    good = s.submit(3, *PATH)
    s.step()
    assert s.state(bad)[1] == mt.MT_EINVAL
    assert s.used() == one
    for _ in range(3):
        s.step()
    assert s.state(good) == (2, mt.MT_OK) and s.used() == 0
    s.free()
    fake.mt_table_free(tables[3])


@pytest.mark.parametrize("slots", [1, 8])
def test_failed_load_does_not_refuse_the_requests_behind_it(fake, slots):
    """A request that fits the budget alone is not refused, nor left out of a
    round, for the memory or the slot of one whose load fails."""
    tables = {3: fake.table(3)}
    s = FakeServer(fake, tables, _used_by_one(fake, tables, 3) + 64, slots)
    fake.fake_poke(16, 8, 2)
    bad = s.submit(3, 4, [0, 2, 2, 2, 2], [1, 1])
    good = s.submit(3, *PATH)
    s.step()
    assert s.state(bad)[1] == mt.MT_EINVAL
    assert s.state(good) == (1, mt.MT_OK)
    for _ in range(2):
        s.step()
    assert s.state(good) == (2, mt.MT_OK) and s.used() == 0
    s.free()
    fake.mt_table_free(tables[3])


@pytest.mark.parametrize("method,want", [(None, []), (0, []), (mt.METHOD_ENUMERATE, [0]),
                                         (mt.METHOD_CELLS, [1]), (1, [1])])
def test_python_server_follows_a_method_asked_for_by_name(fake, monkeypatch, method, want):
    from paper_1804_09741_gb300 import server

    class Table:
        handle = fake.table(3)

    class Recording:
        calls = []

        def __getattr__(self, name):
            if name == "mt_server_set_method":
                return lambda h, m: self.calls.append(m) or fake.mt_server_set_method(h, m)
            return getattr(fake, name)
    Recording.calls = []
    monkeypatch.setattr(server, "load_library", Recording)
    srv = server.Server({3: Table}) if method is None else server.Server({3: Table}, method=method)
    assert Recording.calls == want
    srv.free()
    fake.mt_table_free(Table.handle)


def test_methods_are_the_abi_values():
    assert (mt.METHOD_ENUMERATE, mt.METHOD_CELLS) == (0, 1)
    assert mt.make_tuning(method=mt.METHOD_CELLS).method == 1


@pytest.mark.parametrize("R", [65535, 65536, 140000])
def test_batches_past_a_grid_dimension(fake, R):
    """The builder's launches have a graph per step of the grid's y dimension,
    which ends at 65,535; a batch of more null graphs (too small to hold a k-set,
    so nothing is counted) is built in parts."""
    g, t = fake.graph(2, [0, 1, 1], [1]), fake.table(3)
    h = ctypes.c_void_p()
    assert fake.mt_batch_create(g, t, R, 1, ctypes.byref(h)) == mt.MT_OK
    seeds = np.zeros(R, np.uint64)
    hist = fake.fake_alloc((R + 1) * 13 * 8)
    fake.log()
    assert fake.mt_batch_run(h.value, seeds.ctypes.data, hist, None, None) == mt.MT_OK
    grids = [re.match(r"launch grid=(\d+)x(\d+)x(\d+) .*k_scatter", e[0]) for e in fake.log()]
    assert sum(int(m[2]) for m in grids if m) == R
    fake.mt_batch_free(h.value)
    fake.mt_graph_free(g)
    fake.mt_table_free(t)
    fake.fake_free(hist)
