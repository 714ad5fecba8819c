"""Orders that the library's host code has to keep and that one GPU cannot show:
which device a free waits for, what a captured count may hold, when a pool may
be trimmed, what a server's budget is charged.  The library's objects are linked
with a CUDA runtime that runs no kernel and logs the calls (fake_cudart/), so
nothing here needs a GPU."""
import ctypes
import glob
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
    if not b.up_to_date():
        if not os.path.exists(b.NVCC):
            pytest.skip("nvcc not available to build the library")
        b.build()
    out = str(tmp_path_factory.mktemp("fake") / "libmotifs_fake.so")
    # -Bsymbolic: the library's calls go to this runtime, whatever else is loaded
    subprocess.check_call([gxx, "-std=c++17", "-O1", "-fPIC", "-shared", "-Wl,-Bsymbolic",
                           "-I", os.path.join(CUDA, "include"),
                           os.path.join(HERE, "fake_cudart", "cudart.cc"),
                           *sorted(glob.glob(os.path.join(b.BUILD, "*.o"))), "-o", out])
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
    with the last handle each device is waited for before its pool is trimmed."""
    fake.cudaSetDevice(1)
    g1, g2 = fake.graph(*PATH), fake.graph(*PATH)
    fake.cudaSetDevice(0)
    g0 = fake.graph(*PATH)
    fake.mt_graph_free(g1)
    fake.mt_graph_free(g0)
    fake.log()
    fake.mt_graph_free(g2)  # the last one
    log = calls(fake.log(), "sync", "free_async", "trim")
    trims = [i for i, e in enumerate(log) if e[0] == "trim"]
    assert {log[i][1] for i in trims} == {0, 1}
    for i in trims:
        last_free = max(j for j, e in enumerate(log[:i]) if e[0] == "free_async")
        assert ("sync", log[i][1]) in [e[:2] for e in log[last_free:i]]
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
