"""The randomisers where their windows and sets change: numbers of attempts
around a window (64) and a buffer of draws (256), graphs so small or dense that
most attempts of a window overlap, sets that fill whole buckets, and arc counts
on both sides of the shared-memory limit, bit for bit against the oracle.  GPU
only."""
import numpy as np
import pytest

import oracle
import synthetic as syn

pytestmark = pytest.mark.gpu

MODELS = ["randomize", "randomize_dyads"]


def check(lib, g, model, seed, attempts):
    r = getattr(lib, model)(lib.graph_from(g), seed, attempts)
    rp, col = r.copy_csr()
    orp, ocol, _ = getattr(oracle, model)(g, seed, attempts)
    np.testing.assert_array_equal(rp, orp)
    np.testing.assert_array_equal(col, ocol)


@pytest.mark.parametrize("model", MODELS)
@pytest.mark.parametrize("attempts", [1, 63, 64, 65, 255, 256, 257, 513])
def test_window_and_buffer_edges(lib, model, attempts):
    lib.load_library()
    check(lib, syn.chung_lu_digraph(300, 1200, 2.2, None, 0.2, 2), model, 11, attempts)


@pytest.mark.parametrize("model", MODELS)
@pytest.mark.parametrize("m,attempts", [(2999, 31), (2999, 33), (2999, 30000), (3000, 30000)])
def test_both_window_widths(lib, model, m, attempts):
    lib.load_library()
    check(lib, syn.chung_lu_digraph(700, m, 2.2, None, 0.2, 4), model, 13, attempts)


@pytest.mark.parametrize("model", MODELS)
@pytest.mark.parametrize("n,p", [(5, 0.5), (8, 0.6), (12, 0.9), (40, 0.5), (90, 0.7)])
def test_overlapping_windows_and_full_buckets(lib, model, n, p):
    lib.load_library()
    g = syn.random_small_digraph(n, p, 0.3, n)
    for seed in (1, 2):
        check(lib, g, model, seed, 20 * g.m)


@pytest.mark.parametrize("model", MODELS)
@pytest.mark.parametrize("m", [16383, 16384, 16385, 17001])
def test_both_sides_of_the_shared_memory_limit(lib, model, m):
    lib.load_library()
    check(lib, syn.chung_lu_digraph(6000, m, 2.3, 150, 0.2, 3), model, 5, 30000)
