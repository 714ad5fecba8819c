"""z-scores with a warp or a thread per class, at numbers of nulls around the 32
lanes, and for classes that no null graph has: the oracle's doubles.  GPU only."""
import numpy as np
import pytest

import oracle
import synthetic as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [3, 4, 5])
@pytest.mark.parametrize("R", [1, 31, 32, 33, 65])
def test_zscores_equal_oracle(lib, k, R):
    lib.load_library()
    g = syn.random_small_digraph(18, 0.2, 0.4, k)
    t = lib.table_build(k)
    dg = lib.graph_from(g)
    b = lib.Batch(dg, t, R, 3 * g.m)
    h, z = b.run(np.arange(1, R + 1, dtype=np.uint64))
    h, z = lib.to_numpy_u64(h), z.cpu().numpy()
    assert b.error() == 0
    if k > 3:  # classes no null has are among them (k = 3 has 13, all met)
        assert (h[1:].sum(axis=0) == 0).any()
    np.testing.assert_array_equal(z, oracle.zscores(h[0], h[1:]))
    b.free()
    t.free()
