"""The k = 6 table's rows, built as permuted copies of the rows above canonical
5-vertex prefixes, against the oracle's canonical forms.  GPU only."""
import numpy as np
import pytest

from gpu_helpers import expected_ids

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def t6(lib):
    lib.load_library()
    t = lib.table_build(6)
    yield t
    t.free()


@pytest.mark.parametrize("prefix", [0, 1, (1 << 20) - 1, (1 << 20) - 2, 0x55555, 0xAAAAA, 0xFF,
                                    0xFFF00, 0x80001, 0x3C0F2])
def test_whole_rows(t6, prefix):
    """Empty, complete, one-way, disconnected and mixed prefixes: all 1,024
    words of the sixth vertex above each."""
    first = prefix << 10
    keys = np.arange(first, first + 1024, dtype=np.uint64)
    np.testing.assert_array_equal(t6.entries(first, 1024), expected_ids(6, keys, t6.class_masks()))
