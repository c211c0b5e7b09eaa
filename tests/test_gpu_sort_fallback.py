"""The radix sort with every tile on the path it takes when the tiles before it stay
silent: it counts the keys before it, from the first of all (few keys) or from its
group's first tile (many)."""
import numpy as np
import pytest

from test_gpu_sort import _sort

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1025, 16385, 311297, 1244000, 1246000, 2500001])
@pytest.mark.parametrize("dtype,bits", [(np.uint32, 10), (np.uint32, 20), (np.uint64, 63)])
def test_every_tile_counts_for_itself(n, dtype, bits):
    rng = np.random.default_rng(n + bits)
    key = rng.integers(0, 1 << bits, n, dtype=dtype)
    key[: n // 3] = key[0]
    order = np.argsort(key, kind="stable")
    k, v = _sort(key, bits, 0)
    assert np.array_equal(k, key[order]) and np.array_equal(v, order)
