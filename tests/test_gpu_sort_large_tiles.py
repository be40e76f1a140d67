"""The sort at the sizes where its passes change to tiles above the full size and
back (456 tiles of 256 threads by 16 and 20 32-bit keys, 608 tiles by 12 and 14
64-bit keys), against numpy's stable sort.  Everything is integer: exact."""
import pytest

from test_gpu_sort_tiles import _check

pytestmark = pytest.mark.gpu

EDGES = [456 * 4096, 608 * 3072, 608 * 3584, 456 * 5120]


@pytest.mark.parametrize("want_keys", [False, True])
@pytest.mark.parametrize("bits", [8, 32, 40, 64])
@pytest.mark.parametrize("n", [n for e in EDGES for n in (e, e + 1)] + [456 * 4096 + 5119])
def test_large_tile_edges(n, bits, want_keys):
    _check(n, bits, 8, want_keys)
