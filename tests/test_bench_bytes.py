"""The bytes that bench.py credits to a sort are those its kernels read and write."""
import os
import re

import pytest

import bench

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_11273_gb300", "csrc")


def _listed(bits, radix):
    """Pass by pass: (key read, index read, key written, index written)."""
    passes = -(-bits // radix)
    if bits <= 32:
        return [(4, 4 * (p > 0), 4 * (p < passes - 1), 4) for p in range(passes)]
    low = 32 // radix  # passes over the low half
    return [(8 if p < low else 4, 4 * (p > 0), 0 if p == passes - 1 else 8 if p < low - 1 else 4, 4)
            for p in range(passes)]


@pytest.mark.parametrize("bits", [1, 8, 16, 17, 24, 32, 33, 36, 40, 48, 63, 64])
@pytest.mark.parametrize("radix", [4, 8])
def test_sort_bytes(bits, radix):
    counting = 8 if bits > 32 else 4
    assert bench.sort_bytes(bits, radix) == counting + sum(map(sum, _listed(bits, radix)))


def test_known_values_and_the_rule_they_follow():
    assert [bench.sort_bytes(*x) for x in ((64, 8), (64, 4), (48, 4), (32, 8))] == [156, 316, 252, 60]
    assert bench.BYTES_SORT == 156
    # the source still drops the low halves after the passes over them
    s = open(os.path.join(CSRC, "rr_sort.cu")).read()
    assert re.search(r"drop = sizeof\(K\) == 8 && !keys_out && pl\.passes > kLowPasses \? kLowPasses - 1", s)
