"""The sort at the sizes where its tile size, its look-back words or its key width
change, against numpy's stable sort, with a workspace of exactly the size asked
for (the bytes after it are checked).  Everything is integer: exact."""
import numpy as np
import pytest
import torch

from paper_2506_11273_gb300 import rr

pytestmark = pytest.mark.gpu

# 456 tiles of 256 threads by 4, 8 and 12 keys; 2^20 keys end the 32-bit look-back words
EDGES = [456 * 1024, 456 * 2048, 1 << 20, 456 * 3072, 456 * 4096]
GUARD = 4096


def _keys(n, bits, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    k = rng.integers(0, 2 ** 64, n, dtype=np.uint64) >> np.uint64(64 - bits)
    k[::3] = k[0]  # long runs of equal keys
    return k


def _check(n, bits, radix, want_keys, seed=1):
    k = _keys(n, bits, seed)
    host = k.view(np.int64) if bits > 32 else k.astype(np.uint32).view(np.int32)
    dk = torch.from_numpy(host).cuda()
    size = rr.rr_sort_workspace_size(n, bits, radix)
    room = torch.full((size + GUARD,), 0xAB, dtype=torch.uint8, device="cuda")
    perm = torch.empty(n, dtype=torch.int32, device="cuda")
    out = torch.empty_like(dk) if want_keys else None
    for _ in range(2):  # the second call finds the first one's words in the workspace
        rr.rr_sort(dk, out, perm, n, bits, radix, room[:size])
    torch.cuda.synchronize()
    want = np.argsort(k, kind="stable")
    assert np.array_equal(rr.u32_to_numpy(perm), want.astype(np.uint32))
    if want_keys:
        assert np.array_equal(rr.keys_to_numpy(out), k[want])
    assert bool((room[size:] == 0xAB).all())
    assert rr.rr_device_error() == 0


@pytest.mark.parametrize("want_keys", [False, True])
@pytest.mark.parametrize("bits", [8, 16, 28, 32, 33, 40, 64])
@pytest.mark.parametrize("n", [n for e in EDGES for n in (e, e + 1)])
def test_tile_size_edges(n, bits, want_keys):
    _check(n, bits, 8, want_keys)


@pytest.mark.parametrize("bits", [3, 4, 8, 32, 36, 64])
@pytest.mark.parametrize("n", [1, 31, 1023, 1024, 1025, 4097, (1 << 20) - 1, 1 << 20])
def test_four_bit_digits(n, bits):
    _check(n, bits, 4, False)


@pytest.mark.parametrize("bits", [32, 64])
@pytest.mark.parametrize("n", [1, 2, 33, 1023, 1024, 1025, 3073, 65537])
def test_small(n, bits):
    _check(n, bits, 8, False)
    _check(n, bits, 8, True, seed=2)
