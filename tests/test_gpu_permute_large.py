"""The reorder of wavefronts that are moved one array after the other (2^21 rays
and more) and of those just below, against numpy's gather, bit for bit."""
import numpy as np
import pytest
import torch

from paper_2506_11273_gb300 import rr

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("payload", [False, True])
@pytest.mark.parametrize("n", [(1 << 21) - 1, 1 << 21, (1 << 21) + 1, 2_500_003])
def test_matches_gather(n, payload):
    rng = np.random.Generator(np.random.PCG64(n))
    o, d = (rng.integers(0, 2 ** 32, (n, 4), dtype=np.uint32) for _ in range(2))  # NaN payloads and all
    p = rng.integers(0, 2 ** 32, n, dtype=np.uint32)
    perm = rng.permutation(n).astype(np.uint32)
    do, dd = (torch.from_numpy(x.view(np.float32)).cuda() for x in (o, d))
    dp, dperm = (torch.from_numpy(x.view(np.int32)).cuda() for x in (p, perm))
    oo, od = torch.empty_like(do), torch.empty_like(dd)
    op = torch.full_like(dp, -1)
    rr.rr_permute(do, dd, dp if payload else None, dperm, oo, od, op if payload else None)
    torch.cuda.synchronize()
    assert np.array_equal(oo.cpu().numpy().view(np.uint32), o[perm])
    assert np.array_equal(od.cpu().numpy().view(np.uint32), d[perm])
    assert np.array_equal(rr.u32_to_numpy(op), p[perm] if payload else np.full(n, 0xFFFFFFFF, np.uint32))
    assert rr.rr_device_error() == 0
